"""Rows per strip of the nodal steps: every choice of the tuner gives the same bits.

Levels just above the narrowest this path takes, whose width leaves a strip nearly empty and whose
height leaves part of a row block; each candidate forced in a child process.  A forced index that is
no candidate would be tuned instead and leave a key in the cache.
"""
import json

import pytest

from test_gpu_tuner import _child

pytestmark = pytest.mark.gpu

CHILD = r"""
import hashlib, json
import numpy as np, torch
import __graft_entry__ as ge
ge.build()
import paper_2304_00337_gb300 as pbs
out = {}
with pbs.Context(0) as ctx:
    for n, m in ((60, 60), (68, 76), (112, 64)):
        geom = pbs.Geometry(np.random.default_rng(1).uniform(1.0, 9.0, (m, n)))
        for prec in (pbs.PBS_FP64, pbs.PBS_MIXED):
            for op, size in (("VCYCLE_NODAL", n * m), ("PROJECT", 2 * n * m)):  # from zero; from an iterate too
                x = torch.from_numpy(np.random.default_rng(2).standard_normal((2, size, 2))).cuda()
                y = torch.zeros_like(x)
                ctx.apply(geom, op, x.data_ptr(), y.data_ptr(), 2, k=(0.4, -1.3),
                          opts=pbs.default_opts(precision=prec, nodal_cycles=2), stream=torch.cuda.current_stream())
                torch.cuda.synchronize()
                out[f"{n} {m} {prec} {op}"] = hashlib.sha256(y.cpu().numpy().tobytes()).hexdigest()
print(json.dumps(out))
"""


def test_rows_do_not_change_a_bit(tmp_path):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    want = None
    for shape in range(5):
        cache = tmp_path / f"tune{shape}.json"
        got = _child({"PBS_TUNE_CACHE": str(cache), "PBS_TUNE": "1", "PBS_TUNE_FORCE": f"node_down={shape},node_up={shape}"},
                     CHILD)
        want = want or got
        assert got == want, shape
        assert not cache.exists() or not any(k.startswith("node_") for k in json.loads(cache.read_text())), shape
