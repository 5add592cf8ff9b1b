"""Choices that an earlier build left in the tuning cache under the nodal steps' plain keys.

There the index of a step with one sweep per side named a tile; the candidates are row strips now, and
an old index must not be taken for one of them: the step is timed again, the old entries stay unread.
"""
import json
import re

import pytest

from test_gpu_tuner import _child

pytestmark = pytest.mark.gpu


def test_old_tile_choices_are_not_read_as_strips(tmp_path):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    cache = tmp_path / "tune.json"
    first = _child({"PBS_TUNE_CACHE": str(cache), "PBS_TUNE": "1"})
    choices = json.loads(cache.read_text())
    keys = [k for k in choices if k.startswith(("node_down|", "node_up|"))]
    assert keys
    plain = re.compile(r"^(node_\w+\|)(?:.*\|)?(\d+x\d+\|c\d+\|.*)$")
    old = {plain.sub(r"\1\2", k): 2 for k in keys}
    # (the other choices stay: another split of the Gram's sums would change the last places)
    cache.write_text(json.dumps({**{k: v for k, v in choices.items() if k not in keys}, **old}))
    second = _child({"PBS_TUNE_CACHE": str(cache), "PBS_TUNE": "1"})
    after = json.loads(cache.read_text())
    assert set(keys) <= set(after) and not set(keys) & set(old)
    assert second["lam"] == first["lam"]  # the rows of a strip do not change a result
