"""Short strips (two and four rows) of the mixed policy's stencil passes: ``strips_short_check.cu``."""
import pytest

from test_gpu_strips import test_strips as _check

pytestmark = pytest.mark.gpu


def test_short_strips(tmp_path):
    _check(tmp_path, "strips_short_check")
