"""FP64 Basin Hopping against stored traces: how each trial ended and the bits of
its energy (tests/golden/record_bh_fp64.py)."""
import json

import pytest

from tests.golden import record_bh_fp64 as R

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def lj():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2510_25938_gb300 import build
    build.build()
    from paper_2510_25938_gb300 import lj_bh
    return lj_bh


@pytest.mark.parametrize("name", sorted(R.CASES))
def test_bh_fp64_trace(lj, name):
    with open(R.PATH) as f:
        want = json.load(f)[name]
    got = R.run(lj, R.CASES[name])
    assert got["status"] == want["status"]
    assert got["energy"] == want["energy"]
