"""Blocks of the three-dimensional slab kernels without grains leave before they
stage anything."""
import pytest

from paper_1908_10793_gb300 import inputs as I
from parity_util import run_gpu
from test_parity_gpu import MIXED

pytestmark = pytest.mark.gpu


def test_blocks_without_grains_stage_nothing():
    """With no grains no block waits for its gas box, so the wait that the
    testing option makes run out is never reached."""
    from paper_1908_10793_gb300 import dust as D
    w = I.sbox3d("small")
    w.q, w.v = [x[:0] for x in w.q], [x[:0] for x in w.v]
    got = run_gpu(w, 1, MIXED, test_wait_timeout=1, feedback=0)
    assert got["rc"] == D.DUST_OK and got["stats"].flags == 0
    assert not got["fixed"].any()
