"""The three-dimensional slab kernels' chunk sums: the 32-bit rounding path is
taken only where the host zone's rest cannot leave 32 bits, so its integers are
those of the 64-bit path; and the carry-free deposit box gives those of the box
of int64 words."""
import numpy as np
import pytest

from paper_1908_10793_gb300 import inputs as I
from parity_util import run_gpu
from test_cube_gpu import _box
from test_parity_gpu import MIXED

pytestmark = pytest.mark.gpu

QUANTUM = 2.0 ** -84
DT, TAU = 1e-6, 1e-5


def _cancelling(dense, impulse, seed=5):
    """8^3 zones (one tile); 128 of them, one in four, hold a chunk of 128
    grains at one place whose impulses, about `impulse` quanta each per unit of
    the drag's share of the momentum, cancel in pairs, so that what is left of
    a sum is the rounding of its partial sums: around 2^31 quanta.  The energy
    stays small.  dense: the other zones are filled with grains at rest (they
    deposit nothing), which makes every block too dense for the 32-bit counters
    and so sends every chunk through the 64-bit rounding."""
    r = np.random.default_rng(seed)
    n, width = 8, 10.0
    edges = [width * np.arange(n + 1.0)] * 3
    zones = np.arange(0, n ** 3, 4)
    q, v = [[], [], []], [[], [], []]
    for z in zones:
        place = np.array([z % n, z // n % n, z // n ** 2]) + 0.5 + r.uniform(-0.45, 0.45, 3)
        for d in range(3):
            half = r.uniform(-1.0, 1.0, 64)
            q[d].append(np.full(128, width * place[d]))
            v[d].append(impulse * QUANTUM * np.concatenate([half, -r.permutation(half)]))
    if dense:
        rest = np.repeat(np.setdiff1d(np.arange(n ** 3), zones), 1800)
        for d, i in enumerate((rest % n, rest // n % n, rest // n ** 2)):
            q[d].append(width * (i + 0.5))
            v[d].append(np.zeros(len(rest)))
    nc = n ** 3
    return I.Workload(
        name="cancelling", geom=I.CARTESIAN, edges=edges, bc=[I.PERIODIC] * 3, weight=I.TSC, species_mass=[1.0],
        species_tau_mode=[I.TAU_CONST], species_tau=[TAU], rho=np.full(nc, 1e-9), vgas=[np.zeros(nc)] * 3,
        q=[np.concatenate(x) for x in q], v=[np.concatenate(x) for x in v], dt=DT, steps=1, feedback=0)


@pytest.mark.parametrize("tile", [(0, 0, 0), (8, 8, 7)])
def test_step_chunks_of_cancelling_impulses(tile):
    scale = 2.0 ** 51 / -np.expm1(-DT / TAU)
    sparse, dense = (run_gpu(_cancelling(d, scale), 1, MIXED, quantum=QUANTUM, tile=tile) for d in (False, True))
    assert np.array_equal(sparse["fixed"], dense["fixed"])


@pytest.mark.parametrize("tile", [(0, 0, 0), (8, 8, 7)])
def test_predictor_chunks_of_cancelling_impulses(tile):
    scale = 2.0 ** 51 / (0.5 * DT / TAU)
    sparse, dense = (run_gpu(_cancelling(d, scale), 1, MIXED, quantum=QUANTUM, tile=tile, gas_predictor=1)
                     for d in (False, True))
    for a, b in zip(sparse["v"], dense["v"]):
        assert np.array_equal(a, b[:len(a)])


@pytest.mark.parametrize("predictor", [0, 1])
def test_deposit_boxes_agree(predictor):
    """About 1170 grains in each of 8^3 zones: one tile's eight parts hold more
    than 65535 grains each (int64 words), the parts of smaller tiles fewer
    (carry-free counters)."""
    w = _box((8, 8, 8), 600001)
    words = run_gpu(w, 2, MIXED, gas_predictor=predictor)
    counters = run_gpu(w, 2, MIXED, gas_predictor=predictor, tile=(4, 3, 5))
    assert np.array_equal(words["fixed"], counters["fixed"])
    for k in ("q", "v"):
        for a, b in zip(words[k], counters[k]):
            assert np.array_equal(a, b)
