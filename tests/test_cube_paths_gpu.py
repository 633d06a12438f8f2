"""The three-dimensional slab kernels where the other tests do not take them:
grains outside their key zone in the curvilinear geometries, the gas predictor
with dense zones and ragged tiles, and the scan and the deposit's clear of large
grids."""
import numpy as np
import pytest

from paper_1908_10793_gb300 import inputs as I
from parity_util import default_quantum, run_gpu, run_oracle, zone_volumes
from test_parity_gpu import MIXED, _grains_per_zone_max, check_against_oracle, compare

pytestmark = pytest.mark.gpu


def _same(a, b):
    assert np.array_equal(a["fixed"], b["fixed"])
    for k in ("q", "v"):
        for x, y in zip(a[k], b[k]):
            assert np.array_equal(x, y, equal_nan=True)


@pytest.mark.parametrize("weight", [I.TSC, I.CIC, I.VOLUME])
@pytest.mark.parametrize("make", [I.cyldisk, I.sphdisk])
def test_curvilinear_strays(make, weight):
    """Every second step pushes grains with the keys of the step before."""
    w = make("small")
    w.weight, w.feedback = weight, 0
    got = run_gpu(w, 2, MIXED, sort_interval=2)
    _same(got, run_gpu(w, 2, MIXED, sort_interval=2, tile=(4, 3, 5)))
    qo, vo, active, dep, _ = run_oracle(w, 2)
    check_against_oracle(w, got, (qo, vo, active, dep), 2, MIXED, w.dt)


@pytest.mark.parametrize("weight", [I.TSC, I.CIC])
@pytest.mark.parametrize("make", [lambda: I.sbox3d("small"), lambda: I.cyldisk("small"), lambda: I.sphdisk("small")])
def test_predictor_dense_zones_and_tile_independent(make, weight):
    """Two zones of 600 and 300 grains among thinly filled ones; the default
    tile has a compiled copy with TSC weights, the others do not."""
    w = make()
    w.weight = weight
    r = np.random.default_rng(11)
    for sel, at in ((slice(0, 600), (3, 5, 2)), (slice(600, 900), (10, 12, 6))):
        for d in range(3):
            e = w.edges[d]
            w.q[d][sel] = e[at[d]] + (e[at[d] + 1] - e[at[d]]) * r.uniform(0.05, 0.95, sel.stop - sel.start)
    nz = _grains_per_zone_max(w) * 27
    dgas = (nz * 0.5 * default_quantum(w, MIXED) / (w.rho * zone_volumes(w))).max()
    compare(w, 2, MIXED, feedback=0, predictor=True, extra_v=8 * dgas)
    got = run_gpu(w, 2, MIXED, feedback=0, gas_predictor=1)
    for tile in ((4, 3, 5), (8, 8, 7)):
        _same(got, run_gpu(w, 2, MIXED, feedback=0, gas_predictor=1, tile=tile))


def test_scan_in_three_kernels_and_large_deposit_clear():
    """More than 4M keys (the scan's chunk sums then take a kernel of their
    own) and a deposit above 16 MB (cleared apart from the scan)."""
    n, grains = 168, 60001
    r = np.random.default_rng(3)
    w = I.sbox3d("small")
    L = 0.2
    w.edges = [I._uniform_edges(-0.5 * L, 0.5 * L, n)] * 3
    w.q = [L * r.uniform(-0.499, 0.499, grains) for _ in range(3)]
    w.v = [1e-3 * r.standard_normal(grains) for _ in range(3)]
    w.rho, w.vgas, w.feedback = np.ones(n ** 3), [1e-3 * r.standard_normal(n ** 3) for _ in range(3)], 0
    got = run_gpu(w, 3, MIXED)
    _same(got, run_gpu(w, 3, MIXED, tile=(7, 6, 5)))
    qo, vo, active, dep, _ = run_oracle(w, 3)
    check_against_oracle(w, got, (qo, vo, active, dep), 3, MIXED, w.dt)
