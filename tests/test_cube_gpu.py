"""The three-dimensional slab kernels at the sizes where they can go wrong:
partial and clipped tiles, one grain, tiles and zones denser than the carry-free
box and the chunk length, strays of stale keys, each set of optional columns;
and the two-dimensional tiles cut into parts.  Each run is compared with the
oracle (the tolerances of test_parity_gpu.py) and, exactly, with a run on
another tile shape: the integers and the grains depend on neither the tile nor
the parts it is cut into."""
import numpy as np
import pytest

from paper_1908_10793_gb300 import inputs as I
from parity_util import run_gpu, run_oracle
from test_parity_gpu import MIXED, check_against_oracle

pytestmark = pytest.mark.gpu


def _box(n, grains, dense=False, species=False, param=False, seed=11):
    w = I.sbox3d("small")
    r = np.random.Generator(np.random.Philox(seed))
    L = 0.2
    w.edges = [I._uniform_edges(-0.5 * L, 0.5 * L, m) for m in n]
    nc = n[0] * n[1] * n[2]
    span = [L / m if dense else L for m in n]  # dense: all in one zone
    w.q = [-0.5 * L + s * (0.05 + 0.9 * r.uniform(0.0, 1.0, grains)) for s in span]
    w.v = [1e-3 * r.standard_normal(grains) for _ in range(3)]
    w.rho, w.vgas = np.ones(nc), [1e-3 * r.standard_normal(nc) for _ in range(3)]
    w.feedback = 0
    if species:
        w.species = (np.arange(grains) % 3).astype(np.uint8)
        w.species_mass = [w.species_mass[0]] * 3
        w.species_tau_mode, w.species_tau = w.species_tau_mode * 3, [0.01, 0.1, 10.0]
    if param:
        w.param = 10.0 ** r.uniform(-3.0, 1.0, grains)
    return w


CASES = {
    "one_grain": (lambda: _box((9, 8, 8), 1), 2, {}),
    "partial_tiles": (lambda: _box((17, 9, 8), 3001), 2, {}),
    "clipped_tile": (lambda: _box((5, 4, 3), 607), 2, {}),
    "dense_zone": (lambda: _box((8, 8, 8), 70001, dense=True), 1, {}),
    "strays": (lambda: _box((16, 24, 9), 9001), 3, {"sort_interval": 2}),
    "species": (lambda: _box((10, 11, 12), 4001, species=True), 2, {}),
    "param": (lambda: _box((10, 11, 12), 4001, param=True), 2, {}),
    "species_param": (lambda: _box((10, 11, 12), 4001, species=True, param=True), 2, {}),
    "box2d_parts": (lambda: I.box2d("small"), 2, {}),
}


@pytest.mark.parametrize("name", list(CASES))
def test_cube_against_oracle_and_another_tile(name):
    make, steps, kw = CASES[name]
    w = make()
    got = run_gpu(w, steps, MIXED, **kw)
    other = run_gpu(w, steps, MIXED, tile=(4, 3, 5), **kw)
    assert np.array_equal(got["fixed"], other["fixed"])
    for k in ("q", "v"):
        for a, b in zip(got[k], other[k]):
            assert np.array_equal(a, b, equal_nan=True)
    qo, vo, active, dep, _ = run_oracle(w, steps)
    check_against_oracle(w, got, (qo, vo, active, dep), steps, MIXED, w.dt)
