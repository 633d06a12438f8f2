"""Grains outside their key zone (keys of the step before, long steps) in the
spherical geometry: their weights are rounded as the general path rounds them.
The digests are those of the kernels that pushed such grains by the general
path's own functions; the inputs use correctly rounded operations only.  And
grains that leave the grid on that path."""
import numpy as np
import pytest

from paper_1908_10793_gb300 import inputs as I
from parity_util import run_gpu
from test_parity_gpu import MIXED

pytestmark = pytest.mark.gpu

# grains left, then the digests of the deposit, the coordinates and the velocities
GOLDEN = {
    I.TSC: [300001, 17895236621238666848, 18198982150415316524, 4090403850151365263, 7676364133412259435,
            16018428006171148288, 2489182679074006067, 16303818644005865493],
    I.CIC: [300001, 18138579055817104153, 504027839889491231, 3689585777722141606, 6548043595270473070,
            9826778709061795840, 7330932351426793475, 7559085779214124654],
    I.VOLUME: [300001, 578741085865350876, 750681188553845444, 2628334482230357729, 8260255384908468922,
               17709446550578528256, 9302544505585562661, 460938810064028904],
}


def _workload(weight):
    r = np.random.Generator(np.random.Philox(17))
    n, grains = (37, 16, 16), 300001
    t = np.arange(n[0] + 1) / n[0]
    edges = [0.5 + 2.5 * (0.6 * t + 0.4 * t * t), 1.25 + 0.640625 * np.arange(n[1] + 1) / n[1],
             6.28125 * np.arange(n[2] + 1) / n[2]]
    x, _, _ = I._grid3(edges)
    nc = len(x)
    vk = 1.0 / np.sqrt(x)
    vgas = [1e-3 * (r.uniform(-1.0, 1.0, nc)) for _ in range(3)]
    vgas[2] = vk * (1.0 + vgas[2])
    q = [e[0] + (e[-1] - e[0]) * r.uniform(0.1, 0.9, grains) for e in edges]
    v = [0.02 * r.uniform(-1.0, 1.0, grains) for _ in range(3)]
    v[2] = v[2] + 1.0 / np.sqrt(q[0])
    return I.Workload(
        name="strays", geom=I.SPHERICAL, edges=edges, bc=[I.OUTFLOW, I.OUTFLOW, I.PERIODIC], weight=weight,
        species_mass=[1e-6], species_tau_mode=[I.TAU_STOKES], species_tau=[1.0], rho=1.0 / x, vgas=vgas, q=q, v=v,
        dt=0.0625, steps=2, feedback=0, param=r.uniform(0.001, 1.0, grains), gm=1.0)


def digest(a):
    a = np.ascontiguousarray(a).view(np.uint64).ravel()
    return int((a * (2 * np.arange(len(a), dtype=np.uint64) + np.uint64(1))).sum(dtype=np.uint64))


def digests(weight):
    got = run_gpu(_workload(weight), 2, MIXED, sort_interval=2)
    alive = ~np.isnan(got["q"][0])
    return [int(alive.sum())] + [digest(got["fixed"])] + [digest(x[alive]) for k in ("q", "v") for x in got[k]]


@pytest.mark.parametrize("weight", [I.TSC, I.CIC, I.VOLUME])
def test_spherical_strays_keep_their_bits(weight):
    assert digests(weight) == GOLDEN[weight]


def test_grains_removed_in_place_keep_their_other_columns():
    """Grains that leave in their first half drift of a step that moves the
    store in place (the step of length zero before it only sorts)."""
    w = I.sbox3d("small")
    w.geom, w.fargo, w.feedback, w.bc = I.CARTESIAN, 0, 0, [I.OUTFLOW] * 3
    w.species_tau_mode = [I.TAU_CONST]
    out = w.q[0] > 0.09
    w.v[0][out] = 10.0
    w.v[1][out] = 0.125
    got = run_gpu(w, 2, MIXED, dt=[0.0, 0.01], sort_interval=2)
    assert out.any() and np.isnan(got["q"][0][out]).all()
    for d in (1, 2):
        assert np.array_equal(got["q"][d][out], w.q[d][out])
