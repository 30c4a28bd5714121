"""Sweeps whose pair data are staged slice by slice, against the oracle.

3.4 million particles on 66^3 cells: 35,937 blocks per colour, two slices.
The oracle compares all pairs, so it gets only the particles of six pockets
(the lowest ids, which are also the lowest ranks of their blocks), around
which the fluid leaves a gap wider than h: nothing outside a pocket touches
it.  The pockets hold ordinary blocks, large ones (more than 256 particles) and
blocks beyond capacity; one lies across the box's faces.  Float64 within 1e-10
of the oracle as in the other sweep tests; the mixed path within 1e-3 of the
largest (float32 arithmetic errors are 1e-5, a misplaced pair is of order
one), and bit for bit alike under every schedule of the colour launches.
"""
import numpy as np
import pytest

import oracle as O
from paper_1707_04232_gb300.inputs import random_box_state

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("needs a CUDA device", allow_module_level=True)

from paper_1707_04232_gb300 import sdpd  # noqa: E402

L, H, N, DT, SEED = 165.0, 2.5, 3_400_000, 0.02, 17
SLICES = 2


@pytest.fixture(scope="module")
def system():
    rng = np.random.default_rng(12)
    centres = np.array([[20.0, 30.0, 40.0], [100.0, 10.0, 70.0], [0.0, 160.0, 80.0],
                        [60.0, 120.0, 20.0], [130.0, 80.0, 130.0], [75.0, 60.0, 150.0]])
    sides = np.array([7.0, 7.0, 7.0, 10.0, 10.0, 6.0])
    pockets = []
    for c, side, n in zip(centres[:3], sides, (343, 343, 343)):
        pockets.append(c + (rng.random((n, 3)) - 0.5) * side)
    for c in centres[3:5]:  # 13^3 on a jittered lattice: 274 per block of cells, 143 neighbours
        x = (np.indices((13, 13, 13)).reshape(3, -1).T + 0.5) / 13 - 0.5
        pockets.append(c + 10.0 * x + rng.normal(0.0, 0.02, x.shape))
    pockets.append(centres[5] + (rng.random((648, 3)) - 0.5) * sides[5])  # 196 neighbours
    q = np.concatenate(pockets)
    n = len(q)
    fluid = np.empty((0, 3))
    while len(fluid) < N - n:
        x = rng.random((N, 3)) * L
        for c, side in zip(centres, sides):
            d = np.abs((x - c + 0.5 * L) % L - 0.5 * L)
            x = x[(d > 0.5 * side + 0.2 + 1.05 * H).any(axis=1)]
        fluid = np.concatenate([fluid, x])
    q = np.concatenate([q, fluid[:N - n]]) % L
    _, p, e = random_box_state(N, 1.0, 1.0, 1.0, 28.5, seed=5)
    return n, q, p, e


def oracle_sweeps(system, scheme, k=2):
    n, q, p, e = system
    P = O.Config(N=n, L=(L,) * 3, K=20.0, scheme=scheme).params()
    _, _, po, eo, _, _ = O.run(P, q[:n], p[:n], e[:n], DT, k, seed=SEED, fd_only=True)
    return po, eo


def sweeps(system, k=2, variant=None, **kw):
    n, q, p, e = system
    s = sdpd.SDPD(N, L, h=H, K=20.0, fd_only=True, **kw)
    if variant is not None:
        s.set_tuning(variant, 128)
    s.set_state(q, p, e)
    before = s.kernel_launches
    s.step(DT, k, seed=SEED)
    assert s.kernel_launches - before == 4 + k * 8 * 3 * SLICES
    assert s.big_blocks().sum() > 0 and s.observables()["status"] == 0
    return s.get_state()[1:]


@pytest.mark.parametrize("scheme", [sdpd.SCHEME_EMS, sdpd.SCHEME_AMS])
def test_float64_slices_match_oracle(system, scheme):
    n = system[0]
    po, eo = oracle_sweeps(system, scheme)
    p, e = sweeps(system, precision=sdpd.FP64, scheme=scheme)
    assert np.abs(p[:n] - po).max() <= 1e-10 * np.abs(po).max()
    assert np.abs(e[:n] - eo).max() <= 1e-10 * eo.max()
    assert (p[n:] != system[2][n:]).any(axis=1).mean() > 0.99  # (and the fluid was swept)


@pytest.mark.parametrize("precision", [sdpd.MIXED, sdpd.FP64])
def test_float32_slices_match_oracle(system, precision):
    n = system[0]
    po, eo = oracle_sweeps(system, sdpd.SCHEME_AMS)
    p, e = sweeps(system, precision=precision, scheme=sdpd.SCHEME_AMS,
                  **({"sweep_f32": True} if precision == sdpd.FP64 else {}))
    assert np.abs(p[:n] - po).max() <= 1e-3 * np.abs(po).max()
    assert np.abs(e[:n] - eo).max() <= 1e-3 * eo.max()


def test_mixed_slices_alike_under_every_schedule(system):
    ref = sweeps(system, precision=sdpd.MIXED)
    for v in (0, 1, 2):
        assert all(np.array_equal(a, b) for a, b in zip(sweeps(system, variant=v, precision=sdpd.MIXED), ref))
