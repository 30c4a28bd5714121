"""Blocks at the edges of the sweep schedule's capacities, against the oracle.

A 2x2x2 cell block is enumerated and scheduled by one of two kernels (up to
256 particles and 2048 owned pairs, up to 512 and 4096), or swept pair by
pair beyond that.  Box sides between two cell counts give blocks of any of
these sizes; the float64 sweep of each must make the oracle's decisions and
end within 1e-10 of it (the bound of the other sweep tests), and the mixed
one must update the same pairs with the same result under every schedule of
the colour launches.
"""
import numpy as np
import pytest

import oracle as O
from paper_1707_04232_gb300.inputs import Workload, lattice_state, random_box_state

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("needs a CUDA device", allow_module_level=True)

from paper_1707_04232_gb300 import sdpd  # noqa: E402


def system(kind):
    """(q, p, eps, box, K, blocks swept pair by pair)."""
    if kind.startswith("lattice"):  # 13: 274.6 per block on average, 14: 343, 19: 254
        w = Workload(n=int(kind[7:]), K=50.0, seed=3)
        return (*lattice_state(w), (w.L,) * 3, w.K, False)
    # random fluids of 413 and (beyond 512) 620 particles per block on average
    box, density = (14.9,) * 3, {"random413": 1.0, "random620": 1.5}[kind]
    N = int(round(box[0] * box[1] * box[2] * density))
    q, p, e = random_box_state(N, 1.0, 1.0, 1.0, 1.5 * 19.0, seed=8)
    return q * np.array(box), p, e, box, 20.0, density > 1.0


@pytest.mark.parametrize("kind", ["lattice13", "lattice14", "lattice19", "random413", "random620"])
def test_block_sizes_match_oracle(kind):
    q, p, e, box, K, big = system(kind)
    N = len(e)
    P = O.Config(N=N, L=box, K=K).params()
    st, po, eo, stats, _ = O.fd_sweep(P, q, p, e, 0.005, 11, 0, records=True)
    s = sdpd.SDPD(N, box, h=2.5, K=K, precision=sdpd.FP64, fd_only=True)
    s.set_state(q, p, e)
    s.step(0.005, 1, seed=11)
    _, pg, eg = s.get_state()
    o = s.observables()
    assert o["n_pairs"] == stats.n_pairs and o["n_accept"] == stats.n_accept
    assert np.abs(pg - po).max() <= 1e-10 * np.abs(po).max()
    assert np.abs(eg - eo).max() <= 1e-10 * eo.max()
    assert (s.big_blocks().sum() > 0) == big
    ref = None
    for v in range(5):
        m = sdpd.SDPD(N, box, h=2.5, K=K, precision=sdpd.MIXED, fd_only=True)
        m.set_tuning(v, 128)
        m.set_state(q, p, e)
        m.step(0.005, 2, seed=11)
        x = m.get_state()
        assert m.observables()["n_pairs"] == 2 * stats.n_pairs
        ref = ref or x
        assert all(np.array_equal(u, w) for u, w in zip(x, ref))


@pytest.mark.parametrize("precision,K,dt", [(sdpd.MIXED, 50.0, 0.05), (sdpd.MIXED, 5.0, 0.45), (sdpd.FP64, 5.0, 0.22)])
def test_tested_one_round_late_is_the_sequential_sweep(precision, K, dt):
    """One block per team (moves made before their test, taken back when it
    rejects them) against two blocks per warp (each round tested before the
    next), float32 pair arithmetic: the same counts and, bit for bit, the same
    state, with moves rejected on the way."""
    w = Workload(n=16, K=K, jitter=0.2, seed=4)
    out = []
    for v in (1, 2):
        s = sdpd.SDPD(w.N, w.L, h=w.h, K=K, precision=precision, fd_only=True, **(
            {"sweep_f32": True} if precision == sdpd.FP64 else {}))
        s.set_tuning(v, 128)
        s.set_state(*lattice_state(w))
        s.step(dt, 3, seed=13)
        o = s.observables()
        out.append((s.get_state(), [o[k] for k in ("n_pairs", "n_accept", "n_reject_bound", "n_reject_metropolis")]))
    assert out[0][1] == out[1][1] and out[0][1][3] > 0
    assert all(np.array_equal(a, b) for a, b in zip(out[0][0], out[1][0]))
