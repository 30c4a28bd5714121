"""What an ensemble's captured graph depends on.

A graph is replayed while nothing that it holds has changed.  Members whose
state changes between two calls with the same time step and seeds must end
where the same system, stepped alone through the same calls, ends: bit for
bit, as the other ensemble tests compare.
"""
import numpy as np
import pytest

from paper_1707_04232_gb300.inputs import Workload, lattice_state, random_box_state

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("needs a CUDA device", allow_module_level=True)

from paper_1707_04232_gb300 import sdpd  # noqa: E402


def same(a, b):
    return all(np.array_equal(x, y) for x, y in zip(a.get_state(), b.get_state()))


@pytest.mark.parametrize("precision", [sdpd.FP64, sdpd.MIXED])
def test_fd_only_member_with_a_new_state_gets_a_new_schedule(precision):
    """The second call's graph is captured with a valid schedule and holds
    none; the third call brings other positions under the same seeds."""
    w = Workload(n=12, K=20.0, seed=1)
    first, second = lattice_state(w), lattice_state(Workload(n=12, K=20.0, jitter=0.3, seed=2))
    handles = [sdpd.SDPD(w.N, w.L, h=w.h, K=w.K, precision=precision, fd_only=True, stream=torch.cuda.Stream())
               for _ in range(4)]
    members, alone = handles[:2], handles[2:]
    for s in handles:
        s.set_state(*first)
    ens = sdpd.SDPDEnsemble(members)
    for seeds, load in (([1, 2], None), ([3, 4], None), ([3, 4], 0), ([3, 4], None), ([3, 4], 1)):
        if load is not None:
            members[load].set_state(*second)
            alone[load].set_state(*second)
        ens.step(0.02, 2, seeds)
        for s, seed in zip(alone, seeds):
            s.step(0.02, 2, seed=seed)
        assert all(same(m, a) for m, a in zip(members, alone))


def test_overflowing_neighbour_lists_after_a_new_state():
    """A fluid with more neighbours than a list row holds (their forces come
    from the cells): the replay after a new state, and after a debug read-out,
    finds the particles of the state's own density pass."""
    N, L = 3000, 10.4
    states = []
    for seed in (1, 2):
        q, p, e = random_box_state(N, 1.0, 1.0, 1.0, 30.0, seed=seed)
        states.append((q * L, p, e))
    member, alone = (sdpd.SDPD(N, L, h=2.5, K=20.0, precision=sdpd.MIXED, scheme=sdpd.SCHEME_NONE,
                               stream=torch.cuda.Stream()) for _ in range(2))
    member.set_state(*states[0])
    alone.set_state(*states[0])
    assert (member.neighbour_counts() > 160).any()
    ens = sdpd.SDPDEnsemble([member])
    for state in (None, states[1], None, states[0]):
        if state is not None:
            member.set_state(*state)
            alone.set_state(*state)
        else:
            member.neighbour_counts()
        ens.step(0.002, 4, [5])
        alone.step(0.002, 4, seed=5)
        assert same(member, alone)


def test_member_with_a_new_workspace():
    """A workspace bound anew holds no state (the call is refused); with a
    state it is the one that is stepped."""
    w = Workload(n=10, K=50.0, seed=3)
    state = lattice_state(w)
    member, alone = (sdpd.SDPD(w.N, w.L, h=w.h, K=w.K, precision=sdpd.MIXED, stream=torch.cuda.Stream())
                     for _ in range(2))
    member.set_state(*state)
    alone.set_state(*state)
    ens = sdpd.SDPDEnsemble([member])
    ens.step(0.005, 2, [9])
    old, member.workspace = member.workspace, torch.empty_like(member.workspace)
    torch.cuda.synchronize()
    assert sdpd.sdpd_bind_workspace(member.h, member.workspace.data_ptr(), member.workspace.numel()) == sdpd.OK
    assert sdpd.sdpd_ensemble_step(ens.e, 0.005, 2, [9]) == sdpd.ERR_NO_STATE
    member.set_state(*state)
    ens.step(0.005, 2, [9])
    alone.step(0.005, 2, seed=9)
    assert same(member, alone)
    del old
