"""What an ensemble's captured graph depends on.

A graph is replayed while nothing that it holds has changed.  Members whose
state changes between two calls with the same time step and seeds must end
where the same system, stepped alone through the same calls, ends: bit for
bit, as the other ensemble tests compare.
"""
import numpy as np
import pytest

from paper_1707_04232_gb300.inputs import Workload, lattice_state

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
