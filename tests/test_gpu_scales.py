"""Float64 density and forces in units far from the usual ones.

The neighbour search looks at batches of candidates and fills the last batch
up; the filling must stay outside whatever the unit of length is.  Lengths
are scaled so that h is 5e18 (its square is within float32's range, in which
the search works) and 2.5e-9, and compared with the oracle at the same scale
within the bound of the other parity tests (1e-12 of the largest).
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


@pytest.mark.parametrize("N", [700, 2433])  # a warp per particle, 8 lanes per particle
@pytest.mark.parametrize("unit", [2e18, 1e-9])
def test_density_and_forces_at_any_unit_of_length(N, unit):
    box = tuple(unit * x for x in (13.0, 14.3, 16.9))
    q, p, e = random_box_state(N, 1.0, 1.0, 1.0, 30.0, seed=N)
    q = q * np.array(box)
    P = O.Config(N=N, L=box, h=2.5 * unit, K=20.0).params()
    rho = O.density(P, q)
    f = O.forces(P, q, rho, e)
    s = sdpd.SDPD(N, box, h=2.5 * unit, K=20.0, precision=sdpd.FP64)
    s.set_state(q, p, e)
    assert (s.neighbour_counts() == O.neighbour_counts(P, q)).all()
    assert np.abs(s.density() - rho).max() <= 1e-12 * rho.max()
    assert np.abs(s.forces() - f).max() <= 1e-12 * np.abs(f).max()


def test_negative_energy_has_no_entropy():
    """A negative internal energy (loaded from the device, where only the
    status tells of it) becomes NaN in a Verlet step, as the oracle's does."""
    N, L = 1000, 10.0
    q, p, e = random_box_state(N, 1.0, 1.0, 1.0, 30.0, seed=6)
    q = q * L
    e[[3, 500]] = -2.0
    P = O.Config(N=N, L=(L,) * 3, K=20.0, scheme=O.SCHEME_NONE).params()
    _, _, _, eo, _, _ = O.run(P, q, p, e, 0.002, 1, seed=1)
    s = sdpd.SDPD(N, L, h=2.5, K=20.0, precision=sdpd.FP64, scheme=sdpd.SCHEME_NONE)
    dev = [torch.from_numpy(x).cuda() for x in (q, p, e)]
    s.set_state(*dev)
    s.step(0.002, 1, seed=1)
    out = [torch.empty_like(x) for x in dev]
    assert sdpd.sdpd_get_state(s.h, *(x.data_ptr() for x in out), 1) == sdpd.ERR_NONPOSITIVE_ENERGY
    eg = out[2].cpu().numpy()
    assert (np.isnan(eg) == np.isnan(eo)).all() and np.isnan(eg).sum() == 2
