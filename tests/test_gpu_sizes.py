"""The sort and the float64 pair passes at the edges of their size rules.

Up to 2048 particles and cells one thread block sorts them, above five
launches do; up to 2432 particles a whole warp shares a particle of the
float64 density and force passes, above 8 lanes do.  Storage order and cells
are compared with the oracle's exactly, densities and forces within the
bounds of the parity tests (1e-12 of the largest in float64, 1e-5 mixed).
The densest box has rows of more than 160 neighbours, whose sums come from the
cells.
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


@pytest.mark.parametrize("N,side", [(1, 10.0), (2, 10.0), (33, 10.0), (2047, 13.0), (2048, 13.0), (2049, 13.0),
                                    (2432, 10.0), (2433, 13.4), (700, 33.0)])
def test_sort_density_and_forces(N, side):
    box = (side, side * 1.1, side * 1.3)
    q, p, e = random_box_state(N, 1.0, 1.0, 1.0, 30.0, seed=N)
    q = q * np.array(box)
    for kernel in (sdpd.KERNEL_LUCY, sdpd.KERNEL_CUBIC):
        P = O.Config(N=N, L=box, K=20.0, kernel=kernel).params()
        rho = O.density(P, q)
        f = O.forces(P, q, rho, e)
        for prec, tol in ((sdpd.FP64, 1e-12), (sdpd.MIXED, 1e-5)):
            s = sdpd.SDPD(N, box, h=2.5, K=20.0, precision=prec, kernel=kernel)
            s.set_state(q, p, e)
            assert np.abs(s.density() - rho).max() <= tol * rho.max()
            assert np.abs(s.forces() - f).max() <= tol * max(np.abs(f).max(), 1e-300)
            if prec == sdpd.FP64:
                assert (s.order() == O.sorted_order(P, q)).all()
                assert (s.cells() == O.cells(P, q)).all()


@pytest.mark.parametrize("N", [700, 2433])
def test_float64_launch_shapes_are_bitwise_alike(N):
    """Block sizes of the passes, set or left alone, on both sides of the line
    of a warp per particle, under every schedule of the colour launches."""
    q, p, e = random_box_state(N, 1.0, 1.0, 1.0, 30.0, seed=N)
    out = []
    for v, pt in ((0, None), (0, 32), (2, 64), (4, 128)):
        s = sdpd.SDPD(N, 13.0, h=2.5, K=20.0, precision=sdpd.FP64)
        if pt is not None:
            s.set_tuning(v, pt)
        s.set_state(q * 13.0, p, e)
        s.step(0.002, 3, seed=3)
        out.append(s.get_state())
    for x in out[1:]:
        assert all(np.array_equal(a, b) for a, b in zip(x, out[0]))
