"""Device memory of large systems (host only: nothing is allocated).

The pair data of a sweep are staged for all colours at once only where that
takes little of the device; beyond 32,768 blocks per colour they take a fixed
slice (134 million pairs of 36 or 76 bytes).  Per particle at unit density the rest is the neighbour lists (640
bytes), the schedule (600 to 900) and the state (300 to 500).
"""
import pytest

from paper_1707_04232_gb300 import sdpd


def workspace(n, **kw):
    p = sdpd.sdpd_params(kB=1.0, eta=1.0, zeta=0.0, c_rho=-1.0, kernel=sdpd.KERNEL_LUCY, scheme=sdpd.SCHEME_EMS,
                         theta=1, **kw)
    st, h = sdpd.sdpd_create(n ** 3, (float(n),) * 3, 1.0, 2.5, p, 50.0, 0)
    assert st == sdpd.OK
    size = sdpd.sdpd_workspace_bytes(h)
    sdpd.sdpd_destroy(h)
    return size


@pytest.mark.parametrize("kw", [{"precision": sdpd.MIXED}, {"precision": sdpd.FP64},
                                {"precision": sdpd.FP64, "sweep_f32": 1}])
def test_large_systems_take_under_1800_bytes_per_particle_and_a_slice(kw):
    for n in (200, 256, 400):
        assert workspace(n, **kw) <= 1800 * n ** 3 + 32768 * 4096 * 76
    assert 2 * workspace(400, **kw) <= 284208 * 2 ** 20  # two of 64 million particles on one device


def test_up_to_there_a_system_stays_below_a_ninth_of_the_device():
    assert 9 * workspace(160, precision=sdpd.FP64) <= 284208 * 2 ** 20


def test_particle_numbers_beyond_a_list_entry_are_refused():
    """A neighbour-list entry keeps 26 bits of the neighbour's index."""
    p = sdpd.sdpd_params(kB=1.0, eta=1.0, zeta=0.0, c_rho=-1.0, kernel=sdpd.KERNEL_LUCY, scheme=sdpd.SCHEME_EMS,
                         precision=sdpd.MIXED, theta=1)
    for N, expect in ((2 ** 26, sdpd.OK), (2 ** 26 + 1, sdpd.ERR_INVALID_ARG)):
        st, h = sdpd.sdpd_create(N, (100.0,) * 3, 1.0, 2.5, p, 50.0, 0)
        assert st == expect
        if h:
            sdpd.sdpd_destroy(h)
