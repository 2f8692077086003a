"""The bounded waits between the generator and chain warps of the paired kernel: one that runs
out ends the launch with the device error word set, and the host reports it."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def M():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__
    __graft_entry__.build()
    from paper_1707_00919_gb300 import muca
    return muca


@pytest.mark.parametrize("L,W", [(8, 45), (8, 9728), (32, 1024), (32, 9728)])
def test_an_expired_wait_is_reported(M, orc, L, W):
    """No try at all: every wait has run out at once, on both sides.  The launch ends (its words
    are whatever the ring holds), the call says so, and other instances go on."""
    from paper_1707_00919_gb300 import _lib as C
    N = L * L
    lnW = np.cumsum(np.random.default_rng(L).normal(0.0, 0.4, N + 1))
    with M.Muca(L, W, 1) as m:
        C.load().muca_testing_no_waits(m._h, 1)
        m.set_weights(lnW)
        m.thermalize_and_record(2 * N + 3, N)
        assert C.load().muca_testing_form(m._h) > 0
        with pytest.raises(M.MucaError) as ex:
            m.get_histogram()
        assert ex.value.code == C.MUCA_EDEVICE and "wait" in str(ex.value)
        with pytest.raises(M.MucaError) as ex:
            m.synchronize()
        assert ex.value.code == C.MUCA_EDEVICE
    with M.Muca(L, 45, 2) as m:
        m.set_weights(lnW)
        m.sweep(1, record=True)
        s, e = orc.init(L, 2, 45)
        H = orc.run(L, 2, s, e, orc.build_table(L, lnW), 0, N, True)
        assert np.array_equal(m.get_histogram(), H) and np.array_equal(m.get_energies(), e)
