"""Launches of many walkers: direct threshold loads only where an SM holds more than two
warps of the kernel per sub-partition at once."""
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


@pytest.mark.parametrize("L,wpb,form", [
    # blocks whose shared memory leaves room for one per SM (6 to 8 warps): loads two ahead
    (44, 192, 0), (40, 224, 0), (28, 256, 0), (32, 256, 0), (60, 32, 0), (64, 192, 0),
    # more than eight warps at once: direct loads
    (44, 160, -1), (40, 160, -1), (36, 160, -1), (32, 160, -1), (28, 160, -1), (20, 256, -1), (8, 256, -1), (4, 32, -1),
])
def test_form_by_resident_warps(M, L, wpb, form):
    import torch
    from paper_1707_00919_gb300 import _lib as C
    W = torch.cuda.get_device_properties(0).multi_processor_count * 8 * 32 + 32
    with M.Muca(L, W, 1, layout=1, walkers_per_block=wpb) as m:
        m.attempts(4, record=False)
        assert C.load().muca_testing_form(m._h) == form
        assert (m.get_energies() >= 0).all()


@pytest.mark.parametrize("layout", [0, 1])
def test_default_counts_are_fixed(M, layout):
    """The walkers per SM of the default count, which decides the chains of an instance created
    without one."""
    import torch
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    counts = {4: 2048, 8: 512 if layout else 768, 12: 2048, 16: 640, 20: 1792, 24: 512, 28: 1120, 32: 320, 36: 512,
              40: 448, 44: 384, 48: 256, 52: 256, 56: 256, 60: 256, 64: 224}
    assert {L: M.muca_optimal_walkers(L, layout)[0] // sms for L in counts} == counts
