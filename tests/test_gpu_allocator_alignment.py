"""Memory that the allocator hook hands out off the kernels' alignment is refused and given
back; memory that is aligned enough for the instance at hand is taken."""
import ctypes

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


@pytest.fixture()
def shifted(M):
    """An allocator whose memory starts `shift` bytes behind a 256-byte boundary."""
    import torch
    from paper_1707_00919_gb300 import _lib as C
    held, state = {}, {"shift": 0}

    def alloc(n, ctx):
        t = torch.empty(n + 256, dtype=torch.uint8, device="cuda")
        p = (t.data_ptr() + 255) // 256 * 256 + state["shift"]
        held[p] = t
        return p

    cb = C.ALLOC_FN(alloc), C.RELEASE_FN(lambda p, ctx: (held.pop(p), None)[1])
    before = M._torch_cb or (C.ALLOC_FN(), C.RELEASE_FN())
    assert C.load().muca_set_allocator(cb[0], cb[1], None) == 0
    yield state, held
    assert C.load().muca_set_allocator(before[0], before[1], None) == 0


def create(C, L, W, layout):
    o = C.muca_options(L, W, 3, layout, 0, 0)
    h = ctypes.c_void_p()
    rc = C.load().muca_create_ex(ctypes.byref(o), ctypes.byref(h))
    if h.value:
        assert C.load().muca_destroy(h) == 0
    return rc


@pytest.mark.parametrize("L,W,layout,shift,ok", [
    (16, 64, 0, 8, False), (16, 48, 0, 4, False), (64, 32, 0, 1, False),
    (16, 64, 1, 4, False), (64, 77, 1, 4, False), (16, 77, 0, 4, False),
    (16, 64, 0, 16, True), (16, 64, 1, 8, True), (64, 77, 1, 8, True), (16, 16, 0, 8, True),
])
def test_instance_memory(M, shifted, L, W, layout, shift, ok):
    from paper_1707_00919_gb300 import _lib as C
    state, held = shifted
    state["shift"] = shift
    assert create(C, L, W, layout) == (0 if ok else C.MUCA_EINVAL)
    assert ok or b"aligned" in C.load().muca_last_error()
    assert not held


def test_batch_and_iteration_memory(M, shifted):
    from paper_1707_00919_gb300 import _lib as C
    state, held = shifted
    with M.Muca(16, 64, 1, torch_allocator=False) as m:
        state["shift"] = 4
        with pytest.raises(M.MucaError) as ex:
            M.Batch([m])
        assert ex.value.code == C.MUCA_EINVAL
        with pytest.raises(M.MucaError) as ex:
            m.iterate_device(M.make_params(max_iterations=1), 1, raise_on_fail=True)
        assert ex.value.code == C.MUCA_EINVAL
        state["shift"] = 8
        with M.Batch([m]) as b:
            b.sweep(1, record=True)
            assert int(m.get_histogram().sum()) == 64 * 256


@pytest.mark.parametrize("L,W,layout", [(16, 77, 0), (48, 33, 0), (32, 64, 1)])
def test_eight_byte_alignment_is_enough(M, orc, shifted, L, W, layout):
    state, held = shifted
    state["shift"] = 8
    N = L * L
    lnW = np.cumsum(np.random.default_rng(L).normal(0.0, 0.4, N + 1))
    with M.Muca(L, W, 4, layout, torch_allocator=False) as m:
        m.set_weights(lnW)
        m.thermalize_and_record(N + 3, 2 * N)
        H, e, lat = m.get_histogram(), m.get_energies(), m.get_lattice()
    s, eo = orc.init(L, 4, W)
    T = orc.build_table(L, lnW)
    orc.run(L, 4, s, eo, T, 0, N + 3, False)
    Ho = orc.run(L, 4, s, eo, T, N + 3, 2 * N, True)
    assert np.array_equal(H, Ho) and np.array_equal(e, eo) and np.array_equal(lat, s)
