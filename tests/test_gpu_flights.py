"""Which form a launch of few walkers takes beside sweeps that are in flight: the paired
kernel only with the device to itself, and again once the others have ended, however the
host came to know of that.  Results do not depend on the form."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

LONG = 20000   # sweeps of L = 32: a third of a second


@pytest.fixture(scope="module")
def M():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__
    __graft_entry__.build()
    from paper_1707_00919_gb300 import muca
    return muca


def paired(m):
    from paper_1707_00919_gb300 import _lib as C
    return C.load().muca_testing_form(m._h) > 0


def test_own_streams(M):
    import torch
    with M.Muca(32, 1024, 1) as a, M.Muca(32, 1024, 2) as b:
        a.sweep(LONG, record=False)
        assert paired(a)
        b.sweep(1, record=False)
        assert not paired(b)
        torch.cuda.synchronize()
        for _ in range(8):   # an overlap is taken to recur for as many launches
            b.sweep(1, record=False)
            assert not paired(b)
        b.sweep(1, record=False)
        assert paired(b)


def test_a_callers_stream(M):
    """Waited for by the caller's own means: the sweeps on it count while they run only."""
    import torch
    st = torch.cuda.Stream()
    with M.Muca(32, 1024, 1, stream=st) as a, M.Muca(32, 1024, 2) as b, M.Muca(32, 1024, 3) as c:
        a.sweep(LONG, record=False)
        assert paired(a)
        b.sweep(1, record=False)
        assert not paired(b)
        st.synchronize()
        c.sweep(1, record=False)
        assert paired(c)


def test_a_captured_launch_is_not_in_flight(M):
    import torch
    st = torch.cuda.Stream()
    with M.Muca(32, 1024, 1, stream=st) as a, M.Muca(32, 1024, 2) as b:
        a.sweep(1, record=False)
        a.synchronize()
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g, stream=st, capture_error_mode="thread_local"):
            a.sweep(1, record=False)
            b.sweep(1, record=False)   # on its own stream: runs now
            assert paired(b)
        lat = a.get_lattice()
        g.replay()
        torch.cuda.synchronize()
        assert np.array_equal(a.get_lattice(), -lat)   # every flip is accepted at ln W = 0


def test_members_of_a_batch_and_after_it(M):
    import torch
    st = torch.cuda.Stream()
    with M.Muca(32, 1024, 1, stream=st) as a, M.Muca(32, 1024, 2) as b, M.Muca(32, 1024, 3) as c:
        with M.Batch([a]) as batch:
            a.sweep(1, record=False)   # by itself, on the batch's stream
            torch.cuda.synchronize()
            b.sweep(1, record=False)
            assert paired(b)
            b.synchronize()
            a.sweep(1, record=False)
            batch.sweep(1, record=False)
        c.sweep(1, record=False)   # closing the batch has waited
        assert paired(c)


def test_batched_sweeps(M):
    import torch
    with M.Muca(32, 1024, 1) as a, M.Muca(32, 1024, 2) as b, M.Muca(32, 1024, 3) as c:
        with M.Batch([a]) as batch:
            batch.sweep(LONG, record=False)
            b.sweep(1, record=False)
            assert not paired(b)
            torch.cuda.synchronize()
            c.sweep(1, record=False)
            assert paired(c)


def test_batched_iteration_in_another_thread(M):
    import threading
    with M.Muca(32, 1024, 1) as a, M.Muca(32, 1024, 2) as b, M.Muca(32, 1024, 3) as c:
        with M.Batch([a]) as batch:
            params = M.make_params(therm_sweeps=LONG, sweeps_per_iter=1, max_iterations=1, flat_threshold=2.0)
            t = threading.Thread(target=batch.iterate_until_flat, args=(params,))
            t.start()
            forms = []
            while t.is_alive():
                b.sweep(1, record=False)
                b.synchronize()
                forms.append(paired(b))
            t.join()
            assert not all(forms)   # the launches before the iteration's own may be
            c.sweep(1, record=False)
            assert paired(c)


def test_allocation_free_sweeps(M):
    import torch
    from paper_1707_00919_gb300 import _lib as C
    L, W, st = 32, 1024, torch.cuda.Stream()
    N = L * L
    zeros = lambda n, t: torch.zeros(n, dtype=t, device="cuda")
    bufs = (torch.ones(N * W, dtype=torch.int8, device="cuda"), zeros(W, torch.int32), zeros(5 * (N + 1), torch.int32),
            zeros(N + 1, torch.int64), zeros(1, torch.int32))   # all spins up, no flip accepted
    r = C.muca_raw_instance(L, 0, W, 1, 0, *(t.data_ptr() for t in bufs))
    torch.cuda.synchronize()
    with M.Muca(L, W, 2) as b, M.Muca(L, W, 3) as c:
        M.muca_batch_sweep_noalloc([r], LONG // 2, False, st.cuda_stream)
        b.sweep(1, record=False)
        assert not paired(b)
        st.synchronize()
        c.sweep(1, record=False)
        assert paired(c)
    assert int(bufs[4].item()) == 0
