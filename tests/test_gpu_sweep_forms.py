"""Every lattice size and every form of the sweep kernel against the oracle, bit for bit:
ranges cut at both ends, ranges inside one row, ragged warps, launches of many warps
(direct threshold loads), batches whose range crosses a step of Philox counter word 1."""
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


def rand_weights(L, seed):
    return np.cumsum(np.random.default_rng(seed).normal(0.0, 0.4, L * L + 1))


@pytest.mark.parametrize("L", range(4, 65, 4))
def test_every_size_and_cut(M, orc, L):
    W, seed, N = 45, 7 + L, L * L
    lnW = rand_weights(L, L)
    # (thermalization, recorded) attempts: inside a row, cut at both ends, ending at a row's
    # end, whole sweeps, a fused launch cut at both ends
    plan = [(0, 3), (1, 0), (0, N + L + 2), (2 * L + 3, 0), (0, 2 * N), (N + 5, N + L - 1)]
    s, e = orc.init(L, seed, W)
    T = orc.build_table(L, lnW)
    t = 0
    with M.Muca(L, W, seed, layout=(L // 4) % 2) as m:
        m.set_weights(lnW)
        for therm, rec in plan:
            m.thermalize_and_record(therm, rec)
            orc.run(L, seed, s, e, T, t, therm, False)
            Ho = orc.run(L, seed, s, e, T, t + therm, rec, True)
            t += therm + rec
            H = m.get_histogram()
            assert np.array_equal(H, Ho if rec else np.zeros(N + 1, dtype=np.uint64))
            assert np.array_equal(m.get_energies(), e)
        assert m.attempt_counter == t
        assert np.array_equal(m.get_lattice(), s)


@pytest.mark.parametrize("L", [4, 8, 12, 24, 28, 32, 48, 60, 64])
@pytest.mark.parametrize("warps_per_sm", [0, 1, 2])
def test_forms_by_walker_count(M, orc, L, warps_per_sm):
    """One and two chain warps per block with their generators, one thread per walker with
    the loads two attempts ahead; a fused launch cut at both ends, then unrecorded rows and a
    recorded part of a row, a ragged last warp."""
    import torch
    W = torch.cuda.get_device_properties(0).multi_processor_count * 32 * warps_per_sm + 77
    seed, N = 11, L * L
    lnW = rand_weights(L, 3 * L)
    T = orc.build_table(L, lnW)
    therm, rec, more, last = 3 * L + 6, 2 * L + 3, 5 * L + 1, L // 2
    with M.Muca(L, W, seed, layout=warps_per_sm % 2) as m:
        m.set_weights(lnW)
        m.set_attempt_counter(5)
        m.thermalize_and_record(therm, rec)
        m.attempts(more, False)
        m.attempts(last, True)
        H, e, lat = m.get_histogram(), m.get_energies(), m.get_lattice()
    assert int(H.sum()) == W * (rec + last)
    Ho = np.zeros(N + 1, dtype=np.uint64)
    whole = L <= 12 or warps_per_sm == 0
    for w0, n in ([(0, W)] if whole else [(0, 64), (W - 77, 77)]):
        s, eo = orc.init(L, seed, n, walker0=w0)
        orc.run(L, seed, s, eo, T, 5, therm, False, walker0=w0)
        orc.run(L, seed, s, eo, T, 5 + therm, rec, True, Ho, walker0=w0)
        orc.run(L, seed, s, eo, T, 5 + therm + rec, more, False, walker0=w0)
        orc.run(L, seed, s, eo, T, 5 + therm + rec + more, last, True, Ho, walker0=w0)
        assert np.array_equal(lat[w0:w0 + n], s)
        assert np.array_equal(e[w0:w0 + n], eo)
    if whole:
        assert np.array_equal(H, Ho)


@pytest.mark.parametrize("L,extra", [(8, 0), (8, 45), (12, 45), (20, 31), (32, 45)])
def test_many_warps(M, orc, L, extra):
    """More than two warps per SM sub-partition: the form with direct loads."""
    import torch
    W = torch.cuda.get_device_properties(0).multi_processor_count * 8 * 32 + 32 + extra
    seed, N = 3, L * L
    lnW = rand_weights(L, 2 * L)
    T = orc.build_table(L, lnW)
    with M.Muca(L, W, seed, layout=1, walkers_per_block=32) as m:
        m.set_weights(lnW)
        m.thermalize_and_record(N + 5, 2 * L + 3)
        H, e, lat = m.get_histogram(), m.get_energies(), m.get_lattice()
    assert int(H.sum()) == W * (2 * L + 3)
    # all walkers where the oracle is quick, else the first and the last ones
    for w0, n in ([(0, W)] if L <= 12 else [(0, 64), (W - 77, 77)]):
        s, eo = orc.init(L, seed, n, walker0=w0)
        orc.run(L, seed, s, eo, T, 0, N + 5, False, walker0=w0)
        Ho = orc.run(L, seed, s, eo, T, N + 5, 2 * L + 3, True, walker0=w0)
        assert np.array_equal(lat[w0:w0 + n], s)
        assert np.array_equal(e[w0:w0 + n], eo)
        if n == W:
            assert np.array_equal(H, Ho)


@pytest.mark.parametrize("L", range(4, 65, 4))
def test_random_order_every_size(M, orc, L):
    """Windows cut by conflicts, chunks of sites, heads and tails inside a Philox block."""
    W, seed, N = 77, 21 + L, L * L
    lnW = rand_weights(L, 5 * L)
    T = orc.build_table(L, lnW)
    s, e = orc.init(L, seed, W)
    t = 0
    with M.Muca(L, W, seed, layout=(L // 4) % 2) as m:
        m.set_weights(lnW)
        m.site_order = M.MUCA_ORDER_RANDOM
        for n, rec in [(1, True), (1, False), (9, True), (4, True), (510, True), (1026, False), (700, True)]:
            m.reset_histogram()
            m.attempts(n, rec)
            Ho = orc.run(L, seed, s, e, T, t, n, rec, site_order=1)
            t += n
            if rec:
                assert np.array_equal(m.get_histogram(), Ho)
            assert np.array_equal(m.get_energies(), e)
        assert np.array_equal(m.get_lattice(), s)


def test_batch_across_counter_word(M):
    """Ranges that cross t = 2^34 inside a batched launch equal the instances run alone."""
    specs = [(8, 70), (24, 33), (64, 40)]
    for back in (2, 100, 64 * 64 + 8):
        alone, together = [], []
        for out in (alone, together):
            inst = [M.Muca(L, W, 5 + L) for L, W in specs]
            for m, (L, _) in zip(inst, specs):
                m.set_weights(rand_weights(L, L))
                m.set_attempt_counter(2**34 - back)
            if out is alone:
                for m in inst:
                    m.sweep(2, record=True)
            else:
                with M.Batch(inst) as b:
                    b.sweep(2, record=True)
            for m in inst:
                out.append((m.get_histogram(), m.get_energies(), m.get_lattice(), m.attempt_counter))
                m.close()
        for x, y in zip(alone, together):
            assert all(np.array_equal(p, q) for p, q in zip(x, y))


@pytest.mark.parametrize("shift", [0, 4, 1])
@pytest.mark.parametrize("L", [4, 8, 12, 20, 32, 36, 60, 64])
def test_lattice_in_and_out(M, L, shift):
    """Lattices given by the user come back unchanged, with their energies, from both
    layouts, also where the allocator's buffer for them starts off a 16-byte boundary."""
    import torch
    from paper_1707_00919_gb300 import _lib as C
    W, N = 71, L * L
    held = {}

    def alloc(n, ctx):
        t = torch.empty(n + 16, dtype=torch.uint8, device="cuda")
        p = t.data_ptr() + (shift if n == W * N else 0)   # the transfer buffer alone
        held[p] = t
        return p

    spins = np.random.default_rng(L).choice(np.array([-1, 1], np.int8), size=(W, N))
    s = spins.reshape(W, L, L).astype(np.int32)
    bonds = (s != np.roll(s, 1, 1)).sum((1, 2)) + (s != np.roll(s, 1, 2)).sum((1, 2))
    cb = C.ALLOC_FN(alloc), C.RELEASE_FN(lambda p, ctx: (held.pop(p), None)[1])
    before = M._torch_cb or (C.ALLOC_FN(), C.RELEASE_FN())
    assert C.load().muca_set_allocator(cb[0], cb[1], None) == 0
    try:
        for layout in (0, 1):
            with M.Muca(L, W, 3, layout) as m:
                m.set_lattice(spins)
                assert np.array_equal(m.get_energies(), bonds // 2)
                assert np.array_equal(np.asarray(m.get_lattice()).reshape(W, N), spins)
    finally:
        assert C.load().muca_set_allocator(before[0], before[1], None) == 0


@pytest.mark.parametrize("specs", [
    [(64, 300), (16, 700), (24, 129)],                  # small items for the longest chains
    [(32, 128), (8, 31)],                               # one item each
    [(8, 257)] * 5 + [(48, 383)],                       # ragged last items, alone and not
    [(16, 40000), (64, 64)],                            # more items than SMs beside one long one
])
def test_batch_item_sizes(M, specs):
    """Every choice of items covers every walker once: a batch equals its instances alone."""
    out = []
    for batched in (False, True):
        inst = [M.Muca(L, W, 50 + i) for i, (L, W) in enumerate(specs)]
        for m, (L, _) in zip(inst, specs):
            m.set_weights(rand_weights(L, 3 * L))
        if batched:
            with M.Batch(inst) as b:
                b.sweep(2, record=True)
        else:
            for m in inst:
                m.sweep(2, record=True)
        out.append([(m.get_histogram(), m.get_energies(), m.get_lattice()) for m in inst])
        for m in inst:
            m.close()
    for x, y in zip(*out):
        assert all(np.array_equal(p, q) for p, q in zip(x, y))
