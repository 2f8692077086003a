"""The one-thread-per-walker forms of the sweep kernel against the oracle, bit for bit, at
every lattice size that reaches them, with the form that ran checked: loads two attempts
ahead, direct loads; spins as bytes in whole and ragged warps, packed rows."""
import functools

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

WALKERS = [(0, 0), (0, 45), (1, 45)]   # (layout, walkers beyond whole warps)


@pytest.fixture(scope="module")
def M():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__
    __graft_entry__.build()
    from paper_1707_00919_gb300 import muca
    return muca


@functools.lru_cache(maxsize=1)
def start(orc, L, seed, W):
    return orc.init(L, seed, W)


def check(M, orc, L, warps_per_sm, extra, layout, wpb, form):
    """A fused launch cut at both ends, unrecorded rows, a recorded part of a row."""
    import torch
    from paper_1707_00919_gb300 import _lib as C
    W = torch.cuda.get_device_properties(0).multi_processor_count * 32 * warps_per_sm + 32 + extra
    seed, N = 40 + L, L * L
    lnW = np.cumsum(np.random.default_rng(L).normal(0.0, 0.4, N + 1))
    T = orc.build_table(L, lnW)
    therm, rec, more, last = 3 * L + 6, 2 * L + 3, 2 * L + 1, L // 2
    with M.Muca(L, W, seed, layout=layout, walkers_per_block=wpb) as m:
        m.set_weights(lnW)
        m.set_attempt_counter(5)
        m.thermalize_and_record(therm, rec)
        assert C.load().muca_testing_form(m._h) == form
        m.attempts(more, False)
        m.attempts(last, True)
        assert C.load().muca_testing_form(m._h) == form
        H, e, lat = m.get_histogram(), m.get_energies(), m.get_lattice()
    s, eo = (x[:W].copy() for x in start(orc, L, seed, W - extra + 45))   # a walker's spins follow from its index
    Ho = np.zeros(N + 1, dtype=np.uint64)
    orc.run(L, seed, s, eo, T, 5, therm, False)
    orc.run(L, seed, s, eo, T, 5 + therm, rec, True, Ho)
    orc.run(L, seed, s, eo, T, 5 + therm + rec, more, False)
    orc.run(L, seed, s, eo, T, 5 + therm + rec + more, last, True, Ho)
    assert np.array_equal(lat, s)
    assert np.array_equal(e, eo)
    assert np.array_equal(H, Ho)


@pytest.mark.parametrize("layout,extra", WALKERS)
@pytest.mark.parametrize("L", range(4, 65, 4))
def test_loads_two_attempts_ahead(M, orc, L, layout, extra):
    check(M, orc, L, 2, extra, layout, 64 if L < 48 else 32, 0)


@pytest.mark.parametrize("layout,extra", WALKERS)
@pytest.mark.parametrize("L", range(4, 45, 4))
def test_direct_loads(M, orc, L, layout, extra):
    check(M, orc, L, 8, extra, layout, 256 if L <= 20 else 128 if L == 24 else 160, -1)


@pytest.mark.parametrize("layout,extra", WALKERS[2:])
@pytest.mark.parametrize("L", [48, 52, 56, 60, 64])
def test_many_walkers_of_large_lattices(M, orc, L, layout, extra):
    """No block size leaves more than eight warps resident."""
    check(M, orc, L, 8, extra, layout, 0, 0)
