"""Batches that exist at the same time."""
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


def test_a_smaller_batch_leaves_the_larger_one_usable(M):
    """The kernel's bound on shared memory serves every batch, whatever was created last."""
    lnW = {L: np.cumsum(np.random.default_rng(L).normal(0.0, 0.4, L * L + 1)) for L in (8, 64)}
    out = []
    for batched in (False, True):
        big, small = M.Muca(64, 300, 1), M.Muca(8, 64, 2)
        for m in (big, small):
            m.set_weights(lnW[m.L])
        if batched:
            with M.Batch([big]) as b, M.Batch([small]) as s:
                b.sweep(2, record=True)
                s.sweep(2, record=True)
                b.sweep(1, record=True)
        else:
            big.sweep(3, record=True)
            small.sweep(2, record=True)
        out.append([x for m in (big, small) for x in (m.get_histogram(), m.get_energies(), m.get_lattice())])
        big.close()
        small.close()
    assert all(np.array_equal(x, y) for x, y in zip(*out))


@pytest.mark.parametrize("L,W", [(8, 64), (32, 700), (64, 300)])
def test_info_reports_the_shared_memory_of_a_launch(M, L, W):
    """Table (a row of zeros behind the energies; 24-byte rows at L = 64, else 28) and the rows
    of a block's walkers."""
    with M.Muca(L, W, 1) as m, M.Batch([m]) as b:
        table = -(-(L * L + 2) * (24 if L == 64 else 28) // 16) * 16
        rows = L * (4 * ((L + 7) // 8) if L <= 32 else 8)
        assert b.info()[2] == table + rows * 256
