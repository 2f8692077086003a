"""Device buffers of the allocation-free batched sweep that are off their alignment are
refused on the host (no launch: no GPU needed, and none of the buffers exists)."""
import ctypes

import pytest


@pytest.fixture(scope="module")
def lib():
    from paper_1707_00919_gb300 import build
    build.build()
    from paper_1707_00919_gb300 import _lib
    return _lib.load()


BASE = 1 << 20   # addresses on every boundary; the lattices below are shorter than a step


@pytest.mark.parametrize("L,layout,W,field,shift", [
    (8, 0, 32, "lattice", 8),           # bytes of whole warps move as 16-byte vectors
    (8, 0, 48, "lattice", 1),
    (32, 0, 16384, "lattice", 4),
    (8, 1, 33, "lattice", 2),           # packed rows: 4-byte words up to L = 32, 8-byte above
    (32, 1, 32, "lattice", 1),
    (48, 1, 5, "lattice", 4),
    (64, 1, 64, "lattice", 2),
    (16, 0, 5, "energy", 2),
    (16, 1, 64, "table", 1),
    (16, 0, 64, "hist", 4),
    (16, 0, 64, "err", 2),
])
def test_misaligned_buffers_are_refused(lib, L, layout, W, field, shift):
    from paper_1707_00919_gb300 import _lib as C
    at = {n: BASE * (i + 1) * 64 for i, n in enumerate(("lattice", "energy", "table", "hist", "err"))}
    at[field] += shift
    r = C.muca_raw_instance(L, layout, W, 1, 0, at["lattice"], at["energy"], at["table"], at["hist"], at["err"])
    assert lib.muca_batch_sweep_noalloc(ctypes.byref(r), 1, 1, 1, None) == C.MUCA_EINVAL
    assert b"aligned" in lib.muca_last_error()
