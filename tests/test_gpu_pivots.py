"""The FP32 LU's pivot rule and reciprocal, on matrices made for it: partial pivoting
inside the 32 x 32 diagonal block by the whole float32 magnitude, the lowest row of the
block among equals, multipliers with the correctly rounded reciprocal."""
import numpy as np
import pytest

from paper_1511_02166_gb300 import inputs
from tests.gpu_util import need_gpu

pytestmark = pytest.mark.gpu

N = 32  # one full diagonal block of the matrix proper, and the border


def factor(blocks, kind):
    """Stored factors [B][33][33] and pivot rows [B][33] of matrices whose leading
    32 x 32 block is given (the border decoupled from it: its Schur complement holds
    the reciprocals of all pivots, and overflows for the smallest ones)."""
    import torch
    from paper_1511_02166_gb300.solver import PanelBatch
    B = len(blocks)
    foil = inputs.naca4(0.02, 0.4, 0.12, N)
    pb = PanelBatch(np.tile(foil, (B, 1)), np.arange(B + 1) * N, np.zeros(B), bucket_width=None)
    A = np.zeros((B, N + 1, N + 1), dtype=np.float32)
    A[:, :N, :N] = blocks
    A[:, N, N] = 1.0
    pb.A_hi.copy_(torch.from_numpy(A).reshape(-1))
    pb.A_lo.zero_()
    pb.info.zero_()
    pb.lu_kind = [kind]
    pb.solve(stage="factor")
    assert pb.info.cpu().tolist() == [0] * B
    return pb.LU.cpu().numpy().reshape(B, N + 1, N + 1), pb.piv.cpu().numpy().reshape(B, N + 1)


@pytest.mark.parametrize("kind", [1, 2])
def test_pivot_is_the_largest_entry_to_the_last_bit(kind):
    need_gpu()
    blocks, want = [], []
    rng = np.random.default_rng(2)
    for bit in range(24):
        for _ in range(8):
            low, high = rng.choice(np.arange(1, N), 2, replace=False)
            a = np.diag(np.full(N, 4.0, np.float32))
            a[0, 0] = 0.5
            a[low, 0] = -1.0
            a[high, 0] = np.float32(1.0) + np.float32(2.0)**-bit
            blocks.append(a)
            want.append(high)
    lu, piv = factor(np.array(blocks), kind)
    assert piv[:, 0].tolist() == want


@pytest.mark.parametrize("kind", [1, 2])
def test_equal_pivots_take_the_lowest_row_of_the_block(kind):
    """Column 0 exchanges rows 0 and r; in column 1 row 0, now at position r, and the
    row at position s < r hold the same magnitude."""
    need_gpu()
    blocks, want = [], []
    for r in range(3, N):
        for s in range(2, r):
            a = np.diag(np.full(N, 4.0, np.float32))
            a[0, 0], a[r, 0] = 1.0, 2.0
            a[1, 1], a[0, 1], a[s, 1] = 0.25, -3.0, 3.0
            blocks.append(a)
            want.append([r, r])
    lu, piv = factor(np.array(blocks), kind)
    assert piv[:, :2].tolist() == want


@pytest.mark.parametrize("kind", [1, 2])
def test_multipliers_take_the_correctly_rounded_reciprocal(kind):
    """Pivots p on the diagonal above rows that hold 2^(e-1) (2^e <= |p|) in their
    column: the multiplier is 2^(e-1) times the reciprocal, exactly, and the stored
    inverse of L its negative.  Pivots from 2^-128 to 2^126."""
    need_gpu()
    rng = np.random.default_rng(7)
    B = 4096
    bits = rng.integers(0x00200001, 0x7e800000, (B, 16), dtype=np.uint32)
    bits[:64] = 0x3f800000 + rng.integers(0, 1 << 23, (64, 16))
    bits[0, :4] = [0x3fffffff, 0x3f800000, 0x00800000, 0x00200001]
    bits[1, :2] = [0x7e7fffff, 0x7e000000]
    bits |= rng.integers(0, 2, (B, 16), dtype=np.uint32) << 31
    p = bits.view(np.float32)
    x = np.ldexp(np.float32(1.0), np.frexp(p)[1] - 2).astype(np.float32)
    blocks = np.tile(np.diag(np.ones(N, np.float32)), (B, 1, 1))
    q = np.arange(16)
    blocks[:, q, q] = p
    blocks[:, q + 16, q] = x
    with np.errstate(over="ignore", under="ignore"):
        want = x * (np.float32(1.0) / p)
    lu, piv = factor(blocks, kind)
    assert (piv[:, :N] == np.arange(N)).all()
    assert np.array_equal((-lu[:, q + 16, q]).view(np.uint32), want.view(np.uint32))
