"""The FP64 to BF16-piece conversion of the tensor-core operands, bit for bit.
With B the identity, C = A B^T in plain BF16 is A's first piece h =
bf16(fl32(a)), and [-h | A] [I | I]^T in split BF16 adds -h, h and then the
second piece, each sum exact in FP32: m = bf16(fl32(a - h))."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def _bf16(x):
    u = np.asarray(x, dtype=np.float64).astype(np.float32).view(np.uint32).astype(np.uint64)
    u = ((u + 0x7FFF + ((u >> 16) & 1)) >> 16) << 16
    return u.astype(np.uint32).view(np.float32).astype(np.float64)


def _values(kind, n, rng):
    """Mantissas at and next to the roundings' ties, exponents in and out of the fast path's range."""
    m = rng.integers(0, 1 << 52, n, dtype=np.uint64)
    z = rng.integers(0, 52, n).astype(np.uint64)
    one = np.uint64(1)
    if kind == "ones":           # a run of ones at the end: just below a tie or a power of two
        m |= (one << z) - one
    elif kind == "zeros":        # few significant bits: exact pieces and exact ties
        m = (m >> z) << z
    elif kind == "ties":         # half an ulp of BF16 (of FP32), plus or minus a little
        low = np.uint64(45 if rng.random() < 0.5 else 29)
        m = (m >> low << low) + (one << (low - one)) + rng.integers(-2, 3, n).astype(np.int64).view(np.uint64)
        m &= (one << np.uint64(52)) - one
    e = rng.integers(1023 - 70, 1023 + 30, n).astype(np.uint64)   # 2^-63 is the range's end
    s = rng.integers(0, 2, n).astype(np.uint64)
    return ((s << np.uint64(63)) | (e << np.uint64(52)) | m).view(np.float64)


@pytest.mark.parametrize("kind", ["random", "ones", "zeros", "ties"])
def test_two_piece_conversion_is_the_two_step_rounding(mpslcc, kind):
    rng = np.random.default_rng(len(kind))
    A = _values(kind, 1000 * 64, rng).reshape(1000, 64)
    A[0, :4] = (0.0, 1.0, -2.0 ** -60, 2.0 ** 100)
    h, eye = _bf16(A), np.eye(64)
    with mpslcc.Context(device=0) as ctx:
        first = ctx.debug_tc_gemm(A, eye, prec=mpslcc.BF16, mode=2)
        second = ctx.debug_tc_gemm(np.hstack([-h, A]), np.hstack([eye, eye]), prec=mpslcc.BF16X3, mode=2)
    assert np.array_equal(first, h)
    assert np.array_equal(second, _bf16(A - h))
