"""The FP64 default against the sum of the absolute products of every element: operands
whose values differ in size along k, so that the digits of the small ones matter.

N terms summed by FP64 FMAs are off by at most N 2^-53 of that sum; the digits may lose
as much, and both round a few times more (the groups of the packed kernel, the classes
of the digits): N + 4."""
import numpy as np
import pytest

from synth import BlockMatrix
from tests import helpers as H

pytestmark = pytest.mark.gpu


def blocks_of(dense, rs, cs, mask=None):
    """The dense matrix in blocks, those where mask is false left out."""
    ro, co = H.offsets(rs), H.offsets(cs)
    mask = np.ones((len(rs), len(cs)), bool) if mask is None else mask
    r, c = np.nonzero(mask)
    v = [dense[ro[i]:ro[i + 1], co[j]:co[j + 1]].T.reshape(-1) for i, j in zip(r, c)]
    return BlockMatrix(np.asarray(rs, np.int32), np.asarray(cs, np.int32), r.astype(np.int32),
                       c.astype(np.int32), np.concatenate(v))


def check(bsm_lib, A, B):
    """Every element of A B by the default kernel; the error against the whole result's norm."""
    with bsm_lib.Context(0) as ctx:
        dA, dB, dC = ctx.from_blocks(A), ctx.from_blocks(B), ctx.empty(A.row_sizes, B.col_sizes)
        st = ctx.multiply(1.0, dA, dB, 0.0, dC, 0.0, blocking=True, stats=True)
        assert st.kept >= 4 * st.c_blocks  # fewer are another kernel's
        got = H.to_dense(BlockMatrix(A.row_sizes, B.col_sizes, *dC.pattern(), dC.values()), np.longdouble)
    a, b = (H.to_dense(M).astype(np.longdouble) for M in (A, B))
    want, size = a @ b, np.abs(a) @ np.abs(b)
    err = np.abs(got - want)
    worst = (err / np.where(size > 0, size, 1)).max() * 2.0 ** 53
    assert worst <= a.shape[1] + 4, f"{float(worst):.3g} x 2^-53 of the sum of absolute products"
    assert not err[size == 0].any()
    return float(np.linalg.norm(err.astype(np.float64)) / np.linalg.norm(want.astype(np.float64)))


# few C blocks (shared out by their tiles) and many; the first block row has one product
@pytest.mark.parametrize("rs,ks,cs", [([13, 13, 13, 5], [13] * 6, [13, 5]), ([17, 33, 8, 9], [16, 5, 8, 9, 1, 7], [16, 8, 33]),
                                      ([5] * 120, [5, 3, 8, 2, 5, 6], [5] * 110), ([13] * 3, [3] * 70, [13, 9])])
@pytest.mark.parametrize("r", [4, 8, 12, 13, 15, 20, 25, 60])
def test_sizes_that_cancel_along_k(bsm_lib, rs, ks, cs, r):
    """A = R D, B = D^-1 S, D powers of two from 2^-r to 2^r: the products are of one size."""
    rng = np.random.default_rng(r + len(rs))
    m, k, n = sum(rs), sum(ks), sum(cs)
    d = np.ldexp(1.0, rng.integers(-r, r + 1, k))
    mask = np.ones((len(rs), len(ks)), bool)
    mask[0, 1:] = False
    A = blocks_of(rng.standard_normal((m, k)) * d, rs, ks, mask)
    B = blocks_of(rng.standard_normal((k, n)) / d[:, None], ks, cs)
    assert check(bsm_lib, A, B) <= 1e-15


@pytest.mark.parametrize("role", ["left", "right"])
@pytest.mark.parametrize("partner", [0.0, 1e-30])
@pytest.mark.parametrize("t", [1e-3, 1e-6, 1e-10, 1e-15, 1e-20])
def test_one_large_value_against_a_small_partner(bsm_lib, role, partner, t):
    """The large value of a row meets zeros or next to nothing: the others decide."""
    rng = np.random.default_rng(5)
    rs, ks, cs = [13, 5, 16, 9], [8, 13, 5, 6, 7], [13, 5, 8]
    m, k, n = sum(rs), sum(ks), sum(cs)
    a, b = rng.standard_normal((m, k)) * t, rng.standard_normal((k, n))
    for at in (3, 10, 37):
        a[:, at] = rng.standard_normal(m)
        b[at] = partner * rng.standard_normal(n)
    if role == "right":
        a, b, rs, cs = b.T.copy(), a.T.copy(), cs, rs
    check(bsm_lib, blocks_of(a, rs, ks), blocks_of(b, ks, cs))


@pytest.mark.parametrize("low", [8, 11, 12])
def test_rows_and_columns_far_below_their_blocks(bsm_lib, low):
    """A row of A and a column of B, each 2^-low of the other rows and columns of its blocks
    but for blocks that do not meet."""
    rng = np.random.default_rng(low)
    rs, ks, cs = [13, 9, 16], [13, 13, 5, 5, 8, 6, 9, 9], [13, 5, 8]
    a = rng.standard_normal((sum(rs), sum(ks)))
    b = rng.standard_normal((sum(ks), sum(cs)))
    keep_a, keep_b = np.ones((len(rs), len(ks)), bool), np.ones((len(ks), len(cs)), bool)
    keep_b[0], keep_a[:, 1] = False, False  # block column 0 of A and block row 1 of B alone are large
    ko = H.offsets(ks)
    a[::3, ko[1]:] *= 2.0 ** -low
    b[:ko[1], ::3] *= 2.0 ** -low
    b[ko[2]:, ::3] *= 2.0 ** -low
    check(bsm_lib, blocks_of(a, rs, ks, keep_a), blocks_of(b, ks, cs, keep_b))


def test_zero_rows_columns_and_blocks(bsm_lib):
    """Exact zeros lose nothing: rows, columns and whole blocks of them."""
    rng = np.random.default_rng(9)
    rs, ks, cs = [13, 5, 16], [13, 5, 5, 8, 6], [13, 5, 8]
    a, b = rng.standard_normal((sum(rs), sum(ks))), rng.standard_normal((sum(ks), sum(cs)))
    a[4], a[20:25], b[:, 3], a[:, 14] = 0.0, 0.0, 0.0, 0.0
    a[:13, :13], b[13:18] = np.diag(np.arange(13.0)), 0.0
    check(bsm_lib, blocks_of(a, rs, ks), blocks_of(b, ks, cs))


def digits(x):
    """The eight signed base-256 digits of x on the scale 1 (x times 2^62 is an integer here)."""
    v = int(x * 2.0 ** 62)
    assert v == x * 2.0 ** 62
    out = []
    for _ in range(7):
        d = (v + 128) % 256 - 128
        out.append(d)
        v = (v - d) >> 8
    return [v] + out[::-1]


@pytest.mark.parametrize("low", [-128, 127])
@pytest.mark.parametrize("rs,cs", [([16], [8]), ([8, 5], [13, 16]), ([16, 33], [5, 32])])
def test_digits_at_their_extreme(bsm_lib, rs, cs, low):
    """144 values of k, as many as are added up in FP32 between two reads, with every digit
    but the first at its extreme: 7 x 2^14 x 144 = 16.5 M of 2^24 on a diagonal. A large value
    on either side that meets a zero sets the scales. The result is that of exact integers
    over the kept digit pairs, rounded once."""
    ks = [8] * 18 + [2]
    x = sum(low * 256 ** (7 - i) for i in range(1, 8)) * 2.0 ** -62
    a, b = np.full((sum(rs), sum(ks)), x), np.full((sum(ks), sum(cs)), x)
    a[:, -2:], b[-2:] = [0.5, 0.0], np.array([[0.0], [0.5]])
    d = digits(x)
    kept = 144 * sum(d[i] * d[j] * 256 ** (14 - i - j) for i in range(8) for j in range(8) if i + j < 9)
    with bsm_lib.Context(0) as ctx:
        A, B = blocks_of(a, rs, ks), blocks_of(b, ks, cs)
        dA, dB, dC = ctx.from_blocks(A), ctx.from_blocks(B), ctx.empty(A.row_sizes, B.col_sizes)
        ctx.multiply(1.0, dA, dB, 0.0, dC, 0.0, blocking=True)
        assert (dC.values() == kept / 2 ** 124).all()  # of integers: rounded to nearest
    # more than FP64 FMAs of the values would give without an error: not by accident
    assert kept != int(x * 2.0 ** 62) ** 2 * 144


@pytest.mark.parametrize("k", [65528, 65529, 70001])
def test_the_longest_k_that_digits_take(bsm_lib, k):
    """8191 octets of k in a block are the digits' limit; longer ones are the packed kernel's."""
    rng = np.random.default_rng(k)
    rs, ks, cs = [5, 3], [k, 9, k, 2, k, 4], [4]
    a, b = rng.standard_normal((sum(rs), sum(ks))), rng.standard_normal((sum(ks), sum(cs)))
    assert check(bsm_lib, blocks_of(a, rs, ks), blocks_of(b, ks, cs)) <= 1e-13
