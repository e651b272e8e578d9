"""The FP64 default on the tensor cores (digits of the operands, exact integer
sums): tile edges, folds of the accumulators, operands that a digit
representation would not hold as FP64 does."""
import numpy as np
import pytest

import synth
from synth import BlockMatrix
from tests import helpers as H

pytestmark = pytest.mark.gpu


def multiply(ctx, A, B, alpha=1.0, beta=0.0, C=None, **kw):
    dA = ctx.from_blocks(A)
    dB = dA if B is A else ctx.from_blocks(B)
    dC = ctx.empty(A.row_sizes, B.col_sizes) if C is None else ctx.from_blocks(C)
    ctx.multiply(alpha, dA, dB, beta, dC, 0.0, blocking=True, **kw)
    out = dC.pattern() + (dC.values(),)
    for m in {id(x): x for x in (dA, dB, dC)}.values():
        m.destroy()
    return out


def full(rng, rs, cs, value):
    """A block matrix without zero blocks, entries value(n)."""
    r, c = np.divmod(np.arange(len(rs) * len(cs)), len(cs))
    n = int(np.sum(rs)) * int(np.sum(cs))
    return BlockMatrix(np.asarray(rs, np.int32), np.asarray(cs, np.int32), r.astype(np.int32),
                       c.astype(np.int32), value(n))


# rows and columns at the edges of the 16 x 8 tiles; k at those of the octets of 8,
# in all 18 octets (one fold of the accumulators), one more, and several folds
@pytest.mark.parametrize("rows", [[1, 7, 8], [9, 15, 16], [17, 24, 33]])
@pytest.mark.parametrize("ks", [[1, 2, 7, 8], [8] * 18, [8] * 18 + [1], [9, 15, 33, 40] * 12])
def test_integers_exact(gpu_ctx, rows, ks):
    """26-bit integers: the sums need more than 53 bits, and are rounded once for
    every 144 values of k, and once more for each such partial sum that is added.
    Each rounding is at most 2^-53 of the sum of the absolute products."""
    rng = np.random.default_rng(len(ks) + sum(rows))
    cols = [1, 7, 8, 9, 16, 17]
    ints = lambda n: rng.integers(-2 ** 26, 2 ** 26, n).astype(np.float64)  # noqa: E731
    A, B = full(rng, rows, ks, ints), full(rng, ks, cols, ints)
    a, b = (H.to_dense(M).astype(np.int64).astype(object) for M in (A, B))
    want, size = a @ b, np.abs(a) @ np.abs(b)
    r, c, v = multiply(gpu_ctx, A, B)
    got = H.to_dense(BlockMatrix(A.row_sizes, B.col_sizes, r, c, v))
    # at most 32 products to a batch, each batch with folds of its own
    octets = sum(-(-k // 8) for k in ks)
    folds = -(-octets // 18) + len(ks) // 32
    bound = 2 * folds
    for x, y, s in zip(got.ravel(), want.ravel(), size.ravel()):
        assert abs(int(x) - y) * 2 ** 53 <= bound * s


@pytest.mark.parametrize("alpha,beta", [(1.0, 0.0), (-0.5, 2.0)])
def test_default_is_exact_on_small_integers_with_c_in(gpu_ctx, oracle_mod, alpha, beta):
    rng = np.random.default_rng(71)
    rs, ks, cs = ([int(x) for x in rng.choice([1, 3, 8, 9, 16, 17], n)] for n in (9, 40, 8))
    A = synth.random_blocks(rng, rs, ks, 0.7, kind="int", shuffle=True)
    B = synth.random_blocks(rng, ks, cs, 0.7, kind="int", shuffle=True)
    C = synth.random_blocks(rng, rs, cs, 0.5, kind="int", shuffle=True)
    ref = oracle_mod.multiply(A, B, alpha=alpha, beta=beta, C=C, eps=0.0)
    r, c, v = multiply(gpu_ctx, A, B, alpha, beta, C)
    assert np.array_equal(r, ref.blk_row) and np.array_equal(c, ref.blk_col)
    assert np.array_equal(v, ref.values)


@pytest.mark.parametrize("what", ["tiny_block", "tiny_row", "nan", "inf", "huge", "denormal", "zero_row",
                                  "tall"])
def test_blocks_that_digits_do_not_hold(gpu_ctx, bsm_lib, oracle_mod, what):
    """One block of A or B outside what its row's scale holds: the C blocks that
    it contributes to come from the FP64 kernel, bit for bit, the others from
    the digit kernel; every C block is within 1e-12 of the oracle's, by itself."""
    rng = np.random.default_rng(72)
    rs = [5, 13, 9, 16, 200 if what == "tall" else 8]
    ks = [5, 13, 8, 6, 5, 13]
    cs = [13, 5, 7]
    normal = rng.standard_normal
    A, B = full(rng, rs, ks, normal), full(rng, ks, cs, normal)
    off = H.block_list_offsets(A)
    b = 1 * len(ks) + 2  # block (1, 2) of A: 13 x 8
    blk = A.values[off[b]:off[b + 1]].reshape(8, 13)
    offb = H.block_list_offsets(B)
    edit = {"tiny_block": lambda: blk.__imul__(1e-6),
            "tiny_row": lambda: blk[:, 3].__imul__(1e-9),
            "nan": lambda: blk.__setitem__((2, 3), np.nan),
            "inf": lambda: blk.__setitem__((2, 3), np.inf),
            "huge": lambda: A.values.__imul__(2.0 ** 400),
            "denormal": lambda: blk.__setitem__((slice(None), 3), 1e-310),
            "zero_row": lambda: blk.__setitem__((slice(None), 3), 0.0),
            "tall": lambda: None}[what]
    edit()
    got = multiply(gpu_ctx, A, B)
    fp64 = multiply(gpu_ctx, A, B, fp64_kernel=bsm_lib.BSM_FP64_PK12)
    assert np.array_equal(got[0], fp64[0]) and np.array_equal(got[1], fp64[1])
    offc = H.block_list_offsets(BlockMatrix(A.row_sizes, B.col_sizes, got[0], got[1], got[2]))
    with np.errstate(all="ignore"):
        ref = oracle_mod.multiply(A, B, eps=0.0)
    rows = {"huge": range(5), "tall": [4], "zero_row": [], "tiny_block": []}.get(what, [1])
    for x, (i, j) in enumerate(zip(got[0], got[1])):
        v, f, o = (a[offc[x]:offc[x + 1]] for a in (got[2], fp64[2], ref.values))
        # a value that is not finite leaves its row without a scale: all its blocks
        assert np.array_equal(v, f, equal_nan=True) == (i in rows), (what, i, j)
        assert np.array_equal(np.isnan(v), np.isnan(o)) and np.array_equal(np.isinf(v), np.isinf(o))
        fine = np.isfinite(o)
        assert H.rel_frobenius(v[fine] / max(1.0, np.abs(o[fine]).max(initial=1.0)),
                               o[fine] / max(1.0, np.abs(o[fine]).max(initial=1.0))) <= 1e-12
    assert len(offb) == len(ks) * len(cs) + 1


@pytest.mark.parametrize("columns", ["all", "one"])
def test_right_operand(gpu_ctx, bsm_lib, oracle_mod, columns):
    """The same for a block of B far below its columns' scales, and for one of its
    columns alone."""
    rng = np.random.default_rng(73)
    rs, ks, cs = [5, 9, 16], [5, 13, 8, 6, 5], [13, 5, 7]
    A, B = full(rng, rs, ks, rng.standard_normal), full(rng, ks, cs, rng.standard_normal)
    off = H.block_list_offsets(B)
    b = 2 * len(cs) + 1  # block (2, 1) of B
    B.values[off[b]:off[b + 1] if columns == "all" else off[b] + ks[2]] *= 1e-7
    got = multiply(gpu_ctx, A, B)
    fp64 = multiply(gpu_ctx, A, B, fp64_kernel=bsm_lib.BSM_FP64_PK12)
    offc = H.block_list_offsets(BlockMatrix(A.row_sizes, B.col_sizes, got[0], got[1], got[2]))
    ref = oracle_mod.multiply(A, B, eps=0.0)
    for x, j in enumerate(got[1]):
        v, f, o = (a[offc[x]:offc[x + 1]] for a in (got[2], fp64[2], ref.values))
        assert np.array_equal(v, f) == (columns == "one" and j == 1)
        assert H.rel_frobenius(v, o) <= 1e-12


def test_wide_range_between_blocks(gpu_ctx, bsm_lib):
    """Blocks of a row and of a column spread over 2^-200 .. 2^200: each C block
    to FP64's precision by itself, exact on integers times powers of two where
    one product decides."""
    rng = np.random.default_rng(75)
    rs, ks, cs = [5, 13, 8], [5, 13, 6, 9, 16, 3], [13, 5]
    ints = lambda n: rng.integers(1, 2 ** 20, n).astype(np.float64)  # noqa: E731
    A, B = full(rng, rs, ks, ints), full(rng, ks, cs, ints)
    offa, offb = H.block_list_offsets(A), H.block_list_offsets(B)
    shift = rng.integers(-200, 200, (len(rs), len(ks)))
    for b in range(len(rs) * len(ks)):
        A.values[offa[b]:offa[b + 1]] *= 2.0 ** int(shift[b // len(ks), b % len(ks)])
    r, c, v = multiply(gpu_ctx, A, B)
    # exact: integers on the common scale 2^-200
    a = H.to_dense(A, dtype=object)
    b = H.to_dense(B, dtype=object)
    a = np.vectorize(lambda x: int(x * 2.0 ** 200), otypes=[object])(a)
    b = np.vectorize(int, otypes=[object])(b)
    want = a @ b
    got = H.to_dense(BlockMatrix(A.row_sizes, B.col_sizes, r, c, v))
    for x, y in zip(got.ravel(), want.ravel()):
        # all terms are positive: one rounding for each of the classes and one for each
        # of their sums (at most 11 + 10 of 2^-53)
        assert abs(int(x * 2.0 ** 200) - y) * 2 ** 53 <= 24 * y


def test_without_memory_for_digits(gpu_ctx, bsm_lib):
    """Contexts side by side: the digit workspace belongs to the context and is
    sized for the operands of each multiply in turn."""
    rng = np.random.default_rng(74)
    with bsm_lib.Context(0) as ctx:
        seen = []
        for sizes in ([13, 5, 5] * 4, [32] * 12, [1] * 30, [13, 5, 5] * 4):
            A = full(np.random.default_rng(len(sizes)), sizes, sizes, rng.standard_normal)
            assert np.array_equal(multiply(ctx, A, A)[2], multiply(gpu_ctx, A, A)[2])
            seen.append(len(A.values))
        assert len(set(seen)) == 3
