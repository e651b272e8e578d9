"""Matrices of few large and of many small blocks: norms by several lanes a block, C
blocks in parts, sums over short runs of blocks."""
import numpy as np
import pytest

import synth
from synth import BlockMatrix
from tests import helpers as H

pytestmark = pytest.mark.gpu


# number of blocks: 16 lanes a block, 4, one, more than one pass
@pytest.mark.parametrize("nblk,top", [(1, 40), (37, 70), (1300, 33), (4800, 20), (9800, 9), (90000, 4)])
def test_norms_are_the_canonical_ones(gpu_ctx, oracle_mod, nblk, top):
    """Every block has to pass a filter at its own canonical norm and none at the
    next larger number: the norms of the blocks sorted, the filter at some of
    them keeps exactly the blocks from there on."""
    rng = np.random.default_rng(nblk)
    n = max(1, int(np.sqrt(nblk)) + 1)
    rs, cs = rng.integers(1, top + 1, n), rng.integers(1, top + 1, n)
    rs[0] = cs[0] = top
    at = np.sort(np.concatenate([[0], 1 + rng.permutation(n * n - 1)[:nblk - 1]]))
    r, c = np.divmod(at, n)
    num = int((rs[r].astype(np.int64) * cs[c]).sum())
    M = BlockMatrix(rs.astype(np.int32), cs.astype(np.int32), r.astype(np.int32), c.astype(np.int32),
                    rng.standard_normal(num))
    norms = oracle_mod.norms(M)
    for eps in [np.sort(norms)[int(q * (nblk - 1))] for q in (0.0, 0.3, 0.7, 1.0)]:
        for e in (eps, np.nextafter(eps, np.inf)):
            D = gpu_ctx.from_blocks(M)
            D.filter(float(e))
            kr, kc = D.pattern()
            keep = ~(norms < e)
            assert np.array_equal(kr, M.blk_row[keep]) and np.array_equal(kc, M.blk_col[keep])
            D.destroy()


# one block; fewer than the warps of the launch; more than one block a warp and step
@pytest.mark.parametrize("n,top,density", [(1, 33, 1.0), (40, 33, 0.5), (170, 4, 0.9)])
def test_sum_of_matrices(gpu_ctx, n, top, density):
    rng = np.random.default_rng(n)
    rs, cs = rng.integers(1, top + 1, n), rng.integers(1, top + 1, n)
    A = synth.random_blocks(rng, rs, cs, density, kind="int", shuffle=True)
    B = synth.random_blocks(rng, rs, cs, density, kind="int", shuffle=True)
    dA, dB = gpu_ctx.from_blocks(A), gpu_ctx.from_blocks(B)
    gpu_ctx.add(-3.0, dA, 2.0, dB)
    r, c = dB.pattern()
    got = H.to_dense(BlockMatrix(A.row_sizes, A.col_sizes, r, c, dB.values()))
    assert np.array_equal(got, 2.0 * H.to_dense(B) - 3.0 * H.to_dense(A))
    for M in (dA, dB):
        M.destroy()


# C blocks of many tiles, few (parts of one tile each, and of several) to many (whole)
@pytest.mark.parametrize("launch", [0, 1])
@pytest.mark.parametrize("n,sizes", [(1, [70]), (3, [33, 100, 1]), (40, [17, 33, 5]), (150, [9, 17])])
def test_parts_of_blocks(gpu_ctx, n, sizes, launch):
    """Small integers, so exact; one block of A in ten has a row of its own scale
    that digits do not hold beside the others (its C blocks go to the packed
    kernel, in parts)."""
    rng = np.random.default_rng(n)
    rs, cs = rng.choice(sizes, n), rng.choice(sizes, n)
    ks = rng.choice(sizes + [3], 7)
    A = synth.random_blocks(rng, rs, ks, 0.8 if n > 1 else 1.0, kind="int")
    B = synth.random_blocks(rng, ks, cs, 0.8 if n > 1 else 1.0, kind="int")
    off = H.block_list_offsets(A)
    for b in range(0, len(A.blk_row), 10):
        blk = A.values[off[b]:off[b + 1]].reshape(-1, A.row_sizes[A.blk_row[b]])
        blk[:, 0] *= 2.0 ** -30
    dA, dB = gpu_ctx.from_blocks(A), gpu_ctx.from_blocks(B)
    dC = gpu_ctx.empty(A.row_sizes, B.col_sizes)
    gpu_ctx.multiply(1.0, dA, dB, 0.0, dC, 0.0, launch=launch, blocking=True)
    r, c = dC.pattern()
    got = H.to_dense(BlockMatrix(A.row_sizes, B.col_sizes, r, c, dC.values()))
    assert np.array_equal(got, H.to_dense(A) @ H.to_dense(B))
    for M in (dA, dB, dC):
        M.destroy()


# rows: one; the most that get the wide thread blocks, one more; past the fused scan
@pytest.mark.parametrize("eps", [0.0, 30.0])
@pytest.mark.parametrize("rows", [1, 455, 456, 457, 2048, 2049])
def test_rows_of_the_symbolic_phase(gpu_ctx, oracle_mod, rows, eps):
    rng = np.random.default_rng(rows)
    rs, ks, cs = rng.integers(1, 4, rows), rng.integers(1, 4, 70), rng.integers(1, 4, 40)
    A = synth.random_blocks(rng, rs, ks, 0.3, kind="int", shuffle=True)
    B = synth.random_blocks(rng, ks, cs, 0.3, kind="int", shuffle=True)
    ref = oracle_mod.multiply(A, B, eps=eps)
    dA, dB = gpu_ctx.from_blocks(A), gpu_ctx.from_blocks(B)
    dC = gpu_ctx.empty(A.row_sizes, B.col_sizes)
    st = gpu_ctx.multiply(1.0, dA, dB, 0.0, dC, eps, stats=True)
    r, c = dC.pattern()
    assert np.array_equal(r, ref.blk_row) and np.array_equal(c, ref.blk_col)
    assert st.kept == ref.kept and st.flops == ref.flops and np.array_equal(dC.values(), ref.values)
    for M in (dA, dB, dC):
        M.destroy()
