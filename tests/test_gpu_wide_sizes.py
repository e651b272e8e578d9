"""Block sizes far beyond those of the blocks that are there: a matrix may have a block row
of 600000 scalars without a block in it. Tile counts are from the largest sizes."""
import numpy as np
import pytest

import synth
from synth import BlockMatrix
from tests import helpers as H

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("empty", [50_000, 600_000])
def test_an_empty_block_row_and_column_of_many_scalars(bsm_lib, empty):
    rng = np.random.default_rng(1)
    ks = [2, 13, 5, 8, 6]
    A = synth.random_blocks(rng, [13, 5], ks, 1.0)
    B = synth.random_blocks(rng, ks, [5, 13], 1.0)
    wide = np.int32(empty)
    rs, cs = np.append(A.row_sizes, wide), np.append(B.col_sizes, wide)
    with bsm_lib.Context(0) as ctx:
        dA = ctx.matrix(rs, A.col_sizes, A.blk_row, A.blk_col, A.values)
        dB = ctx.matrix(B.row_sizes, cs, B.blk_row, B.blk_col, B.values)
        dC = ctx.empty(rs, cs)
        for _ in range(2):
            st = ctx.multiply(1.0, dA, dB, 0.0, dC, 0.0, blocking=True, stats=True)
            assert st.kept >= 4 * st.c_blocks  # the default for many products a C block
            r, c = dC.pattern()
            got = H.to_dense(BlockMatrix(A.row_sizes, B.col_sizes, r, c, dC.values()))
            a, b = H.to_dense(A), H.to_dense(B)
            # FP64 FMAs and the digits: (N + 4) 2^-53 of the sum of absolute products, and
            # the reference's own N 2^-53
            assert (np.abs(got - a @ b) <= (2 * sum(ks) + 4) * 2.0 ** -53 * (np.abs(a) @ np.abs(b))).all()
