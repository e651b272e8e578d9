"""The per-block split kernel: tile shapes, ragged ends of k, more products than one
lookup holds, and the runs of C blocks that are stored together."""
import numpy as np
import pytest
import torch

import synth
from tests import helpers as H

pytestmark = pytest.mark.gpu


# rows x columns of C within 8 x 8, 16 x 8, 8 x 16, 16 x 16, and beyond (several tiles; of
# more values than a run gathers); k of one value to the largest, 60 products
@pytest.mark.parametrize("rows,cols", [((1, 7, 8), (3, 8)), ((9, 16), (1, 8)), ((2, 8), (9, 16)),
                                       ((13, 16), (15, 16)), ((17, 24, 32), (5, 23, 32))])
@pytest.mark.parametrize("ks", [(1,), (4, 5, 8), (9, 13, 16, 32)])
@pytest.mark.parametrize("prec,launch,with_c", [(1, 0, False), (1, 1, True), (2, 0, True), (2, 1, False)])
def test_tiles_and_runs(gpu_ctx, rows, cols, ks, prec, launch, with_c):
    """Small integers: every slice product and sum is exact, so are C and its copy in
    host memory."""
    rng = np.random.default_rng(sum(rows) + sum(ks))
    rs, kk, cs = rng.choice(rows, 13), rng.choice(ks, 60), rng.choice(cols, 11)
    A = synth.random_blocks(rng, rs, kk, 0.8, kind="int", shuffle=True)
    B = synth.random_blocks(rng, kk, cs, 0.8, kind="int", shuffle=True)
    C = synth.random_blocks(rng, rs, cs, 0.5, kind="int", shuffle=True) if with_c else None
    alpha, beta = (-2.0, 3.0) if with_c else (1.0, 0.0)
    host = torch.full((int(rs.sum()) * int(cs.sum()),), float("nan"), dtype=torch.float64,
                      pin_memory=True).numpy()
    dA, dB = gpu_ctx.from_blocks(A), gpu_ctx.from_blocks(B)
    dC = gpu_ctx.from_blocks(C) if with_c else gpu_ctx.empty(rs, cs)
    gpu_ctx.multiply(alpha, dA, dB, beta, dC, 0.0, precision=prec, launch=launch, host_out=host,
                     blocking=True)
    r, c = dC.pattern()
    got = dC.values()
    want = alpha * H.to_dense(A) @ H.to_dense(B) + (beta * H.to_dense(C) if with_c else 0.0)
    assert np.array_equal(H.to_dense(synth.BlockMatrix(rs, cs, r, c, got)), want)
    assert np.array_equal(host[:len(got)], got)
    for M in (dA, dB, dC):
        M.destroy()
