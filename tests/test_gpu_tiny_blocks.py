"""The kernel for tiny C blocks with few products: its runs of blocks and their stores."""
import numpy as np
import pytest
import torch

import synth
from tests import helpers as H

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("launch", [0, 1])
@pytest.mark.parametrize("alpha,with_c", [(1.0, False), (-3.0, False), (2.0, True)])
@pytest.mark.parametrize("top", [2, 4, 5, 6, 7, 8, 11])
def test_g8_runs_and_host_copy(gpu_ctx, bsm_lib, top, alpha, with_c, launch):
    """g8 with the host copy: C blocks gathered over runs (blocks of a run that lie
    apart, as in the per-stack lists; blocks without products; more products than a
    run lists; a run with blocks past the kernel's tile, top 11; partly filled last
    runs). Integer inputs: the values are exact, and the host
    copy equals them."""
    rng = np.random.default_rng(50 + top)
    sizes = np.arange(1, top + 1)
    rs, ks, cs = rng.choice(sizes, 61), rng.choice(sizes, 70), rng.choice(sizes, 47)
    A = synth.random_blocks(rng, rs, ks, 0.25, kind="int", shuffle=True)
    B = synth.random_blocks(rng, ks, cs, 0.2, kind="int", shuffle=True)
    C = synth.random_blocks(rng, rs, cs, 0.3, kind="int", shuffle=True) if with_c else None
    beta = -1.0 if with_c else 0.0
    host = torch.full((int(rs.sum()) * int(cs.sum()),), float("nan"), dtype=torch.float64,
                      pin_memory=True).numpy()
    dA, dB = gpu_ctx.from_blocks(A), gpu_ctx.from_blocks(B)
    dC = gpu_ctx.from_blocks(C) if with_c else gpu_ctx.empty(rs, cs)
    gpu_ctx.multiply(alpha, dA, dB, beta, dC, 0.0, launch=launch, host_out=host, blocking=True,
                     fp64_kernel=bsm_lib.BSM_FP64_G8)
    r, c = dC.pattern()
    got = dC.values()
    want = alpha * H.to_dense(A) @ H.to_dense(B) + (beta * H.to_dense(C) if with_c else 0.0)
    assert np.array_equal(H.to_dense(synth.BlockMatrix(rs, cs, r, c, got)), want)
    assert np.array_equal(host[:len(got)], got)
    for M in (dA, dB, dC):
        M.destroy()


@pytest.mark.parametrize("alpha", [-1.0, 2.0 ** -520, -2.0 ** 40, 1.7, -0.0])
def test_g8_alpha(gpu_ctx, bsm_lib, alpha):
    """alpha at the stores (with results that are denormal, zeros, infinities and values
    that are not numbers): the bits are those of a multiplication of the sums."""
    rng = np.random.default_rng(9)
    rs = rng.choice([1, 3, 5], 30)
    A = synth.random_blocks(rng, rs, rs, 0.4, kind="normal")
    off = H.block_list_offsets(A)
    for b in range(0, len(A.blk_row), 5):
        A.values[off[b]:off[b + 1]] *= 2.0 ** -260
    A.values[off[7]] = np.inf
    A.values[off[9]] = np.nan
    A.values[off[11]:off[12]] = 0.0
    out = []
    dA = gpu_ctx.from_blocks(A)
    for a in (1.0, alpha):
        dC = gpu_ctx.empty(A.row_sizes, A.col_sizes)
        gpu_ctx.multiply(a, dA, dA, 0.0, dC, 0.0, fp64_kernel=bsm_lib.BSM_FP64_G8, blocking=True)
        out.append(dC.values())
        dC.destroy()
    dA.destroy()
    with np.errstate(all="ignore"):
        want = out[0] * alpha
    assert np.array_equal(out[1], want, equal_nan=True)
    assert np.array_equal(np.signbit(out[1])[~np.isnan(want)], np.signbit(want)[~np.isnan(want)])
