"""With a second destination in host memory the C blocks of the kernels for tiny blocks and
of the split precisions leave in runs, without one block by block or tile by tile. Both
give the same bits."""
import numpy as np
import pytest
import torch

import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("alpha,beta", [(1.0, 0.0), (-0.7, 0.0), (1.0, 1.0), (0.3, -2.0)])
@pytest.mark.parametrize("top", [1, 4, 5, 6, 8, 13])
def test_with_and_without_a_host_copy(gpu_ctx, bsm_lib, top, alpha, beta):
    rng = np.random.default_rng(top)
    rs, ks, cs = (rng.choice(np.arange(1, top + 1), n) for n in (150, 160, 140))
    A = synth.random_blocks(rng, rs, ks, 0.1, shuffle=True)
    B = synth.random_blocks(rng, ks, cs, 0.1, shuffle=True)
    C = synth.random_blocks(rng, rs, cs, 0.2, shuffle=True)
    host = torch.full((int(rs.sum()) * int(cs.sum()),), float("nan"), dtype=torch.float64,
                      pin_memory=True).numpy()
    dA, dB = gpu_ctx.from_blocks(A), gpu_ctx.from_blocks(B)
    out = []
    for h in (host, None):
        dC = gpu_ctx.from_blocks(C)
        gpu_ctx.multiply(alpha, dA, dB, beta, dC, 0.0, host_out=h, blocking=True,
                         fp64_kernel=bsm_lib.BSM_FP64_G8)
        out.append(dC.values())
        dC.destroy()
    assert np.array_equal(out[0], out[1])
    assert np.array_equal(host[:len(out[0])], out[0])
    for M in (dA, dB):
        M.destroy()


@pytest.mark.parametrize("alpha,beta", [(1.0, 0.0), (-0.7, 0.0), (1.0, 1.0), (0.3, -2.0)])
@pytest.mark.parametrize("sizes", [[1, 2, 5], [6, 8, 9], [13, 16], [17, 23, 32], [1, 8, 9, 16, 17, 32]])
@pytest.mark.parametrize("n", [20, 180])  # few C blocks, shared out by their tiles, and many
@pytest.mark.parametrize("precision", [1, 2])
def test_split_with_and_without_a_host_copy(gpu_ctx, precision, n, sizes, alpha, beta):
    rng = np.random.default_rng(sizes[0] + n)
    rs, ks, cs = (rng.choice(sizes, k) for k in (n, n + 5, n - 3))
    A = synth.random_blocks(rng, rs, ks, 0.1, shuffle=True)
    B = synth.random_blocks(rng, ks, cs, 0.1, shuffle=True)
    C = synth.random_blocks(rng, rs, cs, 0.2, shuffle=True)
    host = torch.full((int(rs.sum()) * int(cs.sum()),), float("nan"), dtype=torch.float64,
                      pin_memory=True).numpy()
    dA, dB = gpu_ctx.from_blocks(A), gpu_ctx.from_blocks(B)
    out = []
    for h in (host, None):
        dC = gpu_ctx.from_blocks(C)
        gpu_ctx.multiply(alpha, dA, dB, beta, dC, 0.0, host_out=h, blocking=True, precision=precision)
        out.append(dC.values())
        dC.destroy()
    assert np.array_equal(out[0], out[1])
    assert np.array_equal(host[:len(out[0])], out[0])
    for M in (dA, dB):
        M.destroy()
