"""The digit workspace of the FP64 default when device memory is short (the cap
BSM_DEVICE_MEMORY_CAP, read once per process: child processes): a multiply that cannot
have it takes the packed kernel, and one that can again is right."""
import json
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

COMMON = r"""
import json, numpy as np, synth
from paper_1705_10218_gb300 import Context, BsmError, BSM_FP64_PK12
from tests import helpers as H
rng = np.random.default_rng(3)

def banded(n, width, size=1):
    i = np.repeat(np.arange(n), width)
    j = i + np.tile(np.arange(width) - width // 2, n)
    keep = (j >= 0) & (j < n)
    s = np.full(n, size, np.int32)
    return synth.BlockMatrix(s, s, i[keep].astype(np.int32), j[keep].astype(np.int32),
                             rng.standard_normal(int(keep.sum()) * size * size))

def ballast(ctx, bytes):
    # matrices of `bytes` (and a little) until the device is full
    side = int((bytes / 8) ** 0.5)
    one = np.array([side], np.int32)
    v = rng.standard_normal(side * side)
    out = []
    while True:
        try:
            out.append(ctx.matrix(one, one, np.zeros(1, np.int32), np.zeros(1, np.int32), v))
        except BsmError as e:
            assert e.name == "NOMEM", e.name
            return out

def multiply(ctx, A, C, kern=None):
    ctx.multiply(1.0, A, A, 0.0, C, 0.0, blocking=True, fp64_kernel=kern)
    return C.values()
"""


def child(code, cap, **more):
    env = dict(os.environ, BSM_DEVICE_MEMORY_CAP=str(cap), **more)
    p = subprocess.run([sys.executable, "-c", COMMON + code], cwd=ROOT, env=env, capture_output=True,
                       text=True, timeout=600)
    assert p.returncode == 0, p.stderr[-2000:]
    return json.loads(p.stdout.strip().splitlines()[-1])


# With a little more memory each time: none of the workspace, its first buffer, the
# next, ... all of it.
STEPS = r"""
A = banded(8000, 9)  # 1 x 1 blocks, up to nine octets of one value each for a C block
D = banded(8000, 1)
with Context(0) as ctx:
    dA, dC = ctx.from_blocks(A), ctx.empty(A.row_sizes, A.col_sizes)
    want = [multiply(ctx, dA, dC, BSM_FP64_PK12) for _ in range(2)][1]  # both of C's buffers
    dD, dE = ctx.from_blocks(D), ctx.empty(A.row_sizes, A.col_sizes)
    multiply(ctx, dD, dE)  # few products: the scales alone
    off, same = [], []
    for m in ballast(ctx, 256 << 10):
        v = multiply(ctx, dA, dC)
        same.append(bool(np.array_equal(v, want)))
        off.append(H.rel_frobenius(v, want))
        m.destroy()
print(json.dumps(dict(same=same, off=off)))
"""


def test_each_buffer_of_the_workspace_refused_in_turn(bsm_lib):
    out = child(STEPS, 48 << 20)
    # without all of it the packed kernel, bit for bit; in the end the digits
    assert out["same"][0] and not out["same"][-1]
    assert max(out["off"]) <= 1e-15


# What a second context can have before and after the first one has taken digits.
TWO = r"""
A = banded(8000, 9)
with Context(0) as one, Context(0) as two:
    dA, dC = one.from_blocks(A), one.empty(A.row_sizes, A.col_sizes)
    want = [multiply(one, dA, dC, BSM_FP64_PK12) for _ in range(2)][1]  # both of C's buffers
    room, off = [], []
    for _ in range(2):
        held = ballast(two, 256 << 10)
        for m in held:
            m.destroy()
        room.append(len(held))
        off.append(H.rel_frobenius(multiply(one, dA, dC), want))
print(json.dumps(dict(room=room, off=off)))
"""


def test_another_context_gets_the_memory_of_the_digits(bsm_lib):
    out = child(TWO, 48 << 20)
    # all of it: the workspace is twice 64 bytes a value, 20 pieces of 256 KiB each
    assert out["room"][1] >= out["room"][0] - 1
    assert max(out["off"]) <= 1e-15


# Two threads, each with a context of its own, at the cap: one takes the other's digits
# back whenever its matrices need the room.
THREADS = r"""
import threading
bad = []

def work(seed):
    rng = np.random.default_rng(seed)
    with Context(0) as ctx:
        for n in [2000, 4000, 3000, 6000, 1000, 5000] * 6:
            A = banded(n, 9)
            A.values[:] = rng.standard_normal(len(A.values))
            try:
                dA, dC = ctx.from_blocks(A), ctx.empty(A.row_sizes, A.col_sizes)
                want = multiply(ctx, dA, dC, BSM_FP64_PK12)
                for _ in range(3):
                    off = H.rel_frobenius(multiply(ctx, dA, dC), want)
                    if not off <= 1e-15:
                        bad.append((seed, n, off))
            except BsmError as e:
                if e.name != "NOMEM":
                    bad.append((seed, n, e.name))
            dA.destroy()
            dC.destroy()

threads = [threading.Thread(target=work, args=(s,)) for s in (1, 2)]
for t in threads:
    t.start()
for t in threads:
    t.join()
print(json.dumps(bad))
"""


@pytest.mark.parametrize("cap", [28, 36, 48])
def test_threads_take_digits_from_each_other(bsm_lib, cap):
    assert child(THREADS, cap << 20) == []


# A tuned choice of the digit kernel (value 6 of the cache file), without and with the memory.
TUNED = r"""
A = banded(8000, 9)
with Context(0) as ctx:
    dA, dC = ctx.from_blocks(A), ctx.empty(A.row_sizes, A.col_sizes)
    want = [multiply(ctx, dA, dC, BSM_FP64_PK12) for _ in range(2)][1]  # both of C's buffers
    held = ballast(ctx, 256 << 10)
    without = multiply(ctx, dA, dC)
    for m in held:
        m.destroy()
    full = multiply(ctx, dA, dC)
print(json.dumps(dict(without=bool(np.array_equal(without, want)), full=bool(np.array_equal(full, want)),
                      off=H.rel_frobenius(full, want))))
"""


def test_a_tuned_digit_kernel_without_memory_is_the_packed_one(bsm_lib, tmp_path):
    cache = tmp_path / "tuned"
    cache.write_text("fp64/all/1,|1,|1, 6 0.0\n")
    out = child(TUNED, 48 << 20, BSM_AUTOTUNE_CACHE=str(cache))
    assert out["without"] and not out["full"] and out["off"] <= 1e-15
