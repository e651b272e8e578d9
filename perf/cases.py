"""The multiplies that a program using this library asks for, as measurable cases.

A case is a kind of system, its size and what the program does with it. The
systems are those of the repository's benchmark and tests: liquid water (atoms
as 13 and 5 wide blocks), amorphous solids (5, 9, 13, 23, 32), fully occupied
matrices of 32 wide blocks, semi-empirical ones (6 wide, 0.05% occupied) and
rectangular ragged ones. The block pattern is the case's own, the values are made
on the GPU from the seed: new inputs are new values on the same system. A
multiply's operands are uploaded by ``prepare``, as a program keeps them between
multiplies, except where the case says that they come new with every pass.
"""
import math

import numpy as np
import torch

import paper_1705_10218_gb300 as bsm
from paper_1705_10218_gb300.sign import sign_iteration

DEV = "cuda" if torch.cuda.is_available() else "cpu"
AMORPHOUS = (5, 9, 13, 23, 32)
AMORPHOUS_P = (0.4, 0.2, 0.2, 0.1, 0.1)
RAGGED = (1, 2, 5, 6, 9, 13, 16, 17, 23, 32, 33)


def listed():
    return [
        # one multiply of the smallest system the request loop serves, its pattern and values read back
        {"name": "water32_call", "kind": "call", "system": "water", "n": 32, "eps": 1e-10},
        # the small water system replayed as a captured graph, values stored to page-locked memory
        {"name": "water64_graph", "kind": "graph", "system": "water", "n": 64, "eps": 1e-10},
        # rectangular operands of ragged blocks, C = beta C + alpha A B with an active filter
        {"name": "ragged_update", "kind": "update", "system": "ragged", "n": 150, "eps": 60.0},
        # a self-consistency step: a new matrix is uploaded, multiplied, and the result read
        {"name": "water512_step", "kind": "step", "system": "water", "n": 512, "eps": 1e-10},
        # the headline system, resident on the device
        {"name": "water2048_fp64", "kind": "multiply", "system": "water", "n": 2048, "eps": 1e-10},
        # the same with the filter dropping products
        {"name": "water1024_filtered", "kind": "multiply", "system": "water", "n": 1024, "eps": 0.3},
        # mixed block sizes up to 32
        {"name": "amorphous1024_fp64", "kind": "multiply", "system": "amorphous", "n": 1024, "eps": 1e-8},
        # every block present
        {"name": "dense64x32_fp64", "kind": "multiply", "system": "dense", "n": 64, "eps": 0.0},
        # very sparse, tiny blocks, about one product per result block
        {"name": "semiempirical20000", "kind": "multiply", "system": "sparse", "n": 20000, "eps": 1e-10},
        # split precision on the tensor cores, three bfloat16 terms
        {"name": "water1024_bf16x3", "kind": "bf16x3", "system": "water", "n": 1024, "eps": 1e-10},
        # independent requests of different sizes through the request loop
        {"name": "server_burst", "kind": "server", "system": "water", "n": 96, "eps": 1e-10},
        # the application itself: two sign iterations with the filter after each
        {"name": "sign_water128", "kind": "sign", "system": "water", "n": 128, "eps": 1e-7},
    ]


# per kind of case: the systems it is used on, the range of n, the range of eps
_RANGES = [
    ("call", "water", (16, 256), (1e-10, 1e-10)),
    ("graph", "water", (16, 256), (1e-10, 1e-10)),
    ("update", "ragged", (20, 200), (1e-10, 100.0)),
    ("step", "water", (64, 1024), (1e-10, 1e-10)),
    ("multiply", "water", (128, 2048), (1e-10, 1e-10)),
    ("multiply", "water", (128, 2048), (0.05, 0.5)),
    ("multiply", "amorphous", (128, 1024), (1e-8, 1e-8)),
    ("multiply", "dense", (8, 80), (0.0, 0.0)),
    ("multiply", "sparse", (2000, 40000), (1e-10, 1e-10)),
    ("bf16x3", "water", (64, 1536), (1e-10, 1e-10)),
    ("tf32x2", "amorphous", (128, 1024), (1e-8, 1e-8)),
    ("server", "water", (32, 256), (1e-10, 1e-10)),
    ("sign", "water", (32, 192), (1e-8, 1e-6)),
]


def draw(rng):
    kind, system, (lo, hi), (e0, e1) = rng.choice(_RANGES)
    n = int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))
    eps = e0 if e0 == e1 else math.exp(rng.uniform(math.log(e0), math.log(e1)))
    return {"kind": kind, "system": system, "n": n, "eps": eps}


# ---------------------------------------------------------------------------
# systems
# ---------------------------------------------------------------------------
class Blocks:
    """A block-sparse matrix: block sizes, sorted block list (rows, cols) and
    values, every block column-major (what Context.from_blocks takes)."""

    def __init__(self, row_sizes, col_sizes, rows, cols, values):
        self.row_sizes = np.asarray(row_sizes, np.int32)
        self.col_sizes = np.asarray(col_sizes, np.int32)
        self.blk_row = rows.to("cpu", torch.int32).numpy()
        self.blk_col = cols.to("cpu", torch.int32).numpy()
        self.values = values.cpu().numpy()


def _gen(seed, salt=0):
    g = torch.Generator(device=DEV)
    g.manual_seed(1000003 * int(seed) + salt)
    return g


def _rand(g, *shape):
    return torch.rand(*shape, generator=g, device=DEV, dtype=torch.float64)


def _pairs(pos, box, cutoff):
    """(i, j, r) with i <= j and minimum-image distance r below the cutoff."""
    n = len(pos)
    out = []
    step = max(1, (1 << 25) // max(n, 1))
    for a in range(0, n, step):
        d = pos[a:a + step, None, :] - pos[None, :, :]
        d -= box * torch.round(d / box)
        r = d.square().sum(-1).sqrt()
        i, j = torch.nonzero(r < cutoff, as_tuple=True)
        keep = i + a <= j
        out.append((i[keep] + a, j[keep], r[i[keep], j[keep]]))
    return tuple(torch.cat(x) for x in zip(*out))


def _geometry(case, which=0):
    """Block sizes of a square system and its upper block list (i, j, scale of
    the entries), with the shift of the diagonal blocks' diagonal."""
    g, n = _gen(which), case["n"]
    if case["system"] == "water":  # density: 64 molecules in a cube of side 12.4
        box = 12.4 * (n / 64.0) ** (1.0 / 3.0)
        o = _rand(g, n, 3) * box
        half = math.radians(104.5) / 2.0
        q = torch.randn(n, 4, generator=g, device=DEV, dtype=torch.float64)
        w, x, y, z = (q / q.norm(dim=1, keepdim=True)).unbind(1)
        c0 = torch.stack((1 - 2 * (y * y + z * z), 2 * (x * y + z * w), 2 * (x * z - y * w)), 1)
        c1 = torch.stack((2 * (x * y - z * w), 1 - 2 * (x * x + z * z), 2 * (y * z + x * w)), 1)
        h0, h1 = (o + 0.96 * (s * math.sin(half) * c0 + math.cos(half) * c1) for s in (1.0, -1.0))
        pos = torch.stack((o, h0, h1), 1).reshape(-1, 3) % box
        i, j, r = _pairs(pos, box, 6.0)
        return np.tile([13, 5, 5], n), i, j, torch.exp(-0.5 * r), 5.0
    if case["system"] == "amorphous":  # 0.1 atoms per cubic angstrom
        box = (n / 0.1) ** (1.0 / 3.0)
        pos = _rand(g, n, 3) * box
        p = torch.tensor(AMORPHOUS_P, device=DEV, dtype=torch.float64)
        kind = torch.multinomial(p, n, replacement=True, generator=g)
        i, j, r = _pairs(pos, box, 7.0)
        return np.asarray(AMORPHOUS)[kind.cpu().numpy()], i, j, torch.exp(-0.4 * r), 5.0
    if case["system"] == "dense":
        i, j = torch.triu_indices(n, n, device=DEV)
        scale = torch.full((len(i),), 1.0 / math.sqrt(32.0 * n), device=DEV, dtype=torch.float64)
        return np.full(n, 32), i, j, scale, 5.0 / math.sqrt(32.0 * n)
    pairs = int(round(5e-4 * n * (n - 1) / 2))  # sparse: 0.05% of the blocks, 6 wide
    i, j = (torch.randint(0, n, (2 * pairs + 16,), generator=g, device=DEV) for _ in range(2))
    key = torch.unique((i * n + j)[i < j])[:pairs]
    d = torch.arange(n, device=DEV)
    key = torch.sort(torch.cat((key, d * n + d))).values
    i, j = key // n, key % n
    return np.full(n, 6), i, j, torch.full((len(i),), 0.3, device=DEV, dtype=torch.float64), 5.0


def _offsets(sr, sc, rows, cols):
    off = torch.zeros(len(rows) + 1, dtype=torch.int64, device=DEV)
    off[1:] = torch.cumsum(sr[rows] * sc[cols], 0)
    return off


def _symmetric(case, seed):
    """The system's matrix: normal entries times the pair's scale, symmetric."""
    sizes, I, J, scale, shift = _geometry(case, case.get("which", 0))
    g = _gen(seed, 1)
    s = torch.as_tensor(np.asarray(sizes), device=DEV, dtype=torch.int64)
    n, off_diag = len(sizes), I != J
    up = torch.arange(len(I), device=DEV)
    rows, cols = torch.cat((I, J[off_diag])), torch.cat((J, I[off_diag]))
    src = torch.cat((up, -1 - up[off_diag]))  # the mirror of upper block b is -1 - b
    order = torch.argsort(rows * n + cols)
    rows, cols, src = rows[order], cols[order], src[order]
    off = _offsets(s, s, rows, cols)
    place, mirror = torch.empty_like(up), torch.full_like(up, -1)
    at = torch.arange(len(src), device=DEV)
    place[src[src >= 0]] = at[src >= 0]
    mirror[-1 - src[src < 0]] = at[src < 0]
    values = torch.empty(int(off[-1]), dtype=torch.float64, device=DEV)
    for a in np.unique(sizes):
        for b in np.unique(sizes):
            sel = torch.nonzero((s[I] == int(a)) & (s[J] == int(b))).flatten()
            if len(sel) == 0:
                continue
            x = torch.randn(len(sel), int(b), int(a), generator=g, device=DEV, dtype=torch.float64)
            x *= scale[sel][:, None, None]
            d = torch.nonzero(I[sel] == J[sel]).flatten()
            if len(d):
                y = x[d] / scale[sel[d]][:, None, None] * (1.0 if shift == 5.0 else shift / 5.0)
                y = torch.triu(y) + torch.triu(y, 1).transpose(1, 2)
                x[d] = y + shift * torch.eye(int(a), device=DEV, dtype=torch.float64)
            run = torch.arange(int(a) * int(b), device=DEV)
            values[off[place[sel]][:, None] + run] = x.reshape(len(sel), -1)
            m = torch.nonzero(mirror[sel] >= 0).flatten()
            if len(m):
                values[off[mirror[sel[m]]][:, None] + run] = x[m].transpose(1, 2).reshape(len(m), -1)
    return Blocks(sizes, sizes, rows, cols, values)


def _random(pattern, g, rs, cs, density):
    mask = _rand(pattern, len(rs), len(cs)) < density
    rows, cols = torch.nonzero(mask, as_tuple=True)
    r, c = (torch.as_tensor(x, device=DEV, dtype=torch.int64) for x in (rs, cs))
    nnz = int((r[rows] * c[cols]).sum())
    return Blocks(rs, cs, rows, cols, torch.randn(nnz, generator=g, device=DEV, dtype=torch.float64))


def _ragged(case, seed):
    p, g, n = _gen(0), _gen(seed, 1), case["n"]
    pick = torch.randint(0, len(RAGGED), (n + (9 * n) // 8 + (7 * n) // 8,), generator=p, device=DEV)
    s = np.asarray(RAGGED)[pick.cpu().numpy()]
    rs, ks, cs = s[:n], s[n:n + (9 * n) // 8], s[n + (9 * n) // 8:]
    return _random(p, g, rs, ks, 0.25), _random(p, g, ks, cs, 0.25), _random(p, g, rs, cs, 0.4)


def _server_systems(case, seed):
    """Eight systems whose sizes fall from n molecules to about an eighth of it."""
    n = case["n"]
    sizes = [n, max(4, n // 8), max(4, (3 * n) // 4), max(4, n // 5), max(4, n // 2), max(4, n // 7),
             max(4, n // 3), max(4, n // 6)]
    return [_symmetric(dict(case, n=m, which=k), 31 * int(seed) + k) for k, m in enumerate(sizes)]


def _sign_system(case, seed):
    """A gapped water matrix scaled into (-1, 1): 100 added to the diagonal of
    the 13 wide blocks, subtracted from that of the 5 wide ones."""
    m = _symmetric(case, seed)
    sr, sc = m.row_sizes[m.blk_row].astype(np.int64), m.col_sizes[m.blk_col].astype(np.int64)
    off = np.concatenate(([0], np.cumsum(sr * sc)))
    for w, shift in ((13, 100.0), (5, -100.0)):
        d = np.nonzero((m.blk_row == m.blk_col) & (sr == w))[0]
        m.values[(off[d][:, None] + np.arange(w) * (w + 1)).reshape(-1)] += shift
    v = np.abs(m.values)  # the largest column sum (= row sum: symmetric)
    col = np.repeat(np.concatenate(([0], np.cumsum(m.col_sizes)))[m.blk_col], sr * sc)
    within = np.arange(len(v)) - np.repeat(off[:-1], sr * sc)
    top = np.bincount(col + within // np.repeat(sr, sr * sc), weights=v).max()
    m.values /= top
    return m


def _result_nnz(A, B, C=None):
    """Values of the result's pattern when nothing is filtered (a bound otherwise)."""
    def mask(M):
        x = torch.zeros(len(M.row_sizes), len(M.col_sizes), device=DEV, dtype=torch.float32)
        x[torch.as_tensor(M.blk_row, device=DEV).long(), torch.as_tensor(M.blk_col, device=DEV).long()] = 1.0
        return x
    if len(A.row_sizes) > 12000:  # very sparse: by its candidate products
        count = np.bincount(A.blk_row, minlength=len(A.row_sizes))
        return int((A.row_sizes[A.blk_row].astype(np.int64) * count[A.blk_col]).sum()) * int(B.col_sizes.max())
    m = (mask(A) @ mask(B)) > 0
    if C is not None:
        m |= mask(C) > 0
    r = torch.as_tensor(A.row_sizes, device=DEV, dtype=torch.float64)
    c = torch.as_tensor(B.col_sizes, device=DEV, dtype=torch.float64)
    return int(r @ (m.double() @ c))


# ---------------------------------------------------------------------------
# what is run
# ---------------------------------------------------------------------------
class State:
    """A program's context, its matrices, and its page-locked result buffer."""

    def __init__(self, case):
        self.case, self.ctx, self.srv, self.hosts = case, None, None, []

    def __del__(self):
        for x in (self.ctx, self.srv):
            if x is not None:
                x.close()


def _host_out(s, nnz):
    t = torch.zeros(max(nnz, 1), dtype=torch.float64, pin_memory=True)
    s.hosts.append(t)
    return t.numpy()


def prepare(case, seed):
    s = State(case)
    kind = case["kind"]
    if kind == "server":
        s.systems = _server_systems(case, seed)
        s.srv = bsm.Server(0, slots=4, hbm_budget=48 << 30)
        return s
    s.ctx = bsm.Context(0)
    if kind == "update":
        A, B, C = _ragged(case, seed)
        s.A, s.B, s.C0 = (s.ctx.from_blocks(x) for x in (A, B, C))
        s.C = s.ctx.empty(A.row_sizes, B.col_sizes)
        s.out = _host_out(s, _result_nnz(A, B, C))
        return s
    M = _sign_system(case, seed) if kind == "sign" else _symmetric(case, seed)
    s.M, s.sizes = M, M.row_sizes
    s.A = s.ctx.from_blocks(M)
    if kind == "sign":
        s.out = _host_out(s, _result_nnz(M, M))
        return s
    s.C = s.ctx.empty(M.row_sizes, M.col_sizes)
    if kind != "call":
        s.out = _host_out(s, _result_nnz(M, M))
    if kind == "step":  # the values of the next step wait in page-locked memory
        v = _host_out(s, len(M.values))
        v[:] = M.values
        M.values = v
    return s


def run(s):
    case, ctx = s.case, s.ctx
    kind, eps = case["kind"], case["eps"]
    if kind == "server":
        ids = [s.srv.submit(M, eps) for M in s.systems]
        while any(s.srv.poll(i)[0] < 2 for i in ids):
            s.srv.progress()
        return [s.srv.take(i) for i in ids]
    if kind == "sign":
        X = sign_iteration(ctx, s.A, s.sizes, 2, eps=eps, filter_eps=100 * eps)
        X.values(out=s.out)
        X.destroy()
        return s.out
    if kind == "update":  # C starts from C0 in every pass
        ctx.add(1.0, s.C0, 0.0, s.C)
        ctx.multiply(-0.5, s.A, s.B, 2.0, s.C, eps, host_out=s.out)
    elif kind == "call":
        ctx.multiply(1.0, s.A, s.A, 0.0, s.C, eps)
        return s.C.pattern() + (s.C.values(),)
    else:
        if kind == "step":
            s.A.assign(s.M.blk_row, s.M.blk_col, s.M.values)
        precision = {"bf16x3": bsm.BSM_PREC_SPLIT_BF16X3, "tf32x2": bsm.BSM_PREC_SPLIT_TF32X2}.get(
            kind, bsm.BSM_PREC_FP64)
        ctx.multiply(1.0, s.A, s.A, 0.0, s.C, eps, precision=precision, graph=kind == "graph",
                     host_out=s.out)
    s.C.nblocks()  # waits for the result
    return s.out  # the result's values, then zeros where the filter left fewer than the buffer holds


# ---------------------------------------------------------------------------
# what a pass cannot do without
# ---------------------------------------------------------------------------
def _count(A, B, C=None):
    """(2mnk over all candidate products, values read, values written)."""
    left, right = (np.bincount(i, weights=s, minlength=len(k)) for i, s, k in (
        (A.blk_col, A.row_sizes[A.blk_row], A.col_sizes), (B.blk_row, B.col_sizes[B.blk_col], A.col_sizes)))
    flops = 2.0 * float((left * A.col_sizes * right).sum())
    read = len(A.values) + (0 if B is A else len(B.values)) + (0 if C is None else len(C.values))
    return flops, read, _result_nnz(A, B, C)


def work(case):
    if case["kind"] == "server":
        parts = [_count(M, M) for M in _server_systems(case, 0)]
    elif case["kind"] == "update":
        parts = [_count(*_ragged(case, 0))]
    else:
        M = _symmetric(case, 0)
        parts = [_count(M, M)]
        if case["kind"] == "sign":  # two multiplies an iteration; the iterate keeps about A's pattern
            parts = [(4 * parts[0][0], parts[0][1], parts[0][1])]
    flops, read, written = (sum(x) for x in zip(*parts))
    return {"bytes": 8.0 * (read + written), "flops": flops}


# ---------------------------------------------------------------------------
# the same in 64 bits by plain torch
# ---------------------------------------------------------------------------
class _T:
    def __init__(self, row_sizes, col_sizes, rows, cols, values):
        as_t = lambda x, dt: torch.as_tensor(x, device=DEV).to(dt)  # noqa: E731
        self.rs, self.cs = as_t(row_sizes, torch.int64), as_t(col_sizes, torch.int64)
        self.rows, self.cols = as_t(rows, torch.int64), as_t(cols, torch.int64)
        self.values = as_t(values, torch.float64)
        self.off = _offsets(self.rs, self.cs, self.rows, self.cols)

    @staticmethod
    def of(M):
        return _T(M.row_sizes, M.col_sizes, M.blk_row, M.blk_col, M.values)

    def norms(self):
        blk = torch.repeat_interleave(torch.arange(len(self.rows), device=DEV), self.off[1:] - self.off[:-1])
        return torch.zeros(len(self.rows), device=DEV, dtype=torch.float64).index_add_(
            0, blk, self.values.square()).sqrt()

    def keep(self, mask):
        el = torch.repeat_interleave(mask, self.off[1:] - self.off[:-1])
        return _T(self.rs, self.cs, self.rows[mask], self.cols[mask], self.values[el])


def _torch_multiply(alpha, A, B, beta, C, eps):
    """beta C + alpha A B over the products whose norms' product is at least eps."""
    count = torch.bincount(B.rows, minlength=len(B.rs))
    start = torch.cumsum(count, 0) - count
    per = count[A.cols]
    a = torch.repeat_interleave(torch.arange(len(A.rows), device=DEV), per)
    first = torch.cumsum(per, 0) - per
    b = start[A.cols[a]] + torch.arange(len(a), device=DEV) - first[a]
    kept = ~(A.norms()[a] * B.norms()[b] < eps)
    a, b = a[kept], b[kept]
    nbc = len(B.cs)
    key = A.rows[a] * nbc + B.cols[b]
    every = key if C is None else torch.cat((key, C.rows * nbc + C.cols))
    blocks, slot = torch.unique(every, return_inverse=True)
    out = _T(A.rs, B.cs, blocks // nbc, blocks % nbc, torch.zeros(0, device=DEV))
    out.values = torch.zeros(int(out.off[-1]), device=DEV, dtype=torch.float64)
    kinds = A.rs[A.rows[a]] * 65536 * 256 + A.cs[A.cols[a]] * 4096 + B.cs[B.cols[b]]
    for kind in torch.unique(kinds).tolist():
        m, k, n = kind // (65536 * 256), kind % (65536 * 256) // 4096, kind % 4096
        sel = torch.nonzero(kinds == kind).flatten()
        mk, kn, mn = (torch.arange(x, device=DEV) for x in (m * k, k * n, m * n))
        for at in range(0, len(sel), 1 << 20):
            p = sel[at:at + (1 << 20)]
            x = A.values[A.off[a[p]][:, None] + mk].reshape(-1, k, m)  # column-major blocks
            y = B.values[B.off[b[p]][:, None] + kn].reshape(-1, n, k)
            u, where = torch.unique(slot[p], return_inverse=True)
            z = torch.zeros(len(u), n * m, device=DEV, dtype=torch.float64)
            z.index_add_(0, where, torch.bmm(y, x).reshape(-1, n * m))
            out.values[out.off[u][:, None] + mn] += z
    out.values *= alpha
    if C is not None:
        blk = slot[len(key):]
        length = C.off[1:] - C.off[:-1]
        within = torch.arange(len(C.values), device=DEV) - torch.repeat_interleave(C.off[:-1], length)
        out.values[torch.repeat_interleave(out.off[blk], length) + within] += beta * C.values
    return out


def _padded(values, n):
    out = np.zeros(max(n, 1))
    out[:len(values)] = values.cpu().numpy()
    return out


def exact(case, seed):
    kind, eps = case["kind"], case["eps"]
    if kind == "server":
        got = [_T.of(M) for M in _server_systems(case, seed)]
        got = [_torch_multiply(1.0, M, M, 0.0, None, eps) for M in got]
        return [(None, None, M.values.cpu().numpy()) for M in got]
    if kind == "update":
        host = _ragged(case, seed)
        A, B, C = (_T.of(M) for M in host)
        return _padded(_torch_multiply(-0.5, A, B, 2.0, C, eps).values, _result_nnz(*host))
    if kind == "sign":
        host = _sign_system(case, seed)
        X = _T.of(host)
        n = torch.arange(len(X.rs), device=DEV)
        for _ in range(2):
            eye = torch.cat([3.0 * torch.eye(int(w), device=DEV, dtype=torch.float64).reshape(-1) for w in X.rs])
            T = _torch_multiply(-1.0, X, X, 1.0, _T(X.rs, X.cs, n, n, eye), eps)
            X = _torch_multiply(0.5, X, T, 0.0, None, eps)
            X = X.keep(X.norms() >= 100 * eps)
        return _padded(X.values, _result_nnz(host, host))
    host = _symmetric(case, seed)
    M = _T.of(host)
    values = _torch_multiply(1.0, M, M, 0.0, None, eps).values
    return (None, None, values.cpu().numpy()) if kind == "call" else _padded(values, _result_nnz(host, host))
