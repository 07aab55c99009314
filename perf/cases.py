"""Timed cases of the ChFSI library: the calls that a user of the package makes.

A case is one call of a public entry point (the filter in each of its arithmetics and
layouts, its reverse mode, the spectral bounds, the Rayleigh-Ritz closure, whole solve
cycles) on operators of the kinds the repository works with: Kronecker-banded grid
operators on g^3 points (half width w, 0.3 potential amplitude, 5% core rows), their
64 x 64 blocked copy, and banded operators in the split storage.  Inputs are drawn on
the GPU from the seed alone; exact() restates each result in 64 bits with torch.
"""
import math

import torch

import paper_2110_15853_gb300 as P

DEV = "cuda"


def listed():
    return [
        # a tiny system (a few atoms): ten launches of well under a thousandth of a second each
        dict(name="filter_f64_tiny", op="filter", layout="csr", g=12, w=2, n=24, m=10, sched="f64*10"),
        # the default call: every step in FP64 on a CSR operator, a mid-size system
        dict(name="filter_f64", op="filter", layout="csr", g=32, w=2, n=512, m=16, sched="f64*16"),
        # two-float steps on a grid that has no blocks (odd edge) and an odd number of states
        dict(name="filter_f32x2_odd", op="filter", layout="csr", g=27, w=3, n=301, m=12, sched="f32x2*12"),
        # the FP64-accurate production filter of a mid-scale system: blocks on the tensor cores
        dict(name="filter_ozaki", op="filter", layout="bsr", g=40, w=3, n=1024, m=20, sched="ozaki*20"),
        # the mixed production schedule on a large system: 40-bit steps closed by FP64-accurate
        # ones, wide stencil, a state count that is no multiple of a tile
        dict(name="filter_ozaki40_large", op="filter", layout="bsr", g=48, w=4, n=1500, m=24,
             sched="ozaki40*20+ozaki*4"),
        # first SCF cycles: BF16 tensor-core steps, then FP64-accurate ones, ragged state count
        dict(name="filter_bf16_ozaki", op="filter", layout="bsr", g=40, w=3, n=700, m=20,
             sched="bf16*16+ozaki*4"),
        # an operator that is dense near the diagonal, in the split storage (ragged last block)
        dict(name="filter_split", op="filter", layout="split", N=20000, band=256, block=1024, n=200, m=10,
             sched="f64*10"),
        # gradient of a loss through the filter, in two-float arithmetic: dX and dH
        dict(name="backward_f32x2", op="backward", layout="csr", g=32, w=2, n=512, m=16, precision="f32x2"),
        # spectral bounds before the first cycle
        dict(name="lanczos", op="lanczos", layout="csr", g=40, w=3, n=1024, steps=20),
        # the default closure (FP64) of a small system
        dict(name="closure_f64_small", op="closure", layout="csr", g=20, w=2, n=96, precision="f64", passes=2),
        # the production closure of a system with thousands of states
        dict(name="closure_ozaki_large", op="closure", layout="bsr", g=40, w=3, n=2400, precision="ozaki", passes=2),
        # whole call: bounds, filter and closure, two cycles, every product on the tensor cores
        dict(name="solve_ozaki", op="solve", layout="hybrid", g=32, w=3, n=640, m=12, cycles=2, sched="ozaki*12",
             precision="ozaki"),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more case: the same entry points, layouts and arithmetics at other sizes."""
    op = rng.choice(["filter"] * 6 + ["backward", "lanczos", "closure", "closure", "solve"])
    w = rng.choice([2, 3, 4])
    if op == "filter":
        layout = rng.choice(["csr", "bsr", "bsr", "split"])
        m = rng.randint(8, 24)
        if layout == "split":
            m = rng.randint(4, 10)
            block = rng.choice([512, 1024, 2048])
            return dict(op=op, layout=layout, N=_log(rng, 4000, 20000), band=block // 4, block=block,
                        n=_log(rng, 24, 200), m=m, sched="f64*%d" % m)
        if layout == "csr":
            kind = rng.choice(["f64", "f32x2", "f32"])
            sched = "%s*%d" % (kind, m) if kind != "f32" else "f32*%d+f64*4" % (m - 4)
            return dict(op=op, layout=layout, g=rng.randint(12, 30), w=w, n=_log(rng, 16, 400), m=m, sched=sched)
        kind = rng.choice(["ozaki", "ozaki40", "bf16"])
        sched = "ozaki*%d" % m if kind == "ozaki" else "%s*%d+ozaki*4" % (kind, m - 4)
        return dict(op=op, layout=layout, g=4 * rng.randint(4, 10), w=w, n=_log(rng, 48, 1400), m=m, sched=sched)
    if op == "backward":
        return dict(op=op, layout="csr", g=rng.randint(12, 28), w=2, n=_log(rng, 16, 400), m=rng.randint(4, 16),
                    precision=rng.choice(["f64", "f32x2"]))
    if op == "lanczos":
        return dict(op=op, layout="csr", g=rng.randint(12, 40), w=rng.choice([2, 3]), n=_log(rng, 16, 1024),
                    steps=rng.randint(10, 20))
    if op == "closure":
        precision = rng.choice(["f64", "f32x2", "ozaki", "ozaki"])
        layout = rng.choice(["csr", "bsr"]) if precision == "ozaki" else "csr"
        top = 2000 if layout == "bsr" else 400
        return dict(op=op, layout=layout, g=4 * rng.randint(4, 9), w=rng.choice([2, 3]), n=_log(rng, 32, top),
                    precision=precision, passes=rng.choice([1, 2]))
    m = rng.randint(8, 16)
    return dict(op=op, layout="hybrid", g=4 * rng.randint(4, 8), w=rng.choice([2, 3]), n=_log(rng, 32, 640), m=m,
                cycles=rng.randint(1, 3), sched="ozaki*%d" % m, precision="ozaki")


# ------------------------------------------------------------------ inputs


def _gen(seed, stream):
    return torch.Generator(device=DEV).manual_seed(seed * 16 + stream)


def _kinetic(d):
    return 2.5 if d == 0 else -1.0 / (1.0 + abs(d)) ** 2


def _grid_entries(g, w, seed):
    """(counts per row, columns, values) of the grid operator, columns ascending per row."""
    N = g ** 3
    r = range(-w, w + 1)
    offs = [(d1, d2, d3) for d1 in r for d2 in r for d3 in r]
    idx = torch.arange(N, device=DEV)
    axes = (idx // (g * g), (idx // g) % g, idx % g)
    inside = [{d: (x + d >= 0) & (x + d < g) for d in r} for x in axes]
    gen = _gen(seed, 0)
    K, centre = len(offs), len(offs) // 2
    vals = torch.empty((K, N), dtype=torch.float64, device=DEV)
    mask = torch.empty((K, N), dtype=torch.bool, device=DEV)
    for k in range(centre, K):
        d1, d2, d3 = offs[k]
        lin = (d1 * g + d2) * g + d3
        kin = 3 * _kinetic(0) if lin == 0 else (_kinetic(d1 + d2 + d3) if (d1 != 0) + (d2 != 0) + (d3 != 0) == 1 else 0.0)
        z = torch.randn(N, dtype=torch.float64, device=DEV, generator=gen)
        z.mul_(0.3 * math.exp(-(d1 * d1 + d2 * d2 + d3 * d3))).add_(kin)
        if lin == 0:
            core = torch.rand(N, device=DEV, generator=gen)
            z += torch.where(core < 0.025, -2.0, 0.0) + torch.where(core > 0.975, 2.0, 0.0)
        vals[k] = z
        mask[k] = inside[0][d1] & inside[1][d2] & inside[2][d3]
        if lin:   # the mirrored entries
            vals[K - 1 - k] = torch.roll(z, lin)
            mask[K - 1 - k] = inside[0][-d1] & inside[1][-d2] & inside[2][-d3]
    lin = torch.tensor([(d1 * g + d2) * g + d3 for d1, d2, d3 in offs], device=DEV, dtype=torch.int32)
    counts = mask.sum(0)
    mask = mask.t().contiguous()
    col = (idx.to(torch.int32)[:, None] + lin[None, :])[mask]
    return counts, col, vals.t().contiguous()[mask]


def _band_entries(N, band, seed):
    """An operator that decays away from the diagonal, with a few far couplings per row."""
    gen = _gen(seed, 1)
    d = torch.arange(0, band + 1, device=DEV)
    z = torch.randn((N, band + 1), dtype=torch.float64, device=DEV, generator=gen)
    z = torch.where(d == 0, 2.5 + 0.1 * z, torch.exp(-d / (band / 4.0)) * (-0.5 + 0.1 * z) * (16.0 / band))
    i = torch.arange(N, device=DEV)
    rows = i[:, None].expand(-1, band + 1)
    cols = rows + d
    keep = cols < N
    rows, cols, v = rows[keep], cols[keep], z[keep]
    off = rows != cols
    fi = torch.randint(0, N, (4 * N,), device=DEV, generator=gen)
    fj = torch.randint(0, N, (4 * N,), device=DEV, generator=gen)
    far = fi + band < fj
    key = torch.unique(fi[far] * N + fj[far])
    fv = 0.01 * torch.randn(key.numel(), dtype=torch.float64, device=DEV, generator=gen)
    fi, fj = key // N, key % N
    rows, cols, v = (torch.cat(t) for t in ((rows, cols[off], fi, fj), (cols, rows[off], fj, fi), (v, v[off], fv, fv)))
    order = torch.argsort(rows * N + cols)
    return torch.bincount(rows, minlength=N), cols[order].to(torch.int32), v[order]


def _row_ptr(counts):
    rp = torch.zeros(counts.numel() + 1, dtype=torch.int64, device=DEV)
    rp[1:] = torch.cumsum(counts, 0)
    return rp


def _blocked(g, counts, col, val, want_csr):
    """The operator in the order of 4 x 4 x 4 sub-cubes: (CsrMatrix or None, BsrMatrix)."""
    N, G = g ** 3, g // 4
    i = torch.arange(N, device=DEV)
    i1, i2, i3 = i // (g * g), (i // g) % g, i % g
    new = (((i1 // 4) * G + i2 // 4) * G + i3 // 4) * 64 + ((i1 % 4) * 4 + i2 % 4) * 4 + i3 % 4
    r, c = torch.repeat_interleave(new, counts), new[col.long()]
    nbr = N // 64
    blocks, where = torch.unique((r // 64) * nbr + c // 64, return_inverse=True)
    bval = torch.zeros(blocks.numel() * 4096, dtype=torch.float64, device=DEV)
    bval[where * 4096 + (r % 64) * 64 + c % 64] = val
    bptr = _row_ptr(torch.bincount(blocks // nbr, minlength=nbr)).to(torch.int32)
    bsr = P.BsrMatrix(bptr, (blocks % nbr).to(torch.int32), bval, nbr)
    if not want_csr:
        return None, bsr
    order = torch.argsort(r * N + c)
    return P.CsrMatrix(_row_ptr(torch.bincount(r, minlength=N)), c[order].to(torch.int32), val[order], N), bsr


def _operator(case, seed, plain=False):
    """The operator in the layout of the case; plain: as a CsrMatrix in the same row order."""
    if case["layout"] == "split":
        N, B = case["N"], case["block"]
        counts, col, val = _band_entries(N, case["band"], seed)
        if plain:
            return P.CsrMatrix(_row_ptr(counts), col, val, N)
        rows = torch.repeat_interleave(torch.arange(N, device=DEV), counts)
        dense = rows // B == col // B
        diag = torch.zeros((N + B - 1) // B * B * B, dtype=torch.float64, device=DEV)
        r, c = rows[dense], col[dense].long()
        diag[(r // B) * B * B + (r % B) * B + c % B] = val[dense]
        ptr = _row_ptr(torch.bincount(rows[~dense], minlength=N))
        return P.SplitMatrix(diag, P.CsrMatrix(ptr, col[~dense], val[~dense], N), B, N)
    counts, col, val = _grid_entries(case["g"], case["w"], seed)
    if case["layout"] == "csr":
        return P.CsrMatrix(_row_ptr(counts), col, val, counts.numel())
    csr, bsr = _blocked(case["g"], counts, col, val, plain or case["layout"] == "hybrid")
    return csr if plain else (bsr if case["layout"] == "bsr" else P.HybridMatrix(csr, bsr))


def _block(N, n, seed, stream):
    x = torch.randn((N, n), dtype=torch.float64, device=DEV, generator=_gen(seed, stream))
    return x.div_(math.sqrt(N))


def _schedule(case):
    return [p for part in case["sched"].split("+") for p in [part.split("*")[0]] * int(part.split("*")[1])]


def _rows(case):
    return case["N"] if case["layout"] == "split" else case["g"] ** 3


# Bounds (a, b, a0) that hold for every seed: the kinetic part's spectrum, widened by the
# potential and the core shifts; a keeps about the wanted share of it (Weyl).
def _bounds(case):
    b, a0 = (4.0, -2.0) if case["layout"] == "split" else (13.5, 1.0)
    return a0 + (b - a0) * max(0.2, min(0.6, (case["n"] / _rows(case)) ** (2.0 / 3.0))), b, a0


def prepare(case, seed):
    op, N, n = case["op"], _rows(case), case["n"]
    H = _operator(case, seed)
    state = dict(case=case, H=H, ws=P.Workspace(DEV))
    if op == "lanczos":
        state["v0"] = torch.randn(N, dtype=torch.float64, device=DEV, generator=_gen(seed, 4))
        return state
    state["X"] = X = _block(N, n, seed, 2)
    if op == "filter":
        state.update(bounds=_bounds(case), out=torch.empty_like(X),
                     schedule=None if set(_schedule(case)) == {"f64"} else _schedule(case))
    elif op == "backward":
        state.update(bounds=_bounds(case), dY=_block(N, n, seed, 3))
    elif op == "closure":   # a filtered block, as the closure gets it
        state["X"] = _plain_filter(_sparse(_operator(case, seed, plain=True)), X, 6, *_bounds(case))
        state.update(psi=torch.empty_like(X), ritz=torch.empty(n, dtype=torch.float64, device=DEV))
    else:
        state.update(schedule=_schedule(case), v0=torch.randn(N, dtype=torch.float64, device=DEV, generator=_gen(seed, 4)))
    return state


def run(state):
    c, H, ws = state["case"], state["H"], state["ws"]
    if c["op"] == "filter":
        return P.filter(H, state["X"], c["m"], *state["bounds"], schedule=state["schedule"], out=state["out"],
                        workspace=ws)
    if c["op"] == "backward":
        return P.filter_backward(H, state["X"], state["dY"], c["m"], *state["bounds"], workspace=ws,
                                 precision=c["precision"])
    if c["op"] == "lanczos":
        return P.lanczos_bounds(H, state["v0"], c["steps"], c["n"], workspace=ws)
    if c["op"] == "closure":
        return P.rayleigh_ritz(H, state["X"], c["passes"], psi=state["psi"], ritz=state["ritz"], workspace=ws,
                               precision=c["precision"])
    return P.solve(H, state["X"], c["m"], c["cycles"], state["v0"], schedule=state["schedule"],
                   rr_precision=c["precision"], workspace=ws)


# ------------------------------------------------------------------ work


def _nnz(case):
    if case["layout"] == "split":
        return case["N"] * (2 * case["band"] + 1) - case["band"] * (case["band"] + 1) + 8 * case["N"]
    g, w = case["g"], case["w"]
    return (g * (2 * w + 1) - w * (w + 1)) ** 3


def work(case):
    """One read of every input and one write of every output, and the flops of the
    definition: 2 nnz n + 5 N n a filter step, 2 nnz n a step of dH, 2 N n^2 a product with
    an n x n matrix, N n^2 a symmetric product, 9 n^3 the eigenproblem."""
    N, n, nnz, op = _rows(case), case["n"], _nnz(case), case["op"]
    h, block = 12.0 * nnz + 8.0 * N, 8.0 * N * n
    step, closure = 2.0 * nnz * n + 5.0 * N * n, 2.0 * nnz * n + 8.0 * N * n * n + 9.0 * n ** 3
    if op == "filter":
        return dict(bytes=h + 2 * block, flops=case["m"] * step)
    if op == "backward":
        return dict(bytes=h + 3 * block + 8.0 * nnz, flops=case["m"] * (2 * step + 2.0 * nnz * n))
    if op == "lanczos":
        return dict(bytes=h + 8.0 * N, flops=case["steps"] * (2.0 * nnz + 4.0 * N * case["steps"]))
    if op == "closure":
        return dict(bytes=h + 2 * block, flops=closure)
    return dict(bytes=h + 2 * block, flops=40.0 * nnz + case["cycles"] * (case["m"] * step + closure))


# ------------------------------------------------------------------ the same in 64 bits


def _sparse(H):
    return torch.sparse_csr_tensor(H.row_ptr, H.col.long(), H.val, (H.n_rows, H.n_rows))


def _coefficients(m, a, b, a0):
    e, c = (b - a) / 2.0, (b + a) / 2.0
    sigma = e / (a0 - c)
    gamma, al, be = 2.0 / sigma, [0.0, sigma / e], [0.0, 0.0]
    for _ in range(2, m + 1):
        nxt = 1.0 / (gamma - sigma)
        al.append(2.0 * nxt / e)
        be.append(sigma * nxt)
        sigma = nxt
    return al, be, c


def _plain_filter(S, X, m, a, b, a0, keep=None):
    al, be, c = _coefficients(m, a, b, a0)
    prev, cur = None, X
    for k in range(1, m + 1):
        if keep is not None:
            keep.append(cur)
        new = al[k] * (S @ cur - c * cur)
        if k >= 2:
            new -= be[k] * prev
        prev, cur = cur, new
    return cur


def _plain_backward(H, X, dY, m, a, b, a0):
    S, ys = _sparse(H), []
    _plain_filter(S, X, m, a, b, a0, keep=ys)
    al, be, c = _coefficients(m, a, b, a0)
    be.append(0.0)
    rows = torch.repeat_interleave(torch.arange(H.n_rows, device=DEV), torch.diff(H.row_ptr))
    col, dH = H.col.long(), torch.zeros_like(H.val)
    part = max(1, (1 << 27) // X.shape[1])
    nxt, bar = None, dY
    for k in range(m, 0, -1):
        for p in range(0, H.nnz, part):
            q = slice(p, p + part)
            dH[q] += al[k] * torch.einsum("pj,pj->p", bar[rows[q]], ys[k - 1][col[q]])
        new = al[k] * (S @ bar - c * bar)
        if nxt is not None:
            new -= be[k + 1] * nxt
        nxt, bar = bar, new
    return bar, dH


def _plain_lanczos(S, v0, steps, n_wanted):
    v = v0 / torch.linalg.vector_norm(v0)
    V, al, be = [v], [], []
    for j in range(steps):
        w = torch.mv(S, V[j])
        al.append(float(torch.dot(V[j], w)))
        w = w - al[j] * V[j] - (be[j - 1] * V[j - 1] if j else 0.0)
        B = torch.stack(V)
        w = w - B.t() @ (B @ w)
        be.append(float(torch.linalg.vector_norm(w)))
        V.append(w / be[j])
    T = torch.diag(torch.tensor(al, dtype=torch.float64)) + sum(
        torch.diag(torch.tensor(be[:-1], dtype=torch.float64), k) for k in (-1, 1))
    theta = torch.linalg.eigvalsh(T)
    a0, b = float(theta[0]), float(theta[-1]) + abs(be[-1])
    return a0 + (b - a0) * (n_wanted / v0.numel()) ** (2.0 / 3.0), b, a0


def _plain_closure(S, Y):
    Q = torch.linalg.qr(Y)[0]
    F = Q.t() @ (S @ Q)
    theta, U = torch.linalg.eigh((F + F.t()) / 2)
    return theta, Q @ U


def exact(case, seed):
    """Ritz vectors have no value of their own (their sign is free): None in their place."""
    state = prepare(case, seed)
    H = _operator(case, seed, plain=True)
    S, op = _sparse(H), case["op"]
    if op == "filter":
        return _plain_filter(S, state["X"], case["m"], *state["bounds"])
    if op == "backward":
        return _plain_backward(H, state["X"], state["dY"], case["m"], *state["bounds"])
    if op == "lanczos":
        return _plain_lanczos(S, state["v0"], case["steps"], case["n"])
    if op == "closure":
        return _plain_closure(S, state["X"])[0], None
    a, b, a0 = _plain_lanczos(S, state["v0"], 20, case["n"])
    psi, history = state["X"], []
    for _ in range(case["cycles"]):
        theta, psi = _plain_closure(S, _plain_filter(S, psi, case["m"], a, b, a0))
        history.append(theta)
        a0, a = float(theta[0]), float(theta[-1])
    return history[-1], None, history
