"""The applies that the performance of this framework is measured on.

A case is one apply of a resident butterfly operator: an operator (its trees, depth and
rank), a direction, a number of right-hand sides, a precision and the kind of buffers.
`listed` gives the named cases, `draw` further ones of the same ranges; `prepare` makes
an operator and its input vectors, `run` applies it once, `work` counts the bytes and
operations no apply can do without, `exact` is the same product in FP64 with torch.

The operators' factors are drawn here: real trees (uniform grids, the polar and the
corona trees of Fourier integral operators, clustered points) with the ranks that a
factorization of that rank limit has, min(r, points of either node), and complex normal
entries scaled so that vectors keep their size from level to level, with decaying
middle singular values.  The host construction of the same operators takes minutes; an
apply reads the same bytes whatever their values.  An operator is a program's resident
weights: it is made once per shape and kept, and `prepare` draws new vectors for it.
"""
import math
from collections import OrderedDict

import numpy as np
import torch

from paper_1509_07925_gb300 import binding as bd

PRECISION = {"auto": bd.MBF_PREC_AUTO, "simt": bd.MBF_PREC_FP32_SIMT, "tf32": bd.MBF_PREC_TF32,
             "bf16x3": bd.MBF_PREC_BF16X3}
KEEP_OPERATORS = 8     # operators kept at a time (a few GB each at most)


def _case(tree, n, L, r, nrhs, dim=2, adjoint=False, precision="auto", kind="op", panels=1):
    return {"tree": tree, "dim": dim, "n": n, "L": L, "r": r, "nrhs": nrhs, "adjoint": adjoint,
            "precision": precision, "kind": kind, "panels": panels}


def listed():
    named = {
        # one transform of a small grid with the operator in cache: latency of a single call
        "dft2_n64_x1": _case("uniform", 64, 4, 16, 1),
        # a few vectors on a small ragged operator, an odd count (an iterative solver's block)
        "polar_n64_x5": _case("polar", 64, 4, 24, 5),
        # the benchmark's operator: one vector forward, and its adjoint (a least-squares step)
        "polar_n256_x1": _case("polar", 256, 6, 24, 1),
        "polar_n256_x1_adjoint": _case("polar", 256, 6, 24, 1, adjoint=True),
        # the largest count that stays on the FP32 path
        "polar_n128_x7": _case("polar", 128, 6, 24, 7),
        # a batch that does not fill a panel of 64 (what a server's batches look like)
        "dft2_n128_x20": _case("uniform", 128, 6, 16, 20),
        # the benchmark's headline: one full panel, forward, adjoint and with TF32 operands
        "polar_n256_x64": _case("polar", 256, 6, 24, 64),
        "polar_n256_x64_adjoint": _case("polar", 256, 6, 24, 64, adjoint=True),
        "polar_n256_x64_tf32": _case("polar", 256, 6, 24, 64, precision="tf32"),
        # three dimensions: wide tiles (c r = 256), half a panel
        "dft3_n32_x32": _case("uniform", 32, 4, 32, 32, dim=3),
        # the multiscale sum: per-corona operators and the dense centre, half a panel
        "msbf_n128_x32": _case("corona", 128, 6, 24, 32, kind="msbf"),
        # panels in page-locked host memory, streamed through the device
        "polar_n256_host_4x64": _case("polar", 256, 6, 24, 64, kind="host", panels=4),
    }
    return [dict(c, name=name) for name, c in named.items()]


def _log_int(rng, lo, hi):
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi + 1)))))))


def draw(rng):
    while True:
        kind = rng.choice(["op"] * 8 + ["msbf", "host"])
        nrhs = _log_int(rng, 1, 128)
        adjoint = kind != "host" and rng.random() < 0.35
        precision = rng.choice(["auto"] * 6 + ["simt", "bf16x3", "tf32"])
        if precision == "tf32" and (adjoint or kind == "msbf"):
            precision = "auto"
        if precision == "simt":
            nrhs = min(nrhs, 16)
        if kind == "msbf":
            n = rng.choice([32, 64, 128])
            c = _case("corona", n, int(math.log2(n)) // 2 * 2, rng.randint(6, 24), nrhs, adjoint=adjoint,
                      precision=precision, kind=kind)
        elif rng.random() < 0.25 and kind == "op":
            n, L = rng.choice([(8, 2), (12, 2), (16, 4), (24, 4), (32, 4)])
            c = _case("uniform", n, L, rng.randint(4, 32), nrhs, dim=3, adjoint=adjoint, precision=precision)
        else:
            n = _log_int(rng, 16, 256)
            Ls = [L for L in (2, 4, 6) if 4 <= n * n // 4 ** (L - 1) <= 224]
            tree = rng.choice(["uniform", "polar", "polar", "points"])
            c = _case(tree, n, rng.choice(Ls), rng.randint(4, 32), nrhs, adjoint=adjoint, precision=precision,
                      kind=kind, panels=rng.randint(2, 4) if kind == "host" else 1)
        if precision == "simt" and _largest_group(c) > 256:
            c["precision"] = "auto"      # beyond what the FP32 path takes
        if _cost(c) <= _cost(_case("uniform", 32, 4, 32, 32, dim=3)):
            return c


def _largest_group(case):
    """Most points in the 2^dim sibling leaves of one node."""
    return max(int(np.diff(off).reshape(-1, 2 ** s[0]).sum(axis=1).max())
               for s in _shapes(case)[0] for off in (s[3][1], s[4][1]))


def _cost(case):
    w = work(case)
    return max(w["bytes"], w["flops"] / 32)


# ----------------------------------------------------------------------------- operators
def _zorder(cell, L):
    """Leaf index in tree order of integer cell coordinates [points][dim] at depth L."""
    idx = np.zeros(cell.shape[0], dtype=np.int64)
    for b in range(L - 1, -1, -1):
        for k in range(cell.shape[1]):
            idx = 2 * idx + ((cell[:, k] >> b) & 1)
    return idx


def _tree(points01, L):
    """(permutation, leaf offsets) of points in [0, 1]^dim, the last cell closed."""
    cell = np.minimum((points01 * 2 ** L).astype(np.int64), 2 ** L - 1)
    leaf = _zorder(cell, L)
    off = np.zeros(2 ** (L * points01.shape[1]) + 1, dtype=np.int64)
    np.cumsum(np.bincount(leaf, minlength=off.size - 1), out=off[1:])
    return np.argsort(leaf, kind="stable"), off


def _grid(n, dim):
    ax = [np.arange(n)] * dim
    return np.stack([a.ravel() for a in np.meshgrid(*ax, indexing="ij")], axis=1)


def _shapes(case):
    """The (dim, L, r, x tree, Omega tree) of each operator of a case, and the natural
    indices of the dense centre (multiscale) or None."""
    dim, n, L, r = case["dim"], case["n"], case["L"], case["r"]
    grid = _grid(n, dim)
    xi = grid - n // 2
    if case["tree"] == "corona":
        out, centre = [], np.ones(n * n, dtype=bool)
        mx = np.abs(xi).max(axis=1)
        t = 0
        while n / 2 ** (t + 2) >= 8:
            half = n / 2 ** (t + 1)
            ids = np.flatnonzero((mx > half / 2) & (mx <= half))
            centre[ids] = False
            Lt = 2 * ((int(math.log2(n)) - t) // 2)
            perm, off = _tree((xi[ids] + half) / (2 * half), Lt)
            out.append((dim, Lt, r, _tree(grid / n, Lt), (ids[perm], off)))
            t += 1
        return out, np.flatnonzero(centre)
    if case["tree"] == "points":
        rng = np.random.default_rng(n)
        xs = rng.random((n * n, dim))
        ws = np.clip(0.5 + 0.2 * rng.standard_normal((n * n, dim)), 0.0, 1.0)
        return [(dim, L, r, _tree(xs, L), _tree(ws, L))], None
    wpts = grid / n
    if case["tree"] == "polar":
        p1 = np.minimum(np.sqrt(2.0) * np.hypot(xi[:, 0], xi[:, 1]) / n, 1.0)
        wpts = np.stack([p1, np.mod(np.arctan2(xi[:, 1], xi[:, 0]) / (2 * np.pi), 1.0)], axis=1)
    return [(dim, L, r, _tree(grid / n, L), _tree(wpts, L))], None


def _ranks(shape):
    """rank[side][l]: [c^l, c^(L-l)] ranks of the node pairs (side 0: X node, Omega node;
    side 1: Omega node, X node), levels h .. L."""
    dim, L, r, (_, xo), (_, wo) = shape
    c = 2 ** dim
    cx = [np.diff(xo).reshape(c ** l, -1).sum(axis=1) for l in range(L + 1)]
    cw = [np.diff(wo).reshape(c ** l, -1).sum(axis=1) for l in range(L + 1)]
    side = lambda a, b: {l: np.minimum(r, np.minimum(a[l][:, None], b[L - l][None, :])) for l in range(L // 2, L + 1)}
    return side(cx, cw), side(cw, cx)


def _block_ranks(rk, l, c):
    """Ranks (outer level l + 1, inner level l) of the transfer blocks of level l, as
    [c^l, c^(L-l-1), c]: of child t of the outer node, and of child tp of the paired one."""
    hi, lo = rk[l + 1], rk[l]
    out = hi.reshape(lo.shape[0], c, hi.shape[1]).transpose(0, 2, 1)
    inn = lo.reshape(lo.shape[0], hi.shape[1], c)
    return out, inn


def _counts(case):
    shapes, centre = _shapes(case)
    nnz = 0
    for s in shapes:
        dim, L, r, (_, xo), (_, wo) = s
        ru, rv = _ranks(s)
        nnz += int((np.diff(xo) * ru[L][:, 0]).sum() + (np.diff(wo) * rv[L][:, 0]).sum())
        for rk in (ru, rv):
            for l in range(L // 2, L):
                o, i = _block_ranks(rk, l, 2 ** dim)
                nnz += int((o.sum(axis=2).astype(np.int64) * i.sum(axis=2)).sum())
    points = case["n"] ** case["dim"]
    return nnz + (points * centre.size if centre is not None else 0), points


def work(case):
    """Each nonzero factor entry read once (8 bytes), each vector read and written once;
    one complex multiply-add (8 operations) per entry and right-hand side."""
    nnz, points = _counts(case)
    vectors = case["nrhs"] * case["panels"]
    return {"bytes": 8 * nnz + 16 * points * vectors, "flops": 8 * nnz * vectors}


def _normal(gen, shape, scale):
    a = torch.randn(*shape, 2, generator=gen, device="cuda", dtype=torch.float64)
    return torch.view_as_complex(a) * (scale / math.sqrt(2.0))


def _factors(shape, seed):
    """Factor arrays (FP64, on the GPU) of one operator in the layout of mbf_factors_t."""
    dim, L, r, (xp, xo), (wp, wo) = shape
    c, h = 2 ** dim, L // 2
    gen = torch.Generator(device="cuda").manual_seed(seed)
    ranks = _ranks(shape)
    dev = lambda a: torch.from_numpy(np.ascontiguousarray(a)).cuda()
    below = lambda rk, R: torch.arange(R, device="cuda") < dev(rk)[..., None]
    tops = [{l: max(1, int(rk[l].max())) for l in rk} for rk in ranks]
    leaf, levels = [], []
    for side, off in ((0, xo), (1, wo)):
        rk, R = ranks[side], tops[side]
        pts = np.diff(off)
        mx = max(1, int(pts.max()))
        m = below(pts, mx)[:, :, None] & below(rk[L][:, 0], R[L])[:, None, :]
        # forward, a U^L row sums over the rank and a (V^L)^* row over the leaf's points
        leaf.append(_normal(gen, m.shape, 1.0 / math.sqrt(R[L] if side == 0 else max(1.0, pts.mean()))) * m)
        lev = []
        for l in range(h, L):
            o, i = _block_ranks(rk, l, c)
            m = below(o, R[l + 1])[:, :, :, :, None, None] & below(i, R[l])[:, :, None, None, :, :]
            fan = c * (R[l] if side == 0 else R[l + 1])
            lev.append(_normal(gen, m.shape, 1.0 / math.sqrt(fan)) * m)
        levels.append(lev)
    Rh = tops[0][h]
    k = torch.arange(Rh, device="cuda", dtype=torch.float64)
    # outputs of the size that a kernel of modulus-one entries gives
    S = 2.0 * math.sqrt(max(1, wp.size)) * torch.exp(-k / 8.0) * below(ranks[0][h], Rh)
    per = lambda side: np.array([tops[side].get(l, 0) for l in range(L + 1)], dtype=np.int32)
    return {"RU": per(0), "RV": per(1), "UL": leaf[0], "VL": leaf[1], "G": levels[0], "H": levels[1], "S": S}


def _operator_seed(case):
    return 1 + case["n"] + 1000 * case["r"] + 100000 * case["L"]


def _centre_kernel(n, centre):
    """exp(2 pi i (x . xi + c(x) |xi|)) with c(x) = (2 + sin 2 pi x1 sin 2 pi x2) / 3, the
    dense centre of a Fourier integral operator: [centre points][n^2]."""
    x = torch.from_numpy(_grid(n, 2)).cuda().double() / n
    xi = torch.from_numpy(_grid(n, 2)[centre] - n // 2).cuda().double()
    cx = (2 + torch.sin(2 * math.pi * x[:, 0]) * torch.sin(2 * math.pi * x[:, 1])) / 3
    phase = xi @ x.T + torch.hypot(xi[:, 0], xi[:, 1])[:, None] * cx[None, :]
    return torch.polar(torch.ones_like(phase), 2 * math.pi * phase)


_operators = OrderedDict()


def _operator(case):
    """The resident operator of a case's shape, made on first use."""
    key = tuple(case[k] for k in ("tree", "dim", "n", "L", "r"))
    if key not in _operators:
        while len(_operators) >= KEEP_OPERATORS:
            _operators.popitem(last=False)
        shapes, centre = _shapes(case)
        n, ops = case["n"] ** case["dim"], []
        for t, s in enumerate(shapes):
            f = _factors(s, _operator_seed(case) + t)
            host = lambda a: a.cpu().numpy()
            hf = bd.HostFactors.from_arrays(s[0], s[1], n, n, s[3][0], s[3][1], s[4][0], s[4][1], f["RU"], f["RV"],
                                            host(f["UL"]), host(f["VL"]), [host(a) for a in f["G"]],
                                            [host(a) for a in f["H"]], host(f["S"]))
            ops.append(bd.Operator(hf))
        if centre is not None:
            _operators[key] = bd.MsBF.create(ops, _centre_kernel(case["n"], centre).cpu().numpy(), centre)
        else:
            _operators[key] = ops[0]
    _operators.move_to_end(key)
    return _operators[key]


# ----------------------------------------------------------------------------- one apply
def _vectors(case, seed):
    """Complex normal vectors [panels][nrhs][points] (complex64, on the GPU)."""
    gen = torch.Generator(device="cuda").manual_seed(seed)
    a = torch.randn(case["panels"], case["nrhs"], case["n"] ** case["dim"], 2, generator=gen, device="cuda")
    return torch.view_as_complex(a / math.sqrt(2.0))


def prepare(case, seed):
    v = _vectors(case, seed)
    if case["kind"] == "host":
        g = v.cpu().pin_memory()
        u = torch.empty_like(g).pin_memory()
    else:
        g = v[0].contiguous()
        u = torch.empty_like(g)
    return {"op": _operator(case), "g": g, "u": u, "nrhs": case["nrhs"], "adjoint": case["adjoint"],
            "precision": PRECISION[case["precision"]], "kind": case["kind"]}


def run(state):
    op, g, u, nrhs, precision = (state[k] for k in ("op", "g", "u", "nrhs", "precision"))
    stream = torch.cuda.current_stream().cuda_stream
    if state["kind"] == "host":
        op.apply_host_batch(g, nrhs, precision, stream, out=u)
    elif state["adjoint"]:
        op.apply_adjoint(g.data_ptr(), u.data_ptr(), nrhs, precision, stream)
    else:
        op.apply(g.data_ptr(), u.data_ptr(), nrhs, precision, stream)
    return u


# ----------------------------------------------------------------------------- FP64 apply
def _leaf_index(perm, off):
    pts = np.diff(off)
    a = np.arange(max(1, int(pts.max())))[None, :]
    idx = np.where(a < pts[:, None], off[:-1, None] + a, 0)
    return torch.from_numpy(perm[idx]).cuda(), torch.from_numpy(a < pts[:, None]).cuda()


def _apply64(shape, f, v, adjoint, points):
    """u = K v ([points][nrhs], FP64), or K^* v, level by level."""
    dim, L, r, (xp, xo), (wp, wo) = shape
    c, h, nr = 2 ** dim, L // 2, v.shape[1]
    # (leaf factor, levels, points) of the side that reads v and of the side that writes u
    src, dst = ("UL", "G", xp, xo), ("VL", "H", wp, wo)
    if not adjoint:
        src, dst = dst, src
    idx, valid = _leaf_index(src[2], src[3])
    y = f[src[0]].mH @ (v[idx] * valid[..., None])
    for l in range(L - 1, h - 1, -1):
        A = f[src[1]][l - h]
        ni, nj, _, R2, _, R1 = A.shape
        z = y.reshape(ni, c, nj, R2, nr).transpose(1, 2).reshape(ni * nj, c * R2, nr)
        y = (A.reshape(ni * nj, c * R2, c * R1).mH @ z).reshape(ni, nj * c, R1, nr)
    # S is indexed (X node, Omega node)
    w = y.transpose(0, 1) * (f["S"].transpose(0, 1) if adjoint else f["S"])[..., None]
    for l in range(h, L):
        A = f[dst[1]][l - h]
        ni, nj, _, R2, _, R1 = A.shape
        o = A.reshape(ni * nj, c * R2, c * R1) @ w.reshape(ni * nj, c * R1, nr)
        w = o.reshape(ni, nj, c, R2, nr).transpose(1, 2).reshape(ni * c, nj, R2, nr)
    idx, valid = _leaf_index(dst[2], dst[3])
    u = torch.zeros(points, nr, dtype=torch.complex128, device="cuda")
    u[idx[valid]] = (f[dst[0]] @ w.reshape(c ** L, -1, nr))[valid]
    return u


def exact(case, seed):
    points = case["n"] ** case["dim"]
    v = _vectors(case, seed).reshape(-1, points).T.to(torch.complex128)
    shapes, centre = _shapes(case)
    u = torch.zeros_like(v)
    for t, s in enumerate(shapes):
        u += _apply64(s, _factors(s, _operator_seed(case) + t), v, case["adjoint"], points)
    if centre is not None:
        K = _centre_kernel(case["n"], centre)
        ids = torch.from_numpy(centre).cuda()
        if case["adjoint"]:
            u[ids] += K.conj() @ v
        else:
            u += K.T @ v[ids]
    u = u.T.contiguous()
    return u.reshape(case["panels"], case["nrhs"], points).cpu() if case["kind"] == "host" else u
