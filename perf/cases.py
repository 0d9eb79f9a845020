"""What this library is used for, as measured cases: batches of small systems
solved on the device through bbs.solve / Handle.solve, uneven batches through a
plan, and the learned initial guess (prediction and training).

Matrices follow the repository's recipe: on every stencil edge {i, j} a draw
s ~ U[-1, 0], a_ij and a_ji = s (1 + U[-0.1, 0.1]) (their mean where a
symmetric matrix is wanted), a_ii = (sum of the row's |a_ij|) (1 + U[lo, hi]),
b ~ U[-1, 1], x0 = 0. The PeleLM shapes take independent entries on a random
structurally symmetric pattern. Everything is drawn on the GPU from the seed.

A solve returns x and the status of every system. The rest of its log is where
and how closely the stopping test was passed (iterations, the last residual):
both follow the last bits of every sum before them (the library promises its
iteration counts to within 2), so they would compare rounding, not results; x
is compared to FP64's own bound.
"""

from __future__ import annotations

import functools
import math

import numpy as np
import torch

from paper_2308_08417_gb300 import bbs
from paper_2308_08417_gb300 import workloads as W

DEV = "cuda"

# Krylov iterations a system of this kind takes to a relative residual of
# 1e-10 (means measured over the batches below; the operation counts need them)
ITERATIONS = {"bicgstab": {"1d3": 22.0, "2d5": 23.0, "2d9": 26.0, "random": 7.5},
              "cg": {"1d3": 32.0, "2d5": 34.0, "2d9": 36.0},
              "gmres": {"1d3": 34.0, "2d5": 36.0, "2d9": 38.0, "random": 11.0},
              "ilu0": {"1d3": 1.0, "2d5": 7.1, "2d9": 7.0},
              "mixed": {"1d3": 40.0, "2d5": 40.0, "2d9": 40.0}}


def listed():
    return [
        # one small call: a handful of tridiagonal systems (the smoke check's
        # batch), where launches and host work count
        dict(name="solve_tiny_csr", kind="solve", method="bicgstab", fmt="csr", stencil="1d3", kx=32, ky=1,
             batch=64, lo=0.05, hi=0.5, call="solve"),
        # the headline: 65,536 systems of a 5-point stencil on a 12 x 12 grid
        dict(name="bicgstab_csr_n144", kind="solve", method="bicgstab", fmt="csr", stencil="2d5", kx=12, ky=12,
             batch=65536, lo=0.05, hi=0.5, call="handle"),
        # the symmetrised copy under CG, on an odd grid with a ragged batch
        dict(name="cg_ell_n143", kind="solve", method="cg", fmt="ell", stencil="2d5", kx=11, ky=13,
             batch=30001, lo=0.05, hi=0.5, call="handle"),
        # restarted GMRES(10) on the headline's systems
        dict(name="gmres_csr_n144", kind="solve", method="gmres", fmt="csr", stencil="2d5", kx=12, ky=12,
             batch=16384, lo=0.05, hi=0.5, call="handle"),
        # BiCGSTAB under ILU(0) on the headline's systems
        dict(name="ilu_csr_n144", kind="solve", method="ilu0", fmt="csr", stencil="2d5", kx=12, ky=12,
             batch=32768, lo=0.05, hi=0.5, call="handle"),
        # reaction systems of a small mechanism (drm19's size and density) over
        # a mesh's cells, stored dense: the smallest systems, the largest batch
        dict(name="bicgstab_dense_n22", kind="solve", method="bicgstab", fmt="dense", stencil="random", n=22,
             nnz=438, batch=131072, lo=0.05, hi=0.5, call="handle"),
        # a large mechanism (isooctane's size and density): long ragged rows
        dict(name="bicgstab_csr_n144_dense_rows", kind="solve", method="bicgstab", fmt="csr", stencil="random",
             n=144, nnz=6135, batch=16384, lo=0.05, hi=0.5, call="handle"),
        # large systems in FP64: a 9-point stencil on a 32 x 32 grid
        dict(name="bicgstab_ell_n1024", kind="solve", method="bicgstab", fmt="ell", stencil="2d9", kx=32, ky=32,
             batch=4096, lo=0.01, hi=0.1, call="handle"),
        # the same systems with FP32 inner solves under FP64 refinement
        dict(name="mixed_ell_n1024", kind="solve", method="mixed", fmt="ell", stencil="2d9", kx=32, ky=32,
             batch=16384, lo=0.01, hi=0.1, call="handle"),
        # systems of every size from 16 to 1024 rows over all three stencils
        dict(name="uneven_n16_1024", kind="uneven", batch=20000, n_min=16, n_max=1024, lo=0.05, hi=0.5),
        # initial guesses of one time step of 16,384 systems
        dict(name="predict_n144", kind="predict", kx=12, ky=12, batch=16384, hidden=256),
        # one training step of the network that predicts them
        dict(name="train_n144", kind="train", n=144, hidden=256, batch=4096, store=65536),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["solve"] * 8 + ["uneven", "predict", "train"])
    if kind == "uneven":
        lo = _log(rng, 16, 64)
        return dict(kind="uneven", batch=_log(rng, 2000, 20000), n_min=lo, n_max=_log(rng, 4 * lo, 1024),
                    lo=0.05, hi=0.5)
    if kind == "predict":
        k = rng.randint(5, 15)
        return dict(kind="predict", kx=k, ky=rng.randint(max(4, k - 3), min(16, k + 3)),
                    batch=_log(rng, 300, 16384), hidden=rng.choice([64, 128, 192, 256]))
    if kind == "train":
        return dict(kind="train", n=_log(rng, 16, 200), hidden=rng.choice([64, 128, 192, 256]),
                    batch=64 * _log(rng, 1, 64), store=_log(rng, 4096, 65536))
    method = rng.choice(["bicgstab"] * 4 + ["cg", "gmres", "ilu0", "mixed"])
    call = rng.choice(["handle", "handle", "solve"])
    if method == "bicgstab" and rng.random() < 0.35:
        name = rng.choice(sorted(W.MECHANISMS))
        _, n, nnz = W.MECHANISMS[name]
        top = min(131072, int(16384 * 6135 / nnz))
        return dict(kind="solve", method=method, fmt=rng.choice(["csr", "dense"]), stencil="random", n=n, nnz=nnz,
                    batch=_log(rng, 64, top), lo=0.05, hi=0.5, call=call)
    stencil = rng.choice(["1d3", "2d5", "2d9"])
    n = _log(rng, 16, 1024 if method != "ilu0" else 400)
    if stencil == "1d3":
        kx, ky = n, 1
    else:
        kx = max(2, int(round(math.sqrt(n) * rng.uniform(0.7, 1.4))))
        ky = max(2, n // kx)
    n = kx * ky
    fmt = "csr" if method == "ilu0" else "ell" if method == "mixed" else rng.choice(["csr", "ell", "csr"])
    # no more rows in all than the large FP64 batch (4,096 x 1,024) has
    top = max(64, min(65536, 4096 * 1024 // n))
    hard = rng.random() < 0.3
    return dict(kind="solve", method=method, fmt=fmt, stencil=stencil, kx=kx, ky=ky, batch=_log(rng, 64, top),
                lo=0.01 if hard else 0.05, hi=0.1 if hard else 0.5, call=call)


# ------------------------------------------------------------------ patterns

_OFFSETS = {"1d3": [(0, -1), (0, 0), (0, 1)],
            "2d5": [(-1, 0), (0, -1), (0, 0), (0, 1), (1, 0)],
            "2d9": [(dy, dx) for dy in (-1, 0, 1) for dx in (-1, 0, 1)]}


def _stencil_slots(stencil, kx, ky):
    """[slots, n] column of each stencil slot of each row, -1 outside the grid (ascending columns)."""
    y, x = np.divmod(np.arange(kx * ky), kx)
    cols = []
    for dy, dx in _OFFSETS[stencil]:
        ok = (y + dy >= 0) & (y + dy < ky) & (x + dx >= 0) & (x + dx < kx)
        cols.append(np.where(ok, (y + dy) * kx + x + dx, -1))
    return np.stack(cols)


@functools.lru_cache(maxsize=64)
def _random_slots(n, nnz):
    """A full diagonal and nnz - n mirrored off-diagonal positions, as [slots, n] columns."""
    rng = np.random.default_rng(1000 * n + nnz)
    iu, ju = np.triu_indices(n, 1)
    pick = rng.permutation(len(iu))[: (nnz - n) // 2]
    on = np.eye(n, dtype=bool)
    on[iu[pick], ju[pick]] = on[ju[pick], iu[pick]] = True
    k = int(on.sum(1).max())
    cols = np.full((k, n), -1)
    for r in range(n):
        c = np.nonzero(on[r])[0]
        cols[: len(c), r] = c
    return cols


def _csr(cols):
    """(row_ptrs, col_idxs, position of each stored entry in the [slots, n] table) of a slot table."""
    ok = (cols >= 0).T
    row_ptrs = np.zeros(cols.shape[1] + 1, dtype=np.int32)
    row_ptrs[1:] = np.cumsum(ok.sum(1))
    r, s = np.nonzero(ok)
    return row_ptrs, cols[s, r].astype(np.int32), s.astype(np.int64) * cols.shape[1] + r


def _slots(case):
    if case["stencil"] == "random":
        return _random_slots(case["n"], case["nnz"])
    return _stencil_slots(case["stencil"], case["kx"], case["ky"])


def _sizes(case):
    cols = _slots(case)
    return cols.shape[1], int((cols >= 0).sum())


# -------------------------------------------------------------------- values

def _gen(seed):
    return torch.Generator(device=DEV).manual_seed(int(seed))


def _uniform(g, lo, hi, *shape):
    return torch.rand(*shape, generator=g, device=DEV, dtype=torch.float64).mul_(hi - lo).add_(lo)


def _edge_values(g, cols, batch, lo, hi, symmetric, paired):
    """[batch, slots, n] values on a slot table (0 outside the pattern)."""
    k, n = cols.shape
    c = torch.as_tensor(cols, device=DEV)
    ok = c >= 0
    row = torch.arange(n, device=DEV)
    diag = c == row
    if paired:  # slot j of row i and slot k - 1 - j of row c share an edge: the upper half draws it
        s = _uniform(g, -1.0, 0.0, batch, k, n)
        v = torch.zeros_like(s)
        for j in range(k):
            if j == k // 2:
                continue
            up = j > k // 2
            at = c[j].clamp(min=0)
            edge = s[:, j] if up else s[:, k - 1 - j][:, at]
            v[:, j] = edge
            f = _uniform(g, -0.1, 0.1, batch, n)
            if not symmetric:
                v[:, j] *= 1.0 + f
        if symmetric:  # the pair's mean: one factor per edge
            f = _uniform(g, -0.1, 0.1, batch, k, n)
            for j in range(k):
                if j != k // 2:
                    v[:, j] *= 1.0 + (f[:, j] if j > k // 2 else f[:, k - 1 - j][:, c[j].clamp(min=0)])
        del s
    else:
        v = _uniform(g, -1.0, 0.0, batch, k, n) * _uniform(g, 0.9, 1.1, batch, k, n)
    v *= (ok & ~diag)
    u = _uniform(g, lo, hi, batch, n)
    a = v.abs().sum(1) * (1.0 + u)
    return v + a[:, None, :] * diag


def _batch(case, seed):
    """(cols [slots, n], values [batch, slots, n], b [batch, n]) of a uniform batch."""
    g = _gen(seed)
    cols = _slots(case)
    v = _edge_values(g, cols, case["batch"], case["lo"], case["hi"], case["method"] == "cg",
                     case["stencil"] != "random")
    return cols, v, _uniform(g, -1.0, 1.0, case["batch"], cols.shape[1])


def _device_batch(fmt, cols, v):
    k, n = cols.shape
    B = v.shape[0]
    row_ptrs, col_idxs, at = _csr(cols)
    nnz = len(col_idxs)
    vals = v.reshape(B, -1)[:, torch.as_tensor(at, device=DEV)]
    longest = int(np.diff(row_ptrs).max())
    if fmt == "csr":
        return bbs.DeviceBatch("csr", n, nnz, longest, torch.as_tensor(row_ptrs, device=DEV),
                               torch.as_tensor(col_idxs, device=DEV), vals)
    rows = np.repeat(np.arange(n), np.diff(row_ptrs))
    if fmt == "ell":  # a row's entries side by side from slot 0, padding after them
        dest = (np.arange(nnz) - np.repeat(row_ptrs[:-1], np.diff(row_ptrs))).astype(np.int64) * n + rows
        ec = np.full(longest * n, -1, dtype=np.int32)
        ec[dest] = col_idxs
        out = torch.zeros(B, longest * n, dtype=torch.float64, device=DEV)
        out[:, torch.as_tensor(dest, device=DEV)] = vals
        return bbs.DeviceBatch("ell", n, nnz, longest, None, torch.as_tensor(ec, device=DEV), out)
    out = torch.zeros(B, n * n, dtype=torch.float64, device=DEV)
    out[:, torch.as_tensor(rows.astype(np.int64) * n + col_idxs, device=DEV)] = vals
    return bbs.DeviceBatch("dense", n, nnz, 0, None, None, out)


def _uneven_grids(case):
    """(kind, kx, ky) of every system: sizes log-uniform, the three stencils in
    equal parts. The grids are the program's (one set per case); the seed draws
    the values on them."""
    rng = np.random.default_rng([case["batch"], case["n_min"], case["n_max"]])
    B = case["batch"]
    n = np.rint(np.exp(rng.uniform(math.log(case["n_min"]), math.log(case["n_max"]), B))).astype(np.int64)
    kind = rng.integers(0, 3, B)
    kx = np.where(kind == 0, n, np.rint(np.sqrt(n)).astype(np.int64))
    ky = np.where(kind == 0, 1, np.maximum(1, n // kx))
    return kind, kx, ky


def _uneven(case, seed):
    """Flat uneven batch: per-system arrays, and the slots of all rows one after another."""
    kind, kx, ky = _uneven_grids(case)
    keys, first, index = np.unique(np.stack([kind, kx, ky], 1), axis=0, return_index=True, return_inverse=True)
    index = index.reshape(-1)
    pats = []
    for kd, x, y in keys.tolist():
        name = ("1d3", "2d5", "2d9")[kd]
        rp, ci, _ = _csr(_stencil_slots(name, x, y))
        pats.append(W.Pattern(x * y, rp, ci, name, x, y))
    n = kx * ky
    nnz = np.array([p.nnz for p in pats], dtype=np.int64)[index]
    vec_off = np.cumsum(n) - n
    val_off = np.cumsum(nnz) - nnz
    t = functools.partial(torch.as_tensor, device=DEV)
    sys = torch.repeat_interleave(torch.arange(case["batch"], device=DEV), t(n))
    N = int(n.sum())
    at = torch.arange(N, device=DEV) - t(vec_off)[sys]
    X, Y, K = t(kx)[sys], t(ky)[sys], t(kind)[sys]
    px, py = at % X, at // X
    g = _gen(seed)
    up = [(0, 1), (1, -1), (1, 0), (1, 1)]
    s = _uniform(g, -1.0, 0.0, 4, N)
    cols = torch.full((9, N), -1, device=DEV)
    v = torch.zeros(9, N, dtype=torch.float64, device=DEV)
    glob = torch.arange(N, device=DEV)
    for o, (dy, dx) in enumerate(_OFFSETS["2d9"]):
        ok = (px + dx >= 0) & (px + dx < X) & (py + dy >= 0) & (py + dy < Y)
        if dx and dy:
            ok &= K == 2
        if dy:
            ok &= K > 0
        c = glob + dy * X + dx
        cols[o] = torch.where(ok, c, -1)
        if (dy, dx) == (0, 0):
            continue
        edge = s[up.index((dy, dx))] if (dy, dx) in up else s[up.index((-dy, -dx))][c.clamp(0, N - 1)]
        v[o] = torch.where(ok, edge * (1.0 + _uniform(g, -0.1, 0.1, N)), 0.0)
    v[4] = v.abs().sum(0) * (1.0 + _uniform(g, case["lo"], case["hi"], N))
    b = _uniform(g, -1.0, 1.0, N)
    return pats, index.astype(np.int32), val_off, vec_off, sys, cols, v, b


# -------------------------------------------------------------------- network

def _mlp_params(g, n, hidden):
    parts = []
    for fan_in, out in ((3 * n, hidden), (hidden, hidden), (hidden, hidden), (hidden, n)):
        bound = 0.5 * math.sqrt(6.0 / fan_in)
        parts.append((torch.rand(out * fan_in, generator=g, device=DEV) * 2 - 1) * bound)
        parts.append((torch.rand(out, generator=g, device=DEV) * 2 - 1) * 0.1)
    return torch.cat(parts)


def _layers(flat, n, hidden):
    got, o = [], 0
    for fan_in, out in ((3 * n, hidden), (hidden, hidden), (hidden, hidden), (hidden, n)):
        w = flat[o:o + out * fan_in].double().view(out, fan_in)
        o += out * fan_in
        got.append((w, flat[o:o + out].double()))
        o += out
    return got


def _train_inputs(case, seed):
    g = _gen(seed)
    n, pad = case["n"], (3 * case["n"] + 63) // 64 * 64
    params = _mlp_params(g, n, case["hidden"])
    feats = torch.zeros(case["store"], pad, dtype=torch.bfloat16, device=DEV)
    feats[:, :3 * n] = torch.randn(case["store"], 3 * n, generator=g, device=DEV).to(torch.bfloat16)
    targets = torch.randn(case["store"], n, generator=g, device=DEV)
    rows = torch.randperm(case["store"], generator=g, device=DEV)[:case["batch"]].to(torch.int32)
    return params, feats, targets, rows


def _predict_inputs(case, seed):
    """One step's batch and the 128 systems the statistics come from, whose
    entries are rounded to multiples of 2^-10 so that their sums are exact."""
    c = dict(case, stencil="2d5", lo=0.05, hi=0.5, method="bicgstab")
    cols, v, b = _batch(c, seed)
    g = _gen(seed + 1)
    x_prev = torch.randn(b.shape, generator=g, device=DEV, dtype=torch.float64) * 0.6
    params = _mlp_params(g, cols.shape[1], case["hidden"])
    m = min(128, case["batch"])
    q = lambda a: torch.round(a * 1024.0) / 1024.0  # noqa: E731
    seen = (q(v[:m]), q(b[:m]), q(x_prev[:m]),
            q(x_prev[:m]) + q(0.05 * torch.randn(m, b.shape[1], generator=g, device=DEV, dtype=torch.float64)))
    return cols, v, b, x_prev, params, seen


# ------------------------------------------------------------------ the cases

def _options(case):
    m = case["method"]
    if m == "mixed":  # the tolerance of the inner solves that the benchmark takes
        return bbs.bbs_default_options(precision="mixed", inner_tol=3e-3)
    if m == "ilu0":
        return bbs.bbs_default_options(precond="ilu0")
    return bbs.bbs_default_options(solver=m)


def prepare(case, seed):
    kind = case["kind"]
    if kind == "solve":
        cols, v, b = _batch(case, seed)
        A = _device_batch(case["fmt"], cols, v)
        del v
        h = bbs.Handle(0)
        if case["call"] == "solve":
            m = case["method"]
            opts = (dict(precision="mixed", inner_tol=3e-3) if m == "mixed" else dict(precond="ilu0") if m == "ilu0"
                    else dict(solver=m))
            return dict(case=case, h=h, A=A, b=b, opts=opts)
        o = _options(case)
        x0 = torch.zeros_like(b)
        return dict(case=case, h=h, A=A, b=b, x0=x0, x=torch.empty_like(b), o=o,
                    log=bbs.Log.empty(A.num_batch, inner=case["method"] == "mixed"), ws=h.workspace(A, o))
    if kind == "uneven":
        pats, index, val_off, vec_off, _, cols, v, b = _uneven(case, seed)
        values = v.t()[(cols >= 0).t()]  # row by row, columns ascending
        vb = W.VarBatch(pats, index, val_off, vec_off, values, b, torch.zeros_like(b))
        h = bbs.Handle(0)
        vd = bbs.VarDeviceBatch.from_varbatch(vb)
        plan = bbs.VarPlan(h, vd, bbs.bbs_default_options())
        return dict(case=case, plan=plan, b=b, x0=torch.zeros_like(b), x=torch.empty_like(b),
                    log=bbs.Log.empty(case["batch"]))
    h = bbs.Handle(0)
    if kind == "predict":
        cols, v, b, x_prev, params, (vs, bs, ps, ns) = _predict_inputs(case, seed)
        A = _device_batch("csr", cols, v)
        mlp = bbs.MLP(h, cols.shape[1], hidden=case["hidden"], max_batch=max(4096, (case["batch"] + 63) // 64 * 64))
        mlp.set_params(params)
        mlp.observe(_device_batch("csr", cols, vs), bs, ps, ns)
        mlp.finalize_stats()
        torch.cuda.synchronize()
        return dict(case=case, mlp=mlp, A=A, b=b, x_prev=x_prev, x0=torch.empty_like(b))
    params, feats, targets, rows = _train_inputs(case, seed)
    mlp = bbs.MLP(h, case["n"], hidden=case["hidden"], max_batch=case["batch"])
    mlp.set_params(params)
    return dict(case=case, mlp=mlp, feats=feats, targets=targets, rows=rows,
                loss=torch.zeros(1, dtype=torch.float32, device=DEV))


def run(s):
    kind = s["case"]["kind"]
    if kind == "solve":
        if s["case"]["call"] == "solve":
            x, log = bbs.solve(s["A"], s["b"], handle=s["h"], **s["opts"])
            return x, log.status
        s["x"].copy_(s["x0"])
        s["h"].solve(s["A"], s["b"], s["x"], s["o"], s["log"], s["ws"])
        return s["x"], s["log"].status
    if kind == "uneven":
        s["x"].copy_(s["x0"])
        s["plan"].solve(s["b"], s["x"], s["log"])
        return s["x"], s["log"].status
    if kind == "predict":
        return s["mlp"].predict(s["A"], s["b"], s["x_prev"], s["x0"])
    s["mlp"].train_step(s["feats"], s["targets"], s["rows"], 1e-3, s["loss"])
    return s["loss"], s["mlp"].get_grads()


def work(case):
    kind, B = case["kind"], case["batch"]
    if kind == "solve":
        n, nnz = _sizes(case)
        stored = n * n if case["fmt"] == "dense" else nnz
        it = ITERATIONS[case["method"]][case["stencil"]]
        if case["method"] == "cg":
            flops = it * (2 * nnz + 13 * n)
        elif case["method"] == "gmres":  # 5.5 basis vectors a step on average: a projection and an update each
            flops = it * (2 * nnz + (5.5 * 4 + 6) * n)
        elif case["method"] == "ilu0":  # two SpMVs and two triangular solves
            flops = it * (8 * nnz + 26 * n)
        else:
            flops = it * (4 * nnz + 26 * n)
        return {"bytes": float(B * (8 * (stored + 3 * n) + 16)), "flops": float(B * flops)}
    if kind == "uneven":
        kd, kx, ky = _uneven_grids(case)
        n = (kx * ky).astype(np.float64)
        edges = np.where(kd == 0, kx - 1, (kx - 1) * ky + kx * (ky - 1))
        nnz = n + 2.0 * edges + np.where(kd == 2, 4.0 * (kx - 1) * (ky - 1), 0.0)
        return {"bytes": float((8 * (nnz + 3 * n) + 16).sum()), "flops": float(22.0 * (4 * nnz + 26 * n).sum())}
    H = case["hidden"]
    n = case["n"] if kind == "train" else case["kx"] * case["ky"]
    weights = 3 * n * H + 2 * H * H + H * n
    if kind == "predict":  # the diagonal, b, x_prev and x0
        return {"bytes": float(B * 4 * n * 8 + 2 * weights), "flops": float(2 * B * weights)}
    # the minibatch's rows; parameters and both moments read and written, the gradients written and copied out
    return {"bytes": float(B * (3 * n * 2 + n * 4) + weights * 4 * 9),
            "flops": float(2 * B * (3 * weights - 3 * n * H))}


# ------------------------------------------------------------- 64-bit results

def _solve64(cols, v, b, dot, inv_diag):
    """Jacobi-BiCGSTAB on flat vectors to the accuracy of 64 bits. cols, v: [slots, rows]; dot(x, y): the
    systems' inner products, spread over their rows."""
    safe = cols.clamp(min=0)

    def mul(x):
        y = torch.zeros_like(x)
        for j in range(cols.shape[0]):
            y.addcmul_(v[j], x[safe[j]])
        return y

    def over(p, q):
        return torch.where(q != 0, p / q, torch.zeros_like(p))

    x = torch.zeros_like(b)
    nb = dot(b, b)
    for _ in range(3):  # restarts polish what the recursion drifted by
        r = b - mul(x)
        rh, p, w = r.clone(), torch.zeros_like(r), torch.zeros_like(r)
        rho = alpha = omega = torch.ones_like(r)
        for it in range(120):
            live = dot(r, r) > 1e-30 * nb
            if it % 8 == 0 and not bool(live.any()):
                break
            rho1 = dot(rh, r)
            p = r + over(rho1 * alpha, rho * omega) * (p - omega * w)
            rho = rho1
            ph = inv_diag * p
            w = mul(ph)
            alpha = torch.where(live, over(rho, dot(rh, w)), 0.0)
            s = r - alpha * w
            sh = inv_diag * s
            t = mul(sh)
            omega = torch.where(live, over(dot(t, s), dot(t, t)), 0.0)
            x = x + alpha * ph + omega * sh
            r = torch.where(live, s - omega * t, r)
            alpha = torch.where(live, alpha, 1.0)
            omega = torch.where(live, omega, 1.0)
    return x


def _forward64(layers, h):
    zs, hs = [], []
    for k, (w, c) in enumerate(layers):
        hs.append(h)
        z = h @ w.t() + c
        zs.append(z)
        h = z if k == 3 else 0.5 * z * (1 + torch.tanh(math.sqrt(2 / math.pi) * (z + 0.044715 * z ** 3)))
    return h, zs, hs


def _gelu_grad64(z):
    u = torch.tanh(math.sqrt(2 / math.pi) * (z + 0.044715 * z ** 3))
    return 0.5 * (1 + u) + 0.5 * z * (1 - u * u) * math.sqrt(2 / math.pi) * (1 + 3 * 0.044715 * z * z)


def exact(case, seed):
    kind = case["kind"]
    if kind == "solve":
        cols, v, b = _batch(case, seed)
        B, k, n = v.shape
        x = torch.empty_like(b)
        step = max(1, min(B, (1 << 23) // n))
        for i in range(0, B, step):
            m = min(step, B - i)
            base = torch.arange(m, device=DEV)[:, None] * n
            c = torch.as_tensor(cols, device=DEV)
            flat = torch.where(c[:, None, :] >= 0, c[:, None, :] + base, -1).reshape(k, -1)
            vv = v[i:i + m].permute(1, 0, 2).reshape(k, -1)
            diag = (flat == torch.arange(m * n, device=DEV)).double().mul(vv).sum(0)

            def dot(p, q, m=m):
                return (p * q).view(m, n).sum(1, keepdim=True).expand(m, n).reshape(-1)

            x[i:i + m] = _solve64(flat, vv, b[i:i + m].reshape(-1), dot, 1.0 / diag).view(m, n)
        return x, torch.zeros(B, dtype=torch.int32)
    if kind == "uneven":
        _, _, _, _, sys, cols, v, b = _uneven(case, seed)
        B = case["batch"]

        def dot(p, q):
            return torch.zeros(B, dtype=torch.float64, device=DEV).index_add_(0, sys, p * q)[sys]

        return _solve64(cols, v, b, dot, 1.0 / v[4]), torch.zeros(B, dtype=torch.int32)
    if kind == "predict":
        cols, v, b, x_prev, params, (vs, bs, ps, ns) = _predict_inputs(case, seed)
        n = cols.shape[1]
        seen = torch.cat([vs[:, 2], bs, ps, ns - ps], 1)  # the diagonal is the middle slot
        mean, var = seen.mean(0), seen.var(0, unbiased=False)
        std = torch.where(var > 1e-12 * mean * mean, var.sqrt(), 1.0)
        f = (torch.cat([v[:, 2], b, x_prev], 1) - mean[:3 * n]) / std[:3 * n]
        out, _, _ = _forward64(_layers(params, n, case["hidden"]), f)
        return x_prev + out * std[3 * n:] + mean[3 * n:]
    params, feats, targets, rows = _train_inputs(case, seed)
    n, r = case["n"], rows.long()
    layers = _layers(params, n, case["hidden"])
    out, zs, hs = _forward64(layers, feats[r][:, :3 * n].double())
    d = out - targets[r].double()
    loss = (d * d).mean().reshape(1)
    d = 2 * d / d.numel()
    grads = []
    for k in (3, 2, 1, 0):
        if k < 3:
            d = d * _gelu_grad64(zs[k])
        grads = [(d.t() @ hs[k]).reshape(-1), d.sum(0)] + grads
        d = d @ layers[k][0]
    return loss, torch.cat(grads)
