"""Workloads of this framework as its users run them, through its public entry points.

Each case is a dict of plain values; ``prepare`` makes what a program has in hand before the
call (the tensor, initial cores, a context or server, output buffers), ``run`` makes one pass
and returns its outputs, ``work`` counts the bytes and operations that no implementation can do
without, and ``exact`` gives the outputs in 64 bits, computed here with torch and numpy alone.

Kinds of case:
  * ``update``  one core update through the per-stage entry points: the distributions of the
                other cores, draws, design rows, fibres, least squares;
  * ``als``     a whole decomposition and its relative error (the use the README shows);
  * ``dense``   one sweep of dense TR-ALS and its relative error, as a program that runs
                Alg. 1 until the error stops changing calls them;
  * ``error``   the relative error of given cores (the termination criterion of Sec. 4.1);
  * ``batched`` many independent problems in one call;
  * ``served``  requests through the continuous-batching server.

Cores of mixed-precision calls carry FP32 accuracy in FP64 buffers (the contraction and the
solves run in FP32), and a program that works on an FP32 tensor keeps FP32 cores: those are
returned as FP32. Cores of FP64 calls are returned as they are.
"""

import math
import random

import numpy as np
import torch

from paper_2010_08581_gb300 import inputs
from paper_2010_08581_gb300 import trals as T

DEV = "cuda"


def _ints(text):
    return tuple(int(v) for v in text.split("x"))


def _text(values):
    return "x".join(str(v) for v in values)


# --------------------------------------------------------------------------------------
# The cases
# --------------------------------------------------------------------------------------
def _update(name, dims, ranks, mode, J, prec):
    return dict(name=name, kind="update", dims=_text(dims), ranks=_text(ranks), mode=mode, J=J,
                prec=prec)


def _als(name, dims, ranks, J, sweeps, prec, sampling="leverage", data="tr", noise=1e-2):
    return dict(name=name, kind="als", dims=_text(dims), ranks=_text(ranks), J=J, sweeps=sweeps,
                prec=prec, sampling=sampling, data=data, noise=noise)


def listed():
    return [
        # The smallest call: one core update of a 40 x 30 x 20 tensor, stage by stage, in FP64
        # (the sizes of the package's smoke check). Launch and host latency is all there is.
        _update("update_small_fp64", (40, 30, 20), (3, 4, 2), 1, 300, "fp64"),
        # A program that drives the stages itself at the benchmark's main size; mode 1 of X is
        # strided, so its fibres are scattered.
        _update("update_500_mixed", (500, 500, 500), (10, 10, 10), 1, 4000, "mixed"),
        # The same at the largest rank the library takes (16, the top of the served range;
        # 256 unknowns per row), odd sizes, contiguous mode.
        _update("update_rank16_mixed", (321, 300, 283), (16, 16, 16), 2, 2560, "mixed"),
        # The benchmark's headline: 500^3 FP32, rank 10, J = 4000, 10 sweeps, then the error.
        _als("als_500_mixed", (500, 500, 500), (10, 10, 10), 4000, 10, "mixed"),
        # The FP64 path: 100^3, rank 5, J = 2000, 10 sweeps, 1e-3 noise, then the error.
        _als("als_100_fp64", (100, 100, 100), (5, 5, 5), 2000, 10, "fp64", noise=1e-3),
        # The largest: an image stack, 256 x 256 x 3 x 2000 FP32 (1.6 GB), smooth content,
        # J = 8000, 20 sweeps; one mode of size 3, one contiguous mode of 2000.
        _als("als_4way_mixed", (256, 256, 3, 2000), (10, 10, 10, 10), 8000, 20, "mixed",
             data="cosine"),
        # High order: 4^10 in 10 modes, rank 10, every unfolding wide (4 x 100), FP64.
        _als("als_10way_fp64", (4,) * 10, (10,) * 10, 2000, 2, "fp64"),
        # Uniform sampling (the variant of Sec. 5, which takes five times the samples) at rank
        # 16 on odd sizes.
        _als("als_uniform_rank16", (321, 300, 283), (16, 16, 16), 12800, 2, "mixed",
             sampling="uniform"),
        # Dense TR-ALS on the headline tensor, one sweep per call with the error after it.
        dict(name="dense_500_mixed", kind="dense", dims="500x500x500", ranks="10x10x10",
             prec="mixed"),
        # The error of given cores on a 5-way tensor of a served shape (uneven modes and ranks).
        dict(name="error_5way", kind="error", dims="37x33x41x29x26", ranks="12x8x14x6x10",
             prec="mixed"),
        # 512 independent small problems in one call (I_n in 32..200, ranks 3..8, J = 10 max L).
        dict(name="batched_512", kind="batched", count=512, shapes=4, sweeps=10, prec="mixed"),
        # A burst of requests to the server: 3- to 5-way, 1e5 to 3e7 entries, ranks 4..16,
        # J = 10 max L, three sweeps each.
        dict(name="served_16", kind="served", count=16, shapes=0, sweeps=3, emax=3e7,
             prec="mixed"),
    ]


def _log_uniform(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def _draw_dims(rng, N, entries, least):
    g = [rng.uniform(-0.5, 0.5) for _ in range(N)]
    m = sum(g) / N
    return tuple(max(least, round(entries ** (1.0 / N) * math.exp(v - m))) for v in g)


def _draw_ranks(rng, dims, lo, hi):
    """Ranks for which every least-squares problem has many more rows than unknowns."""
    N = len(dims)
    ranks = [rng.randint(lo, hi) for _ in range(N)]
    numel = math.prod(dims)
    for k in range(N):
        while 6 * ranks[k - 1] * ranks[k] > numel // dims[k] and max(ranks[k - 1], ranks[k]) > 2:
            big = k - 1 if ranks[k - 1] > ranks[k] else k
            ranks[big] -= 1
    return tuple(ranks)


def _lmax(ranks):
    return max(ranks[k - 1] * ranks[k] for k in range(len(ranks)))


def draw(rng):
    """One more case of the ranges above."""
    kind = rng.choice(("update", "update", "als", "als", "als", "dense", "error", "batched",
                       "served"))
    if kind == "update":
        prec = rng.choice(("fp64", "mixed", "mixed"))
        N = rng.choice((3, 3, 4, 5))
        dims = _draw_dims(rng, N, _log_uniform(rng, 2e4, 1e7 if prec == "fp64" else 1.2e8), 6)
        ranks = _draw_ranks(rng, dims, 2, 10 if prec == "fp64" else 16)
        J = max(64, int(_lmax(ranks) * rng.uniform(6, 40)))
        c = _update("", dims, ranks, rng.randrange(N), J, prec)
    elif kind == "als":
        flavour = rng.choice(("mixed", "mixed", "fp64", "uniform"))
        N = rng.choice((3, 3, 4))
        top = {"mixed": 1.2e8, "fp64": 4e6, "uniform": 6e7}[flavour]
        dims = _draw_dims(rng, N, _log_uniform(rng, 1e5, top), 12)
        ranks = _draw_ranks(rng, dims, 3, {"mixed": 11, "fp64": 8, "uniform": 16}[flavour])
        J = int(_lmax(ranks) * rng.uniform(12, 45))
        c = _als("", dims, ranks, J, rng.randint(1, 2 if flavour == "uniform" else 10),
                 "fp64" if flavour == "fp64" else "mixed",
                 "uniform" if flavour == "uniform" else "leverage")
    elif kind == "dense":
        N = rng.choice((3, 3, 4))
        dims = _draw_dims(rng, N, _log_uniform(rng, 1e5, 1.2e8), 12)
        c = dict(kind=kind, dims=_text(dims), ranks=_text(_draw_ranks(rng, dims, 3, 16)),
                 prec="mixed")
    elif kind == "error":
        prec = rng.choice(("fp64", "mixed", "mixed"))
        N = rng.choice((3, 4, 5))
        dims = _draw_dims(rng, N, _log_uniform(rng, 1e5, 1e7 if prec == "fp64" else 1.2e8), 4)
        c = dict(kind=kind, dims=_text(dims), ranks=_text(_draw_ranks(rng, dims, 3, 16)),
                 prec=prec)
    elif kind == "batched":
        c = dict(kind=kind, count=int(_log_uniform(rng, 16, 400)), shapes=rng.randrange(1, 10 ** 6),
                 sweeps=rng.randint(1, 8), prec="mixed")
    else:
        c = dict(kind=kind, count=rng.randint(3, 16), shapes=rng.randrange(1, 10 ** 6),
                 sweeps=rng.randint(1, 4), emax=_log_uniform(rng, 1e6, 3e7), prec="mixed")
    c.pop("name", None)
    return c


# --------------------------------------------------------------------------------------
# What a program has in hand
# --------------------------------------------------------------------------------------
def _dtype(case):
    return torch.float64 if case["prec"] == "fp64" else torch.float32


def _prec(case):
    return T.TR_PREC_FP64 if case["prec"] == "fp64" else T.TR_PREC_MIXED


def _tensor(case, seed):
    """The data tensor: a random tensor ring plus noise, or smooth content."""
    dims = _ints(case["dims"])
    if case.get("data") == "cosine":
        return inputs.cosine_sum(dims, seed, device=DEV, dtype=_dtype(case))
    return inputs.tr_plus_noise(dims, _ints(case["ranks"]), seed, case.get("noise", 1e-2),
                                device=DEV, dtype=_dtype(case))[0]


def _start_cores(case, seed):
    """N(0, 1) initial cores, FP64, slice-major (I, Rl, Rr)."""
    cores = inputs.random_cores(_ints(case["dims"]), _ints(case["ranks"]), seed + 1)
    return [inputs.slice_major(c).to(DEV) for c in cores]


def _near_cores(case, seed):
    """The cores that made the tensor, 2 % off: what a converged decomposition holds."""
    cores = inputs.random_cores(_ints(case["dims"]), _ints(case["ranks"]), seed)
    off = inputs.random_cores(_ints(case["dims"]), _ints(case["ranks"]), seed + 1)
    return [inputs.slice_major(c + 0.02 * e).to(DEV) for c, e in zip(cores, off)]


def _others(N, k):
    return [(k + 1 + m) % N for m in range(N - 1)]


def _flat_cores(shapes):
    """One FP64 buffer for many cores, each on a 256-byte boundary, and the views."""
    sizes = [(math.prod(s) + 31) // 32 * 32 for s in shapes]
    flat = torch.zeros(sum(sizes), dtype=torch.float64, device=DEV)
    views, at = [], 0
    for s, n in zip(shapes, sizes):
        views.append(flat[at:at + math.prod(s)].view(s))
        at += n
    return flat, views


def _core_shapes(dims, ranks):
    return [(dims[k], ranks[k - 1], ranks[k]) for k in range(len(dims))]


def _batch(case):
    """Sizes of a batch: three modes of 32 to 200, ranks of 3 to 8."""
    r = random.Random(case["shapes"])
    return [(tuple(r.randint(32, 200) for _ in range(3)), tuple(r.randint(3, 8) for _ in range(3)))
            for _ in range(case["count"])]


def _requests(case):
    return inputs.serving_requests(case["count"], case["shapes"], emax=case["emax"])


def prepare(case, seed):
    kind = case["kind"]
    s = dict(case=case, seed=seed)
    if kind == "served":
        reqs = _requests(case)
        s["server"] = T.Server(max_slots=max(8, case["count"]), arena_bytes=2 << 30,
                               max_sweeps=case["sweeps"], fit_tol=0.0)
        s["reqs"] = []
        for i, r in enumerate(reqs):
            X, _ = inputs.tr_plus_noise(r["dims"], r["ranks"], seed * 1009 + i, 1e-2, device=DEV)
            flat, views = _flat_cores(_core_shapes(r["dims"], r["ranks"]))
            s["reqs"].append((X, r["ranks"], r["J"], seed + i, views, flat))
        torch.cuda.synchronize()
        s["server"].start()
        return s
    s["ctx"] = T.Context(0)
    if kind == "batched":
        shapes = _batch(case)
        s["flat"], views = _flat_cores([c for d, r in shapes for c in _core_shapes(d, r)])
        s["probs"] = [dict(X=inputs.tr_plus_noise(d, r, seed * 1009 + i, 1e-3, device=DEV)[0],
                           ranks=r, J=10 * _lmax(r), seed=seed + i, cores=views[3 * i:3 * i + 3])
                      for i, (d, r) in enumerate(shapes)]
        return s
    dims, ranks = _ints(case["dims"]), _ints(case["ranks"])
    s["X"] = _tensor(case, seed)
    if kind == "error":
        s["cores"] = _near_cores(case, seed)
        return s
    s["init"] = _start_cores(case, seed)
    if kind == "update":
        k, J, dt, N = case["mode"], case["J"], _dtype(case), len(dims)
        s["p"] = [torch.empty(d, dtype=torch.float64, device=DEV) for d in dims]
        s["cdf"] = [torch.empty(d, dtype=torch.float64, device=DEV) for d in dims]
        s["idx"] = torch.empty((J, N - 1), dtype=torch.int32, device=DEV)
        s["w"] = torch.empty(J, dtype=torch.float64, device=DEV)
        s["A"] = torch.empty((J, ranks[k - 1] * ranks[k]), dtype=dt, device=DEV)
        s["Y"] = torch.empty((J, dims[k]), dtype=dt, device=DEV)
        s["core"] = torch.empty((dims[k], ranks[k - 1], ranks[k]), dtype=torch.float64, device=DEV)
        return s
    s["cores"] = T.empty_cores(dims, ranks, device=DEV)
    if case.get("sampling") == "uniform":
        T.tr_set_sampling(s["ctx"], T.TR_SAMPLING_UNIFORM)
    return s


# --------------------------------------------------------------------------------------
# One pass
# --------------------------------------------------------------------------------------
def _kept(case, cores):
    return list(cores) if case["prec"] == "fp64" else [c.float() for c in cores]


def _going_on(call):
    """A singular update keeps its core and the decomposition goes on; the status says so."""
    try:
        call()
    except T.TrError as e:
        if e.status != T.TR_ERR_SINGULAR:
            raise


def run(s):
    case = s["case"]
    kind = case["kind"]
    if kind == "served":
        srv = s["server"]
        tickets = [srv.submit(X, ranks, J, seed, cores) for X, ranks, J, seed, cores, _ in s["reqs"]]
        fits = []
        for t in tickets:
            fits.append(srv.wait(t)["fit"])
            srv.release(t)
        return [flat.float() for *_, flat in s["reqs"]] + fits
    ctx, prec = s["ctx"], _prec(case)
    if kind == "batched":
        _going_on(lambda: T.tr_als_sampled_batched(ctx, s["probs"], case["sweeps"], prec))
        return [s["flat"].float()]
    dims, ranks, X = _ints(case["dims"]), _ints(case["ranks"]), s["X"]
    if kind == "error":
        return [T.tr_rel_error(ctx, X, ranks, s["cores"])]
    if kind == "update":
        k, J = case["mode"], case["J"]
        for m in _others(len(dims), k):
            T.tr_leverage(ctx, s["init"][m], s["p"][m], s["cdf"][m])
        T.tr_sample(ctx, k, dims, s["p"], s["cdf"], J, s["seed"], k, s["idx"], s["w"])
        T.tr_subchain(ctx, k, dims, ranks, s["init"], s["idx"], s["w"], s["A"])
        T.tr_gather(ctx, X, k, s["idx"], s["w"], s["Y"])
        T.tr_solve(ctx, s["A"], s["Y"], ranks[k - 1], ranks[k], prec, s["core"])
        out = [s["p"][m] for m in _others(len(dims), k)] + [s["cdf"][m] for m in _others(len(dims), k)]
        return out + [s["idx"], s["w"], s["A"], s["Y"]] + _kept(case, [s["core"]])
    if kind == "dense":
        _going_on(lambda: T.tr_als(ctx, X, ranks, 1, s["seed"], prec, s["cores"],
                                   init_cores=s["init"]))
    else:
        _going_on(lambda: T.tr_als_sampled(ctx, X, ranks, case["J"], case["sweeps"], s["seed"],
                                           prec, s["cores"], init_cores=s["init"]))
    err = T.tr_rel_error(ctx, X, ranks, s["cores"])
    return _kept(case, s["cores"]) + [err]


# --------------------------------------------------------------------------------------
# What a pass cannot do without
# --------------------------------------------------------------------------------------
def _split_k(dims, ranks):
    """The fewest products per entry of a reconstruction: the rank pair at the cheapest cut."""
    return min(ranks[-1] * ranks[m] for m in range(len(dims) - 1))


def _ls_flops(J, L, I):
    return J * L * (L + 2 * I) + L ** 3 / 3 + 2 * L * L * I


def _sampled_work(dims, ranks, J, sweeps, es, leverage):
    """Bytes of the fibres read (each of the J rows of X once per update) and of the cores;
    operations of the rows, the normal equations, the solves and the leverage scores."""
    b = f = 0.0
    for k in range(len(dims)):
        L, I = ranks[k - 1] * ranks[k], dims[k]
        others = _others(len(dims), k)
        chain = sum(2 * ranks[k] * ranks[m - 1] * ranks[m] for m in others[1:])
        b += sweeps * J * I * es + 8 * I * L * (sweeps + 1)
        f += sweeps * (J * chain + _ls_flops(J, L, I))
        if leverage:
            f += sweeps * (2 * I * L * L + L ** 3 / 3)
    return b, f


def work(case):
    kind = case["kind"]
    if kind == "served":
        b = f = 0.0
        for r in _requests(case):
            n = math.prod(r["dims"])
            x, y = _sampled_work(r["dims"], r["ranks"], r["J"], case["sweeps"], 4, True)
            b += x + case["sweeps"] * 4 * n
            f += y + case["sweeps"] * 2 * n * _split_k(r["dims"], r["ranks"])
        return dict(bytes=b, flops=f)
    if kind == "batched":
        each = [_sampled_work(d, r, 10 * _lmax(r), case["sweeps"], 4, True)
                for d, r in _batch(case)]
        return dict(bytes=sum(b for b, _ in each), flops=sum(f for _, f in each))
    dims, ranks = _ints(case["dims"]), _ints(case["ranks"])
    es = 8 if case["prec"] == "fp64" else 4
    n = math.prod(dims)
    core_bytes = 8 * sum(math.prod(c) for c in _core_shapes(dims, ranks))
    error = dict(bytes=n * es + core_bytes, flops=2 * n * _split_k(dims, ranks))
    if kind == "error":
        return error
    if kind == "update":
        k, J = case["mode"], case["J"]
        L, I = ranks[k - 1] * ranks[k], dims[k]
        others = _others(len(dims), k)
        lev = [(dims[m], ranks[m - 1] * ranks[m]) for m in others]
        chain = sum(2 * ranks[k] * ranks[m - 1] * ranks[m] for m in others[1:])
        b = J * I * es * 2 + J * L * es + core_bytes + J * (8 + 4 * (len(dims) - 1))
        f = J * chain + _ls_flops(J, L, I) + sum(2 * a * c * c + c ** 3 / 3 for a, c in lev)
        return dict(bytes=b, flops=f)
    if kind == "dense":
        f = sum(n // dims[k] * (2 * ranks[k] * ranks[k - 1] * ranks[k - 2])
                + _ls_flops(n // dims[k], ranks[k - 1] * ranks[k], dims[k])
                for k in range(len(dims)))
        return dict(bytes=len(dims) * n * es + 2 * core_bytes + error["bytes"],
                    flops=f + error["flops"])
    b, f = _sampled_work(dims, ranks, case["J"], case["sweeps"], es,
                         case["sampling"] == "leverage")
    return dict(bytes=b + error["bytes"], flops=f + error["flops"])


# --------------------------------------------------------------------------------------
# The same in 64 bits, with torch alone
# --------------------------------------------------------------------------------------
def _philox(c0, c1, c2, c3, k0, k1):
    """Philox4x32-10 (Salmon et al., SC'11) on int64 tensors that hold 32-bit words."""
    M = 0xFFFFFFFF
    for r in range(10):
        p0, p1 = c0 * 0xD2511F53, c2 * 0xCD9E8D57      # the low 64 bits of the products
        c0, c1, c2, c3 = (((p1 >> 32) & M) ^ c1 ^ k0, p1 & M, ((p0 >> 32) & M) ^ c3 ^ k1, p0 & M)
        k0, k1 = (k0 + 0x9E3779B9) & M, (k1 + 0xBB67AE85) & M
    return c0, c1, c2, c3


def _uniforms(J, npos, seed, update_id):
    """u[j][m]: the top 53 bits of words (2(m%2), 2(m%2)+1) of block (j, m/2, update id)."""
    j = torch.arange(J, dtype=torch.int64, device=DEV)
    cols = []
    for m in range(npos):
        z = torch.zeros_like(j)
        w = _philox(j, z + m // 2, z + (update_id & 0xFFFFFFFF), z + (update_id >> 32),
                    seed & 0xFFFFFFFF, (seed >> 32) & 0xFFFFFFFF)
        hi, lo = (w[2], w[3]) if m % 2 else (w[0], w[1])
        cols.append(((hi << 21) | (lo >> 11)).double() * 2.0 ** -53)
    return torch.stack(cols, 1)


def _distribution(core):
    """p and CDF from the leverage scores of the core's I x (Rl Rr) unfolding."""
    G = core.reshape(core.shape[0], -1)
    U, S, _ = torch.linalg.svd(G, full_matrices=False)
    keep = S > max(G.shape) * np.finfo(np.float64).eps * S.max()
    ell = (U[:, keep] ** 2).sum(1)
    p = ell / ell.sum()
    return p, torch.cumsum(p, 0)


def _draws(ps, cdfs, dims, k, J, seed, update_id, uniform):
    others = _others(len(dims), k)
    u = _uniforms(J, len(others), seed, update_id)
    idx, q = [], torch.ones(J, dtype=torch.float64, device=DEV)
    for m, mode in enumerate(others):
        if uniform:
            i = (u[:, m] * dims[mode]).long().clamp(max=dims[mode] - 1)
            q = q / dims[mode]
        else:
            i = torch.searchsorted(cdfs[mode], u[:, m].contiguous(), right=True)
            i = i.clamp(max=dims[mode] - 1)
            q = q * ps[mode][i]
        idx.append(i)
    return torch.stack(idx, 1), 1.0 / torch.sqrt(J * q)


def _rows(cores, k, idx):
    """Slice products around the ring, column a + Rl b = entry (b, a)."""
    others = _others(len(cores), k)
    S = cores[others[0]][idx[:, 0]]
    for m, mode in enumerate(others[1:], 1):
        S = torch.bmm(S, cores[mode][idx[:, m]])
    return S.reshape(S.shape[0], -1)


def _fibres(X, k, idx):
    at = [None] * X.dim()
    for m, mode in enumerate(_others(X.dim(), k)):
        at[mode] = idx[:, m][:, None]
    at[k] = torch.arange(X.shape[k], device=DEV)[None, :]
    return X[tuple(at)].double()


def _ls_core(A, Y, Rl, Rr):
    """The minimiser of ||A Z - Y|| by a QR factorisation, as a core (I, Rl, Rr)."""
    Q, R = torch.linalg.qr(A)
    Z = torch.linalg.solve_triangular(R, Q.T @ Y, upper=True)
    return Z.T.reshape(-1, Rr, Rl).transpose(1, 2).contiguous()


def _error(X, cores):
    """||TR - X|| / ||X||, in slabs along the first mode."""
    right = cores[1]                                   # (P, R_0, R_j), built mode by mode
    for c in cores[2:]:
        right = torch.einsum("pab,ibc->piac", right, c).reshape(-1, right.shape[1], c.shape[2])
    W = right.permute(2, 1, 0).reshape(-1, right.shape[0])          # (R_last R_0) x P
    left = cores[0].reshape(cores[0].shape[0], -1)                  # I_0 x (R_last R_0)
    se = sx = 0.0
    Xm = X.reshape(X.shape[0], -1)
    for i in range(0, X.shape[0], 64):
        x = Xm[i:i + 64].double()
        se += float((left[i:i + 64] @ W - x).square().sum())
        sx += float(x.square().sum())
    return math.sqrt(se / sx)


def _dense_core(X, cores, k):
    """Alg. 1's core update: every row, weight 1, the normal equations in slabs of rows."""
    dims = X.shape
    N = len(dims)
    L = cores[k].shape[1] * cores[k].shape[2]
    P = math.prod(dims) // dims[k]
    modes = [m for m in range(N) if m != k]
    Xk = X.movedim(k, N - 1)
    M = torch.zeros((L, L), dtype=torch.float64, device=DEV)
    B = torch.zeros((L, dims[k]), dtype=torch.float64, device=DEV)
    flat = Xk.reshape(P, dims[k])
    for r in range(0, P, 65536):
        rest = torch.arange(r, min(P, r + 65536), device=DEV)
        at = {}
        for m in reversed(modes):
            at[m] = rest % dims[m]
            rest = rest // dims[m]
        A = _rows(cores, k, torch.stack([at[m] for m in _others(N, k)], 1))
        M += A.T @ A
        B += A.T @ flat[r:r + 65536].double()
    Z = torch.cholesky_solve(B, torch.linalg.cholesky(M))
    return Z.T.reshape(dims[k], cores[k].shape[2], cores[k].shape[1]).transpose(1, 2).contiguous()


def exact(case, seed):
    """None where draws follow cores that were rounded to FP32 (mixed decompositions by
    leverage scores: a rounding that moves one draw moves every core after it)."""
    kind = case["kind"]
    if kind in ("batched", "served"):
        return None
    if kind == "als" and case["prec"] == "mixed" and case["sampling"] == "leverage":
        return None
    dims, ranks = _ints(case["dims"]), _ints(case["ranks"])
    N = len(dims)
    X = _tensor(case, seed)
    if kind == "error":
        return [_error(X, _near_cores(case, seed))]
    cores = _start_cores(case, seed)
    if kind == "update":
        k, J = case["mode"], case["J"]
        ps, cdfs = [None] * N, [None] * N
        for m in _others(N, k):
            ps[m], cdfs[m] = _distribution(cores[m])
        idx, w = _draws(ps, cdfs, dims, k, J, seed, k, False)
        A = _rows(cores, k, idx) * w[:, None]
        Y = _fibres(X, k, idx) * w[:, None]
        out = [ps[m] for m in _others(N, k)] + [cdfs[m] for m in _others(N, k)]
        return out + [None, w, A, Y, _ls_core(A, Y, ranks[k - 1], ranks[k])]
    if kind == "dense":
        for k in range(N):
            cores[k] = _dense_core(X, cores, k)
        return cores + [_error(X, cores)]
    uniform = case["sampling"] == "uniform"
    ps, cdfs = [None] * N, [None] * N
    if not uniform:
        for k in range(1, N):
            ps[k], cdfs[k] = _distribution(cores[k])
    for s in range(case["sweeps"]):
        for k in range(N):
            idx, w = _draws(ps, cdfs, dims, k, case["J"], seed, s * N + k, uniform)
            A = _rows(cores, k, idx) * w[:, None]
            Y = _fibres(X, k, idx) * w[:, None]
            cores[k] = _ls_core(A, Y, ranks[k - 1], ranks[k])
            if not uniform:
                ps[k], cdfs[k] = _distribution(cores[k])
    return cores + [_error(X, cores)]
