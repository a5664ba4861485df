"""What a user of libsymnmf runs, as cases that can be timed and compared.

Each case is one call sequence through the public entry points
(``paper_2607_24518_gb300.symnmf``, the names of include/symnmf.h): a solve,
a gradient, a dependence build, rolling windows, spherical K-means, a
monitor's objective, a batch of solves, and the way from an FP32 matrix to a
first gradient in FP8 storage.  Sizes are those of the bench workloads and
the tests (n = 512 and 20000, k = 8 / 32 / 64, T = 500, batches of handles
with restarts) and generic ones between, odd sizes included.

Inputs are absolute correlations of a market-and-sectors factor model, drawn
on the GPU from the seed; ``exact`` repeats each path in 64-bit torch from
the same inputs.
"""
from __future__ import annotations

import math

import torch

from paper_2607_24518_gb300 import symnmf as L

DT = {"f32": L.F32, "bf16": L.BF16, "fp8": L.FP8E4M3}
ES = {"f32": 4, "bf16": 2, "fp8": 1}
METHODS = {"adagrad": L.ADAGRAD, "rmsprop": L.RMSPROP, "piecewise": L.PIECEWISE_ADAGRAD,
           "row_svrg": L.ROW_SVRG, "block_svrg": L.BLOCK_SVRG_ADAPTGROW, "admm": L.ADMM}
# the library's default learning rates, but for RMSprop: its default takes
# ten iterations from H_0 straight to H = 0 at these sizes
ETA = {"rmsprop": 1e-3, "piecewise": 1.0}
TILE = 128


def _hp(method):
    return L.symnmf_hparams_default(METHODS[method], eta=ETA.get(method, 2.0))


def listed():
    return [
        # the smallest solve of the test suite, to where its trajectory is
        # compared: many short iterations, launches and latency count
        {"name": "solve_512", "kind": "solve", "n": 512, "k": 8, "dtype": "f32",
         "method": "adagrad", "iters": 50, "pitch": "tight"},
        # a universe of some thousand series handed over as it is: an odd
        # number of columns, rows without any alignment
        {"name": "solve_odd_3001", "kind": "solve", "n": 3001, "k": 10, "dtype": "f32",
         "method": "adagrad", "iters": 20, "pitch": "tight"},
        # the headline workload: full-batch AdaGrad on the FP32 matrix
        {"name": "solve_20000_f32", "kind": "solve", "n": 20000, "k": 32, "dtype": "f32",
         "method": "adagrad", "iters": 10, "pitch": "tight"},
        # the largest rank, the other first-order method, half the storage
        {"name": "solve_20000_k64_bf16", "kind": "solve", "n": 20000, "k": 64, "dtype": "bf16",
         "method": "rmsprop", "iters": 10, "pitch": "tight"},
        # the sampled method of the large FP8 runs: full passes and block
        # steps in turn
        {"name": "svrg_50000_fp8", "kind": "solve", "n": 50000, "k": 64, "dtype": "fp8",
         "method": "block_svrg", "iters": 10, "pitch": "tight"},
        # a caller with its own optimizer: gradient and objective at H
        {"name": "grad_30000_k64", "kind": "grad", "n": 30000, "k": 64, "dtype": "f32",
         "pitch": "tight"},
        # the solver's input from data: n variables, T = 500 observations
        {"name": "dependence_20000", "kind": "dependence", "n": 20000, "T": 500, "dtype": "f32",
         "center": True},
        # rolling windows: the next window's matrix into the handle, then a
        # few iterations from the factor at hand
        {"name": "rolling_10000", "kind": "rolling", "n": 10000, "k": 32, "T": 250,
         "dtype": "bf16", "iters": 10},
        # hard clusters of the same matrix
        {"name": "kmeans_20000", "kind": "kmeans", "n": 20000, "k": 32, "dtype": "bf16",
         "iters": 5, "pitch": "tight"},
        # a monitor's objective beside a solve, without allocation
        {"name": "monitor_10000", "kind": "monitor", "n": 10000, "k": 32, "dtype": "f32",
         "pitch": "tight"},
        # several instances of unequal size, two restarts each in one
        # handle, stepped together
        {"name": "batch_8", "kind": "batch", "count": 8, "n": 8000, "k": 16, "restarts": 2,
         "dtype": "bf16", "iters": 10},
        # a new problem in FP8 storage: quantise, open a handle, ||S||^2,
        # first gradient, close
        {"name": "store_12000", "kind": "store", "n": 12000, "k": 32, "src": "f32"},
    ]


def _logint(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["solve", "solve", "solve", "grad", "dependence", "rolling", "kmeans",
                       "monitor", "batch", "store"])
    dtype = rng.choice(["f32", "bf16", "fp8"])
    pitch = rng.choice(["tight", "padded"])
    if kind == "solve":
        n = _logint(rng, 300, 20000)
        return {"kind": kind, "n": n, "k": _logint(rng, 2, 64), "dtype": dtype,
                "method": rng.choice(sorted(METHODS)),
                "iters": 10 if n > 5000 else rng.randint(10, 30), "pitch": pitch}
    if kind == "grad":
        return {"kind": kind, "n": _logint(rng, 1000, 28000), "k": _logint(rng, 2, 64),
                "dtype": dtype, "pitch": pitch}
    if kind == "dependence":
        return {"kind": kind, "n": _logint(rng, 500, 20000), "T": _logint(rng, 40, 1000),
                "dtype": dtype, "center": rng.random() < 0.7}
    if kind == "rolling":
        return {"kind": kind, "n": _logint(rng, 500, 10000), "k": _logint(rng, 4, 64),
                "T": _logint(rng, 60, 500), "dtype": dtype, "iters": 10}
    if kind == "kmeans":
        return {"kind": kind, "n": _logint(rng, 1000, 18000), "k": _logint(rng, 4, 64),
                "dtype": dtype, "iters": rng.randint(2, 5), "pitch": pitch}
    if kind == "monitor":
        return {"kind": kind, "n": _logint(rng, 500, 20000), "k": _logint(rng, 2, 64),
                "dtype": dtype, "pitch": pitch}
    if kind == "batch":
        R = rng.choice([1, 2, 4])
        return {"kind": kind, "count": rng.randint(2, 8), "n": _logint(rng, 1000, 8000),
                "k": R * rng.randint(3, 64 // R), "restarts": R, "dtype": dtype, "iters": 10}
    return {"kind": kind, "n": _logint(rng, 1000, 12000), "k": _logint(rng, 2, 64),
            "src": rng.choice(["f32", "bf16"])}


# ------------------------------------------------------------------ inputs
def _gen(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed))
    return g


def _observations(n, T, seed):
    """T x n returns: market loadings U[0.4, 0.8], 24 sectors of loadings
    U[0, 0.5] at 10% density, unit noise."""
    g = _gen(seed)
    load = torch.zeros(25, n, device="cuda")
    load[0] = 0.4 + 0.4 * torch.rand(n, device="cuda", generator=g)
    on = torch.rand(24, n, device="cuda", generator=g) < 0.1
    load[1:] = 0.5 * torch.rand(24, n, device="cuda", generator=g) * on
    z = torch.randn(T, 25, device="cuda", generator=g)
    Y = torch.randn(T, n, device="cuda", generator=g)
    return Y.addmm_(z, load).mul_(0.01)


def _angles(n, T, seed):
    """T x n non-negative rows of unit norm: the angular parts of heavy-tailed
    exceedances, as the TPDM takes them."""
    g = _gen(seed)
    A = 0.2 + 0.8 * torch.rand(16, n, device="cuda", generator=g)
    A *= torch.rand(16, n, device="cuda", generator=g) < 0.2
    A[0] += 0.05
    X = torch.rand(T, 16, device="cuda", generator=g).clamp_min_(1e-6).pow_(-0.5) @ A
    return X / X.norm(dim=1, keepdim=True)


def _abs_corr(n, seed):
    """n x n |correlation| in FP32, exactly symmetric, unit diagonal, over a
    window of 128 observations."""
    X = _observations(n, 128, seed)
    X = X - X.mean(dim=0)
    X = X / X.norm(dim=0)
    S = X.T @ X
    S.abs_().clamp_(max=1.0)
    for r in range(0, n, 4096):
        e = min(n, r + 4096)
        S[e:, r:e] = S[r:e, e:].T
        D = S[r:e, r:e]
        D.copy_(torch.triu(D, 1) + torch.triu(D, 1).T)
    S.fill_diagonal_(1.0)
    return S


def _quantise(S):
    """E4M3 codes of S (same storage shape, uint8) and the power-of-two scale
    of every 128 x 128 tile: the smallest with max|tile| / scale <= 448."""
    n = S.shape[0]
    nt = -(-n // TILE)
    q = torch.empty(n, n, dtype=torch.uint8, device="cuda")
    sc = torch.empty(nt, nt, dtype=torch.float32, device="cuda")
    for t in range(nt):
        r, e = t * TILE, min(n, (t + 1) * TILE)
        row = torch.zeros(e - r, nt * TILE, device="cuda")
        row[:, :n] = S[r:e]
        amax = row.abs().amax(dim=0).reshape(nt, TILE).amax(dim=1)
        m, x = torch.frexp(amax)
        x = x - 9 + (m > 0.875).to(x.dtype)
        s = torch.where(amax > 0, torch.ldexp(torch.ones_like(amax), x), torch.ones_like(amax))
        sc[t] = s
        row /= s.repeat_interleave(TILE)
        q[r:e] = row[:, :n].to(torch.float8_e4m3fn).view(torch.uint8)
    return q, sc


def _dequantise(q, sc):
    n = q.shape[0]
    S = torch.empty(n, n, dtype=torch.float64, device="cuda")
    for t in range(sc.shape[0]):
        r, e = t * TILE, min(n, (t + 1) * TILE)
        S[r:e] = q[r:e].view(torch.float8_e4m3fn).to(torch.float64)
        S[r:e] *= sc[t].double().repeat_interleave(TILE)[:n]
    return S


def _stored(S32, dtype, pitch):
    """The matrix as the caller stores it: (tensor, row pitch, scales)."""
    n = S32.shape[0]
    scales = None
    if dtype == "bf16":
        S = S32.to(torch.bfloat16)
    elif dtype == "fp8":
        S, scales = _quantise(S32)
    else:
        S = S32
    lds = n
    if pitch == "padded":  # rows on 16-byte boundaries
        lds = -(-n * ES[dtype] // 16) * 16 // ES[dtype]
        if lds != n:
            P = torch.zeros(n, lds, dtype=S.dtype, device="cuda")
            P[:, :n] = S
            S = P
    return S, lds, scales


def _stored64(case, seed):
    S32 = _abs_corr(case["n"], seed)
    if case["dtype"] == "f32":
        return S32.double()
    if case["dtype"] == "bf16":
        return S32.to(torch.bfloat16).double()
    return _dequantise(*_quantise(S32))


def _h0(n, k, seed, mean=0.3):
    """H_0 ~ U[0, sqrt(mean(S) / k)]"""
    g = _gen(seed * 2654435761 + 17)
    return torch.rand(n, k, device="cuda", generator=g) * math.sqrt(mean / k)


def _labels0(S32, k, seed):
    """Initial clusters: every row joins the seed row it depends on most."""
    rows = torch.randperm(S32.shape[0], generator=_gen(seed + 5), device="cuda")[:k]
    return S32[:, rows].argmax(dim=1).to(torch.int32)


class _Handle:
    """A solver handle that goes with the state that holds it."""

    def __init__(self, S, n, lds, k, dtype, scales=None, stream=None):
        self.keep = (S, scales, stream)
        self.h = (L.symnmf_create(S, n, k, DT[dtype]) if lds == n else
                  L.symnmf_create_ld(S, n, lds, k, DT[dtype]))
        if scales is not None:
            L.symnmf_set_tile_scales(self.h, scales, scales.shape[1])
        if stream is not None:
            L.symnmf_set_stream(self.h, stream)

    def __del__(self):
        if getattr(self, "h", None) is not None:
            L.symnmf_destroy(self.h)
            self.h = None


def _batch_sizes(case):
    """Unequal sizes from n / 4 to n, and the rank of each (the restarts of
    one instance side by side)."""
    c = case["count"]
    return [case["n"] // 4 + (3 * case["n"] // 4) * (i + 1) // c for i in range(c)]


def prepare(case, seed):
    kind, n = case["kind"], case["n"]
    st = {"case": case}
    new = lambda *shape, dt=torch.float32: torch.empty(*shape, dtype=dt, device="cuda")  # noqa: E731
    if kind in ("solve", "grad", "kmeans"):
        k = case["k"]
        S32 = _abs_corr(n, seed)
        if kind == "kmeans":
            st["labels0"] = _labels0(S32, k, seed)
            st["labels"] = new(n, dt=torch.int32)
        S, lds, scales = _stored(S32, case["dtype"], case["pitch"])
        del S32
        st["handle"] = _Handle(S, n, lds, k, case["dtype"], scales)
        st["H0"] = _h0(n, k, seed)
        if kind != "kmeans":
            st["out"] = [new(n, k) for _ in range(3)]
        if kind == "solve":
            st["hp"] = _hp(case["method"])
        if kind == "grad":
            L.symnmf_set_H(st["handle"].h, st["H0"])
    elif kind == "dependence":
        st["Y"] = (_observations if case["center"] else _angles)(n, case["T"], seed)
        st["lds"] = -(-n * ES[case["dtype"]] // 16) * 16 // ES[case["dtype"]]
        tdt = {"f32": torch.float32, "bf16": torch.bfloat16, "fp8": torch.uint8}[case["dtype"]]
        st["S"] = torch.zeros(n, st["lds"], dtype=tdt, device="cuda")
        nt = -(-n // TILE)
        st["scales"] = new(nt, nt) if case["dtype"] == "fp8" else None
        st["norm"] = new(1, dt=torch.float64)
    elif kind == "rolling":
        T, k = case["T"], case["k"]
        st["stride"] = max(1, T // 5)
        st["Y"] = _observations(n, T + st["stride"], seed)
        es = ES[case["dtype"]]
        st["lds"] = -(-n * es // 16) * 16 // es
        tdt = {"f32": torch.float32, "bf16": torch.bfloat16, "fp8": torch.uint8}[case["dtype"]]
        S = torch.zeros(n, st["lds"], dtype=tdt, device="cuda")
        nt = -(-n // TILE)
        scales = new(nt, nt) if case["dtype"] == "fp8" else None
        L.symnmf_build_dependence(st["Y"], T, n, n, 1, DT[case["dtype"]], S, st["lds"], scales, nt)
        st["S"], st["scales"] = S, scales
        st["handle"] = _Handle(S, n, st["lds"], k, case["dtype"], scales)
        st["H0"] = _h0(n, k, seed)
        st["hp"] = _hp("adagrad")
        st["out"] = [new(n, k) for _ in range(2)]
    elif kind == "monitor":
        S32 = _abs_corr(n, seed)
        st["norm"] = float(S32.double().square().sum())
        st["S"], st["lds"], st["scales"] = _stored(S32, case["dtype"], case["pitch"])
        st["H"] = _h0(n, case["k"], seed)
        st["f"] = new(1, dt=torch.float64)
    elif kind == "batch":
        st["items"] = []
        for i, m in enumerate(_batch_sizes(case)):
            S, lds, scales = _stored(_abs_corr(m, seed + 101 * i), case["dtype"], "padded")
            hd = _Handle(S, m, lds, case["k"], case["dtype"], scales, torch.cuda.Stream())
            L.symnmf_set_restarts(hd.h, case["restarts"])
            st["items"].append((hd, _h0(m, case["k"], seed + i), new(m, case["k"]),
                                new(m, case["k"])))
        st["hps"] = [_hp("piecewise") for _ in st["items"]]
    else:
        S = _abs_corr(n, seed)
        st["S"] = S if case["src"] == "f32" else S.to(torch.bfloat16)
        nt = -(-n // TILE)
        st["lds"] = -(-n // 16) * 16
        st["q"] = torch.zeros(n, st["lds"], dtype=torch.uint8, device="cuda")
        st["scales"], st["sumsq"] = new(nt, nt), new(nt, nt, dt=torch.float64)
        st["H"], st["G"] = _h0(n, case["k"], seed), new(n, case["k"])
    torch.cuda.synchronize()
    return st


# --------------------------------------------------------------------- run
def run(st):
    case = st["case"]
    kind, n = case["kind"], case["n"]
    if kind == "solve":
        h, (H, acc, g) = st["handle"].h, st["out"]
        L.symnmf_set_H(h, st["H0"])
        _, stats = L.symnmf_step(h, st["hp"], case["iters"])
        L.symnmf_get_H(h, H)
        L.symnmf_get_buffer(h, L.BUF_ACC, acc)
        L.symnmf_get_buffer(h, L.BUF_GRAD, g)
        return {"H": H, "acc": acc, "grad": g, "E": stats.E, "kkt": stats.kkt}
    if kind == "grad":
        h, G = st["handle"].h, st["out"][0]
        L.symnmf_grad(h, G)
        f, E = L.symnmf_objective(h)
        return {"G": G, "f": f, "E": E}
    if kind == "dependence":
        L.symnmf_build_dependence(st["Y"], case["T"], n, n, int(case["center"]),
                                  DT[case["dtype"]], st["S"], st["lds"], st["scales"],
                                  -(-n // TILE), st["norm"])
        return {"S": st["S"], "scales": st["scales"], "norm": st["norm"]}
    if kind == "rolling":
        h, T = st["handle"].h, case["T"]
        L.symnmf_set_H(h, st["H0"])
        L.symnmf_window_update(h, st["Y"][st["stride"]:], T, n, 1, st["S"], st["lds"],
                               st["scales"], -(-n // TILE))
        _, stats = L.symnmf_step(h, st["hp"], case["iters"])
        L.symnmf_get_H(h, st["out"][0])
        L.symnmf_get_buffer(h, L.BUF_ACC, st["out"][1])
        return {"H": st["out"][0], "acc": st["out"][1], "E": stats.E}
    if kind == "kmeans":
        stats, _ = L.symnmf_spkmeans(st["handle"].h, st["labels0"], st["labels"], case["iters"],
                                     0.0, trace=False)
        return {"labels": st["labels"], "J": stats.J}
    if kind == "monitor":
        L.symnmf_objective_noalloc(st["S"], n, st["lds"], DT[case["dtype"]], st["scales"],
                                   -(-n // TILE), st["H"], case["k"], st["norm"], st["f"])
        return {"f": st["f"]}
    if kind == "batch":
        for hd, H0, _, _ in st["items"]:
            L.symnmf_set_H(hd.h, H0)
        _, stats = L.symnmf_batch_step([it[0].h for it in st["items"]], st["hps"], case["iters"])
        for hd, _, H, acc in st["items"]:
            L.symnmf_get_H(hd.h, H)
            L.symnmf_get_buffer(hd.h, L.BUF_ACC, acc)
        return {"H": [it[2] for it in st["items"]], "acc": [it[3] for it in st["items"]],
                "E": [s.E for s in stats]}
    nt = -(-n // TILE)
    L.symnmf_quantize_fp8(st["S"], DT[case["src"]], n, n, n, st["q"], st["lds"], st["scales"], nt,
                          st["sumsq"])
    h = L.symnmf_create_ld(st["q"], n, st["lds"], case["k"], L.FP8E4M3)
    L.symnmf_set_tile_scales(h, st["scales"], nt)
    norm = L.symnmf_get_norm(h)
    L.symnmf_set_H(h, st["H"])
    L.symnmf_grad(h, st["G"])
    L.symnmf_destroy(h)
    return {"q": st["q"], "scales": st["scales"], "sumsq": st["sumsq"], "norm": norm, "G": st["G"]}


# -------------------------------------------------------------------- work
def work(case):
    kind, n = case["kind"], case["n"]
    k = case.get("k", 0)
    if kind == "solve":
        # S once per full pass; a block step needs phi of it, a row step half
        share = {"row_svrg": 0.55, "block_svrg": 0.75}.get(case["method"], 1.0)
        one = ES[case["dtype"]] * n * n * share + 16 * n * k
        return {"bytes": case["iters"] * one, "flops": case["iters"] * share * 2.0 * n * n * k}
    if kind == "grad":
        return {"bytes": 2.0 * ES[case["dtype"]] * n * n + 12.0 * n * k, "flops": 4.0 * n * n * k}
    if kind == "dependence":
        return {"bytes": 4.0 * case["T"] * n + ES[case["dtype"]] * n * n,
                "flops": 1.0 * n * n * case["T"]}
    if kind == "rolling":
        # the window's matrix written once and read by every iteration
        it = case["iters"]
        return {"bytes": (1.0 + it) * ES[case["dtype"]] * n * n + 4 * case["T"] * n
                + it * 16 * n * k, "flops": 1.0 * n * n * case["T"] + it * 2.0 * n * n * k}
    if kind == "kmeans":
        return {"bytes": case["iters"] * 2.0 * ES[case["dtype"]] * n * n,
                "flops": case["iters"] * 2 * 2.0 * n * n * k}
    if kind == "monitor":
        return {"bytes": 1.0 * ES[case["dtype"]] * n * n + 4.0 * n * k, "flops": 2.0 * n * n * k}
    if kind == "batch":
        n2 = float(sum(m * m for m in _batch_sizes(case)))
        return {"bytes": case["iters"] * ES[case["dtype"]] * n2,
                "flops": case["iters"] * 2.0 * n2 * k}
    # source read once, codes written once and read by ||S||^2 and the gradient
    return {"bytes": (ES[case["src"]] + 3.0) * n * n, "flops": 2.0 * n * n * k}


def tolerance(case):
    """About four times what the paths were seen to differ from their 64-bit
    values: FP32 sums of FP32 / BF16 products (3e-6 in gradients and states;
    after RMSprop's and ADMM's steps the gradient is a small difference of its
    terms, 1e-4 off), H as two E4M3 pieces with FP8 storage (8e-5; 7e-3 and
    single entries of ADMM's dual 0.1 off), the long tensor-core sums of the
    dependence matrix (1.5e-5), the monitor's FP64 cross-tile sums (6e-9).
    BF16 values may round to the next one, E4M3 codes and the labels of near
    ties likewise."""
    kind, dtype = case["kind"], case.get("dtype", "fp8")
    if kind == "monitor":
        return {"rel": 2.5e-8}
    if kind == "kmeans":
        return {"rel": 1e-4, "differ": 5e-3}
    if kind == "dependence":
        return ({"rel": 6e-4, "max": 1e-2} if dtype == "bf16" else
                {"rel": 6e-5, "max": 1e-3, "differ": 1e-3})
    if case.get("method") in ("rmsprop", "admm"):
        return {"rel": 0.025, "max": 0.4} if dtype == "fp8" else {"rel": 5e-4, "max": 1e-2}
    return {"rel": 4e-4, "max": 1e-2} if dtype == "fp8" else {"rel": 1.2e-5, "max": 1e-2}


# ------------------------------------------------------------------- exact
_M64 = (1 << 64) - 1


def _sample(t, stream, nb, m):
    """m of nb blocks for iteration t (seed 0): SplitMix64 draws, partial
    Fisher-Yates, sorted."""
    def mix(z):
        z = ((z ^ (z >> 30)) * 0xBF58476D1CE4E5B9) & _M64
        z = ((z ^ (z >> 27)) * 0x94D049BB133111EB) & _M64
        return z ^ (z >> 31)
    st = (t * 0xBF58476D1CE4E5B9 + stream * 0x94D049BB133111EB) & _M64
    perm, m = list(range(nb)), min(m, nb)
    for d in range(m):
        u = mix((st + (d + 1) * 0x9E3779B97F4A7C15) & _M64)
        j = d + u % (nb - d)
        perm[d], perm[j] = perm[j], perm[d]
    return sorted(perm[:m])


def _rows_of(blocks, n):
    return torch.cat([torch.arange(b * TILE, min(n, (b + 1) * TILE), device="cuda")
                      for b in blocks])


def _solve64(S, H, method, iters, norm=None, restarts=1):
    """The solver of the appendix in 64 bits: (H, accumulator, last gradient,
    E and KKT measure of the last check, t % 10 == 0)."""
    n, k = H.shape
    H = H.double()
    A, M = torch.zeros_like(H), torch.zeros_like(H)
    norm = float(S.square().sum()) if norm is None else norm
    mask = torch.ones(k, k, dtype=torch.float64, device="cuda")
    if restarts > 1:
        b = torch.arange(k, device="cuda") // (k // restarts)
        mask = (b[:, None] == b[None, :]).double()
    eta = ETA.get(method, 2.0)
    eps = 1e-8 if method == "rmsprop" else 1e-10
    period = {"row_svrg": 10, "block_svrg": 2}.get(method, 1)
    nb = -(-n // TILE)
    E = kkt = float("nan")
    mu = g = None
    for t in range(iters):
        if t % period == 0 or t % 10 == 0:
            P = S @ H
            gram = (H.T @ H) * mask
            g = 4.0 * (H @ gram - P)
            mu = g
            if t % 10 == 0:
                f = restarts * norm - 2.0 * float((H * P).sum()) + float(gram.square().sum())
                E = f / (restarts * norm)
                kkt = float(torch.where(H > 0, g, g.clamp(max=0.0)).norm()) / (n * k)
        elif method == "row_svrg":
            I = _rows_of(_sample(t, 0, nb, -(-math.ceil(0.5 * n) // TILE)), n)
            g = mu.clone()
            g[I] = 4.0 * (H[I] @ ((H.T @ H) * mask) - S[I] @ H)
        else:
            m = -(-math.ceil(math.sqrt(0.5) * n) // TILE)
            I, J = (_rows_of(_sample(t, s, nb, m), n) for s in (1, 2))
            g, est = mu.clone(), torch.zeros_like(mu)
            g[I] = 0.0
            g[J] = 0.0
            SIJ = S[I][:, J]
            est[I] += 2.0 * (H[I] @ ((H[J].T @ H[J]) * mask) - SIJ @ H[J])
            est[J] += 2.0 * (H[J] @ ((H[I].T @ H[I]) * mask) - SIJ.T @ H[I])
            del SIJ
            g += est
        if method == "admm":
            inv = torch.linalg.inv(2.0 * (H.T @ H) * mask
                                   + 500.0 * torch.eye(k, dtype=torch.float64, device="cuda"))
            x = (2.0 * P + 500.0 * (H - A)) @ inv + A
            H = x.clamp(min=0.0)
            A = x - H
        elif method == "rmsprop":
            A = 0.99 * A + 0.01 * g * g
            M = 0.5 * M + eta * g / (A.sqrt() + eps)
            H = (H - M).clamp(min=0.0)
        else:
            A = A + g * g
            H = (H - eta * g / (A.sqrt() + eps)).clamp(min=0.0)
    return H, A, g, E, kkt


def _depend64(Y, center):
    Y = Y.double()
    if center:
        Y = Y - Y.mean(dim=0)
    d = Y.square().sum(dim=0)
    Y = Y / torch.where(d > 0, d.sqrt(), torch.ones_like(d))
    S = Y.T @ Y
    S.abs_().clamp_(max=1.0).fill_diagonal_(1.0)
    return S


def exact(case, seed):
    kind, n = case["kind"], case["n"]
    if kind == "solve":
        H, A, g, E, kkt = _solve64(_stored64(case, seed), _h0(n, case["k"], seed), case["method"],
                                   case["iters"])
        return {"H": H, "acc": A, "grad": g, "E": E, "kkt": kkt}
    if kind == "grad":
        S, H = _stored64(case, seed), _h0(n, case["k"], seed).double()
        P, gram, norm = S @ H, H.T @ H, float(S.square().sum())
        f = norm - 2.0 * float((H * P).sum()) + float(gram.square().sum())
        return {"G": 4.0 * (H @ gram - P), "f": f, "E": f / norm}
    if kind == "dependence":
        S = _depend64((_observations if case["center"] else _angles)(n, case["T"], seed),
                      case["center"])
        norm = S.square().sum().reshape(1)
        es = ES[case["dtype"]]
        lds = -(-n * es // 16) * 16 // es
        if case["dtype"] == "fp8":  # codes are whole numbers: no 64-bit value
            nt = -(-n // TILE)
            pad = torch.zeros(n, nt * TILE, dtype=torch.float64, device="cuda")
            pad[:, :n] = S
            del S
            rows = torch.stack([pad[r * TILE:(r + 1) * TILE].amax(dim=0) for r in range(nt)])
            m, x = torch.frexp(rows.reshape(nt, nt, TILE).amax(dim=2).float())
            x = x - 9 + (m > 0.875).to(x.dtype)
            return {"S": None, "scales": torch.ldexp(torch.ones_like(m), x).double(), "norm": norm}
        if case["dtype"] == "bf16":
            S = S.to(torch.bfloat16).double()
            norm = S.square().sum().reshape(1)
        out = torch.zeros(n, lds, dtype=torch.float64, device="cuda")
        out[:, :n] = S
        return {"S": out, "scales": None, "norm": norm}
    if kind == "rolling":
        T, stride = case["T"], max(1, case["T"] // 5)
        S = _depend64(_observations(n, T + stride, seed)[stride:], True)
        if case["dtype"] == "bf16":
            S = S.to(torch.bfloat16).double()
        elif case["dtype"] == "fp8":
            S = _dequantise(*_quantise(S.float()))
        H, A, _, E, _ = _solve64(S, _h0(n, case["k"], seed), "adagrad", case["iters"])
        return {"H": H, "acc": A, "E": E}
    if kind == "kmeans":
        lab = _labels0(_abs_corr(n, seed), case["k"], seed).long()
        S = _stored64(case, seed)
        S /= S.norm(dim=1, keepdim=True)
        J = float("nan")
        for _ in range(case["iters"]):
            B = torch.zeros(n, case["k"], dtype=torch.float64, device="cuda")
            B[torch.arange(n, device="cuda"), lab] = 1.0
            C = S.T @ B  # S has unit rows here: column k sums cluster k's rows
            nc = C.norm(dim=0)
            cos = S @ torch.where(nc > 0, C / nc, torch.zeros_like(C))
            best, to = cos.max(dim=1)
            J, done = float((1.0 - best).sum()), bool((to == lab).all())
            lab = to
            if done:
                break
        return {"labels": None, "J": J}
    if kind == "monitor":
        S32 = _abs_corr(n, seed)
        norm = float(S32.double().square().sum())
        del S32
        S, H = _stored64(case, seed), _h0(n, case["k"], seed).double()
        f = norm - 2.0 * float((H * (S @ H)).sum()) + float((H.T @ H).square().sum())
        return {"f": torch.tensor([f], dtype=torch.float64)}
    if kind == "batch":
        Hs, As, Es = [], [], []
        for i, m in enumerate(_batch_sizes(case)):
            S = _stored64({"n": m, "dtype": case["dtype"]}, seed + 101 * i)
            H, A, _, E, _ = _solve64(S, _h0(m, case["k"], seed + i), "piecewise", case["iters"],
                                     restarts=case["restarts"])
            Hs.append(H)
            As.append(A)
            Es.append(E)
        return {"H": Hs, "acc": As, "E": Es}
    S32 = _abs_corr(n, seed)
    if case["src"] == "bf16":
        S32 = S32.to(torch.bfloat16).float()
    q, sc = _quantise(S32)
    nt = -(-n // TILE)
    pad = torch.zeros(nt * TILE, nt * TILE, dtype=torch.float64, device="cuda")
    pad[:n, :n] = S32
    sumsq = pad.reshape(nt, TILE, nt, TILE).square().sum(dim=(1, 3))
    del S32, pad
    S, H = _dequantise(q, sc), _h0(n, case["k"], seed).double()
    return {"q": None, "scales": sc.double(), "sumsq": sumsq, "norm": float(S.square().sum()),
            "G": 4.0 * (H @ (H.T @ H) - S @ H)}
