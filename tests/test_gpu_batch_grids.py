"""Handles stepped together take fewer CTAs per row tile the more tiles all of
them have.  Enough tiles that this binds (240 and more in all: down to one CTA
per row tile, where a handle alone takes several) against stepping every handle
alone: the same sums in another FP32 order.  AdaGrad runs with eta = 0.1 and
eps = 1e3, so a step moves an entry by at most eta / eps times the difference of
its gradients (with the default eps the first step is the gradient's sign).
Rows of S H are below 0.2 * 8000, so gradients differ by less than 2^-20 * 4 *
1600 = 6e-3, ten steps by 6e-6.  And once the others have stopped, the one left
runs as if it were alone, bit for bit."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


@pytest.fixture(scope="module")
def L():
    from paper_2607_24518_gb300 import build
    build.build()
    from paper_2607_24518_gb300 import symnmf
    return symnmf


def _matrix(n, seed):
    A = np.random.default_rng(seed).random((n, 6))
    return torch.tensor(np.minimum(1.0, A @ A.T / 3), dtype=torch.float32, device=DEV)


def _handle(L, S, k, dtype, keep):
    n = S.shape[0]
    if dtype == "fp8":
        nt, lds = -(-n // 128), -(-n // 16) * 16
        q = torch.zeros(n, lds, dtype=torch.uint8, device=DEV)
        sc = torch.zeros(nt, nt, device=DEV)
        L.symnmf_quantize_fp8(S, L.F32, n, n, n, q, lds, sc, nt, None)
        torch.cuda.synchronize()
        h = L.symnmf_create_ld(q, n, lds, k, L.FP8E4M3)
        L.symnmf_set_tile_scales(h, sc, nt)
        keep.append((q, sc))
        return h
    T = S.to({"f32": torch.float32, "bf16": torch.bfloat16}[dtype])
    keep.append(T)
    return L.symnmf_create(T, n, k, {"f32": L.F32, "bf16": L.BF16}[dtype])


def _H(L, h, n, k):
    out = torch.empty(n, k, device=DEV)
    L.symnmf_get_H(h, out)
    torch.cuda.synchronize()
    return out


@pytest.mark.parametrize("dtype,k,ns", [("f32", 8, (4000,) * 8), ("f32", 64, (3992, 2000, 4096) * 3),
                                        ("bf16", 32, (4000, 7992, 1000) * 3), ("fp8", 16, (3984, 8000) * 4),
                                        ("fp8", 64, (4000,) * 8)])
def test_batch_of_many_tiles_equals_handles_alone(L, dtype, k, ns):
    assert sum(-(-n // 128) for n in ns) >= 240
    mats = {n: _matrix(n, n) for n in set(ns)}
    keep, hs = [], []
    H0 = [torch.tensor(np.random.default_rng(i).uniform(0, 0.2, (n, k)), dtype=torch.float32, device=DEV)
          for i, n in enumerate(ns)]
    streams = [torch.cuda.Stream() for _ in ns]
    hp = L.symnmf_hparams_default(L.ADAGRAD, eta=0.1, eps=1e3)
    try:
        for n, st in zip(ns, streams):
            h = _handle(L, mats[n], k, dtype, keep)
            hs.append(h)
            L.symnmf_set_stream(h, st)
        torch.cuda.synchronize()
        for h, h0 in zip(hs, H0):
            L.symnmf_set_H(h, h0)
        torch.cuda.synchronize()
        L.symnmf_batch_step(hs, [hp] * len(hs), 10)
        together = [_H(L, h, n, k) for h, n in zip(hs, ns)]
        for h, n, h0, got in zip(hs, ns, H0, together):
            L.symnmf_set_H(h, h0)
            L.symnmf_step(h, hp, 10)
            alone = _H(L, h, n, k)
            assert float((got - alone).abs().max()) <= 6e-6
            assert float((got - h0).abs().max()) >= 1e-3  # it moved
    finally:
        for h in hs:
            L.symnmf_destroy(h)


@pytest.mark.parametrize("dtype,n,k", [("f32", 4000, 8), ("bf16", 8000, 32)])
def test_the_last_one_running_gets_its_grid_back(L, dtype, n, k):
    """Seven handles meet the stopping rule at their second check; the eighth
    goes on.  Its state after twelve iterations equals two in the batch and
    ten alone."""
    S = _matrix(n, 1)
    keep, hs, got = [], [], []
    H0 = torch.tensor(np.random.default_rng(2).uniform(0, 0.2, (n, k)), dtype=torch.float32, device=DEV)
    streams = [torch.cuda.Stream() for _ in range(8)]
    go = L.symnmf_hparams_default(L.ADAGRAD, eta=0.1)
    stop = L.symnmf_hparams_default(L.ADAGRAD, eta=0.1, tau_E=1e30, tau_g=1e30, tau_stag=1e30, warmup=0,
                                    check_interval=1)
    try:
        for st in streams:
            h = _handle(L, S, k, dtype, keep)
            hs.append(h)
            L.symnmf_set_stream(h, st)
        for split in (False, True):
            torch.cuda.synchronize()
            for h in hs:
                L.symnmf_set_H(h, H0)
            torch.cuda.synchronize()
            _, outs = L.symnmf_batch_step(hs, [stop] * 7 + [go], 2 if split else 12)
            assert [o.converged for o in outs] == [1] * 7 + [0]
            if split:
                L.symnmf_step(hs[7], go, 10)
            got.append(_H(L, hs[7], n, k))
    finally:
        for h in hs:
            L.symnmf_destroy(h)
    assert torch.equal(got[0], got[1])
