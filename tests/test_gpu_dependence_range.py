"""The dependence builder at the edges of its FP16 pieces and of its tile
list: columns whose magnitudes differ by 60 powers of ten (each has its own
power-of-two scale), columns without variance, outliers that push the other
entries of a column towards FP16's subnormals, and sizes around the group of
16 row tiles, the 256-column blocks and the 128-observation transposes.
Bounds as derived in test_gpu_dependence.py with the FP16 chain length:
2^-22 from the pieces plus 4 units of 2^-24 for each of the 3 T' / 16 chained
MMAs."""
import numpy as np
import pytest
import torch

from oracle import dependence_oracle as D
from oracle import symnmf_oracle as O

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


@pytest.fixture(scope="module")
def L():
    from paper_2607_24518_gb300 import build
    build.build()
    from paper_2607_24518_gb300 import symnmf
    return symnmf


def tol(T):
    Tp = (T + 31) // 32 * 32
    return 2.0 ** -22 + 4.0 * (3 * Tp / 16) * 2.0 ** -24


@pytest.mark.parametrize("center", [0, 1])
def test_columns_of_any_magnitude(L, center):
    T, n = 200, 420
    rng = np.random.default_rng(center)
    Y = rng.standard_normal((T, 6)) @ rng.random((6, n)) + rng.standard_normal((T, n))
    Y = np.abs(Y) if not center else Y
    Y *= 10.0 ** rng.integers(-30, 18, size=n)
    Y[17, ::7] *= 1e4          # an outlier 1e4 times the rest of its column
    Y[:, 5] = 0.0
    Y[:, 200] = 3.0 if center else 0.0
    Y = Y.astype(np.float32)
    S = torch.full((n, n), -1.0, device=DEV)
    L.symnmf_build_dependence(torch.tensor(Y, device=DEV), T, n, n, center, L.F32, S, n)
    got = S.double().cpu().numpy()
    C = Y.astype(np.float64)
    if center:  # the builder centres in FP32
        C = (Y - Y.astype(np.float64).mean(0).astype(np.float32)).astype(np.float64)
    nrm = np.sqrt((C * C).sum(0))
    C = C / np.where(nrm > 0, nrm, 1.0)
    ref = np.minimum(1.0, np.abs(C.T @ C))
    np.fill_diagonal(ref, 1.0)
    assert np.max(np.abs(got - ref)) <= tol(T)
    assert np.array_equal(got, got.T)


@pytest.mark.parametrize("T", [3, 64, 1100])
def test_columns_of_a_level_whose_sum_leaves_fp32(L, T):
    """Means are FP64 sums: a column at 1e37 or 3e38 has a finite mean although
    64 of its entries add up to more than FP32 holds.  (T = 3: at most one
    entry a thread; 64: four; 1100: more than a run of 64.)"""
    n = 72
    rng = np.random.default_rng(T)
    Y = rng.standard_normal((T, 4)) @ rng.random((4, n)) + rng.standard_normal((T, n))
    level = np.array([1.0, 1e20, 5e36, 1e37, -1e37, 3e38, -3e38])[np.arange(n) % 7]
    Y = (level * (1.0 + 0.02 * np.clip(Y, -5, 5))).astype(np.float32)
    assert np.isfinite(Y).all()
    S = torch.full((n, n), -1.0, device=DEV)
    L.symnmf_build_dependence(torch.tensor(Y, device=DEV), T, n, n, 1, L.F32, S, n)
    C = (Y - Y.astype(np.float64).mean(0).astype(np.float32)).astype(np.float64)  # centred in FP32
    C /= np.sqrt((C * C).sum(0))
    ref = np.minimum(1.0, np.abs(C.T @ C))
    np.fill_diagonal(ref, 1.0)
    got = S.double().cpu().numpy()
    assert np.max(np.abs(got - ref)) <= tol(T)


@pytest.mark.parametrize("out", ["f32", "bf16", "fp8"])
@pytest.mark.parametrize("T,n", [(2, 128), (128, 256), (129, 257), (31, 2048), (33, 2049), (160, 4353)])
def test_tile_list_and_mirrors(L, T, n, out):
    rng = np.random.default_rng(n)
    Y = (rng.standard_normal((T, 4)) @ rng.random((4, n)) + rng.standard_normal((T, n))).astype(np.float32)
    es, dt = {"f32": (4, torch.float32), "bf16": (2, torch.bfloat16), "fp8": (1, torch.uint8)}[out]
    lds, nt = -(-n * es // 16) * 16 // es, -(-n // 128)
    S = torch.full((n, lds), 77, dtype=dt, device=DEV)
    sc = torch.zeros(nt, nt, device=DEV)
    L.symnmf_build_dependence(torch.tensor(Y, device=DEV), T, n, n, 1,
                              {"f32": L.F32, "bf16": L.BF16, "fp8": L.FP8E4M3}[out], S, lds, sc, nt)
    ref = torch.tensor(D.dependence(Y.astype(np.float64), True), device=DEV)
    if out == "fp8":
        got = S[:, :n].contiguous().view(torch.float8_e4m3fn).double()
        scale = sc.double().repeat_interleave(128, 0)[:n].repeat_interleave(128, 1)[:, :n]
        assert bool((torch.log2(sc) == torch.log2(sc).round()).all())
        got = got * scale
        step = torch.clamp(2.0 ** torch.floor(torch.log2(got.clamp_min(1e-30))) / 8, min=0) + scale * 2.0 ** -9
        assert bool(((got - ref).abs() <= tol(T) + 0.51 * step).all())
    else:
        got = S[:, :n].double()
        bound = tol(T) + (2.0 ** -9 if out == "bf16" else 0.0)
        assert float((got - ref).abs().max()) <= bound
    assert torch.equal(got, got.T)
    assert bool((S[:, n:].float() == 77).all())


@pytest.mark.parametrize("out,es", [("f32", 4), ("bf16", 2), ("fp8", 1)])
def test_rows_on_16_but_not_on_32_bytes(L, out, es):
    """Rows on 16-byte boundaries only take 16-byte stores: the same entries
    as with rows on 32-byte boundaries."""
    T, n = 64, 300
    Y = torch.tensor(np.random.default_rng(3).standard_normal((T, n)), dtype=torch.float32, device=DEV)
    dt = {"f32": torch.float32, "bf16": torch.bfloat16, "fp8": torch.uint8}[out]
    got = []
    for pitch, off in ((320 * 4, 0), (320 * 4 + 16, 0), (320 * 4, 16)):
        lds = pitch // es
        flat = torch.zeros(n * lds + 64, dtype=dt, device=DEV)
        S = flat[off // es:off // es + n * lds].view(n, lds)
        sc = torch.zeros(3, 3, device=DEV)
        L.symnmf_build_dependence(Y, T, n, n, 1, {"f32": L.F32, "bf16": L.BF16, "fp8": L.FP8E4M3}[out],
                                  S, lds, sc, 3)
        got.append((S[:, :n].float(), sc))
        assert not bool((S[:, n:].float() != 0).any())
    for S, sc in got[1:]:
        assert torch.equal(S, got[0][0]) and torch.equal(sc, got[0][1])
