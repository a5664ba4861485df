"""Sums of squares of S in FP64 accuracy: ||S||^2 of a handle and the tile sums
of the quantiser, and through the objective of a Lloyd step the row norms of
spherical K-means, at the edges of their 16-entry groups, 64-entry runs and
512-column chunks, for aligned and unaligned rows, for values that leave the
FP32 words for the FP64 sum and for tile scales that are no powers of two.
Reference: numpy in FP64.  Bound: a run of 64 entries rounds only in its third
word, 128 times at most 2^-58 of 64 cap^2 with cap at most twice the largest
entry: 2^-43 of its square if every rounding were the worst and all went one
way.  A run of uniform entries (their cubes) sums to 21 (9) such squares, so
2^-46; one or two entries do not reach the third word, and FP64 sums over n <=
2100 terms add less."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu
DEV = "cuda:0"
REL = 2.0 ** -46


@pytest.fixture(scope="module")
def L():
    from paper_2607_24518_gb300 import build
    build.build()
    from paper_2607_24518_gb300 import symnmf
    return symnmf


@pytest.mark.parametrize("dtype", ["f32", "bf16", "fp8"])
@pytest.mark.parametrize("n,pad", [(1, 0), (15, 1), (129, 0), (512, 0), (513, 15), (2049, 7)])
@pytest.mark.parametrize("scale", [1.0, 1e25, 1e-25])
def test_norm_of_a_handle(L, n, pad, dtype, scale):
    rng = np.random.default_rng(n + pad)
    lds = n + pad
    S = torch.zeros(n, lds, device=DEV)
    S[:, :n] = torch.tensor(rng.random((n, n)), dtype=torch.float32, device=DEV)
    if dtype == "fp8":
        nt = -(-n // 128)
        q = (S * 448).to(torch.float8_e4m3fn)
        # powers of two, times a factor that is none for two of the three scales
        sc = torch.tensor(scale * 2.0 ** rng.integers(-8, 0, (nt, nt)), dtype=torch.float32, device=DEV)
        h = L.symnmf_create_ld(q.view(torch.uint8), n, lds, 4, L.FP8E4M3)
        L.symnmf_set_tile_scales(h, sc, nt)
        tile = sc.double().cpu().numpy().repeat(128, 0)[:n].repeat(128, 1)[:, :n]
        S64 = q[:, :n].to(torch.float64).cpu().numpy() * tile
    else:
        S = (S * scale).to({"f32": torch.float32, "bf16": torch.bfloat16}[dtype])
        h = L.symnmf_create_ld(S, n, lds, 4, {"f32": L.F32, "bf16": L.BF16}[dtype])
        S64 = S[:, :n].double().cpu().numpy()
    try:
        ref = float(np.sum(S64 * S64))
        assert abs(L.symnmf_get_norm(h) - ref) <= REL * ref
    finally:
        L.symnmf_destroy(h)


def test_norm_when_the_largest_entry_comes_last(L):
    """Entries that grow along a row by 2^60 in all raise the bound of the runs
    again and again; zeros and entries below 2^-40 come first."""
    n = 700
    rng = np.random.default_rng(5)
    S = (rng.random((n, n)) * 2.0 ** np.linspace(-50, 10, n)[None, :]).astype(np.float32)
    S[:, :40] = 0.0
    for M in (S, S[:, ::-1].copy(), np.where(rng.random((n, n)) < 0.01, S, np.float32(0))):
        h = L.symnmf_create(torch.tensor(M, device=DEV), n, 4, L.F32)
        try:
            ref = float(np.sum(M.astype(np.float64) ** 2))
            assert abs(L.symnmf_get_norm(h) - ref) <= 2.0 ** -43 * ref
        finally:
            L.symnmf_destroy(h)


@pytest.mark.parametrize("src", ["f32", "bf16"])
@pytest.mark.parametrize("rows,cols,ld,ldq", [(1, 1, 1, 1), (128, 128, 128, 128), (130, 257, 257, 260),
                                              (257, 131, 133, 131), (64, 516, 520, 517)])
@pytest.mark.parametrize("scale", [1.0, 1e25])
def test_quantiser_tiles(L, rows, cols, ld, ldq, src, scale):
    from oracle import symnmf_oracle as O
    rng = np.random.default_rng(rows + cols)
    tdt = {"f32": torch.float32, "bf16": torch.bfloat16}[src]
    S = torch.tensor(scale * rng.random((rows, ld)) ** 3, dtype=torch.float32, device=DEV).to(tdt)
    nr, nc = -(-rows // 128), -(-cols // 128)
    q = torch.zeros(rows, ldq, dtype=torch.uint8, device=DEV)
    sc = torch.zeros(nr, nc, device=DEV)
    ss = torch.zeros(nr, nc, dtype=torch.float64, device=DEV)
    L.symnmf_quantize_fp8(S, {"f32": L.F32, "bf16": L.BF16}[src], rows, cols, ld, q, ldq, sc, nc, ss)
    torch.cuda.synchronize()
    S64 = S[:, :cols].double().cpu().numpy()
    codes = q.view(torch.float8_e4m3fn).double().cpu().numpy()
    for i in range(nr):
        for j in range(nc):
            T = S64[i * 128:(i + 1) * 128, j * 128:(j + 1) * 128]
            s = O.tile_scale(float(T.max()))
            assert float(sc[i, j]) == s
            ref = float(np.sum(T * T))
            assert abs(float(ss[i, j]) - ref) <= REL * ref
            np.testing.assert_array_equal(codes[i * 128:i * 128 + T.shape[0], j * 128:j * 128 + T.shape[1]],
                                          O.e4m3_round(T / s))
    assert not bool((q[:, cols:] != 0).any())


@pytest.mark.parametrize("dtype", ["f32", "bf16"])
@pytest.mark.parametrize("n,pad", [(130, 0), (517, 3), (2050, 6)])
def test_row_norms_through_one_lloyd_step(L, n, pad, dtype):
    """J = sum_i (1 - cos_i) after one step from known labels takes ||s_i||
    of every row."""
    from oracle import spkmeans_oracle as KM
    rng = np.random.default_rng(n)
    tdt = {"f32": torch.float32, "bf16": torch.bfloat16}[dtype]
    S = torch.zeros(n, n + pad, dtype=tdt, device=DEV)
    A = rng.random((n, 3))
    S[:, :n] = torch.tensor(A @ A.T / 3, dtype=torch.float32, device=DEV).to(tdt)
    lab = (np.arange(n) % 3).astype(np.int32)
    h = L.symnmf_create_ld(S, n, n + pad, 3, {"f32": L.F32, "bf16": L.BF16}[dtype])
    try:
        out = torch.empty(n, dtype=torch.int32, device=DEV)
        _, J = L.symnmf_spkmeans(h, torch.tensor(lab, device=DEV), out, 1)
        _, ref, _ = KM.lloyd_step(S[:, :n].double().cpu().numpy(), lab, 3)
        assert abs(J[0] - ref) <= 1e-5 * n
    finally:
        L.symnmf_destroy(h)
