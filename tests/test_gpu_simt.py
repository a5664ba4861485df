"""The exact-FP32 product at the edges of its tiles (128 rows, 32-column
chunks, a ring of four), for rows of any pitch and a base that is aligned to
the element only, all storage types and padded ranks; and the stand-alone
epilogue behind it (gradient, one step of every method, objective).
Reference: the FP64 oracle on the stored values; FP32 sums of n terms in
chains of at most n / 4 FMAs, held to 1e-5 as everywhere."""
import numpy as np
import pytest
import torch

from oracle import symnmf_oracle as O

pytestmark = pytest.mark.gpu
DEV = "cuda:0"
REL = 1e-5


@pytest.fixture(scope="module")
def L():
    from paper_2607_24518_gb300 import build
    build.build()
    from paper_2607_24518_gb300 import symnmf
    return symnmf


def _handle(L, n, k, dtype, seed):
    """A handle on an n x n matrix whose base lies one element past an
    aligned address and whose pitch is odd; its values in FP64; and H."""
    rng = np.random.default_rng(seed)
    A = rng.random((n, 4))
    S64 = np.minimum(1.0, (A @ A.T) / 2)
    lds = n + 1 + (n % 2)
    tdt = {"f32": torch.float32, "bf16": torch.bfloat16, "fp8": torch.float8_e4m3fn}[dtype]
    flat = torch.zeros(n * lds + 1, dtype=torch.float32, device=DEV)
    V = flat[1:].view(n, lds)
    V[:, :n] = torch.tensor(S64 * (256.0 if dtype == "fp8" else 1.0), dtype=torch.float32, device=DEV)
    V[:, n:] = 3.0  # what lies between the rows must not enter
    q = flat.to(tdt)
    keep = [q, q[1:]]
    base = (q.view(torch.uint8) if dtype == "fp8" else q)[1:]
    h = L.symnmf_create_ld(base, n, lds, k, {"f32": L.F32, "bf16": L.BF16, "fp8": L.FP8E4M3}[dtype])
    vals = q[1:].view(n, lds)[:, :n].to(torch.float64).cpu().numpy()
    if dtype == "fp8":
        nt = -(-n // 128)
        sc = torch.tensor(2.0 ** rng.integers(-9, -7, (nt, nt)), dtype=torch.float32, device=DEV)
        L.symnmf_set_tile_scales(h, sc, nt)
        keep.append(sc)
        vals = vals * sc.double().cpu().numpy().repeat(128, 0)[:n].repeat(128, 1)[:, :n]
    H = rng.uniform(0, 0.3, (n, k)).astype(np.float32)
    Hd = torch.tensor(H, device=DEV)
    L.symnmf_set_H(h, Hd)
    assert L.symnmf_get_impl(h) == 1
    return h, vals, H.astype(np.float64), keep


@pytest.mark.parametrize("dtype", ["f32", "bf16", "fp8"])
@pytest.mark.parametrize("n,k", [(1, 1), (31, 8), (33, 9), (127, 16), (129, 17), (257, 33), (385, 64), (1001, 5)])
def test_gradient_and_objective(L, n, k, dtype):
    h, S, H, keep = _handle(L, n, k, dtype, seed=n + k)
    try:
        G = torch.empty(n, k, device=DEV)
        L.symnmf_grad(h, G)
        f, _ = L.symnmf_objective(h)
        scale = 4.0 * (np.linalg.norm(S @ H) + np.linalg.norm(H @ (H.T @ H)))
        ref = 4.0 * (H @ (H.T @ H) - S @ H)
        assert np.linalg.norm(G.double().cpu().numpy() - ref) <= REL * scale
        want = np.sum(S * S) - 2.0 * np.sum(H * (S @ H)) + np.sum((H.T @ H) ** 2)
        assert abs(f - want) <= 1e-6 * (np.sum(S * S) + np.sum((H.T @ H) ** 2))
    finally:
        L.symnmf_destroy(h)


@pytest.mark.parametrize("method", [0, 1, 5])
@pytest.mark.parametrize("n,k", [(1, 3), (129, 8), (300, 11), (257, 33), (140, 64)])
def test_one_step_of_the_stand_alone_epilogue(L, n, k, method):
    h, S, H, keep = _handle(L, n, k, "f32", seed=n + k)
    try:
        over = {"rho": 50.0} if method == 5 else {"eta": 0.1}
        L.symnmf_step(h, L.symnmf_hparams_default(method, **over), 3)
        hp = O.HParams.paper(method)
        for key, v in over.items():
            setattr(hp, key, v)
        s = O.Solver(S, H, hp)
        s.run(3)
        for which, ref in ((L.BUF_H, s.H), (L.BUF_ACC, s.A)):
            got = torch.empty(n, k, device=DEV)
            L.symnmf_get_buffer(h, which, got)
            tol = 1e-4 * (np.linalg.norm(ref) + (np.linalg.norm(s.H) if method == 5 else 0.0))
            assert np.linalg.norm(got.double().cpu().numpy() - ref) <= tol
    finally:
        L.symnmf_destroy(h)


@pytest.mark.parametrize("n,k", [(129, 8), (300, 11), (257, 33), (400, 64)])
def test_tile_scalars_of_the_stand_alone_epilogue_are_fp64_sums(L, n, k):
    """With H = 0 the gradient is 0 and the accumulator stays as it is, so the
    record's sum(G) is the sum of what was put there: 2^50 once per tile,
    several 3 * 2^25 and many ones.  They need 51 bits, one thread holds one of
    them at most (rows below 32 and every fourth column of a tile), and an FP64
    sum of them is exact."""
    h, _, _, keep = _handle(L, n, k, "f32", seed=n)
    try:
        L.symnmf_set_H(h, torch.zeros(n, k, device=DEV))
        A = np.zeros((n, k), dtype=np.float32)
        rng = np.random.default_rng(k)
        for r0 in range(0, n, 128):
            rows = min(32, n - r0)
            v = rng.choice(np.array([1.0, 3 * 2.0 ** 25, 0.0]), size=(rows, -(-k // 4)))
            v[rng.integers(rows), rng.integers(v.shape[1])] = 2.0 ** 50
            A[r0:r0 + rows, ::4] = v
        L.symnmf_set_buffer(h, L.BUF_ACC, torch.tensor(A, device=DEV))
        L.symnmf_step(h, L.symnmf_hparams_default(L.ADAGRAD), 1)
        assert L.symnmf_get_trace(h)[-1].sumA == float(A.astype(np.float64).sum())
    finally:
        L.symnmf_destroy(h)


@pytest.mark.parametrize("n,k", [(38000, 64), (38000, 20), (16700, 64), (700, 64)])
def test_chains_of_the_objective_without_a_handle(L, n, k):
    """An FP32 chain of m equal terms rounds by at most m / 2 * 2^-24 of its sum
    (half a unit of a partial sum, whose average is half the sum), and equal
    terms come near that.  Eight column shares bound a chain by 128 columns of
    ceil(tiles / 8) tiles, however many shares a call takes; 32 FMAs of the dot
    with H, 35 of a Gram partial (twice, as its square) and slack add 256."""
    s, t = 0.640625, np.float32(0.0809360146522522)
    S = torch.full((n, n), s, dtype=torch.bfloat16, device=DEV)
    H = torch.full((n, k), float(t), device=DEV)
    f = torch.zeros(1, dtype=torch.float64, device=DEV)
    L.symnmf_objective_noalloc(S, n, n, L.BF16, None, 0, H, k, 0.0, f)
    tr = float(n) * n * k * s * float(t) ** 2
    g2 = (k * n * float(t) ** 2) ** 2
    m = 128 * -(-(-(-n // 128)) // 8)
    assert abs(float(f[0]) - (g2 - 2.0 * tr)) <= (m / 2 + 256) * 2.0 ** -24 * 2.0 * tr
