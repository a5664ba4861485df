"""Block-SVRG's three products and its Grams start as the launch before them
leaves the SMs; under a cap of CTAs they run one after the other.  A cap of one
SM less than the GPU has leaves the grids of small matrices as they are, so both
orders must give the same state bit for bit."""
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


@pytest.mark.parametrize("phi", [0.1, 0.5, 0.9])
@pytest.mark.parametrize("n,k,dtype", [(130, 3, "f32"), (300, 8, "bf16"), (700, 32, "f32"), (1100, 64, "f32"),
                                       (1500, 16, "fp8"), (1500, 64, "bf16"), (1400, 64, "fp8")])
def test_chained_equals_one_after_the_other(L, n, k, dtype, phi):
    rng = np.random.default_rng(n + k)
    A = rng.random((n, 6))
    S = torch.tensor(np.minimum(1.0, A @ A.T / 3), dtype=torch.float32, device=DEV)
    nt, sc = -(-n // 128), None
    lds = -(-n // 16) * 16
    tdt = {"f32": torch.float32, "bf16": torch.bfloat16, "fp8": torch.float8_e4m3fn}[dtype]
    q = torch.zeros(n, lds, dtype=torch.float32, device=DEV)
    q[:, :n] = S * (256.0 if dtype == "fp8" else 1.0)
    q = q.to(tdt)
    base = q.view(torch.uint8) if dtype == "fp8" else q
    H = torch.tensor(rng.uniform(0, 0.3, (n, k)), dtype=torch.float32, device=DEV)
    hp = L.symnmf_hparams_default(L.BLOCK_SVRG_ADAPTGROW, eta=0.1, phi0=phi, snapshot_period=5,
                                  block_rows=128)
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    got = []
    for cap in (0, sms - 1):
        h = L.symnmf_create_ld(base, n, lds, k, {"f32": L.F32, "bf16": L.BF16, "fp8": L.FP8E4M3}[dtype])
        try:
            if dtype == "fp8":
                sc = torch.full((nt, nt), 2.0 ** -8, dtype=torch.float32, device=DEV)
                L.symnmf_set_tile_scales(h, sc, nt)
            L.symnmf_set_ctas(h, cap)
            L.symnmf_set_H(h, H)
            L.symnmf_step(h, hp, 24)
            bufs = [torch.empty(n, k, device=DEV) for _ in range(3)]
            for which, b in zip((L.BUF_H, L.BUF_ACC, L.BUF_SNAPSHOT), bufs):
                L.symnmf_get_buffer(h, which, b)
            got.append([b.cpu() for b in bufs])
        finally:
            L.symnmf_destroy(h)
    assert torch.isfinite(got[0][0]).all()
    for a, b in zip(*got):
        assert torch.equal(a, b)
