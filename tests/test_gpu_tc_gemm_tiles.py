"""Tensor-core GEMM over its tile widths (64, 128, 256 columns, chosen by how
many tiles the product has) and both FP32 store paths (TMA for 16-byte aligned
rows of D, direct otherwise), against the FP64 product of the same BF16 values:
|D - D_exact| <= 4 K 2^-24 (|A| |B|^T), and nothing written outside D."""
from __future__ import annotations

import pytest

from paper_1811_11679_gb300 import hande

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("m,n,k,ldd,shift", [
    (300, 40, 200, 40, 0), (4000, 129, 72, 132, 0), (12000, 100, 96, 104, 0),     # 64, 64 and 128 columns
    (20000, 250, 64, 256, 0), (20000, 250, 64, 251, 0), (20000, 250, 64, 256, 1),  # 256: TMA, ragged, unaligned
    (38, 256, 1000, 256, 0), (1, 512, 8, 512, 0)])
def test_gemm_tiles_and_store_paths(m, n, k, ldd, shift):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    g = torch.Generator(device="cuda").manual_seed(m + n + k)
    a = torch.randn((m, (k + 7) // 8 * 8), generator=g, device="cuda").to(torch.bfloat16)[:, :k]
    b = torch.randn((n, (k + 7) // 8 * 8), generator=g, device="cuda").to(torch.bfloat16)[:, :k]
    flat = torch.full((m * ldd + 64,), 7.0, dtype=torch.float32, device="cuda")
    d = flat[shift:shift + m * ldd].view(m, ldd)[:, :n]
    hande.gemm_bf16(a, b, out=d)
    torch.cuda.synchronize()
    exact = a.double() @ b.double().T
    bound = 4.0 * k * 2.0 ** -24 * (a.double().abs() @ b.double().abs().T) + 1e-30
    assert torch.all((d.double() - exact).abs() <= bound)
    d.fill_(7.0)
    assert torch.all(flat == 7.0)
