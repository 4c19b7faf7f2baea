"""Tensor-core GEMM on each tile width with each FP32 store path, the shapes
chosen so that the width rule (the widest tile that still gives every one of 152
SMs a tile) takes the width named here; test_launch_order.py checks that it does.
TMA stores need D and its rows on 16 bytes and a multiple of four columns, else
the store is direct.  Against the FP64 product of the same BF16 values: products
are exact in FP32, so |D - D_exact| <= 4 K 2^-24 (|A| |B|^T); nothing outside D
is written."""
from __future__ import annotations

import pytest

from paper_1811_11679_gb300 import hande

# tile columns, m, n, k, row stride of D, offset of D in elements
SHAPES = [
    (128, 20000, 100, 96, 104, 0),     # TMA, columns beyond N clipped
    (128, 20000, 99, 96, 101, 0),      # direct
    (128, 20000, 128, 72, 132, 1),     # direct: D off 16 bytes
    (256, 20000, 252, 64, 256, 0),     # TMA, columns clipped
    (256, 20000, 256, 136, 256, 0),    # TMA, whole tiles
    (256, 20000, 250, 64, 251, 0),     # direct
    # several tiles per SM, and warps of the last tile wholly past M
    (256, 39000, 252, 136, 256, 0), (256, 39000, 250, 136, 251, 0),
    (128, 39000, 100, 200, 100, 0), (64, 39000, 40, 200, 40, 0), (64, 39000, 38, 200, 38, 0),
]


@pytest.mark.gpu
@pytest.mark.parametrize("width,m,n,k,ldd,shift", SHAPES)
def test_width_and_store_path(width, m, n, k, ldd, shift):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    g = torch.Generator(device="cuda").manual_seed(m + n + k)
    pad = (k + 7) // 8 * 8
    a = torch.randn((m, pad), generator=g, device="cuda").to(torch.bfloat16)[:, :k]
    b = torch.randn((n, pad), generator=g, device="cuda").to(torch.bfloat16)[:, :k]
    flat = torch.full((m * ldd + 64,), 7.0, dtype=torch.float32, device="cuda")
    d = flat[shift:shift + m * ldd].view(m, ldd)[:, :n]
    for _ in range(2):   # the same bits twice
        first = d.clone()
        hande.gemm_bf16(a, b, out=d)
        torch.cuda.synchronize()
    assert torch.equal(first, d)
    exact = a.double() @ b.double().T
    bound = 4.0 * k * 2.0 ** -24 * (a.double().abs() @ b.double().abs().T) + 1e-30
    assert torch.all((d.double() - exact).abs() <= bound)
    d.fill_(7.0)
    assert torch.all(flat == 7.0)


@pytest.mark.gpu
@pytest.mark.parametrize("m,n,k", [(128 * 38 + 8, 2048, 64), (128 * 152 + 96, 252, 64), (128 * 304 + 1, 252, 72)])
def test_last_tile_past_the_rows_leaves_the_tile_before_alone(m, n, k):
    """CTAs that walk a whole tile and then one with warps wholly past M, which
    store nothing, many times over (the error bound as above)."""
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    g = torch.Generator(device="cuda").manual_seed(m)
    a = torch.randn((m, k), generator=g, device="cuda").to(torch.bfloat16)
    b = torch.randn((n, k), generator=g, device="cuda").to(torch.bfloat16)
    exact = a.double() @ b.double().T
    bound = 4.0 * k * 2.0 ** -24 * (a.double().abs() @ b.double().abs().T) + 1e-30
    status = torch.zeros(1, dtype=torch.int32, device="cuda")
    bad = torch.zeros((), dtype=torch.int64, device="cuda")
    for _ in range(200):
        d = hande.gemm_bf16(a, b, status=status)
        bad += ((d.double() - exact).abs() > bound).sum()
    torch.cuda.synchronize()
    assert status.item() == 0
    assert bad.item() == 0
