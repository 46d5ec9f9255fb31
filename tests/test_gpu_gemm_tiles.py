"""lsp_linear at the edges of the projection GEMM's tiles: token counts around one and two
accumulators, outputs around the 32-feature store chunk and without a tensor map (odd row
pitch), walks over several items with one and with two accumulator sets."""
import numpy as np
import pytest
import torch

from tests.gpu_common import f64, lsp_lib

pytestmark = pytest.mark.gpu

CASES = [
    # M, N, K, dtype, splits
    (128, 1000, 128, "bf16", 1),      # one full accumulator, ragged last tile
    (129, 1004, 136, "bf16", 2),      # two accumulators of 72 tokens, ragged k
    (144, 33, 64, "bf16", 1),         # odd row pitch: per-thread stores, one feature past a chunk
    (256, 4099, 192, "bf16", 3),      # odd row pitch over split partials
    (257, 2050, 64, "bf16", 1),       # two token groups, pitch no multiple of 16 bytes
    (512, 20000, 128, "bf16", 1),     # two groups walked, one accumulator set
    (7, 40016, 192, "bf16", 1),       # few tokens, walked with two sets
    (100, 39999, 64, "bf16", 1),      # the same without a tensor map
    (1, 17, 64, "bf16", 1),
    (200, 12000, 96, "f32", 3),       # tf32, two accumulators, walked
    (130, 1001, 36, "f32", 1),
]


@pytest.mark.parametrize("M,N,K,dt,splits", CASES)
def test_linear_tile_edges(M, N, K, dt, splits):
    lsp = lsp_lib()
    g = torch.Generator().manual_seed(M + 3 * N + K)
    tdt = torch.bfloat16 if dt == "bf16" else torch.float32
    X = torch.randn(M, K, generator=g).to(tdt)
    W = (torch.randn(N, K, generator=g) * 0.05).to(tdt)
    buf = torch.full((M * N + 8192,), float("nan"), device="cuda")     # the tail must stay untouched
    nbytes = lsp.lsp_linear_workspace_bytes(M, N, splits)
    ws = torch.full((nbytes + 4096,), 0xFF, dtype=torch.uint8, device="cuda")
    lsp.lsp_linear(X.cuda(), W.cuda(), buf, M, N, K, lsp.LSP_DTYPE_BF16 if dt == "bf16" else lsp.LSP_DTYPE_F32,
                   splits, ws, nbytes)
    torch.cuda.synchronize()
    assert torch.isnan(buf[M * N:]).all() and (ws[nbytes:] == 0xFF).all()
    ref = f64(X) @ f64(W).T
    err = np.abs(f64(buf[:M * N].view(M, N)) - ref).max()
    # the bounds of the library's other linear tests: bf16 operands are exact in fp32 sums,
    # tf32 keeps 10 mantissa bits of each operand
    assert err <= (1e-5 if dt == "bf16" else 4e-3) * np.abs(ref).max(), err
