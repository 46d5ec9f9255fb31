"""lsp_linear where no tensor map describes the output -- a row pitch or an address off a 16-byte
boundary: rows copied in bulk between the boundaries (one item a CTA) or stored from
registers (a walk over items), for every remainder of the pitch and of the address."""
import numpy as np
import pytest
import torch

from tests.gpu_common import f64, lsp_lib

pytestmark = pytest.mark.gpu

CASES = [
    # M, N, K, dtype, splits
    (1, 1, 64, "bf16", 1), (5, 2, 64, "bf16", 1), (3, 3, 128, "bf16", 2), (16, 5, 64, "bf16", 1),    # shorter than a vector
    (17, 31, 64, "f32", 1), (33, 33, 64, "bf16", 1), (16, 30001, 64, "bf16", 1),
    (128, 8190, 128, "bf16", 1), (129, 8191, 128, "bf16", 1),        # one accumulator, and two
    (206, 30561, 96, "bf16", 1),                                     # rows of several passes
    (256, 33999, 64, "bf16", 1), (300, 4999, 64, "f32", 1),          # two token groups
    (23, 17919, 256, "bf16", 4), (100, 39997, 64, "bf16", 1),        # walks over items
    (512, 30002, 64, "bf16", 1),
]


@pytest.mark.parametrize("M,N,K,dt,splits", CASES)
@pytest.mark.parametrize("offset", [0, 1, 2, 3])
def test_linear_rows_off_the_boundary(M, N, K, dt, splits, offset):
    lsp = lsp_lib()
    g = torch.Generator(device="cuda").manual_seed(M + 3 * N + K)
    tdt = torch.bfloat16 if dt == "bf16" else torch.float32
    X = torch.randn(M, K, generator=g, device="cuda").to(tdt)
    W = (torch.randn(N, K, generator=g, device="cuda") * 0.05).to(tdt)
    buf = torch.full((M * N + 8192,), float("nan"), device="cuda")   # what lies around Y stays as it is
    nbytes = lsp.lsp_linear_workspace_bytes(M, N, splits)
    ws = torch.full((nbytes + 4096,), 0xFF, dtype=torch.uint8, device="cuda")
    Y = buf[offset:offset + M * N]
    lsp.lsp_linear(X, W, Y, M, N, K, lsp.LSP_DTYPE_BF16 if dt == "bf16" else lsp.LSP_DTYPE_F32, splits, ws, nbytes)
    torch.cuda.synchronize()
    assert torch.isnan(buf[:offset]).all() and torch.isnan(buf[offset + M * N:]).all() and (ws[nbytes:] == 0xFF).all()
    ref = X.double() @ W.double().T
    err = (Y.view(M, N).double() - ref).abs().max().item()
    # the bounds of the library's other linear tests
    assert err <= (1e-5 if dt == "bf16" else 4e-3) * ref.abs().max().item(), err
