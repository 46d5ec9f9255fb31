"""Verification with the rows read only up to each request's first rejection (the launches of
large calls), at rejections in every position, none, and at the first; several calls on one
state (its counters reset themselves); rows behind the rejection hold NaN."""
import numpy as np
import pytest
import torch

from tests.gpu_common import lsp_lib
from tests.test_gpu_verify import _compare, _shape

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("T", [1.0, 0.0])
@pytest.mark.parametrize("C,B,V", [(20, 16, 40000), (64, 8, 50000), (64, 7, 33008)])
def test_rejection_at_every_position(T, C, B, V):
    lsp = lsp_lib()
    s = _shape(C, B, V)
    g = torch.Generator().manual_seed(C + V)
    zt = torch.randn(C, B + 1, V, generator=g) * 2.0
    zq = zt[:, :B].clone()                            # q = p: every candidate is accepted
    y = zt[:, :B].argmax(-1).to(torch.int32)
    want = [(b * 5) % (B + 1) for b in range(C)]      # request b: rejected at want[b] (B: nowhere)
    ztg, zqg = zt.clone(), zq.clone()
    for b, j in enumerate(want):
        if j == B:
            continue
        tok = int(y[b, j])
        zt[b, j, tok] = ztg[b, j, tok] = -60.0        # p(y) = 0 at that position
        ztg[b, j + 1:] = float("nan")                 # nothing behind it is part of the answer
        zqg[b, j + 1:] = float("nan")
    st = lsp.lsp_state_create(lsp.make_config(s))
    try:
        dz, dq, dy = ztg.cuda(), zqg.cuda(), y.cuda()
        prev = None
        for _ in range(3):
            acc = torch.full((C,), -1, dtype=torch.int32, device="cuda")
            tok = torch.full((C,), -1, dtype=torch.int32, device="cuda")
            lsp.lsp_verify(st, dz, dq, dy, lsp.make_sample_params(temperature=T, seed=77, rnd=5), acc, tok)
            torch.cuda.synchronize()
            got = (acc.cpu().numpy(), tok.cpu().numpy())
            assert got[0].tolist() == want
            if prev is not None:
                assert np.array_equal(got[1], prev[1])
            prev = got
        assert lsp.lsp_get_error(st) == (lsp.LSP_OK, 0)
        exact = _compare(s, zt, zq, y.numpy(), T, 77, 5, *got)
        assert exact >= C - 3
        # a candidate outside the vocabulary is reported and rejected
        dy[0, 0] = V
        lsp.lsp_verify(st, dz, dq, dy, lsp.make_sample_params(temperature=T, seed=77, rnd=5), acc, tok)
        assert lsp.lsp_get_error(st) == (lsp.LSP_ERR_STATE, lsp.LSP_DEV_BAD_TOKEN)
    finally:
        lsp.lsp_state_destroy(st)
