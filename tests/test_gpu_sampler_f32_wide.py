"""The fp32 one-launch sampler where a CTA's slice of W_c fits only without padding between the rows."""
import numpy as np
import pytest
import torch

import oracle
from tests.gpu_common import f64, lsp_lib
from paper_2609_37029_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("V", [233472, 240000])            # the widest slice with padding on 152 SMs, and one without
def test_wide_f32_vocabulary_takes_one_launch(V):
    lsp = lsp_lib()
    C, B, rc = 2, 3, 32
    s = synth.LspShape("fw", C=C, B=B, L=1, D=1, H=128, nq=2, nkv=2, d=64, F=64, V=V, W=16, R=4, rc=rc, dtype="f32")
    st = lsp.lsp_state_create(lsp.make_config(s))
    small = lsp.lsp_state_create(lsp.make_config(s.with_(V=1024)))
    try:
        assert lsp.lsp_round_launches(st) == lsp.lsp_round_launches(small)
        g = torch.Generator().manual_seed(V)
        z0 = torch.randn(C, B, V, generator=g) * 2.0
        Ec, Wc = (torch.randn(V, rc, generator=g) * 0.3 for _ in range(2))
        prev = torch.randint(0, V, (C,), generator=g, dtype=torch.int32)
        toks = torch.full((C, B), -1, dtype=torch.int32, device="cuda")
        zout = torch.full((C, B, V), float("nan"), device="cuda")
        lsp.lsp_sample(st, z0.cuda(), prev.cuda(), Ec.cuda(), Wc.cuda(), lsp.make_sample_params(0.0), toks, zout)
        toks_g, z_g = toks.cpu().numpy(), f64(zout)
        for b in range(C):
            t_o, z_o, marg = oracle.sample_block(f64(z0[b]), int(prev[b]), f64(Ec), f64(Wc), 0.0, 0, 0, b, forced_prev=toks_g[b])
            np.testing.assert_allclose(z_g[b], z_o, rtol=0, atol=2e-5 * np.abs(z_o).max())
            sel = marg > 1e-2
            assert np.array_equal(toks_g[b][sel], t_o[sel])
        assert lsp.lsp_get_error(st) == (lsp.LSP_OK, 0)
    finally:
        lsp.lsp_state_destroy(st)
        lsp.lsp_state_destroy(small)
