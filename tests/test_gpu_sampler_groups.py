"""The one-launch sampler at the edges of its request groups (eight), vocabulary tiles (32 rows),
CTAs (fewer than requests at the smallest vocabularies) and slots (one step; the
logits not written), with a state whose launches follow one another and without one."""
import numpy as np
import pytest
import torch

import oracle
from tests.gpu_common import f64, lsp_lib
from paper_2609_37029_gb300 import synth

pytestmark = pytest.mark.gpu

CASES = [
    # C, B, V, rc, temperature
    (1, 16, 4096, 64, 1.0),
    (8, 3, 8208, 32, 0.7),      # V = 16 mod 32: the last tile is half full
    (9, 5, 8208, 64, 0.0),      # a second group of one request
    (16, 4, 48, 64, 1.0),       # two CTAs lead eight requests each
    (3, 1, 16, 32, 0.0),        # one step, one half tile
    (17, 4, 33008, 64, 1.0),    # groups of 16 and 1 in two launches
    (2, 7, 155648, 64, 1.0),    # the widest slice a CTA takes
]


@pytest.mark.parametrize("C,B,V,rc,temperature", CASES)
@pytest.mark.parametrize("noalloc", [False, True])
def test_sampler_edges(C, B, V, rc, temperature, noalloc):
    lsp = lsp_lib()
    s = synth.LspShape("sg", C=C, B=B, L=1, D=1, H=128, nq=1, nkv=1, d=128, F=64, V=V, W=16, R=16, rc=rc)
    st = None if noalloc else lsp.lsp_state_create(lsp.make_config(s))
    try:
        g = torch.Generator().manual_seed(C + V)
        z0 = torch.randn(C, B, V, generator=g) * 2.0
        Ec, Wc = ((torch.randn(V, rc, generator=g) * 0.5).bfloat16() for _ in range(2))
        prev = torch.randint(0, V, (C,), generator=g, dtype=torch.int32)
        sp = lsp.make_sample_params(temperature, seed=0x1234ABCD5678, rnd=9)
        zg, pg, eg, wg = z0.cuda(), prev.cuda(), Ec.cuda(), Wc.cuda()

        def call(tokens, logits):
            if noalloc:
                lsp.lsp_sample_noalloc(zg, pg, eg, wg, lsp.LSP_DTYPE_BF16, C, B, V, rc, sp, tokens, logits)
            else:
                lsp.lsp_sample(st, zg, pg, eg, wg, sp, tokens, logits)

        toks = torch.full((C, B), -1, dtype=torch.int32, device="cuda")
        zout = torch.full((C, B, V), float("nan"), device="cuda")
        call(toks, zout)
        for _ in range(3):                            # launches after launches, without the logits
            again = torch.full_like(toks, -1)
            call(again, None)
            assert torch.equal(again, toks)
        assert torch.equal(zg, z0.cuda())             # the base logits stay as they are
        toks_g, z_g = toks.cpu().numpy(), f64(zout)
        for b in range(C):
            t_o, z_o, marg = oracle.sample_block(f64(z0[b]), int(prev[b]), f64(Ec), f64(Wc), temperature,
                                                 0x1234ABCD5678, 9, b, forced_prev=toks_g[b])
            # fp32 sums of exact bf16 products: the bound of the library's other sampler tests
            np.testing.assert_allclose(z_g[b], z_o, rtol=0, atol=2e-5 * np.abs(z_o).max())
            sel = marg > 1e-2
            assert np.array_equal(toks_g[b][sel], t_o[sel]), (b, toks_g[b], t_o, marg)
        if st:
            assert lsp.lsp_get_error(st) == (lsp.LSP_OK, 0)
    finally:
        if st:
            lsp.lsp_state_destroy(st)
