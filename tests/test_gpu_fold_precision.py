"""Relative error of the folded summary against 64 bits: no larger than the kernel that a
call took before it went to the tcgen05 fold.  Two bf16 parts of the weights leave 2^-18 / sqrt(3)
= 2.2e-6 on a weight, and, weights and values being random, on the norm of m; three leave 2^-26.
With fp32 sums in between the bound is 1e-6: it fails with two parts."""
import numpy as np
import pytest
import torch

import oracle
from tests.gpu_common import export_state, f64, lsp_lib
from paper_2609_37029_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("rep,R,rows,prefill", [(5, 8, 1126, False), (4, 7, 2048, False), (8, 5, 700, False),
                                                (4, 16, 120, False), (4, 16, 84, True), (5, 8, 1999, True),
                                                (8, 16, 4096, True), (4, 16, 65, True)])
def test_summary_error_against_64_bits(rep, R, rows, prefill):
    lsp = lsp_lib()
    s = synth.LspShape("fold", C=1, B=16, L=2, D=1, H=256, nq=2 * rep, nkv=2, d=128, F=256, V=1024, W=40, R=R, rc=16)
    st = lsp.lsp_state_create(lsp.make_config(s))
    try:
        w = synth.make_weights(s, seed=3)
        lsp.lsp_state_init(st, w["G"].cuda())
        ost = oracle.state_init(s)
        k, v, h = synth.make_features(s, rows, seed=8)
        if prefill:
            lsp.lsp_prefill(st, 0, k[0].contiguous().cuda(), v[0].contiguous().cuda(), h[0].contiguous().cuda())
        else:
            lsp.lsp_view_update(st, k.cuda(), v.cuda(), h.cuda(), torch.tensor([rows], dtype=torch.int32).cuda())
        oracle.view_update(s, ost, f64(w["G"]), f64(k), f64(v), f64(h), np.array([rows], dtype=np.int32))
        m = export_state(lsp, st, s)["m"].double().numpy()
        assert np.linalg.norm(m - ost.m) < 1e-6 * np.linalg.norm(ost.m)
    finally:
        lsp.lsp_state_destroy(st)
