"""Prefills of at most 128 rows take one kernel of their own; at the edges of its 16-row
steps, with windows shorter and longer than the prefix, and without each part of the interface."""
import numpy as np
import pytest
import torch

import oracle
from tests.gpu_common import check_view_state, f64, lsp_lib
from paper_2609_37029_gb300 import synth

pytestmark = pytest.mark.gpu


def _shape(**kw):
    base = dict(C=2, B=16, L=3, D=1, H=256, nq=10, nkv=2, d=128, F=256, V=1024, W=40, R=16, rc=16)
    return synth.LspShape("pf", **{**base, **kw})


@pytest.mark.parametrize("t", [1, 2, 15, 16, 17, 64, 65, 100, 127, 128])
@pytest.mark.parametrize("kw", [{}, {"W": 5, "R": 7}, {"W": 300, "nq": 2}, {"R": 0}, {"W": 0, "no_boundary": True}])
def test_small_prefill_matches_oracle(t, kw):
    lsp = lsp_lib()
    s = _shape(**kw)
    st = lsp.lsp_state_create(lsp.make_config(s))
    try:
        w = synth.make_weights(s, seed=3)
        lsp.lsp_state_init(st, w["G"].cuda() if w["G"].numel() else None)
        ost, Gn = oracle.state_init(s), f64(w["G"])
        k, v, h = synth.make_features(s, 90, seed=4)
        acc = np.array([90, 90], dtype=np.int32)                # both requests hold a prefix; one is replaced
        lsp.lsp_view_update(st, k.cuda(), v.cuda(), None if s.no_boundary else h.cuda(), torch.tensor(acc).cuda())
        oracle.view_update(s, ost, Gn, f64(k), f64(v), f64(h), acc)
        k, v, h = synth.make_features(s, t, seed=200 + t)
        lsp.lsp_prefill(st, 1, k[1].contiguous().cuda(), v[1].contiguous().cuda(),
                        None if s.no_boundary else h[1].contiguous().cuda())
        one = s.with_(C=1)
        fresh = oracle.state_init(one)
        oracle.view_update(one, fresh, Gn, f64(k[1:]), f64(v[1:]), f64(h[1:]), np.array([t], dtype=np.int32))
        ost.eta[1], ost.m[1], ost.t[1] = fresh.eta[0], fresh.m[0], fresh.t[0]
        ost.hb[1] = fresh.hb[0]
        ost.win_k[1], ost.win_v[1] = fresh.win_k[0], fresh.win_v[0]
        torch.cuda.synchronize()
        check_view_state(lsp, st, ost, s)
        assert lsp.lsp_get_error(st) == (lsp.LSP_OK, 0)
    finally:
        lsp.lsp_state_destroy(st)


@pytest.mark.parametrize("t", [128, 129])
def test_rows_off_a_16_byte_boundary_are_refused(t):
    lsp = lsp_lib()
    s = _shape()
    st = lsp.lsp_state_create(lsp.make_config(s))
    try:
        w = synth.make_weights(s, seed=3)
        lsp.lsp_state_init(st, w["G"].cuda())
        n = s.L * t * s.nkv * s.d
        ok = torch.zeros(n + 8, dtype=torch.bfloat16, device="cuda")
        h = torch.zeros(s.L, t, s.H, dtype=torch.bfloat16, device="cuda")
        for k, v in ((ok[1:n + 1], ok[:n]), (ok[:n], ok[1:n + 1])):
            with pytest.raises(lsp.LspError):
                lsp.lsp_prefill(st, 0, k.view(s.L, t, s.nkv, s.d), v.view(s.L, t, s.nkv, s.d), h)
    finally:
        lsp.lsp_state_destroy(st)
