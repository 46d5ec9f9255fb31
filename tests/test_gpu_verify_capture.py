"""Greedy verification in its two forms -- one launch, or two where the call is captured or its
rows are many: a captured call replayed on new inputs, and a call of the host, decide as the
oracle does, in turn on one state (they share its counters)."""
import pytest
import torch

import oracle
from tests.gpu_common import f64, lsp_lib
from paper_2609_37029_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("C,B,V", [(1, 1, 16), (4, 16, 2048), (3, 7, 32016), (9, 16, 65600)])   # the last: two launches either way
def test_captured_greedy_verification(C, B, V):
    lsp = lsp_lib()
    s = synth.LspShape("vc", C=C, B=B, L=1, D=1, H=128, nq=1, nkv=1, d=128, F=64, V=V, W=16, R=16, rc=16)
    st = lsp.lsp_state_create(lsp.make_config(s))
    try:
        g = torch.Generator().manual_seed(C * B + V)
        zt = torch.empty(C, B + 1, V, device="cuda")
        zq = torch.zeros(C, B, V, device="cuda")
        y = torch.empty(C, B, dtype=torch.int32, device="cuda")
        acc, nxt = (torch.empty(C, dtype=torch.int32, device="cuda") for _ in range(2))
        sp = lsp.make_sample_params(0.0)

        def inputs():
            z = torch.randn(C, B + 1, V, generator=g)
            t = z[:, :B].argmax(-1).to(torch.int32)
            for b in range(C):                              # a wrong candidate somewhere, or none
                i = int(torch.randint(0, B + 1, (1,), generator=g))
                if i < B:
                    t[b, i] = (t[b, i] + 1) % V
            zt.copy_(z)
            y.copy_(t)
            return z, t

        def check(z, t):
            torch.cuda.synchronize()
            for b in range(C):
                r, n = oracle.verify_block(f64(z[b]), torch.zeros(B, 1).numpy(), t[b].numpy(), 0.0, 0, 0, b)[:2]
                assert (int(acc[b]), int(nxt[b])) == (r, n), b

        inputs()
        run = lambda: lsp.lsp_verify(st, zt, zq, y, sp, acc, nxt)
        run()
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph):
            run()
        for call in (graph.replay, run, graph.replay, graph.replay, run, run):
            want = inputs()
            call()
            check(*want)
        assert lsp.lsp_get_error(st) == (lsp.LSP_OK, 0)
    finally:
        lsp.lsp_state_destroy(st)
