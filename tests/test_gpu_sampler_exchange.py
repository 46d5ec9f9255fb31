"""The one-launch sampler's exchange of keys: where the choice between leaders and direct reads
lies, for each layout of the direct words (up to four requests a group, and more), where both
take turns in one call, and past the point where the 12-bit step tags come round again."""
import pytest
import torch

from tests.gpu_common import lsp_lib
from tests.test_gpu_sampler_groups import test_sampler_edges as _edges
from paper_2609_37029_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("C,B,V,rc,temperature", [
    (1, 4, 10240, 64, 1.0),     # 32 CTAs of ten tiles
    (2, 3, 10224, 32, 0.0),
    (3, 5, 5120, 64, 0.7),
    (4, 4, 10240, 64, 0.0),
    (5, 3, 992, 64, 1.0),       # 31 CTAs
    (8, 4, 10240, 32, 0.0),
    (8, 4, 10256, 64, 1.0),     # one tile more: leaders
    (9, 4, 8192, 64, 1.0),      # two groups: 32 CTAs of eight tiles
    (11, 3, 8192, 64, 0.0),
    (16, 3, 8208, 64, 0.0),     # one tile more: leaders
    (20, 4, 9008, 64, 1.0),     # leaders for the first 16 requests, direct reads for the other four
])
@pytest.mark.parametrize("noalloc", [False, True])
def test_exchange_edges(C, B, V, rc, temperature, noalloc):
    _edges(C, B, V, rc, temperature, noalloc)


@pytest.mark.parametrize("C,V,dtype", [(16, 20000, "bf16"), (17, 9008, "bf16"), (3, 2048, "bf16"), (2, 4096, "f32")])
def test_tags_come_round(C, V, dtype):
    """300 launches of 16 steps: the 4096 tags are used up after 256.  The same inputs give the
    same tokens every time."""
    lsp = lsp_lib()
    B = 16
    s = synth.LspShape("sg", C=C, B=B, L=1, D=1, H=128, nq=1, nkv=1, d=128, F=64, V=V, W=16, R=16, rc=64, dtype=dtype)
    st = lsp.lsp_state_create(lsp.make_config(s))
    try:
        g = torch.Generator(device="cuda").manual_seed(V)
        # two sets of logits in turn, so that a stale key would be another token
        zs = [torch.randn(C, B, V, generator=g, device="cuda") * 2.0 for _ in range(2)]
        Ec, Wc = ((torch.randn(V, 64, generator=g, device="cuda") * 0.5).to(s.torch_dtype) for _ in range(2))
        prev = torch.randint(0, V, (C,), generator=g, dtype=torch.int32, device="cuda")
        sp = lsp.make_sample_params(1.0, seed=77, rnd=1)
        out = torch.full((300, C, B), -1, dtype=torch.int32, device="cuda")
        for i in range(300):
            lsp.lsp_sample(st, zs[i % 2], prev, Ec, Wc, sp, out[i], None)
        torch.cuda.synchronize()
        assert torch.equal(out, out[:2].repeat(150, 1, 1)) and not torch.equal(out[0], out[1])
        assert lsp.lsp_get_error(st) == (lsp.LSP_OK, 0)
    finally:
        lsp.lsp_state_destroy(st)
