"""The fp32 attention's forms in whole rounds against the oracle: two, four and eight queries a CTA
(more than two where that makes more CTAs than SMs), a ragged last group, rows with and
without padding, and rows in chunks where they do not fit; windows not yet full, and wrapped."""
import pytest

from tests.gpu_common import lsp_lib
from tests.test_gpu_round import _run_rounds
from paper_2609_37029_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("C,B,W,R", [
    (1, 5, 64, 16),       # two queries a CTA, the last group of one
    (8, 5, 64, 16),       # four, the last group of one
    (8, 7, 48, 8),        # four, the last group of three
    (8, 16, 64, 16),      # eight
    (6, 1, 32, 4),        # one query
    (2, 8, 410, 16),      # rows without padding
    (2, 8, 500, 16),      # rows in chunks
])
def test_f32_round(C, B, W, R):
    s = synth.LspShape("f32a", C=C, B=B, L=2, D=2, H=256, nq=8, nkv=2, d=64, F=256, V=1024, W=W, R=R, rc=16, dtype="f32")
    _run_rounds(lsp_lib(), s, (W // 2, W + 37))
