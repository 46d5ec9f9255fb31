"""Long view updates (a chunk of a prefix in one call) take the segmented tcgen05 fold;
checked against the oracle at the edges of its 128-row blocks, for every head grouping it
is instantiated for, and where a later block raises the scores' reference."""
import numpy as np
import pytest
import torch

import oracle
from tests.gpu_common import check_view_state, f64, fold_chunk, lsp_lib
from paper_2609_37029_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def lsp():
    return lsp_lib()


def _shape(rep=4, nkv=2, **kw):
    base = dict(C=3, B=16, L=2, D=1, H=256, nq=rep * nkv, nkv=nkv, d=128, F=256, V=1024, W=40, R=16, rc=16)
    return synth.LspShape("fold", **{**base, **kw})


def _run(lsp, s, chunks, atol=1e-4, edit=None):
    """Fold each chunk (capacity, accepted counts) on the GPU and in the oracle; rows past the
    accepted count hold NaN on the GPU side (they must not be read into any result)."""
    st = lsp.lsp_state_create(lsp.make_config(s))
    try:
        w = synth.make_weights(s, seed=3)
        lsp.lsp_state_init(st, w["G"].cuda())
        ost, Gn = oracle.state_init(s), f64(w["G"])
        for n, (rows, acc) in enumerate(chunks):
            k, v, h = synth.make_features(s, rows, seed=70 + n)
            if edit:
                edit(k, v)
            for b, a in enumerate(acc):
                k[b, :, a:] = v[b, :, a:] = h[b, :, a:] = float("nan")
            fold_chunk(lsp, st, ost, s, Gn, k, v, h, torch.tensor(acc, dtype=torch.int32))
        torch.cuda.synchronize()
        check_view_state(lsp, st, ost, s, atol)
        assert lsp.lsp_get_error(st) == (lsp.LSP_OK, 0)
    finally:
        lsp.lsp_state_destroy(st)


@pytest.mark.parametrize("acc", [[1, 0, 128], [127, 129, 256], [300, 1, 257], [0, 0, 0]])
def test_fold_block_edges(lsp, acc):
    _run(lsp, _shape(), [(300, acc), (260, [min(a, 260) for a in reversed(acc)])])


@pytest.mark.parametrize("rep", range(1, 9))
def test_fold_head_groupings(lsp, rep):
    _run(lsp, _shape(rep=rep, R=16 if rep % 2 else 7), [(400, [400, 131, 2])])


@pytest.mark.parametrize("variant", [{"W": 0}, {"W": 256}, {"no_boundary": True}, {"C": 40, "B": 8, "L": 3, "W": 16}])
def test_fold_variants(lsp, variant):
    s = _shape(**variant)
    acc = [(37 * b) % 641 for b in range(s.C)]          # many units and shares of uneven length
    _run(lsp, s, [(640, [min(a, 640) for a in acc])])


def test_fold_moves_the_reference(lsp):
    """Keys grow along the prefix, so that later blocks pass the first block's maximum by far
    more than the slack.  Scores reach |s| <= 64: fp32 products and sums leave <= 64 * 2^-20 on
    each, twice (weight and normaliser), times |v| <= 4: 5e-4."""
    def grow(k, v):
        k *= torch.linspace(0.2, 180.0, k.shape[2]).view(1, 1, -1, 1, 1)
    _run(lsp, _shape(), [(700, [700, 390, 150])], atol=5e-4, edit=grow)


def test_fold_reports_a_bad_count_and_leaves_that_request(lsp):
    s = _shape()
    st = lsp.lsp_state_create(lsp.make_config(s))
    try:
        w = synth.make_weights(s, seed=3)
        lsp.lsp_state_init(st, w["G"].cuda())
        ost = oracle.state_init(s)
        k, v, h = synth.make_features(s, 300, seed=5)
        lsp.lsp_view_update(st, k.cuda(), v.cuda(), h.cuda(), torch.tensor([200, 301, -1], dtype=torch.int32).cuda())
        assert lsp.lsp_get_error(st) == (lsp.LSP_ERR_STATE, lsp.LSP_DEV_BAD_DELTA)
        oracle.view_update(s, ost, f64(w["G"]), f64(k), f64(v), f64(h), np.array([200, 0, 0], dtype=np.int32))
        check_view_state(lsp, st, ost, s)
    finally:
        lsp.lsp_state_destroy(st)
