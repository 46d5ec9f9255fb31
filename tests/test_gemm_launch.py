"""How the projection GEMM is launched, host logic only (no GPU): every token row and weight row in
exactly one item, and the shared memory, tensor memory and tensor-map boxes that a CTA of it may use."""
import pytest

SHAPES = [(4096, 4096), (6144, 4096), (4096, 12288), (12288, 4096), (151936, 4096), (151936, 5120), (17408, 5120),
          (64, 256), (1, 64), (1183, 7016), (30561, 416), (257, 20480)]


@pytest.fixture(scope="module")
def lsp():
    from paper_2609_37029_gb300 import build
    build.build()
    from paper_2609_37029_gb300 import lsp as mod
    return mod


def test_qwen3_8b_round(lsp):
    info = lambda *a: lsp.lsp_gemm_launch_info(lsp.LSP_DTYPE_BF16, *a, 152)
    gu = info(256, 12288, 4096, 1, 0)                      # gate/up: one group of 256 tokens
    assert (gu.token_groups, gu.tokens_per_group, gu.accumulators, gu.splits) == (1, 256, 2, 1)
    for n, k, splits in [(6144, 4096, 3), (4096, 4096, 4), (4096, 12288, 9)]:
        a = info(256, n, k, 0, 0)
        assert (a.splits, a.token_groups, a.tokens_per_group) == (splits, 1, 256)
        assert a.splits == lsp.lsp_gemm_plan_info(lsp.LSP_DTYPE_BF16, 256, n, k, 0, 152)[0]
    head = info(256, 151936, 4096, 0, 1)                   # the LM head is walked by one CTA an SM
    assert head.ctas == 152 < head.tiles
    assert info(512, 17408, 5120, 1, 0).token_groups == 2


@pytest.mark.parametrize("N,K", SHAPES)
@pytest.mark.parametrize("swiglu", [0, 1])
@pytest.mark.parametrize("dtype", ["bf16", "f32"])
def test_launch_covers_and_fits(lsp, N, K, swiglu, dtype):
    dt, es = (lsp.LSP_DTYPE_BF16, 2) if dtype == "bf16" else (lsp.LSP_DTYPE_F32, 4)
    kblocks = -(-K * es // 128)
    for sms in (152, 148, 8):
        for M in list(range(1, 513, 7)) + [16, 17, 112, 128, 129, 144, 145, 256, 257, 272, 273, 511, 512]:
            for splits in (0,) if swiglu else (0, 1, 3):
                a = lsp.lsp_gemm_launch_info(dt, M, N, K, swiglu, splits, sms)
                what = (M, splits, sms)
                # token rows: groups of 16 x, each of one or two accumulators of at most 128 and 8 x
                assert a.token_groups * a.tokens_per_group >= M > (a.token_groups - 1) * a.tokens_per_group, what
                assert a.tokens_per_group % 16 == 0 and a.tokens_per_group <= 256 and a.accumulators in (1, 2), what
                per_acc = a.tokens_per_group // a.accumulators
                assert per_acc * a.accumulators == a.tokens_per_group and per_acc <= 128 and per_acc % 8 == 0, what
                # weight rows: UMMA N in steps of 16, tensor-map boxes of at most 256 rows
                feats = a.tile_rows // 2 if swiglu else a.tile_rows
                assert a.tile_rows % 16 == 0 and 16 <= a.tile_rows <= 256 and a.tiles * feats >= N > (a.tiles - 1) * feats, what
                assert swiglu or a.tile_rows % 32 == 0, what
                assert not swiglu or a.tile_rows % 32 == 16, what    # rows of an odd number of 16-byte vectors
                assert 1 <= a.splits <= kblocks and (splits == 0 or a.splits == min(splits, kblocks)), what
                items = a.tiles * a.token_groups * a.splits
                walk = a.ctas != items
                assert not walk or (a.ctas == sms < items and not swiglu), what
                # shared memory: both rings, the staging of a walk, 1 KB of alignment
                assert 2 <= a.weight_stages <= 8 and 2 <= a.activation_stages <= 8, what
                assert a.tokens_per_group > 128 or a.weight_stages == a.activation_stages, what
                ring = (a.weight_stages * a.tile_rows + a.activation_stages * a.tokens_per_group) * 128
                assert ring + (32768 if walk else 0) + 1024 < a.smem_bytes <= 227 * 1024, what
                # an accumulator's 128 lanes read from the last stage's second tile on
                assert (a.activation_stages * a.tokens_per_group - per_acc + 128) * 128 < a.smem_bytes, what
                # tensor memory: a power of two that holds every set
                cols = a.accumulator_sets * a.accumulators * -(-a.tile_rows // 32) * 32
                assert cols <= a.tmem_columns <= 512 and a.tmem_columns & (a.tmem_columns - 1) == 0 and a.tmem_columns >= 32, what
                assert a.accumulator_sets == 1 or walk, what
                if swiglu:                                       # the output tile is staged over the rings
                    assert a.tokens_per_group * feats * es <= ring, what


def test_bad_arguments(lsp):
    for args in [(0, 128, 128, 0, 0, 152), (513, 128, 128, 0, 0, 152), (16, 0, 128, 0, 0, 152), (16, 128, 0, 0, 0, 152),
                 (16, 128, 128, 0, -1, 152), (16, 128, 128, 0, 0, 0),
                 (16, 128, 100, 0, 0, 152),                      # K x 2 no multiple of 16 bytes
                 (16, 128, 128, 1, 2, 152)]:                     # gate/up takes no splits
        with pytest.raises(lsp.LspError):
            lsp.lsp_gemm_launch_info(lsp.LSP_DTYPE_BF16, *args)
    with pytest.raises(lsp.LspError):
        lsp.lsp_gemm_launch_info(7, 16, 128, 128, 0, 0, 152)
