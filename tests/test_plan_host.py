"""Which kernels a configuration takes (host arithmetic; no GPU)."""
import ctypes

import pytest

import paper_1409_5705_b200 as S

TILES, PAIRS, FEW = 1, 2, 3


def bf16(rows, cols, samples, workers=1, **more):
    return S.make_config(S.MLR, rows, cols, workers, samples // workers, 0.05, S.PREC_BF16, **more)


def test_arguments():
    cfg = bf16(64, 256, 128)
    assert S.sfb_get_plan(cfg, 128)[0] == TILES and S.sfb_get_plan(cfg, 32)[0] == FEW
    for n in (0, 129):
        with pytest.raises(S.SfbError):
            S.sfb_get_plan(cfg, n)
    assert S.lib().sfb_get_plan(ctypes.byref(cfg), 1, None, None, None) == -1
    assert S.sfb_get_plan(S.make_config(S.MLR, 64, 256, 1, 8, 0.1, S.PREC_TF32X3), 8) == (4, 1, 0)
    assert S.sfb_get_plan(S.make_config(S.MLR, 64, 256, 1, 8, 0.1, S.PREC_FP32_FFMA), 8) == (0, 1, 0)


# Logits where pairs of CTAs take longer than forward_kernel: many classes with few features, whose softmax has twice the partials to
# merge; two and a half rounds of short tiles; a few tiles of a long contraction, which clusters of eight cut as well.
@pytest.mark.parametrize("rows,cols,samples", [(36_667, 912, 364), (78_798, 1_716, 156), (44_790, 2_884, 237), (121, 3_772, 180),
                                               (3, 6_764, 244), (89, 6_608, 533), (9_760, 200, 300), (190, 708, 513)])
def test_logits_that_pairs_would_slow_down(rows, cols, samples):
    assert S.sfb_get_plan(bf16(rows, cols, samples), samples)[0] == TILES


# ... and where they are the faster ones: uneven rounds of long tiles, clusters that are not all resident.
@pytest.mark.parametrize("rows,cols,samples", [(10_000, 20_000, 1_024), (10_000, 4_000, 512), (20_000, 4_000, 256), (281, 7_060, 146),
                                               (2_220, 2_588, 144), (873, 2_800, 634)])
def test_logits_on_pairs(rows, cols, samples):
    assert S.sfb_get_plan(bf16(rows, cols, samples), samples)[0] == PAIRS


# Up to 64 samples: the kernel of few samples, but in a worker's call for more than 40 with fewer than 12 k-blocks, and for the longest
# contractions of a few tiles.
@pytest.mark.parametrize("rows,cols,samples,call,step", [
    (64, 64, 40, True, True), (64, 64, 41, False, True), (300, 708, 64, True, True), (300, 704, 64, False, True), (3_048, 268, 56, False, True),
    (107, 84, 44, False, True), (4_999, 3_004, 64, True, True), (4_999, 3_004, 65, False, False), (512, 18_000, 8, True, True),
    (512, 18_004, 8, False, False), (513, 24_000, 64, True, True)])
def test_logits_of_few_samples(rows, cols, samples, call, step):
    assert (S.sfb_get_plan(bf16(rows, cols, 2 * samples, workers=2), samples)[0] == FEW) == call
    assert (S.sfb_get_plan(bf16(rows, cols, samples), samples)[0] == FEW) == step


# The softmax in one launch: up to 128 samples (64 with more than 6,000 features) and eight partials, all of the context's samples at once.
@pytest.mark.parametrize("rows,cols,samples,merged", [(64, 256, 128, 1), (64, 256, 129, 0), (64, 6_000, 128, 1), (64, 6_004, 65, 0),
                                                      (64, 6_004, 64, 1), (256, 256, 16, 1), (257, 256, 16, 0)])
def test_softmax_in_one_launch(rows, cols, samples, merged):
    assert S.sfb_get_plan(bf16(rows, cols, samples), samples)[2] == merged
    if samples > 1:
        assert S.sfb_get_plan(bf16(rows, cols, samples), samples - 1)[2] == 0


# Products of pairs of words of fewer tiles than pairs of CTAs: narrow tiles are cut although they have few k-blocks, products that drain their
# accumulator at every k-block (sparse coding in fp32 mode) into more parts than others.
def test_parts_of_products_of_words():
    dml = S.make_config(S.DML, 28, 1_656, 1, 193, 1e-3, S.PREC_BF16)
    assert S.sfb_get_plan(dml, 193)[:2] >= (5, 2)
    assert S.sfb_get_plan(S.make_config(S.DML, 137, 1_592, 7, 15, 1e-3, S.PREC_BF16), 15)[1] > 1
    assert S.sfb_get_plan(S.make_config(S.DML, 500, 8_000, 1, 256, 1e-3, S.PREC_BF16), 256)[1] < 31
    assert S.sfb_get_plan(S.make_config(S.DML, 1_000, 20_000, 16, 64, 1e-3, S.PREC_BF16), 1_024)[1] >= 2


# The form of the coder where forms round differently.  bf16: two products an iteration where W^T W would have larger errors (five iterations
# of 3,445 x 3,172, K = 156: the codes 5.1e-6 from 64 bits, 7.8e-6 on W^T W); fp32: pairs of words rather than two products of FMAs, W^T W
# in fp64 rather than either where it is the faster one.
@pytest.mark.parametrize("rows,cols,samples,iters,prec,product", [
    (3_445, 3_172, 156, 5, S.PREC_BF16, 5), (8_078, 84, 10, 5, S.PREC_BF16, 5), (10_000, 5_000, 512, 20, S.PREC_BF16, 6),
    (4_960, 820, 29, 5, S.PREC_FP32, 5), (1_130, 1_156, 251, 20, S.PREC_FP32, 5), (198, 1_408, 685, 5, S.PREC_FP32, 5),
    (5_521, 116, 82, 5, S.PREC_FP32, 7), (2_000, 1_000, 128, 20, S.PREC_FP32, 7), (1_720, 1_148, 230, 20, S.PREC_FP32, 7)])
def test_form_of_the_coder(rows, cols, samples, iters, prec, product):
    cfg = S.make_config(S.SC, rows, cols, 1, samples, 1e-3, prec, sc_ista_iters=iters, sc_prox=1, sc_lipschitz=1.0)
    assert S.sfb_get_plan(cfg, samples)[0] == product


# Room for parts of tiles only where some call's logits take pairs of CTAs that leave some.
def test_workspace_of_the_logits_on_pairs():
    size = lambda *a, **k: S.sfb_workspace_bytes(bf16(*a, **k))  # noqa: E731
    assert size(64, 256, 129) - size(64, 256, 128) < 100_000
    rows, cols, K = 325_000, 10_000, 1_024             # operands, logits, probabilities, samples (staged, fp32, bf16, label sums), partials
    need = rows * 10_048 * 2 + K * rows * 6 + K * cols * 14 + K * rows // 256 * 8
    assert need < size(rows, cols, K) < need + 10_000_000
    cfg = bf16(10_000, 20_000, 1_024)
    assert S.sfb_get_plan(cfg, 1_024)[:2] == (PAIRS, 2)
    assert size(10_000, 20_000, 1_024, workers=16) > 10_000 * 20_032 * 2 + 1_024 * (10_000 * 6 + 20_000 * 14) + 19_000_000
