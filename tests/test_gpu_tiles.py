"""GPU parity of kernels that a size selects and the other files' shapes do not reach: the streamed
pooling, every tile of the projection shortcut, the pipelined k-bit pack kernel with each number of
planes, the box filter with four outputs per thread.  Edges of tiles, remainders, ragged tensors."""
import numpy as np
import pytest
import torch

import paper_1603_05279_b200 as X
from test_gpu_bgrad import test_binary_gradient_backward_parity as backward_parity
from test_gpu_fused import test_fused_binactiv_parity as fused_parity
from test_gpu_options import _index_of_planes
from test_gpu_options import test_kbit_block_parity as kbit_block_parity
from test_gpu_parity import test_block_parity as block_parity
from util import GuardSet, assert_close, dev, host, unpack_weights

pytestmark = pytest.mark.gpu


def sms():
    return torch.cuda.get_device_properties(0).multi_processor_count


def rng(seed):
    return np.random.Generator(np.random.Philox(seed))


# (N, C, H, W, k, stride, pad): a last chunk of one plane and a tensor that is not a multiple of four
# floats; several planes per chunk; clipped windows; the largest planes that are streamed
@pytest.mark.parametrize("relu", [False, True])
@pytest.mark.parametrize("case", [(11, 256, 36, 34, 3, 2, 1), (9, 301, 30, 37, 2, 3, 1), (24, 128, 35, 35, 4, 3, 3),
                                  (40, 90, 21, 23, 5, 2, 4), (7, 400, 30, 31, 7, 2, 3), (40, 90, 21, 23, 6, 2, 3),
                                  (90, 129, 11, 12, 1, 2, 0),
                                  (197, 193, 9, 7, 2, 2, 0), (150, 256, 13, 13, 3, 2, 0),
                                  (10, 256, 27, 27, 3, 2, 1), (3, 805, 38, 40, 5, 3, 2)])
def test_streamed_maxpool_is_exact(oracle, case, relu):
    N, C, H, W, k, s, p = case
    x = rng(sum(case)).standard_normal((N, C, H, W)).astype(np.float32)
    want = oracle.maxpool2d(x, k, s, p, relu=relu)
    gs = GuardSet()
    out = gs.new("out", want.shape)
    X.xnor_maxpool2d(dev(x), k, s, p, relu, out)
    X.xnor_check_device()
    gs.check()
    assert np.array_equal(host(out), want)


# tiles of 64 x 32 (the first two, with tails of pixels, channels and filters, and the fifth), 128 x 64 (the two
# between) and 32 x 16 by the rule of launch_shortcut_conv1x1 on 148 SMs; planes of odd size
@pytest.mark.parametrize("case", [(14, 131, 29, 29, 250, 2), (13, 45, 17, 14, 230, 1),
                                  (64, 64, 28, 28, 130, 1), (40, 70, 57, 55, 96, 2), (16, 128, 28, 28, 256, 2),
                                  (5, 70, 15, 13, 90, 1), (2, 256, 14, 14, 512, 2), (1, 33, 9, 9, 40, 2)])
def test_shortcut_tiles(oracle, case):
    N, C, H, W, Co, s = case
    g = rng(sum(case))
    x = g.standard_normal((N, C, H, W)).astype(np.float32)
    w = (0.05 * g.standard_normal((Co, C))).astype(np.float32)
    gs = GuardSet()
    out = gs.new("out", (N, Co, (H - 1) // s + 1, (W - 1) // s + 1))
    X.xnor_shortcut_conv1x1(dev(x), dev(w), s, out)
    gs.check()
    assert_close(host(out), oracle.shortcut_conv1x1(x, w.reshape(Co, C, 1, 1), s), "shortcut")


# one warp per pixel group and groups shared by warps; channel tails; 16- and 4-byte copies
@pytest.mark.parametrize("kbits", [2, 3, 4, 5, 7])
@pytest.mark.parametrize("case", [(90, 40, 28, 28, 3, 1), (2, 300, 10, 14, 5, 2), (3, 70, 9, 11, 3, 1)])
def test_kbit_pack(oracle, case, kbits):
    N, C, H, W, k, p = case
    g = rng(sum(case) + kbits)
    x = (0.6 * g.standard_normal((N, C, H, W))).astype(np.float32)
    scale = (1.0 + 0.2 * g.standard_normal(C)).astype(np.float32)
    shift = (0.2 * g.standard_normal(C)).astype(np.float32)
    d = X.make_desc(N, C, H, W, 8, k, k, 1, p)
    gs = GuardSet()
    planes = gs.new("x_planes", (kbits, N, H, W, (C + 31) // 32), torch.int32)
    _, A0, K0 = X.alloc_binactiv(d)
    A, K = gs.like("A", A0), gs.like("K", K0)
    X.xnor_binactiv_kbit(dev(x), dev(scale), dev(shift), d, kbits, planes, A, K)
    gs.check()
    y = oracle.bn_affine(x, scale, shift)
    codes = 2 * _index_of_planes(host(planes), C) - (2 ** kbits - 1)
    assert np.array_equal(codes, oracle.quantize_k(y, kbits).astype(np.int64))
    A_or = oracle.channel_abs_mean(y)
    assert_close(host(A), A_or, "A")
    assert_close(host(K), oracle.box_filter(A_or, k, k, 1, p), "K")


# the decision points themselves and their neighbours, whole and partial channel words
@pytest.mark.parametrize("kbits", [1, 2, 3, 4, 5])
@pytest.mark.parametrize("C,H", [(64, 8), (43, 8), (64, 7)])
def test_kbit_decision_points(oracle, kbits, C, H):
    levels = 2 ** kbits - 1
    tau = np.array([(2 * j - 1) / levels - 1 for j in range(1, levels + 1)], np.float32)
    edges = np.concatenate([tau, np.nextafter(tau, np.float32(-9)), np.nextafter(tau, np.float32(9)),
                            np.array([0.0, -0.0, 1, -1, 3, -3, np.inf, -np.inf], np.float32)])
    x = rng(kbits + C).choice(edges, (2, C, H, H)).astype(np.float32)
    d = X.make_desc(2, C, H, H, 8, 1, 1, 1, 0)
    gs = GuardSet()
    planes = gs.new("x_planes", (kbits, 2, H, H, (C + 31) // 32), torch.int32)
    _, A, K = X.alloc_binactiv(d)
    X.xnor_binactiv_kbit(dev(x), None, None, d, kbits, planes, A, K)
    gs.check()
    codes = 2 * _index_of_planes(host(planes), C) - levels
    assert np.array_equal(codes, oracle.quantize_k(x, kbits).astype(np.int64))


# pixels not a multiple of the 128 of a warp, images ending inside a run; one to five channel words, tails
@pytest.mark.parametrize("kbits", [1, 2])
@pytest.mark.parametrize("case", [(83, 100, 28, 29, 1, 0), (83, 33, 29, 28, 1, 0), (70, 130, 30, 32, 3, 1),
                                  (300, 16, 12, 19, 3, 1), (66, 64, 32, 32, 1, 0)])
def test_wide_pack(oracle, case, kbits):
    test_kbit_pack(oracle, case, kbits)


# max|g| by a cluster per image (74 images and up on 148 SMs), images of odd size and of one chunk per thread
@pytest.mark.parametrize("shape", [(75, 33, 5, 5, 17, 3, 1), (74, 32, 21, 19, 101, 3, 1)])
def test_gradient_maximum_of_many_images(oracle, shape):
    backward_parity(oracle, shape)


# two bit planes per pass in every schedule, an even and an odd number of passes; channel tails, both phases
@pytest.mark.parametrize("engine", [X.XNOR_ENGINE_UMMA_SINGLE, X.XNOR_ENGINE_UMMA_STREAM, X.XNOR_ENGINE_UMMA_PAIR,
                                    X.XNOR_ENGINE_UMMA_PAIR_STREAM])
@pytest.mark.parametrize("kbits", [2, 4, 5])
@pytest.mark.parametrize("shape", [(16, 70, 19, 18, 64, 3, 2, 1), (12, 128, 20, 21, 160, 3, 1, 1), (4, 33, 8, 8, 16, 1, 1, 0)])
def test_kbit_two_planes_per_pass(oracle, shape, kbits, engine):
    kbit_block_parity(oracle, shape, kbits, engine)


@pytest.mark.parametrize("valid", [False, True])
@pytest.mark.parametrize("case", [(190, 2, 56, 56, 3, 1), (260, 2, 55, 44, 5, 2), (300, 1, 51, 48, 5, 0),
                                  (360, 1, 37, 50, 3, 0)])
def test_box_filter_rows(oracle, case, valid):
    N, C, H, W, k, p = case
    Ho, Wo = H + 2 * p - k + 1, W + 2 * p - k + 1
    assert Wo % 4 == 0 and (Ho * Wo + 255) // 256 * N > 16 * sms()         # four outputs per thread from here on
    x = rng(sum(case)).standard_normal((N, C, H, W)).astype(np.float32)
    d = X.make_desc(N, C, H, W, 8, k, k, 1, p, X.XNOR_FLAG_K_VALID_TAPS if valid else 0)
    gs = GuardSet()
    xp, A, K = (gs.like(n, t) for n, t in zip(("x_packed", "A", "K"), X.alloc_binactiv(d)))
    X.xnor_binactiv(dev(x), None, None, d, xp, A, K)
    gs.check()
    A_or = oracle.channel_abs_mean(x)
    assert_close(host(A), A_or, "A")
    want = oracle.box_filter_valid_taps(A_or, k, k, 1, p) if valid else oracle.box_filter(A_or, k, k, 1, p)
    assert_close(host(K), want, "K")


# fused, the schedule the planner takes: resident in several slabs of few K-steps, streaming with two warps per
# quarter of the lanes, small problems in slabs of 64
@pytest.mark.parametrize("case,resident,slabs,filters,parts", [
    ((40, 16, 14, 14, 544, 1, 1, 0, 3, 1, 1, True), 1, 3, 192, 9),
    ((30, 16, 9, 19, 288, 3, 2, 1, 1, 1, 0, False), 1, 3, 96, 9),
    ((60, 416, 14, 13, 384, 1, 2, 0, 3, 1, 1, True), 0, 3, 128, 6),
    ((1, 352, 9, 9, 224, 3, 1, 1, 3, 1, 1, False), 1, 4, 64, 8),
    ((2, 33, 7, 5, 96, 3, 1, 1, 3, 2, 1, True), 1, 2, 64, 4)])
def test_fused_schedules(oracle, case, resident, slabs, filters, parts):
    N, C, H, W, Co, k, s, p = case[:8]
    d = X.make_desc(N, C, H, W, Co, k, k, s, p)
    plan = X.xnor_conv2d_plan(d, fused=True)
    assert (plan.resident, plan.slabs, plan.slab_filters) == (resident, slabs, filters)
    assert X.xnor_conv2d_binactiv_parts(d) == parts
    fused_parity(oracle, case, X.XNOR_ENGINE_AUTO)


# the plain convolution: several resident slabs of few K-steps, streaming because it is faster, pairs streaming
# slabs of more than 128 filters (and of 256, with one accumulator, where a pair has one item), and both sides
# of the 16 slabs that a small problem may keep resident
@pytest.mark.parametrize("shape,resident,pair,slabs,filters", [
    ((30, 33, 31, 30, 428, 1, 1, 2, 0), 1, 0, 2, 224), ((16, 128, 28, 28, 256, 3, 3, 2, 1), 1, 0, 2, 128),
    ((136, 944, 8, 19, 512, 1, 1, 1, 0), 0, 0, 4, 128), ((11, 544, 22, 37, 178, 3, 3, 1, 1), 0, 1, 1, 192),
    ((40, 300, 14, 13, 250, 7, 7, 1, 3), 0, 1, 1, 256),
    ((170, 90, 15, 16, 256, 5, 5, 1, 2), 1, 1, 2, 128), ((42, 320, 21, 22, 200, 3, 3, 2, 1), 0, 1, 2, 128),
    ((1, 256, 7, 7, 256, 1, 1, 1, 0), 1, 0, 16, 16), ((1, 256, 7, 7, 272, 1, 1, 1, 0), 0, 0, 17, 16),
    ((1, 512, 7, 7, 512, 3, 3, 1, 1), 1, 0, 16, 32), ((1, 512, 7, 7, 528, 3, 3, 1, 1), 0, 0, 17, 32)])
def test_plain_schedules(oracle, shape, resident, pair, slabs, filters):
    N, C, H, W, Co, kh, kw, s, p = shape
    plan = X.xnor_conv2d_plan(X.make_desc(N, C, H, W, Co, kh, kw, s, p))
    assert (plan.resident, plan.pair, plan.slabs, plan.slab_filters) == (resident, pair, slabs, filters)
    block_parity(oracle, shape, X.XNOR_ENGINE_AUTO)


# several items per CTA, drained in chunks of 64 filters that the warps of a lane quarter take in turn: one to
# four chunks, a short last chunk, turns that move on from item to item, filters beyond C_out, warps that skip items.
# Items of few K-steps: resident with three warps per quarter (single CTAs, pairs), streaming with two
@pytest.mark.parametrize("engine", [X.XNOR_ENGINE_AUTO, X.XNOR_ENGINE_UMMA_STREAM, X.XNOR_ENGINE_UMMA_PAIR])
@pytest.mark.parametrize("residual", [False, True])
@pytest.mark.parametrize("Co,k", [(16, 1), (48, 3), (70, 1), (80, 1), (112, 3), (144, 3), (200, 1), (240, 1)])
def test_drained_chunks(oracle, Co, k, residual, engine):
    N, C, H, W = 160, 16, 23, 24
    d = X.make_desc(N, C, H, W, Co, k, k, 1, k // 2)
    g = rng(Co + k)
    x = g.standard_normal((N, C, H, W)).astype(np.float32)
    w = g.standard_normal((Co, C, k, k)).astype(np.float32)
    res = g.standard_normal((N, Co, H, W)).astype(np.float32) if residual else None
    wp, alpha = X.alloc_weights(Co, C, k, k)
    xp, A, K = X.alloc_binactiv(d)
    gs = GuardSet()
    out = gs.like("out", X.alloc_out(d))
    X.xnor_binarize_weights(dev(w), wp, alpha)
    X.xnor_binactiv(dev(x), None, None, d, xp, A, K)
    X.xnor_set_engine(engine)
    try:
        X.xnor_conv2d_forward(xp, wp, alpha, K, None if res is None else dev(res), d, out)
    finally:
        X.xnor_set_engine(X.XNOR_ENGINE_AUTO)
    X.xnor_check_device()
    gs.check()
    assert_close(host(out), oracle.xnor_block(x, w, 1, k // 2, None, None, res).out, "out")


# The remaining schedules of the drain, through both lean store branches (acc_out absent, with and without a
# residual), against the CUDA cores bit for bit and the oracle on the outer images: streaming and streaming pairs with one
# draining warp per quarter (64 K-steps and more), two and three chunks per item, four items per CTA; pairs
# streaming short items, two chunks of 4 + 2 groups; one slab of 256 filters with one accumulator
@pytest.mark.parametrize("residual", [False, True])
@pytest.mark.parametrize("shape,engine,resident,pair,slabs,filters", [
    ((100, 256, 28, 28, 128, 3, 1, 1), X.XNOR_ENGINE_UMMA_STREAM, 0, 0, 1, 128),
    ((100, 256, 28, 28, 128, 3, 1, 1), X.XNOR_ENGINE_UMMA_PAIR_STREAM, 0, 1, 1, 128),
    ((60, 490, 35, 30, 190, 3, 1, 1), X.XNOR_ENGINE_AUTO, 0, 1, 1, 192),
    ((100, 64, 28, 28, 96, 3, 1, 1), X.XNOR_ENGINE_UMMA_PAIR_STREAM, 0, 1, 1, 96),
    ((40, 300, 14, 13, 256, 7, 1, 3), X.XNOR_ENGINE_AUTO, 0, 1, 1, 256)])
def test_drain_of_streamed_items(oracle, shape, engine, resident, pair, slabs, filters, residual):
    N, C, H, W, Co, k, s, p = shape
    d = X.make_desc(N, C, H, W, Co, k, k, s, p)
    g = rng(Co + k)
    x = g.standard_normal((N, C, H, W)).astype(np.float32)
    w = g.standard_normal((Co, C, k, k)).astype(np.float32)
    wp, alpha = X.alloc_weights(Co, C, k, k)
    xp, A, K = X.alloc_binactiv(d)
    gs = GuardSet()
    want = X.alloc_out(d)
    out = gs.like("out", want)
    res = dev(g.standard_normal(tuple(out.shape)).astype(np.float32)) if residual else None
    X.xnor_binarize_weights(dev(w), wp, alpha)
    X.xnor_binactiv(dev(x), None, None, d, xp, A, K)
    try:
        X.xnor_set_engine(engine)
        plan = X.xnor_conv2d_plan(d, residual=residual)
        assert (plan.resident, plan.pair, plan.slabs, plan.slab_filters) == (resident, pair, slabs, filters)
        X.xnor_conv2d_forward(xp, wp, alpha, K, res, d, out)
        X.xnor_set_engine(X.XNOR_ENGINE_POPC)
        X.xnor_conv2d_forward(xp, wp, alpha, K, res, d, want)
    finally:
        X.xnor_set_engine(X.XNOR_ENGINE_AUTO)
    X.xnor_check_device()
    gs.check()
    assert torch.equal(out, want)
    for n in (0, N - 1):
        r = oracle.xnor_block(x[n:n + 1], w, s, p, residual=None if res is None else host(res[n:n + 1]))
        assert_close(host(out[n:n + 1]), r.out, "out, image %d" % n)


# fused, four items and more per CTA: chunks of 4 + 2 groups over three warps (resident, single CTAs and pairs) and
# two (streaming), 4 + 4 + 2 and 6 + 4; from 96 K-steps one warp per quarter with a chunk of six groups
@pytest.mark.parametrize("engine", [X.XNOR_ENGINE_UMMA_SINGLE, X.XNOR_ENGINE_UMMA_STREAM, X.XNOR_ENGINE_UMMA_PAIR,
                                    X.XNOR_ENGINE_UMMA_PAIR_STREAM])
@pytest.mark.parametrize("case", [(100, 64, 28, 28, 96, 3, 1, 1, 3, 1, 1, True), (100, 40, 28, 27, 160, 1, 1, 0, 1, 1, 0, False),
                                  (50, 704, 28, 28, 192, 3, 1, 1, 1, 1, 0, False)])
def test_fused_drain_of_many_items(oracle, case, engine):
    fused_parity(oracle, case, engine)


# CTA pairs: what the warps of one CTA announce to the issuing thread of the other is there when the MMA reads it.  Many
# launches of many items, resident (one and several slabs) and streaming, the inputs changing from launch to launch
# so that nothing left over from the one before can pass: bit for bit what the CUDA cores give
@pytest.mark.parametrize("engine", [X.XNOR_ENGINE_UMMA_PAIR, X.XNOR_ENGINE_UMMA_PAIR_STREAM])
@pytest.mark.parametrize("shape", [(40, 384, 13, 13, 384, 3, 1), (64, 64, 28, 28, 96, 3, 1), (24, 512, 14, 14, 224, 3, 2),
                                   (64, 128, 14, 14, 512, 1, 1)])
def test_pairs_are_repeatably_exact(shape, engine):
    N, C, H, W, Co, k, s = shape
    d = X.make_desc(N, C, H, W, Co, k, k, s, k // 2)
    g = torch.Generator(device="cuda")
    g.manual_seed(sum(shape))

    def normal(*size):
        return torch.randn(size, generator=g, device="cuda")

    layers = []
    for _ in range(3):
        wp, alpha = X.alloc_weights(Co, C, k, k)
        xp, A, K = X.alloc_binactiv(d)
        X.xnor_binarize_weights(normal(Co, C, k, k), wp, alpha)
        X.xnor_binactiv(normal(N, C, H, W), None, None, d, xp, A, K)
        layers.append((xp, wp, alpha, K, X.alloc_out(d)))
    outs = [X.alloc_out(d) for _ in range(30)]
    try:
        X.xnor_set_engine(X.XNOR_ENGINE_POPC)
        for xp, wp, alpha, K, want in layers:
            X.xnor_conv2d_forward(xp, wp, alpha, K, None, d, want)
        X.xnor_set_engine(engine)
        assert X.xnor_conv2d_plan(d).pair
        for i, out in enumerate(outs):
            xp, wp, alpha, K, _ = layers[i % 3]
            X.xnor_conv2d_forward(xp, wp, alpha, K, None, d, out)
    finally:
        X.xnor_set_engine(X.XNOR_ENGINE_AUTO)
    X.xnor_check_device()
    assert all(torch.equal(out, layers[i % 3][4]) for i, out in enumerate(outs))


# how a patch is built: one to thirteen channel words (five and more that are no multiple of four go one by one when
# streaming), both strides, planes of more and of less than four columns (a
# patch then touches more rows than a warp has lanes), the ragged end of the packed tensor; patches of one or two
# items per CTA, which all patch warps build
@pytest.mark.parametrize("engine", [X.XNOR_ENGINE_AUTO, X.XNOR_ENGINE_UMMA_STREAM, X.XNOR_ENGINE_UMMA_PAIR])
@pytest.mark.parametrize("shape", [
    (70, 20, 9, 1, 16, 1, 1, 1, 0), (70, 33, 5, 2, 16, 3, 3, 1, 1), (150, 70, 3, 3, 24, 3, 3, 1, 1),
    (90, 128, 7, 4, 16, 3, 3, 2, 1), (41, 161, 5, 3, 32, 3, 2, 1, 1), (3, 64, 41, 33, 20, 3, 3, 2, 1),
    (5, 96, 17, 19, 40, 5, 5, 2, 2), (3, 31, 29, 40, 16, 3, 3, 2, 0), (7, 190, 13, 11, 48, 1, 1, 2, 0),
    (37, 100, 15, 17, 77, 5, 5, 1, 2), (60, 40, 29, 30, 64, 3, 3, 2, 1), (36, 64, 27, 28, 100, 3, 3, 1, 1),
    (9, 167, 35, 35, 288, 1, 1, 1, 0), (2, 392, 23, 24, 112, 3, 3, 2, 1), (4, 352, 9, 2, 48, 3, 3, 1, 1), (1, 200, 21, 3, 32, 1, 1, 2, 0)])
def test_patches(oracle, shape, engine):
    block_parity(oracle, shape, engine)


# words of a filter around whole batches of 32 (8 warps, four words each), tails of channels
@pytest.mark.parametrize("C,k", [(32, 5), (768, 1), (800, 1), (980, 1), (1024, 1), (1030, 1), (45, 4), (200, 3), (225, 3), (1, 7)])
def test_weight_words(oracle, C, k):
    w = rng(C + k).standard_normal((5, C, k, k)).astype(np.float32)
    wp0, alpha0 = X.alloc_weights(5, C, k, k)
    gs = GuardSet()
    wp, alpha = gs.like("w_packed", wp0), gs.like("alpha", alpha0)
    X.xnor_binarize_weights(dev(w), wp, alpha)
    gs.check()
    B, want = oracle.binarize_weights(w)
    assert np.array_equal(unpack_weights(host(wp), C, k, k), B)
    assert_close(host(alpha), want, "alpha")
