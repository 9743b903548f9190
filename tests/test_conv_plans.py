"""How the convolution calls run a shape (xnor_conv2d_plan): host logic, no GPU needed."""
import pytest

import paper_1603_05279_b200 as X
from paper_1603_05279_b200 import binding as B
from paper_1603_05279_b200 import workloads as wl
from paper_1603_05279_b200.runner import LayerBuffers


def plan(N, C, H, W, Co, k, stride=1, pad=None, kbits=1, fused=False, residual=False):
    return X.xnor_conv2d_plan(X.make_desc(N, C, H, W, Co, k, k, stride, k // 2 if pad is None else pad), kbits, fused,
                              residual)


@pytest.fixture(autouse=True)
def default_engine():
    yield
    X.xnor_set_engine(B.XNOR_ENGINE_AUTO)


# kernels for 1 .. 7 bit planes: in pairs on the tensor cores; one by one where the rows of two do not fit
# beside each other, and on the CUDA cores (stride 3, or by choice)
@pytest.mark.parametrize("shape,engine,tensor,launches", [
    ((4, 128, 28, 28, 128, 3, 1, 1), B.XNOR_ENGINE_AUTO, 1, [1, 1, 2, 2, 3, 3, 4]),
    ((32, 897, 36, 40, 135, 5, 1, 1), B.XNOR_ENGINE_AUTO, 1, [1, 2, 3, 4, 5, 6, 7]),
    ((4, 128, 28, 28, 128, 3, 3, 1), B.XNOR_ENGINE_AUTO, 0, [1, 2, 3, 4, 5, 6, 7]),
    ((4, 128, 28, 28, 128, 3, 1, 1), B.XNOR_ENGINE_POPC, 0, [1, 2, 3, 4, 5, 6, 7]),
])
def test_launches_of_a_kbit_convolution(shape, engine, tensor, launches):
    X.xnor_set_engine(engine)
    plans = [plan(*shape, kbits=k) for k in range(1, 8)]
    assert [p.launches for p in plans] == launches
    assert all(p.tensor_cores == tensor for p in plans)
    N, C, H, W, Co, k, stride, pad = shape
    for kbits in (2, 3):
        L = LayerBuffers(wl.ConvShape("s", N, C, H, W, Co, k, stride, pad, 1.0), device="meta", variant="kbit", kbits=kbits)
        assert L.launches() == 1 + L.binactiv_launches() + launches[kbits - 1]


def test_plan_refuses_what_the_calls_refuse():
    for bad in (dict(kbits=0), dict(kbits=8), dict(kbits=2, fused=True)):
        with pytest.raises(X.XnorError):
            plan(4, 64, 8, 8, 64, 3, **bad)
    with pytest.raises(X.XnorError):
        plan(1, 8, 5, 5, 4, 3, kbits=2)               # 25 words per plane
    with pytest.raises(X.XnorError):
        plan(1, 8, 5, 5, 40, 3, fused=True)           # the next layer's words are not whole


def schedule(p):
    return ("pair " if p.pair else "") + ("resident" if p.resident else "streaming"), p.slabs, p.slab_filters


def test_fused_slabs_stay_resident():
    """The fused epilogue outweighs a patch per slab, however few K-steps a slab has."""
    assert schedule(plan(58, 16, 34, 34, 768, 1, fused=True)) == ("resident", 4, 192)
    assert schedule(plan(60, 64, 55, 53, 384, 3, stride=2, fused=True)) == ("resident", 2, 192)


@pytest.mark.parametrize("shape,warps", [((60, 416, 14, 13, 384, 1, 2, 0), 2),       # 7 K-steps
                                         ((42, 976, 55, 27, 192, 3, 1, 1), 1)])      # 140
def test_fused_streaming_drains_short_items_with_two_warps(shape, warps):
    p = plan(*shape, fused=True)
    assert not p.resident
    N, C, H, W, Co, k, stride, pad = shape
    assert X.xnor_conv2d_binactiv_parts(X.make_desc(N, C, H, W, Co, k, k, stride, pad)) == p.slabs * warps


@pytest.mark.parametrize("shape,expected", [
    ((190, 67, 51, 51, 428, 1, 2, 0), ("resident", 2, 224)),          # the drain is the longest part: three warps
    ((79, 80, 49, 49, 912, 3, 2, 1), ("resident", 4, 240)),
    ((255, 272, 7, 7, 768, 1, 2, 0), ("resident", 4, 192)),           # one patch each either way
    ((256, 128, 28, 28, 256, 3, 2, 1), ("streaming", 2, 128)),        # the patch is: built once per tile
    ((136, 944, 8, 19, 512, 1, 1, 0), ("streaming", 4, 128)),          # (pairs, where they fit, do not change that)
    ((155, 432, 9, 9, 513, 1, 1, 0), ("resident", 3, 176)),
    ((61, 112, 28, 28, 272, 3, 2, 1), ("resident", 2, 144)), ((72, 192, 48, 48, 400, 1, 2, 0), ("streaming", 4, 112))])
def test_slabs_of_few_steps_are_resident_where_that_is_faster(shape, expected):
    assert schedule(plan(*shape)) == expected


def test_a_residual_favours_the_three_draining_warps():
    assert schedule(plan(37, 544, 51, 47, 256, 1)) == ("streaming", 2, 128)
    assert schedule(plan(37, 544, 51, 47, 256, 1, residual=True)) == ("resident", 2, 128)


@pytest.mark.parametrize("shape,expected", [
    ((1, 352, 9, 9, 224, 3, 1, 1), ("resident", 4, 64)), ((2, 33, 7, 5, 96, 3, 1, 1), ("resident", 2, 64)),
    ((2, 448, 46, 46, 416, 3, 1, 1), ("pair resident", 5, 96))])       # no slabs beyond the two that spread it
def test_small_fused_problems_are_spread(shape, expected):
    assert schedule(plan(*shape, fused=True)) == expected


@pytest.mark.parametrize("shape,expected", [
    ((2, 928, 38, 38, 912, 5, 1, 2), ("pair streaming", 5, 192)),      # 65 items for 74 pairs instead of 104
    ((12, 544, 22, 53, 176, 3, 1, 1), ("pair streaming", 1, 192)),     # as long, and half the items
    ((113, 544, 27, 5, 576, 5, 1, 2), ("pair streaming", 5, 128))])    # seven short rounds beat four long ones
def test_pairs_stream_the_slabs_that_save_rounds(shape, expected):
    assert schedule(plan(*shape)) == expected


def test_a_small_problem_keeps_one_item_per_sm():
    """59 tiles: slabs of 32 filters are two items per SM, which two bit planes are worth and one is not."""
    shape = (12, 256, 23, 23, 120, 5, 1, 2)
    assert plan(*shape, kbits=2).resident and not plan(*shape).resident
    assert not plan(3, 480, 51, 51, 192, 3).resident
