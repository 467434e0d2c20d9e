"""The 3x3 layer's kernels at the channel counts where their pipelines take another depth (stages, chunks per stage, an odd 64
input channels in the last accumulator) and at the edges of their tiles, against sums over the stored operands."""
import numpy as np
import pytest

import oracle
import synth_inputs as si
import paper_2003_10735_b200 as st
from test_gpu_bf16 import dev, make_ctx, problem, rel_l2

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.fixture(autouse=True)
def side_stream():
    s = torch.cuda.Stream()
    with torch.cuda.stream(s):
        yield s
    s.synchronize()


def taps(x):
    """[9][c][h][w]: the input under each tap, zeros outside the map"""
    h, w = x.shape[1:]
    p = np.pad(x, ((0, 0), (1, 1), (1, 1)))
    return np.stack([p[:, dy:dy + h, dx:dx + w] for dy in range(3) for dx in range(3)])


@pytest.mark.parametrize("c_in,ch,h,w", [
    (64, 64, 1, 1), (64, 64, 5, 33), (192, 64, 61, 67), (128, 128, 4, 32), (192, 128, 7, 95), (320, 64, 9, 31),
    (64, 192, 6, 34), (128, 256, 3, 65), (256, 256, 101, 161),
    # items of two tiles, the last of a row with one tile on the map; more of them than a GPU has SMs; 301 whole items, the last five cut in two
    (64, 64, 145, 200), (192, 128, 97, 200), (64, 64, 180, 320), (64, 128, 104, 344),
])
def test_forward_and_weight_gradient_of_the_stored_operands(c_in, ch, h, w):
    C = 5
    theta = si.initial_head_params(c_in, ch, C, 2)
    nw = ch * c_in * 9
    theta[nw:nw + ch] = np.linspace(-0.2, 0.3, ch)
    feat, T = problem(3, c_in, C, h, w)
    ctx = make_ctx(c_in, ch, C, h, w, theta)
    st.st_set_frozen_features(ctx, 0, dev(feat)); st.st_teacher_labels(ctx, 0, dev(T))
    st.st_distill_step(ctx, 1)
    hd = st.st_read_tensor(ctx, 0, st.ST_TENSOR_HIDDEN).reshape(ch, h, w)
    dh = st.st_read_tensor(ctx, 0, st.ST_TENSOR_HIDDEN_GRAD).reshape(ch, -1).astype(np.float64)
    g = st.st_read_tensor(ctx, 0, st.ST_TENSOR_PARAM_GRAD)[:nw].reshape(ch, c_in, 9)
    X = taps(oracle.round_bf16(feat).astype(np.float64)).reshape(9, c_in, h * w)
    W1 = oracle.round_bf16(theta[:nw]).astype(np.float64).reshape(ch, c_in, 9)
    ref = np.maximum(sum(W1[:, :, t] @ X[t] for t in range(9)) + theta[nw:nw + ch, None].astype(np.float64), 0).reshape(ch, h, w)
    assert (np.abs(hd - ref) <= 2.0 ** -8 * np.abs(ref) + 1e-5 * np.abs(ref).max()).all()
    assert rel_l2(g, np.stack([dh @ X[t].T for t in range(9)], axis=2)) <= 1e-5
    st.st_destroy(ctx)


@pytest.mark.parametrize("c_in,blocks,h,w", [
    (64, ((64, 0), (64, 64)), 1, 1), (64, ((64, 64), (64, 0)), 17, 9), (128, ((128, 0), (64, 0)), 16, 8), (64, ((128, 64), (128, 0)), 33, 23),
    (64, ((192, 0), (64, 0)), 18, 41), (64, ((256, 0), (64, 0)), 97, 150), (64, ((64, 0), (64, 0)), 180, 200),
    (64, ((64, 0), (64, 0)), 145, 200), (64, ((128, 0), (64, 0)), 97, 200), (64, ((64, 0), (64, 0)), 180, 320),
])
def test_gradient_passed_back_at_the_edges_of_its_tiles(c_in, blocks, h, w):
    """The first block's gradient, masked by its own ReLU, and its bias gradient, against sums over the second block's gradient as
    stored: a lone pixel, one row and column beyond a tile of 16 x 8, whole tiles, items of one tile, items cut into
    ranges of channels, and, in the last three cases, items of two tiles: 25 columns of tiles, so that the last item of a row has one
    on the map, and 240 items, so that a block walks several."""
    C, rng = 5, np.random.default_rng(1)
    shapes, prev = [], c_in
    for co, cs in blocks:
        shapes.append((co, prev + cs)); prev = co
    theta = []
    for co, ci in shapes:
        theta += [rng.standard_normal(co * ci * 9) * np.sqrt(2 / (9 * ci)), np.linspace(-0.2, 0.3, co)]
    theta += [rng.standard_normal(C * prev) * np.sqrt(2 / prev), np.zeros(C)]
    ctx = st.st_init_head(c_in=c_in, n_classes=C, feat_h=h, feat_w=w, gemm_precision=1, lr=0.01, blocks=blocks,
                          cuda_stream=torch.cuda.current_stream().cuda_stream, init_params=np.concatenate(theta).astype(np.float32))
    feat, T = problem(3, c_in, C, h, w)
    st.st_set_frozen_features(ctx, 0, dev(feat)); st.st_teacher_labels(ctx, 0, dev(T))
    for b, (_, cs) in enumerate(blocks):
        if cs:
            st.st_set_skip_features(ctx, 0, b, dev(np.maximum(rng.standard_normal((cs, h, w)), 0).astype(np.float32)))
    st.st_distill_step(ctx, 1)
    read = lambda which, c: st.st_read_tensor(ctx, 0, which).reshape(c, h, w)
    (c1, i1), (c2, i2) = shapes
    out1, d1 = read(st.ST_TENSOR_HIDDEN_FIRST, c1), read(st.ST_TENSOR_HIDDEN_GRAD_FIRST, c1)
    d2 = read(st.ST_TENSOR_HIDDEN_GRAD, c2).astype(np.float64)
    W2 = oracle.round_bf16(np.asarray(theta[2], np.float32)).astype(np.float64).reshape(c2, i2, 9)[:, :c1]
    back = taps(d2).reshape(9, c2, h * w)                       # under tap t: d2 at the pixel shifted by t; the transpose mirrors the taps
    ref = sum(W2[:, :, 8 - t].T @ back[t] for t in range(9)).reshape(c1, h, w) * (out1 > 0)
    assert (np.abs(d1 - ref) <= 2.0 ** -8 * np.abs(ref) + 1e-5 * max(np.abs(ref).max(), 1e-30)).all()
    g = st.st_read_tensor(ctx, 0, st.ST_TENSOR_PARAM_GRAD)[c1 * i1 * 9:][:c1]
    assert rel_l2(g, ref.sum((1, 2))) <= 1e-5
    st.st_destroy(ctx)


@pytest.mark.parametrize("c_in,co,cs,h,w", [
    (64, 64, 0, 9, 70), (64, 64, 128, 4, 32), (128, 64, 64, 5, 33), (192, 128, 0, 21, 31), (64, 64, 192, 30, 64), (128, 128, 192, 47, 61),
])
def test_weight_gradient_of_an_odd_64_input_channels(c_in, co, cs, h, w):
    """The last 64 of an odd number of channel blocks, whose first two vertical taps are one product: from the previous output and from a skip
    input, maps of one chunk of 4 x 32 pixels, of ragged ones, of several to a range."""
    C, rng = 5, np.random.default_rng(4)
    ci = c_in + cs
    theta = np.concatenate([rng.standard_normal(co * ci * 9) * np.sqrt(2 / (9 * ci)), np.linspace(-0.2, 0.3, co),
                            rng.standard_normal(C * co) * np.sqrt(2 / co), np.zeros(C)]).astype(np.float32)
    ctx = st.st_init_head(c_in=c_in, n_classes=C, feat_h=h, feat_w=w, gemm_precision=1, lr=0.01, blocks=((co, cs),),
                          cuda_stream=torch.cuda.current_stream().cuda_stream, init_params=theta)
    feat, T = problem(3, c_in, C, h, w)
    skip = np.maximum(rng.standard_normal((cs, h, w)), 0).astype(np.float32)
    st.st_set_frozen_features(ctx, 0, dev(feat)); st.st_teacher_labels(ctx, 0, dev(T))
    if cs:
        st.st_set_skip_features(ctx, 0, 0, dev(skip))
    st.st_distill_step(ctx, 1)
    dh = st.st_read_tensor(ctx, 0, st.ST_TENSOR_HIDDEN_GRAD).reshape(co, -1).astype(np.float64)
    g = st.st_read_tensor(ctx, 0, st.ST_TENSOR_PARAM_GRAD)[:co * ci * 9].reshape(co, ci, 9)
    X = taps(oracle.round_bf16(np.concatenate([feat, skip])).astype(np.float64)).reshape(9, ci, h * w)
    for t in range(9):
        ref = dh @ X[t].T
        assert rel_l2(g[:, :, t], ref) <= 1e-5 and rel_l2(g[:, -64:, t], ref[:, -64:]) <= 1e-5, t
    st.st_destroy(ctx)
