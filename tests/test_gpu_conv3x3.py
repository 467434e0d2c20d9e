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
