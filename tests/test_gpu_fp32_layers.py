"""fp32 convolutions and the many-class loss kernel against the oracle at the sizes where their tilings can go wrong:
tile edges and remainders, the channel counts at which another instantiation takes over, two streams."""
import numpy as np
import pytest

import oracle
import synth_inputs as si
import paper_2003_10735_b200 as st
from test_gpu_parity import check_weights, rand_problem, run_both

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.fixture(autouse=True)
def side_stream():
    s = torch.cuda.Stream()
    with torch.cuda.stream(s):
        yield s
    s.synchronize()


@pytest.mark.parametrize("c_in,ch,C,h,w", [
    (1, 0, 4, 4, 32), (33, 0, 5, 5, 33),           # 1x1: 4 / 16 output channels per warp, one tile / one pixel over
    (31, 9, 17, 3, 31), (35, 25, 48, 8, 64),       # 3x3: a group of 8 and one channel, four groups; 17 and 48 classes
    (64, 65, 49, 9, 65),                           # two blocks of output channels in every kernel
    (2, 3, 33, 141, 451),                          # many-class loss: 7 node rows and two warps per cell row, ragged
    (3, 0, 255, 4, 30), (3, 0, 34, 13, 61),        # ... 4 node rows and three warps
])
def test_fp32_steps_at_tile_edges(c_in, ch, C, h, w):
    feat, T = rand_problem(5, c_in, C, h, w, blobs=h * w < 5000)
    theta = si.initial_head_params(c_in, ch, C, 4)
    K = 2 if h * w < 5000 else 1
    ctx, head, loss, ref_loss, conf, masks, lab = run_both((c_in, ch, C, h, w, 0.05, 0.9), feat, T, theta, K, 0, want_conf=True)
    np.testing.assert_allclose(loss, ref_loss, rtol=1e-4)
    check_weights(ctx, head, theta, max_rel=1e-5, mean_abs=1e-5, upd_rel=2e-4)
    for k in range(K):
        ref_conf, _, _ = oracle.agreement(lab, masks[k], C)
        assert conf[k].sum() == lab.size
        assert np.abs(conf[k] - ref_conf).sum() <= 2 * max(2, lab.size // 2000)       # near-ties of the upsampled logits
    st.st_destroy(ctx)


@pytest.mark.parametrize("c_in,C,h,w", [
    (32, 5, 4, 32), (33, 16, 5, 33), (64, 17, 9, 31),          # one / two input channels per lane; the last lanes' second channel missing
    (65, 16, 7, 64), (65, 17, 3, 65), (128, 33, 8, 32),        # two / four, by the classes too; a full tile of 128 channels
    (129, 49, 2, 30), (200, 20, 37, 70),                       # one channel of a second tile; several chunks per pixel range, odd rows
])
def test_fp32_classifier_gradient_at_channel_edges(c_in, C, h, w):
    """The 1x1 weight and bias gradients where the number of input channels per lane changes.  One step without momentum moves a
    parameter by lr times its gradient, a sum of h * w products in fp32: in any order within h * w * 2^-24 of the sum of their
    sizes, against 64 bits (2590 pixels: 1.6e-4; roundings of either sign leave far less)."""
    feat, T = rand_problem(7, c_in, C, h, w, blobs=True)
    theta = si.initial_head_params(c_in, 0, C, 4)
    ctx, head, loss, ref_loss, conf, masks, lab = run_both((c_in, 0, C, h, w, 0.05, 0.0), feat, T, theta, 1, 0, want_conf=True)
    np.testing.assert_allclose(loss, ref_loss, rtol=1e-4)
    check_weights(ctx, head, theta, max_rel=1e-5, mean_abs=1e-5, upd_rel=2e-4)
    st.st_destroy(ctx)


@pytest.mark.parametrize("h,w", [(6, 40), (141, 451)])
def test_many_classes_steep_logits(h, w):
    """Logits that change by hundreds between neighbouring nodes (exact per-pixel maxima), labels out of range."""
    c_in, C = 2, 40
    rng = np.random.default_rng(3)
    f = (rng.random((h, w)) < 0.5).astype(np.float32)
    feat = np.stack([f, 1.0 - f])
    W = rng.standard_normal((C, 2)).astype(np.float32)
    W[0, 0] = W[39, 1] = 300.0
    theta = np.concatenate([W.ravel(), np.zeros(C, np.float32)])
    lab = rng.integers(0, C, (4 * h, 4 * w)).astype(np.uint8)
    ctx = st.st_init_head(c_in=c_in, n_classes=C, feat_h=h, feat_w=w, lr=1e-4, init_params=theta,
                          cuda_stream=torch.cuda.current_stream().cuda_stream)
    st.st_set_frozen_features(ctx, 0, feat)
    st.st_set_labels(ctx, 0, lab)
    loss, conf = np.zeros(1, np.float32), np.zeros((1, C, C), np.int64)
    st.st_distill_step(ctx, 1, loss, conf)
    torch.cuda.current_stream().synchronize()
    head = oracle.Head(c_in, 0, C, lr=1e-4, theta=theta)
    ref, mask = oracle.distill_step(head, feat, lab)
    assert abs(loss[0] - ref) <= 1e-4 * abs(ref)
    got = np.empty(ctx.n_params, np.float32)
    st.st_pack_updated_params(ctx, 0, got)
    assert np.linalg.norm((got - theta) - (head.theta - theta)) <= 2e-3 * np.linalg.norm(head.theta - theta)
    ref_conf, _, _ = oracle.agreement(lab, mask, C)
    assert np.abs(conf[0] - ref_conf).sum() <= 2 * max(2, lab.size // 1000)
    st.st_destroy(ctx)
