"""Both backward products of the classifier behind a trained hidden layer (one kernel) at the sizes where its tiling can go
wrong: a lone pixel, tile edges, odd groups of 64 channels, several tiles per block, several streams."""
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


@pytest.mark.parametrize("ch,C,h,w,S", [
    (64, 2, 1, 1, 1), (128, 32, 1, 127, 1), (192, 5, 8, 16, 2), (256, 9, 3, 43, 1), (256, 32, 155, 157, 1), (64, 21, 140, 163, 2),
])
def test_products_of_the_stored_operands(ch, C, h, w, S):
    c_in = 64
    theta = si.initial_head_params(c_in, ch, C, 2)
    theta[ch * c_in * 9:ch * c_in * 9 + ch] = np.linspace(-0.2, 0.3, ch)
    ctx = make_ctx(c_in, ch, C, h, w, np.tile(theta, S), S=S)
    for s in range(S):
        feat, T = problem(8 + s, c_in, C, h, w)
        st.st_set_frozen_features(ctx, s, dev(feat)); st.st_teacher_labels(ctx, s, dev(T))
    st.st_distill_step(ctx, 1)
    W2 = oracle.round_bf16(theta[ch * c_in * 9 + ch:][:C * ch].reshape(C, ch)).astype(np.float64)
    for s in range(S):
        hd = st.st_read_tensor(ctx, s, st.ST_TENSOR_HIDDEN).reshape(ch, h * w).astype(np.float64)
        dz = oracle.round_bf16(st.st_read_tensor(ctx, s, st.ST_TENSOR_LOGIT_GRAD)).reshape(C, h * w).astype(np.float64)
        dh = st.st_read_tensor(ctx, s, st.ST_TENSOR_HIDDEN_GRAD).reshape(ch, h * w)
        g = st.st_read_tensor(ctx, s, st.ST_TENSOR_PARAM_GRAD)[ch * c_in * 9:]
        ref = (W2.T @ dz) * (hd > 0)
        np.testing.assert_allclose(dh, ref, rtol=2.0 ** -7, atol=1e-6 * max(np.abs(ref).max(), 1e-30))
        assert rel_l2(g[:ch], ref.sum(1)) <= 1e-5
        assert rel_l2(g[ch:ch + C * ch], (dz @ hd.T).ravel()) <= 1e-5
    st.st_destroy(ctx)
