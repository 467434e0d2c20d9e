"""The update's sums of partial weight gradients, in the ways that the number of weights and of partial sums choose: a thread group's lanes
and batches (8, 16, 32 or 64 lanes), layers that are streamed, layers whose rows are no whole vectors; SGD and Adam.  Reference: the
step worked out in 64 bits from the gradient that the update says it has applied, and that gradient against a context whose streams share
the launch (bit for bit) and against the sum over the nodes."""
import numpy as np
import pytest

import oracle
import synth_inputs as si
import paper_2003_10735_b200 as st
from test_gpu_bf16 import dev, problem, rel_l2

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("c_in,ch,C,h,w,bf16", [
    (256, 0, 21, 180, 320, 1),       # 286 partial sums of 5376 weights: 32 groups
    (64, 0, 2, 9, 32, 1),            # two of 128: most groups have none
    (64, 64, 3, 60, 70, 1),          # 36864 weights: a handful of partial sums, 4 groups of 64
    (64, 64, 3, 120, 200, 1),        # more: 8 groups of 32
    (64, 64, 3, 180, 320, 1),
    (64, 192, 3, 60, 100, 1),        # 110592 weights: streamed, the classifier's in the grouped part
    (48, 0, 7, 40, 61, 0),           # fp32
    (27, 20, 5, 31, 33, 0),          # fp32, 4860 weights
    (27, 21, 5, 31, 33, 0),          # fp32, 5103: no whole vectors
])
@pytest.mark.parametrize("adam", [0, 1])
def test_step_from_the_applied_gradient(c_in, ch, C, h, w, bf16, adam):
    theta = si.initial_head_params(c_in, ch, C, 2)
    feat, T = problem(3, c_in, C, h, w)
    stream = torch.cuda.Stream()
    grads, after = [], []
    with torch.cuda.stream(stream):
        for S in (1, 3):
            ctx = st.st_init_head(n_streams=S, c_in=c_in, c_hidden=ch, n_classes=C, feat_h=h, feat_w=w, gemm_precision=bf16, lr=0.01, momentum=0.0 if adam else 0.5,
                                  optimizer=adam, cuda_stream=stream.cuda_stream, init_params=np.stack([theta] * S))
            for s in range(S):
                st.st_set_frozen_features(ctx, s, dev(feat)); st.st_teacher_labels(ctx, s, dev(T))
            st.st_distill_step(ctx, 1)
            grads += [st.st_read_tensor(ctx, s, st.ST_TENSOR_PARAM_GRAD) for s in range(S)]
            for s in range(S):
                p = np.empty(ctx.n_params, np.float32)
                st.st_pack_updated_params(ctx, s, p)
                after.append(p)
            if S == 1 and ch == 0:
                dz = st.st_read_tensor(ctx, 0, st.ST_TENSOR_LOGIT_GRAD).reshape(C, -1)
            st.st_destroy(ctx)
    assert all(g.tobytes() == grads[0].tobytes() for g in grads) and all(p.tobytes() == after[0].tobytes() for p in after)
    g = grads[0].astype(np.float64)
    if adam:     # first step: m / c1 = g, v / c2 = g^2 up to the rounding of the stored moments, 2^-24 each
        step = 0.01 * g / (np.abs(g) + 1e-8)
    else:
        step = 0.01 * g
    want = theta.astype(np.float64) - step
    # one rounding of the parameter, and of the step's factors
    assert (np.abs(after[0] - want) <= 2.0 ** -24 * np.abs(want) * 1.01 + 2.0 ** -21 * np.abs(step) + 1e-30).all()
    if ch == 0:
        X = (oracle.round_bf16(feat) if bf16 else feat).astype(np.float64).reshape(c_in, -1)
        z = (oracle.round_bf16(dz) if bf16 else dz).astype(np.float64)
        assert rel_l2(grads[0][:C * c_in], (z @ X.T).ravel()) <= 1e-5
