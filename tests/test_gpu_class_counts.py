"""Every class count has its own instantiation of the loss kernel: loss, gradient, confusion matrix and student mask of each
against the oracle in double, on the kernel's own logits, for every way a head takes through it."""
import numpy as np
import pytest

import oracle
import synth_inputs as si
import paper_2003_10735_b200 as st
from test_gpu_bf16 import dev, make_ctx, packed, problem, rel_l2

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.fixture(autouse=True)
def side_stream():
    s = torch.cuda.Stream()
    with torch.cuda.stream(s):
        yield s
    s.synchronize()


@pytest.mark.parametrize("C", range(2, 33))
@pytest.mark.parametrize("ch,h,w,prec,steep", [
    (0, 9, 32, 1, 0.0), (0, 17, 37, 1, 4.0),            # logits multiplied inside the kernel; steep: cells off the fast path too
    (64, 9, 36, 1, 0.0), (64, 8, 31, 1, 0.0),           # stored logits: tile copy / plain loads
    (0, 11, 41, 0, 4.0),                                # fp32 gradient
])
def test_one_step_at_every_class_count(C, ch, h, w, prec, steep):
    c_in = 64
    feat, T = problem(C, c_in, C, h, w)
    theta = si.initial_head_params(c_in, ch, C, C)
    if steep:                                           # two thirds of the logits change by tens between neighbouring nodes
        theta[:C * c_in].reshape(C, c_in)[::3, 0] += steep * 10
    labels = oracle.teacher_labels(T)
    labels[2, 3], labels[-1, -1] = C - 1, 0
    for want_conf in (False, True):                     # two instantiations
        ctx = make_ctx(c_in, ch, C, h, w, theta, prec=prec)
        st.st_set_frozen_features(ctx, 0, dev(feat)); st.st_set_labels(ctx, 0, dev(labels))
        mask = np.zeros((4 * h, 4 * w), np.uint8)
        st.st_student_mask(ctx, 0, mask)
        loss, conf = np.zeros((1, 1), np.float32), np.zeros((1, 1, C, C), np.int64)
        st.st_distill_step(ctx, 1, loss, conf if want_conf else None)
        torch.cuda.current_stream().synchronize()
        z = st.st_read_tensor(ctx, 0, st.ST_TENSOR_LOGITS).reshape(C, h, w).astype(np.float64)
        u = oracle.upsample(z, 4)
        ref, g, _ = oracle.softmax_ce(u, labels)
        dz = oracle.upsample_adjoint(g, 4)
        assert abs(loss[0, 0] - ref) <= 1e-5 * ref      # sums of fp32 terms whose exponentials are good to 5e-6
        assert rel_l2(st.st_read_tensor(ctx, 0, st.ST_TENSOR_LOGIT_GRAD), dz.ravel()) <= 2e-5
        # the weight gradient: what the step itself wrote of the logit gradient (bf16 with tensor cores: 2^-9 a value at most)
        a = st.st_read_tensor(ctx, 0, st.ST_TENSOR_HIDDEN if ch else st.ST_TENSOR_FEATURES).reshape(-1, h * w).astype(np.float64)
        grad = st.st_read_tensor(ctx, 0, st.ST_TENSOR_PARAM_GRAD)[-C * (a.shape[0] + 1):]
        assert rel_l2(grad[:-C], (dz.reshape(C, -1) @ a.T).ravel()) <= (2.0 ** -9 if prec else 2e-5)
        assert rel_l2(grad[-C:], dz.sum((1, 2))) <= 1e-4 * max(1.0, np.abs(dz).sum() / np.linalg.norm(dz.sum((1, 2))) / 100)
        # masks and counts: the largest interpolated logit, near-ties either way
        best = u.argmax(0)
        top = np.take_along_axis(u, best[None], 0)[0]
        def tied(m): return np.take_along_axis(u, m[None].astype(np.int64), 0)[0] >= top - 1e-4 * np.maximum(1.0, np.abs(top))
        assert tied(mask).all()
        if want_conf:
            want = oracle.confusion(labels, best.astype(np.uint8), C)
            want = want[0] if isinstance(want, tuple) else want
            assert conf.sum() == labels.size and np.array_equal(conf[0, 0].sum(1), want.sum(1))
            assert np.abs(conf[0, 0] - want).sum() <= 2 * max(2, labels.size // 1000)
        st.st_destroy(ctx)
