"""The loss kernel that multiplies its own logits, where a block works on several tiles: more tiles than fit the GPU at once, of
several streams, some of them ended (Train).  A stream's results are those of a context that has this stream alone, bit for bit,
which the oracle tests cover."""
import numpy as np
import pytest

import synth_inputs as si
import paper_2003_10735_b200 as st
from test_gpu_contexts import packed

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.fixture(autouse=True)
def side_stream():
    s = torch.cuda.Stream()
    with torch.cuda.stream(s):
        yield s
    s.synchronize()


def context(streams, c_in, C, h, w, **kw):
    """Stream s of the context is problem streams[s]."""
    thetas = np.concatenate([si.initial_head_params(c_in, 0, C, 100 + q) for q in streams])
    ctx = st.st_init_head(n_streams=len(streams), c_in=c_in, c_hidden=0, n_classes=C, feat_h=h, feat_w=w, gemm_precision=1, lr=0.1,
                          momentum=0.9, cuda_stream=torch.cuda.current_stream().cuda_stream, init_params=thetas, **kw)
    for s, q in enumerate(streams):
        feat = np.maximum(np.random.default_rng(q).standard_normal((c_in, h, w)), 0).astype(np.float32)
        if q % 3 == 0:
            feat[0] *= 60                                          # cells off the fast path
        labels = si.voronoi_map(4 * h, 4 * w, 9, C, 300 + q)
        st.st_set_frozen_features(ctx, s, feat); st.st_set_labels(ctx, s, labels)
    return ctx


# classes: fewest; prefetching blocks with an odd and the largest count; blocks of one tile with the smallest and the largest
@pytest.mark.parametrize("C", [2, 9, 22, 23, 32])
@pytest.mark.parametrize("c_in,weight", [(64, 0), (192, 4)])
def test_streams_that_share_blocks(C, c_in, weight):
    S, K, h, w = 13, 3, 58, 83                                     # 27 tiles a stream, 351 in all; ragged in both directions
    kw = dict(object_weight=weight, object_radius=3) if weight else {}
    ctx = context(range(S), c_in, C, h, w, **kw)
    loss, conf = np.zeros((S, K), np.float32), np.zeros((S, K, C, C), np.int64)
    student = [packed(ctx, s) for s in range(S)]
    st.st_distill_step(ctx, K, loss)
    plain = [packed(ctx, s) for s in range(S)]
    for s in range(S):
        st.st_apply_update(ctx, s, student[s])
    with_conf = np.zeros((S, K), np.float32)
    st.st_distill_step(ctx, K, with_conf, conf)
    met = np.zeros((S, K + 1)); n_upd = np.zeros(S, np.int32); best = np.zeros(S)
    st.st_train_key_frame(ctx, 2.0, K, n_upd, best, met)
    threshold = float(np.sort(met[:, 0])[S // 2])                  # half of the streams end at once
    st.st_train_key_frame(ctx, threshold, K, n_upd, best, met)
    trained = [packed(ctx, s) for s in range(S)]
    st.st_destroy(ctx)
    assert 0 < (n_upd == 0).sum() < S
    for q in (0, 1, 6, S - 1):
        one = context([q], c_in, C, h, w, **kw)
        l1, c1 = np.zeros((1, K), np.float32), np.zeros((1, K, C, C), np.int64)
        st.st_distill_step(one, K, l1)
        assert packed(one).tobytes() == plain[q].tobytes() and l1[0].tobytes() == loss[q].tobytes()
        st.st_apply_update(one, 0, student[q])
        st.st_distill_step(one, K, l1, c1)
        assert l1[0].tobytes() == with_conf[q].tobytes() and (c1[0] == conf[q]).all()
        m1, u1, b1 = np.zeros((1, K + 1)), np.zeros(1, np.int32), np.zeros(1)
        st.st_train_key_frame(one, 2.0, K, u1, b1, m1)
        st.st_train_key_frame(one, threshold, K, u1, b1, m1)
        assert u1[0] == n_upd[q] and b1[0] == best[q] and (m1[0] == met[q]).all()
        assert packed(one).tobytes() == trained[q].tobytes()
        st.st_destroy(one)


@pytest.mark.parametrize("blocks,c_in,C,h,w,first", [
    (((64, 0),), 64, 5, 9, 32, 0), (((192, 0),), 64, 21, 30, 61, 0), (((256, 0),), 64, 32, 23, 95, 0),
    (((64, 64), (128, 0)), 64, 13, 24, 40, 0), (((64, 0), (64, 64)), 128, 19, 17, 47, 1), (((128, 0),), 64, 23, 19, 33, 1),
])
def test_behind_blocks_as_with_a_forward_of_its_own(blocks, c_in, C, h, w, first, monkeypatch):
    """A classifier behind blocks (some or all of them frozen): the loss kernel multiplies its logits, or (ST_FUSED_FORWARD=0) reads
    those of a kernel of its own.  Same products in the same order, so the first step's logits agree bit for bit; sums of
    exponentials are shifted by another maximum and round differently in the last place."""
    S, K = 2, 3

    def run(fused):
        if not fused:
            monkeypatch.setenv("ST_FUSED_FORWARD", "0")
        rng = np.random.default_rng(7)
        prev, n = c_in, 0
        theta = []
        for _ in range(S):
            prev = c_in
            for co, cs in blocks:
                theta.append(rng.standard_normal(co * (prev + cs) * 9) * np.sqrt(2.0 / ((prev + cs) * 9))); theta.append(np.zeros(co))
                prev = co
            theta.append(rng.standard_normal(C * prev) * np.sqrt(2.0 / prev)); theta.append(rng.standard_normal(C) * 0.1)
        ctx = st.st_init_head(n_streams=S, c_in=c_in, n_classes=C, feat_h=h, feat_w=w, gemm_precision=1, lr=0.05, momentum=0.9, blocks=blocks,
                              first_trained=first, cuda_stream=torch.cuda.current_stream().cuda_stream,
                              init_params=np.concatenate(theta).astype(np.float32))
        monkeypatch.delenv("ST_FUSED_FORWARD", raising=False)
        for s in range(S):
            st.st_set_frozen_features(ctx, s, np.maximum(rng.standard_normal((c_in, h, w)), 0).astype(np.float32))
            for b, (_, cs) in enumerate(blocks):
                if cs:
                    st.st_set_skip_features(ctx, s, b, np.maximum(rng.standard_normal((cs, h, w)), 0).astype(np.float32))
            st.st_set_labels(ctx, s, si.voronoi_map(4 * h, 4 * w, 9, C, 300 + s))
        out = {}
        one = np.zeros((S, 1), np.float32)
        st.st_distill_step(ctx, 1, one)
        out["z"] = [st.st_read_tensor(ctx, s, st.ST_TENSOR_LOGITS) for s in range(S)]
        loss, conf = np.zeros((S, K), np.float32), np.zeros((S, K, C, C), np.int64)
        st.st_distill_step(ctx, K, loss, conf)
        out["loss"], out["conf"] = np.concatenate([one, loss], 1), conf
        out["theta"] = [st_packed(ctx, s) for s in range(S)]
        n_upd, best, met = np.zeros(S, np.int32), np.zeros(S), np.zeros((S, K + 1))
        st.st_train_key_frame(ctx, 2.0, K, n_upd, best, met)
        out["met"] = met
        out["z_train"] = [st.st_read_tensor(ctx, s, st.ST_TENSOR_LOGITS) for s in range(S)]
        out["launches"] = st.st_launch_count(ctx)
        st.st_destroy(ctx)
        return out

    def st_packed(ctx, s):
        out = np.empty(ctx.n_params, np.float32)
        n = st.st_pack_updated_params(ctx, s, out)
        return out[:n // 4] if isinstance(n, int) and n else out

    a, b = run(True), run(False)
    assert a["launches"] < b["launches"]
    np.testing.assert_allclose(a["loss"], b["loss"], rtol=2e-5)     # K steps whose bf16 roundings fall the other way now and then
    np.testing.assert_allclose(a["met"], b["met"], atol=2e-3)
    assert np.abs(a["conf"] - b["conf"]).sum(axis=(2, 3)).max() <= 2 * max(4, 16 * h * w // 1000)
    for s in range(S):
        assert a["z"][s].tobytes() == b["z"][s].tobytes()
        for k in ("theta", "z_train"):
            assert np.linalg.norm(a[k][s] - b[k][s]) <= 5e-3 * np.linalg.norm(b[k][s])
