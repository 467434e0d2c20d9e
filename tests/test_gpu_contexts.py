"""What a context must not depend on: other contexts in the process, the number of streams beside a stream, the buffers that
results are asked for in, and what it has been asked before."""
import numpy as np
import pytest

import synth_inputs as si
import paper_2003_10735_b200 as st

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.fixture(autouse=True)
def side_stream():
    s = torch.cuda.Stream()
    with torch.cuda.stream(s):
        yield s
    s.synchronize()


def make(c_in, ch, C, h, w, S=1, prec=0, seed=0, **kw):
    """A context with inputs; stream s has the same student, features and labels whatever S is."""
    thetas = [si.initial_head_params(c_in, ch, C, 100 + seed + s) for s in range(S)]
    ctx = st.st_init_head(n_streams=S, c_in=c_in, c_hidden=ch, n_classes=C, feat_h=h, feat_w=w, gemm_precision=prec,
                          lr=kw.pop("lr", 0.1), momentum=kw.pop("momentum", 0.9),
                          cuda_stream=torch.cuda.current_stream().cuda_stream, init_params=np.concatenate(thetas), **kw)
    for s in range(S):
        rng = np.random.default_rng(seed + s)
        st.st_set_frozen_features(ctx, s, np.maximum(rng.standard_normal((c_in, h, w)), 0).astype(np.float32))
        st.st_set_labels(ctx, s, si.voronoi_map(4 * h, 4 * w, 9, C, 300 + seed + s))
    return ctx


def packed(ctx, s=0):
    out = np.empty(ctx.n_params, np.float32)
    st.st_pack_updated_params(ctx, s, out)
    return out


# ---- where packed buffers lie
@pytest.mark.parametrize("where", ["pinned", "device", "ordinary"])
@pytest.mark.parametrize("offset", [0, 1, 2, 3, 4, 13])        # bytes of a message in front of the buffer
@pytest.mark.parametrize("ch,prec", [(0, 1), (64, 1), (9, 0)])
def test_packed_buffers_at_any_address(ch, prec, offset, where):
    """Packed buffers are bytes: behind a header of any length they give and take the same parameters."""
    server, client = make(64, ch, 5, 12, 20, prec=prec, seed=1), make(64, ch, 5, 12, 20, prec=prec, seed=2)
    st.st_distill_step(server, 2)
    want, n = packed(server).tobytes(), server.n_params * 4
    message = torch.full((n + offset + 16,), 0x5a, dtype=torch.uint8)
    message = message.pin_memory() if where == "pinned" else message.cuda() if where == "device" else message
    lib = st.load_library()
    st._check(lib.st_pack_updated_params(server.handle, 0, message.data_ptr() + offset, n, None), server)
    got = message.cpu().numpy()
    assert got[offset:offset + n].tobytes() == want
    assert (got[:offset] == 0x5a).all() and (got[offset + n:] == 0x5a).all()
    st._check(lib.st_apply_update(client.handle, 0, message.data_ptr() + offset, n), client)
    assert packed(client).tobytes() == want
    st.st_destroy(server)
    st.st_destroy(client)


# ---- the number of streams
@pytest.mark.parametrize("c_in,ch,C,h,w,prec", [
    (33, 9, 5, 40, 70, 0), (96, 48, 40, 24, 40, 0), (5, 0, 4, 61, 90, 0), (64, 0, 21, 45, 80, 0),
    (64, 64, 5, 24, 40, 1), (64, 192, 5, 45, 80, 1), (128, 0, 21, 45, 80, 1),      # the second: another form of the 1x1 forward for 16 streams
])
def test_results_of_a_stream_do_not_depend_on_its_neighbours(c_in, ch, C, h, w, prec):
    K = 2
    one = make(c_in, ch, C, h, w, 1, prec)
    want = np.zeros((1, K), np.float32)
    st.st_distill_step(one, K, want)
    for S in (2, 5, 16):
        many = make(c_in, ch, C, h, w, S, prec)
        loss = np.zeros((S, K), np.float32)
        st.st_distill_step(many, K, loss)
        assert packed(many).tobytes() == packed(one).tobytes(), S
        assert loss[0].tobytes() == want[0].tobytes(), S
        st.st_destroy(many)
    st.st_destroy(one)


# ---- other contexts
@pytest.mark.parametrize("first,second,ch,prec", [(24, 22, 0, 1), (32, 29, 64, 1), (8, 5, 0, 0), (120, 60, 0, 0), (255, 33, 0, 0), (32, 9, 0, 0)])
def test_a_later_context_of_fewer_classes_takes_nothing_from_an_earlier_one(first, second, ch, prec):
    c_in, h, w = 64, 20, 40
    want = {}
    for C in (first, second):
        ctx = make(c_in, ch, C, h, w, prec=prec)
        conf = np.zeros((1, 2, C, C), np.int64)
        st.st_distill_step(ctx, 2, None, conf)
        want[C] = (packed(ctx).tobytes(), conf, st.st_agreement(ctx, 0))
        st.st_destroy(ctx)
    a, b = make(c_in, ch, first, h, w, prec=prec), make(c_in, ch, second, h, w, prec=prec)
    for ctx, C in ((a, first), (b, second)):
        conf = np.zeros((1, 2, C, C), np.int64)
        st.st_distill_step(ctx, 2, None, conf)
        np.testing.assert_array_equal(conf, want[C][1])
        assert packed(ctx).tobytes() == want[C][0]
        assert st.st_agreement(ctx, 0) == want[C][2]
        st.st_destroy(ctx)


# ---- the buffers that results are asked for in, and what a context has been asked before
def test_losses_reach_any_buffer():
    """The same steps with the losses asked for in one device buffer again and again, in two in turn, in a part of one, in pinned
    and in ordinary memory, and not at all."""
    K, S = 3, 2
    ctx = make(64, 0, 5, 12, 20, S, prec=1, momentum=0.0)
    start = [packed(ctx, s) for s in range(S)]
    a, b = (torch.zeros((S, K), device="cuda") for _ in range(2))
    part = torch.zeros(S * K + 3, device="cuda")
    pinned, ordinary = torch.zeros((S, K)).pin_memory(), np.zeros((S, K), np.float32)
    want = None
    for buf in (None, a, a, b, a, b, part[3:], pinned, ordinary, a, None, pinned):
        for s in range(S):
            st.st_apply_update(ctx, s, start[s])
        if buf is not None:
            buf.fill(0) if buf is ordinary else buf.zero_()
        st.st_distill_step(ctx, K, buf)
        torch.cuda.current_stream().synchronize()
        if buf is None:
            continue
        got = buf.copy() if buf is ordinary else buf.cpu().numpy().reshape(S, K)
        want = got.copy() if want is None else want
        assert got.tobytes() == want.tobytes()
    assert (want > 0).all() and len(set(want.ravel())) == S * K and part[:3].sum() == 0
    st.st_destroy(ctx)


def test_a_threshold_that_changes_holds_no_memory():
    """A server that adapts its threshold: the calls replay one graph (0.6 MB of device memory each would be 48 MB in all)."""
    ctx = make(64, 0, 5, 12, 20, prec=1, momentum=0.0)
    start, K = packed(ctx), 63

    def train(threshold):
        st.st_apply_update(ctx, 0, start)
        n, metrics = np.zeros(1, np.int32), np.zeros((1, K + 1))
        st.st_train_key_frame(ctx, threshold, K, n, None, metrics)
        return n[0], metrics[0]

    n, want = train(2.0)                                          # never met: every update is made
    assert n == K
    held = torch.cuda.mem_get_info()[0]
    for i in range(80):
        n, got = train(2.0 + i / 1024)
        assert n == K and got.tobytes() == want.tobytes()
    assert held - torch.cuda.mem_get_info()[0] < 8 << 20
    for threshold in (0.0, 0.5 * (want[0] + want.max()), want.max()):      # each call goes by its own threshold
        past = [i for i in range(K + 1) if (want[i] > threshold if i else not want[0] < threshold)]
        n, got = train(threshold)
        assert n == (past[0] if past else K)
        np.testing.assert_array_equal(got[:n + 1], want[:n + 1])
    st.st_destroy(ctx)


def test_more_step_counts_than_graphs_are_kept():
    ctx = make(64, 0, 5, 12, 20, prec=1, momentum=0.0)
    start, want = packed(ctx), np.zeros((1, 40), np.float32)
    st.st_distill_step(ctx, 40, want)
    for n in [*range(1, 41), *range(1, 41), 40, 39, 1]:           # 32 graphs are kept: in the second round all have been given back
        loss = np.zeros((1, n), np.float32)
        st.st_apply_update(ctx, 0, start)
        st.st_distill_step(ctx, n, loss)
        assert loss.tobytes() == want[:, :n].tobytes(), n
    st.st_destroy(ctx)
