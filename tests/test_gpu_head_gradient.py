"""Weight gradient of a one-layer head, formed by the loss kernel tile by tile: compared with the sum over all nodes in 64 bits of
the same bf16 operands, at channel counts of one to four 64-channel blocks (an odd one has half of a 128-channel product to
itself), class counts around the limits of the tensor-memory reads and of the fused form, maps of one tile, of ragged tiles and of
many more tiles than blocks, several streams."""
import numpy as np
import pytest
import torch

import paper_2003_10735_b200 as st

pytestmark = pytest.mark.gpu


def bf16(x):
    return torch.from_numpy(x).to(torch.bfloat16).to(torch.float64).numpy()


@pytest.mark.parametrize("c_in,C,h,w,S", [
    (64, 2, 9, 32, 1),            # the smallest map that takes this form: two rows of tiles, the second with two own rows
    (64, 16, 14, 60, 2),          # whole tiles
    (128, 17, 15, 61, 1),         # one row and one column more
    (192, 21, 22, 47, 3),         # an odd 64-channel block
    (256, 24, 29, 95, 1),         # the most classes that are multiplied here
    (256, 25, 29, 95, 1),         # one more: the weight gradient is a kernel of its own
    (128, 5, 70, 150, 16),        # 800 tiles: several per group
    (256, 13, 100, 200, 4),       # 420 tiles of two 128-channel products
])
def test_weight_gradient_against_64_bits(c_in, C, h, w, S):
    rng = np.random.default_rng(1000 * c_in + C)
    stream = torch.cuda.Stream()
    theta = (rng.standard_normal((S, C * c_in + C)) * 0.05).astype(np.float32)
    feats = np.maximum(rng.standard_normal((S, c_in, h, w)), 0).astype(np.float32)
    labels = rng.integers(0, C, (S, 4 * h, 4 * w), dtype=np.uint8)
    with torch.cuda.stream(stream):
        ctx = st.st_init_head(n_streams=S, c_in=c_in, n_classes=C, feat_h=h, feat_w=w, gemm_precision=1, lr=0.01,
                              cuda_stream=stream.cuda_stream, init_params=theta)
        for s in range(S):
            st.st_set_frozen_features(ctx, s, feats[s])
            st.st_set_labels(ctx, s, labels[s])
        st.st_distill_step(ctx, 1)
        got = [st.st_read_tensor(ctx, s, st.ST_TENSOR_PARAM_GRAD) for s in range(S)]
        dz = [st.st_read_tensor(ctx, s, st.ST_TENSOR_LOGIT_GRAD) for s in range(S)]
        st.st_destroy(ctx)
    tiles = ((h + 6) // 7) * ((w + 29) // 30)
    for s in range(S):
        x, g = bf16(feats[s]).reshape(c_in, -1), bf16(dz[s]).reshape(C, -1)
        want, size = g @ x.T, np.abs(g) @ np.abs(x).T
        # products of two bf16 values are exact in fp32; one rounding per 16 nodes of a tile (its 224 in 14 products of inner depth 4),
        # then one per partial sum of a thread group (tiles / 16) and per group (16)
        roundings = 14 + 4 + tiles / 16 + 16
        err = np.abs(got[s][:C * c_in].reshape(C, c_in) - want)
        assert (err <= roundings * 2.0 ** -23 * size + 1e-30).all(), (err / size).max()
