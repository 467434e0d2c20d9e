"""What the speed of this framework is measured on: the work its users have it do, through its public entry points.

A case is one pass of one of four tasks:

  key_frame  one key frame of every client stream: install the stream's student, cache the frozen part's output and the
             skip inputs, reduce the teacher's logits to labels, K optimisation steps, pack the updated part, measure
             student/teacher agreement; the label map is wanted as well.  Results stay on the device (the pass does not wait
             for the GPU).
  train      the same with Algorithm 1's control (metric, best student, threshold) in place of the fixed K steps and with
             the results a server sends off (updated part, metrics) delivered to host memory, so that the pass waits.
  predict    the client's side: install the updated part that has arrived in host memory, cache a frame's features,
             predict its mask.
  agreement  confusion matrix and mean IoU of two given masks.

Every pass starts from the same student (st_apply_update: the one the client has), so that all passes do the same work.
The inputs are on the device, where the teacher and the frozen part of the student leave them.
"""
import math

import torch

import paper_2003_10735_b200 as st

_DEFAULTS = {
    "task": "key_frame", "streams": 1, "c_in": 256, "hidden": 0, "blocks": "", "classes": 21, "feat_h": 180, "feat_w": 320,
    "steps": 8, "bf16": True, "adam": False, "lr": 0.01, "momentum": 0.9, "object_weight": 0, "object_radius": 0,
}


def _case(name=None, **kw):
    c = dict(_DEFAULTS, **kw)
    return dict(c, name=name) if name else c


def listed():
    return [
        # ComputeMetric alone, as on the client's own frames: two masks of a 720p frame, the smallest call there is
        _case("masks 720p", task="agreement"),
        # the client at 720p: an update arrives, the next frame is segmented
        _case("predict 720p", task="predict"),
        # a small head in plain fp32 on small frames, one step: launches and host work count
        _case("360p fp32 one step", c_in=64, classes=4, feat_h=90, feat_w=160, steps=1, bf16=False, momentum=0.0),
        # small frames on tensor cores: the kernels are a few microseconds each
        _case("360p 1x1", c_in=128, feat_h=90, feat_w=160),
        # the headline workload: 720p, one 1x1 layer, eight steps
        _case("720p 1x1"),
        # the server loop on it: Algorithm 1 with the paper's optimiser, threshold and MAX_UPDATES, results to the host
        _case("train 720p 1x1", task="train", adam=True),
        # 720p with a hidden 3x3 layer: dense contractions forward and backward
        _case("720p two layers", hidden=256, lr=0.005),
        # the largest frame: 1080p, two layers, sixteen steps
        _case("1080p two layers", hidden=256, classes=19, feat_h=270, feat_w=480, steps=16, lr=0.005),
        # sixteen clients served together
        _case("720p 16 streams", streams=16),
        # the trained back part in the paper's own shape: two blocks with skip inputs, Adam, weighted loss, Algorithm 1
        _case("train 720p stack", task="train", c_in=128, blocks="128+64,64+64", adam=True, lr=0.001, object_weight=5, object_radius=8),
        # odd sizes: frames of a cropped, resized camera, three clients, a narrow hidden layer
        _case("odd sizes 3 streams", streams=3, c_in=192, hidden=128, classes=13, feat_h=101, feat_w=187, steps=4),
        # channel and class counts that only the fp32 path takes
        _case("fp32 many classes", c_in=96, hidden=48, classes=81, feat_h=90, feat_w=160, steps=4, bf16=False),
    ]


def draw(rng):
    while True:
        c = _drawn(rng)
        if _cost(c) <= max(_cost(k) for k in listed()):
            return c


def _log_int(rng, lo, hi):
    return round(math.exp(rng.uniform(math.log(lo), math.log(hi))))


def _drawn(rng):
    task = rng.choice(("key_frame", "key_frame", "key_frame", "train", "train", "predict", "agreement"))
    feat_h = _log_int(rng, 45, 270)
    kw = dict(task=task, feat_h=feat_h, feat_w=round(feat_h * rng.uniform(1.2, 2.1)), classes=_log_int(rng, 2, 32),
              steps=_log_int(rng, 1, 16))
    if task == "agreement":
        return _case(**kw)
    if task != "predict":
        kw["streams"] = _log_int(rng, 1, 16)
        kw.update(rng.choice((dict(), dict(momentum=0.0), dict(adam=True))))
        if rng.random() < 0.3:
            kw.update(object_weight=rng.randint(2, 5), object_radius=rng.randint(0, 16))
    head = rng.choice(("1x1", "1x1", "hidden", "stack", "fp32"))
    if head == "fp32":
        kw.update(bf16=False, c_in=_log_int(rng, 16, 256), hidden=rng.choice((0, _log_int(rng, 16, 128))))
        if not kw.get("object_weight"):
            kw["classes"] = _log_int(rng, 2, 150)
    elif head == "stack":
        kw["c_in"] = 64 * rng.randint(1, 2)
        kw["blocks"] = "%d+%d,%d+%d" % (64 * rng.randint(1, 2), 64 * rng.randint(0, 2), 64 * rng.randint(1, 2), 64 * rng.randint(0, 2))
    else:
        kw["c_in"] = 64 * rng.randint(1, 4 if head == "hidden" else 8)
        kw["hidden"] = 64 * rng.randint(1, 4) if head == "hidden" else 0
    return _case(**kw)


# ---- sizes -------------------------------------------------------------------------------------------------------
def _blocks(c):
    return [tuple(int(v) for v in b.split("+")) for b in c["blocks"].split(",") if b]


def _layers(c):
    """(output channels, input channels, taps, channels of the input that the layer before it has produced) in forward order."""
    prev, made, out = c["c_in"], 0, []
    for co, cs in _blocks(c) or ([(c["hidden"], 0)] if c["hidden"] else []):
        out.append((co, prev + cs, 9, made))
        prev = made = co
    return out + [(c["classes"], prev, 1, made)]


def _pixels(c):
    return c["feat_h"] * c["feat_w"], 16 * c["feat_h"] * c["feat_w"]


def _forward_flops(c):
    return 2.0 * _pixels(c)[0] * sum(co * ci * taps for co, ci, taps, _ in _layers(c))


def work(case):
    c = case
    p, P = _pixels(c)
    if c["task"] == "agreement":
        return {"bytes": 2.0 * P + 8 * c["classes"] ** 2 + 8, "flops": 0.0}
    n_params = sum(co * (ci * taps + 1) for co, ci, taps, _ in _layers(c))
    c_inputs = c["c_in"] + sum(b[1] for b in _blocks(c))
    inputs = 4.0 * c_inputs * p + 4.0 * n_params
    mask = _forward_flops(c) + 4.0 * c["classes"] * P                     # interpolate and compare every class of every pixel
    if c["task"] == "predict":
        return {"bytes": inputs + P, "flops": mask}
    # a step: forward, weight gradients, the gradient passed back to what a trained layer has produced, and per class and
    # frame pixel 20 operations of the loss (interpolation, exponential, sum, normalisation, adjoint)
    back = 2.0 * p * sum(co * made * taps for co, _, taps, made in _layers(c))
    step = 2.0 * _forward_flops(c) + back + 20.0 * c["classes"] * P
    return {"bytes": c["streams"] * (inputs + 4.0 * c["classes"] * P + P + 4.0 * n_params),
            "flops": c["streams"] * (c["steps"] * step + mask)}


def _cost(c):
    """Rough seconds of a pass, to keep drawn cases below the largest listed one."""
    w, (p, P) = work(c), _pixels(c)
    steps = c["streams"] * c["steps"] if c["task"] in ("key_frame", "train") else 1
    per_pixel = 1e-12 * c["classes"] * P * steps
    return w["bytes"] / 3e12 + w["flops"] / (5e14 if c["bf16"] else 5e12) + per_pixel


def tolerance(case):
    if case["task"] == "agreement":
        return "exact"
    if case["task"] == "predict":
        return {"rel": 0.0, "differ": 1e-3}                               # near-ties of the upsampled logits
    # bf16 operands: a weight or a gradient rounded the other way now and then, and what K steps make of it; fp32: the order
    # of the sums, and the metric, a count of pixels of which one or two near-ties fall the other way.  Adam divides by the
    # size of the gradient: a parameter whose gradient all but cancels moves by its sign.
    rel = 5e-3 if case["bf16"] else 1e-4
    return {"rel": rel, "max": 0.5 if case["adam"] else 40 * rel}


# ---- inputs ------------------------------------------------------------------------------------------------------
_stream = None


def _cuda_stream():
    """One CUDA stream for everything, as in a process that serves its clients from one queue."""
    global _stream
    if _stream is None:
        _stream = torch.cuda.Stream()
    return _stream


def _class_map(g, H, W, n_regions, n_classes):
    """Regions of one class each (nearest of n_regions random points), uint8 [H][W]: a segmented frame."""
    pts = torch.rand((n_regions, 2), generator=g, device="cuda") * torch.tensor([H, W], device="cuda", dtype=torch.float32)
    ys, xs = torch.arange(H, device="cuda", dtype=torch.float32)[:, None], torch.arange(W, device="cuda", dtype=torch.float32)[None, :]
    best, cls = torch.full((H, W), float("inf"), device="cuda"), torch.zeros((H, W), dtype=torch.uint8, device="cuda")
    for r in range(n_regions):
        d = (ys - pts[r, 0]) ** 2 + (xs - pts[r, 1]) ** 2
        cls.masked_fill_(d < best, r % n_classes)
        best = torch.minimum(best, d)
    return cls


def _features(g, n, h, w, low=None):
    """ReLU(N(0, 1)); with `low` (class per feature pixel) channel c is raised where the frame shows class c, as a frozen
    part's output that tells something about the frame."""
    x = torch.randn((n, h, w), generator=g, device="cuda").relu_()
    if low is not None:
        x.scatter_add_(0, (low.long() % n)[None], torch.full((1, h, w), 3.0, device="cuda"))
    return x


def _student(g, c):
    """Packed parameters: He-normal weights and zero biases; every layer leans toward passing its input channels on, so that
    the classes can be told apart like by a student that has seen the stream before."""
    parts = []
    for co, ci, taps, _ in _layers(c):
        wt = torch.randn((co, ci, taps), generator=g, device="cuda") * math.sqrt(2.0 / (ci * taps))
        wt[torch.arange(co), torch.arange(co) % ci, taps // 2] += 0.5 if taps == 1 else 1.0
        parts += [wt.reshape(-1), torch.zeros(co, device="cuda")]
    return torch.cat(parts)


def prepare(case, seed):
    c = case
    h, w, C, S = c["feat_h"], c["feat_w"], c["classes"], c["streams"]
    H, W = 4 * h, 4 * w
    with torch.cuda.stream(_cuda_stream()):
        g = torch.Generator(device="cuda")
        g.manual_seed(seed)
        state = {"case": c, "conf": torch.zeros((C, C), dtype=torch.int64, device="cuda"),
                 "miou": torch.zeros(S, dtype=torch.float64, device="cuda")}
        if c["task"] == "agreement":
            # a prediction whose region borders are a few pixels off, with one per cent of stray pixels
            label = _class_map(g, H, W, 64, C)
            stray = torch.rand((H, W), generator=g, device="cuda") < 0.01
            noise = torch.randint(0, C, (H, W), generator=g, device="cuda", dtype=torch.uint8)
            state.update(label=label, pred=torch.where(stray, noise, torch.roll(label, (3, 5), (0, 1))))
            # masks need no student; the smallest head gives the context that st_agreement is called on
            state["ctx"] = st.st_init_head(c_in=1, n_classes=C, feat_h=h, feat_w=w, cuda_stream=_cuda_stream().cuda_stream,
                                           init_params=torch.zeros(2 * C, device="cuda"))
            return state
        feats, skips, logits, students = [], [], [], []
        for _ in range(S):
            cls = _class_map(g, H, W, 64, C)
            feats.append(_features(g, c["c_in"], h, w, cls[2::4, 2::4]))
            skips.append([_features(g, cs, h, w) if cs else None for _, cs in _blocks(c)])
            if c["task"] != "predict":
                t = torch.randn((C, H, W), generator=g, device="cuda").mul_(0.5)
                logits.append(t.scatter_add_(0, cls.long()[None], torch.full((1, H, W), 4.0, device="cuda")))
            students.append(_student(g, c))
        students = torch.stack(students)
        ctx = st.st_init_head(
            n_streams=S, c_in=c["c_in"], c_hidden=c["hidden"], n_classes=C, feat_h=h, feat_w=w, gemm_precision=int(c["bf16"]),
            lr=c["lr"], momentum=0.0 if c["adam"] else c["momentum"], optimizer=int(c["adam"]),
            object_weight=c["object_weight"], object_radius=c["object_radius"], blocks=_blocks(c),
            cuda_stream=_cuda_stream().cuda_stream, init_params=students)
        state.update(ctx=ctx, feats=feats, skips=skips, logits=logits, students=students)
        if c["task"] != "predict":
            state["labels"] = torch.zeros((S, H, W), dtype=torch.uint8, device="cuda")
        if c["task"] == "predict":
            state.update(update=students[0].cpu().pin_memory(), mask=torch.zeros((H, W), dtype=torch.uint8, device="cuda"))
        elif c["task"] == "train":
            state.update(packed=torch.zeros((S, ctx.n_params)).pin_memory(), best=torch.zeros(S, dtype=torch.float64).pin_memory(),
                         metrics=torch.zeros((S, c["steps"] + 1), dtype=torch.float64).pin_memory())
        else:
            state.update(packed=torch.zeros((S, ctx.n_params), device="cuda"), losses=torch.zeros((S, c["steps"]), device="cuda"))
        torch.cuda.current_stream().synchronize()
    return state


# ---- one pass ----------------------------------------------------------------------------------------------------
def run(state):
    c, ctx = state["case"], state["ctx"]
    if c["task"] == "agreement":
        st.st_agreement(ctx, 0, state["pred"], state["label"], state["conf"], miou_out=state["miou"])
        return {"conf": state["conf"], "miou": state["miou"]}
    if c["task"] == "predict":
        st.st_apply_update(ctx, 0, state["update"])
        _set_inputs(state, ctx, 0)
        st.st_student_mask(ctx, 0, state["mask"])
        return state["mask"]
    for s in range(c["streams"]):
        st.st_apply_update(ctx, s, state["students"][s])
        _set_inputs(state, ctx, s)
        st.st_teacher_labels(ctx, s, state["logits"][s], state["labels"][s])
    if c["task"] == "train":
        st.st_train_key_frame(ctx, 0.8, c["steps"], None, state["best"], state["metrics"])
        for s in range(c["streams"]):
            st.st_pack_updated_params(ctx, s, state["packed"][s])
        return {k: state[k] for k in ("packed", "best", "metrics", "labels")}
    st.st_distill_step(ctx, c["steps"], state["losses"])
    for s in range(c["streams"]):
        st.st_pack_updated_params(ctx, s, state["packed"][s])
        st.st_agreement(ctx, s, miou_out=state["miou"][s:s + 1])
    return {k: state[k] for k in ("packed", "losses", "miou", "labels")}


def _set_inputs(state, ctx, s):
    st.st_set_frozen_features(ctx, s, state["feats"][s])
    for b, x in enumerate(state["skips"][s]):
        if x is not None:
            st.st_set_skip_features(ctx, s, b, x)
