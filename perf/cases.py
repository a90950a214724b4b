"""The work this framework is used for, as measurable cases: scoring batches of frames, stepping video
streams in the closed loop forward -> select, the branched arrangement, the isolated fused linear, the
adapter-set selection by itself and the training-time context construction.

A case is a dict of plain values.  `prepare` makes what a program holds before the call (inputs on the GPU
from the seed; the model, whose weights depend on the case alone, is built once and kept, as a serving
process keeps it), `run` makes one pass through the public entry points and returns everything it wrote.
"""
from __future__ import annotations

import numpy as np
import torch

from paper_2507_14959_b200 import binding

#: width, heads, MLP width of the backbones (12 blocks, 16-pixel patches, 64-wide heads)
BACKBONES = {"deit_tiny": (192, 3, 768), "deit_small": (384, 6, 1536), "vit_base": (768, 12, 3072)}
LAYERS = 12
PATCH_DIM = 3 * 16 * 16
MAX_SET = 3                       # adapters of a frame: 1 / 2 / 3 with probability 0.6 / 0.3 / 0.1
MEAN_SET = 1.5
LINEAR_MAX_SET = 8                # the isolated linear: 1 to 8 adapters of 128 per frame
LINEAR_ADAPTERS = 128
SETS_IN_TURN = 4                  # host set lists used in turn: consecutive batches differ in some frames' sets
TAU, SCORE_THR = 0.6, 0.5


def listed():
    return [
        # one camera on the small embedded model, adapters on query and value of the last two blocks: the
        # smallest call there is, where latency and launches count
        {"name": "stream_tiny_1", "path": "stream", "model": "deit_tiny", "img": 224, "frames": 1, "classes": 80,
         "adapters": 11, "rank": 16, "last_blocks": 2, "own_stream": True},
        # sixteen cameras at the large image size (577 tokens), every block adapted, closed loop
        {"name": "stream_base384_16", "path": "stream", "model": "vit_base", "img": 384, "frames": 16, "classes": 800,
         "adapters": 64, "rank": 16, "last_blocks": 12, "own_stream": True},
        # a request with a single frame on the large backbone
        {"name": "batch_base_1", "path": "batch", "model": "vit_base", "img": 224, "frames": 1, "classes": 800,
         "adapters": 32, "rank": 16, "last_blocks": 12, "own_stream": False},
        # an odd, middling batch on the large backbone
        {"name": "batch_base_37", "path": "batch", "model": "vit_base", "img": 224, "frames": 37, "classes": 800,
         "adapters": 32, "rank": 16, "last_blocks": 12, "own_stream": False},
        # the production batch on the large backbone: the largest call
        {"name": "batch_base_256", "path": "batch", "model": "vit_base", "img": 224, "frames": 256, "classes": 800,
         "adapters": 32, "rank": 16, "last_blocks": 12, "own_stream": True},
        # the middle backbone with low-rank adapters, a batch of 64 frames
        {"name": "batch_small_64", "path": "batch", "model": "deit_small", "img": 224, "frames": 64, "classes": 160,
         "adapters": 16, "rank": 8, "last_blocks": 12, "own_stream": False},
        # the cheap placement with one branch per active adapter behind a shared trunk
        {"name": "branched_base_96", "path": "branched", "model": "vit_base", "img": 224, "frames": 96, "classes": 800,
         "adapters": 32, "rank": 16, "last_blocks": 2, "own_stream": False},
        # the fused linear alone: few frames, wide sets of rank-16 adapters
        {"name": "linear_qkv_16", "path": "linear", "k_in": 768, "n_out": 2304, "frames": 16, "rank": 16,
         "zipf": False, "epilogue": 0},
        # many frames, high rank, clustered sets, GELU
        {"name": "linear_fc1_64_r64", "path": "linear", "k_in": 768, "n_out": 3072, "frames": 64, "rank": 64,
         "zipf": True, "epilogue": 1},
        # the long contraction with a residual on the largest batch
        {"name": "linear_fc2_256", "path": "linear", "k_in": 3072, "n_out": 768, "frames": 256, "rank": 16,
         "zipf": False, "epilogue": 2},
        # the selection for many streams at once
        {"name": "select_2048", "path": "select", "frames": 2048, "classes": 800, "adapters": 64, "copy": True},
        # contexts from the label sets of a training set (the size of COCO's training images)
        {"name": "contexts_118287", "path": "contexts", "frames": 118287, "classes": 80, "size": 5, "contexts": 45,
         "overlap": True},
    ]


def _log_int(rng, lo, hi):
    return int(round(lo * (hi / lo) ** rng.random()))


def draw(rng):
    path = rng.choice(["stream", "batch", "batch", "branched", "linear", "linear", "select", "contexts"])
    if path == "linear":
        k_in, n_out, epilogue = rng.choice([(768, 2304, 0), (768, 3072, 1), (3072, 768, 2), (768, 768, 2), (384, 1152, 0),
                                            (1536, 384, 2), (192, 768, 1)])
        return {"path": path, "k_in": k_in, "n_out": n_out, "frames": _log_int(rng, 1, 256),
                "rank": rng.choice([4, 8, 16, 24, 32, 64]), "zipf": rng.random() < 0.5, "epilogue": epilogue}
    if path == "select":
        return {"path": path, "frames": _log_int(rng, 1, 2048), "classes": rng.choice([80, 160, 601, 800]),
                "adapters": rng.choice([11, 16, 32, 64]), "copy": rng.random() < 0.5}
    if path == "contexts":
        return {"path": path, "frames": _log_int(rng, 2000, 250000), "classes": rng.choice([80, 160, 365, 601, 800]),
                "size": rng.choice([2, 3, 5, 10, 15]), "contexts": rng.choice([11, 26, 45, 50]),
                "overlap": rng.random() < 0.5}
    model = rng.choice(["deit_tiny", "deit_small", "vit_base"])
    img = 384 if rng.random() < 0.25 else 224
    most = {"deit_tiny": 256, "deit_small": 256, "vit_base": 192}[model] // (4 if img == 384 else 1)
    if path == "stream":
        most //= 2
    if path == "branched":
        most = most * 2 // 3
    return {"path": path, "model": model, "img": img, "frames": _log_int(rng, 1, most),
            "classes": rng.choice([80, 160, 800]), "adapters": rng.choice([4, 11, 16, 32, 64]),
            "rank": rng.choice([4, 8, 16, 32]), "last_blocks": 2 if path == "branched" else rng.choice([2, 12, 12]),
            "own_stream": rng.random() < 0.5}


# ---- inputs -----------------------------------------------------------------------------------------
def _generator(seed):
    return torch.Generator(device="cuda").manual_seed(seed)


def _normal(gen, shape, std, mean=0.0):
    """bf16-representable values, as float32 on the host (what the model constructor takes)."""
    return (torch.randn(shape, generator=gen, device="cuda") * std + mean).bfloat16().float().cpu().numpy()


def _shapes(model):
    d, _, m = BACKBONES[model]
    return ((d, 3 * d), (d, d), (d, m), (m, d))


def _groups(classes, adapters):
    """Class subsets of the adapters: a partition, in which every tenth class is also listed by the next adapter."""
    per = max(1, classes // adapters)
    groups = [[(per * a + j) % classes for j in range(per)] for a in range(adapters)]
    for k in range(0, classes, 10):
        other = groups[(k // per + 1) % adapters]
        if k not in other:
            other.append(k)
    return [np.asarray(sorted(set(g)), dtype=np.int32) for g in groups]


def _build_model(case, max_frames):
    d, heads, m = BACKBONES[case["model"]]
    tokens, classes = (case["img"] // 16) ** 2 + 1, case["classes"]
    gen = _generator(20250714)
    # The base head of a trained multi-label classifier is confident: a few classes are well above the score
    # threshold and the rest well below it (six standard deviations of a logit), so that rounding does not
    # decide which labels a frame has.
    head_b = np.full(classes, -6.0 * 0.02 * d ** 0.5, dtype=np.float32)
    head_b[[3 % classes, classes // 2, classes - 7]] *= -1.0
    backbone = {
        "patch_w": _normal(gen, (PATCH_DIM, d), 0.02), "patch_b": _normal(gen, (d,), 0.02),
        "cls": _normal(gen, (d,), 0.02), "pos": _normal(gen, (tokens, d), 0.02),
        "ln1_g": _normal(gen, (LAYERS, d), 0.02, 1.0), "ln1_b": _normal(gen, (LAYERS, d), 0.02),
        "qkv_w": _normal(gen, (LAYERS, d, 3 * d), 0.02), "qkv_b": _normal(gen, (LAYERS, 3 * d), 0.02),
        "proj_w": _normal(gen, (LAYERS, d, d), 0.02), "proj_b": _normal(gen, (LAYERS, d), 0.02),
        "ln2_g": _normal(gen, (LAYERS, d), 0.02, 1.0), "ln2_b": _normal(gen, (LAYERS, d), 0.02),
        "fc1_w": _normal(gen, (LAYERS, d, m), 0.02), "fc1_b": _normal(gen, (LAYERS, m), 0.02),
        "fc2_w": _normal(gen, (LAYERS, m, d), 0.02), "fc2_b": _normal(gen, (LAYERS, d), 0.02),
        "lnf_g": _normal(gen, (d,), 0.02, 1.0), "lnf_b": _normal(gen, (d,), 0.02),
        "head_w": _normal(gen, (d, classes), 0.02), "head_b": head_b,
    }
    model = binding.Model(img=case["img"], d=d, layers=LAYERS, heads=heads, mlp=m, n_classes=classes, backbone=backbone,
                          max_adapters=case["adapters"], max_rank=case["rank"], max_set=MAX_SET, max_frames=max_frames)
    r = case["rank"]
    for a, ids in enumerate(_groups(classes, case["adapters"])):
        A, B = [None] * (4 * LAYERS), [None] * (4 * LAYERS)
        for i in range(4 * (LAYERS - case["last_blocks"]), 4 * LAYERS):
            k, n = _shapes(case["model"])[i % 4]
            if case["last_blocks"] == LAYERS or i % 4 == 0:      # the cheap placement adapts query and value only
                A[i], B[i] = _normal(gen, (k, r), 0.02), _normal(gen, (r, n), 0.02)
                if case["last_blocks"] < LAYERS:
                    B[i][:, d:2 * d] = 0.0
        acc = 0.5 + 0.5 * torch.rand(len(ids), generator=gen, device="cuda").cpu().numpy()
        model.register_adapter(a, rank=r, scale=32.0 / r, A=A, B=B, class_ids=ids,
                               head_w=_normal(gen, (d, len(ids)), 0.02), head_b=_normal(gen, (len(ids),), 0.02), acc=acc)
    model.set_cover(TAU)
    return model


def _build_linear(case):
    gen = _generator(20250714)
    k, n, r = case["k_in"], case["n_out"], case["rank"]
    lin = binding.Linear(_normal(gen, (k, n), 0.02), _normal(gen, (n,), 0.02), max_adapters=LINEAR_ADAPTERS, max_rank=r,
                         max_set=LINEAR_MAX_SET, max_frames=case["frames"], tokens=197, epilogue=case["epilogue"])
    for a in range(LINEAR_ADAPTERS):
        lin.register(a, r, 32.0 / r, _normal(gen, (k, r), 0.02), _normal(gen, (r, n), 0.02))
    return lin


_kept = {}                        # the one model or linear in use, as a serving process holds it
_streams = []


def _keep(key, build):
    if key not in _kept:
        _kept.clear()
        _kept[key] = build()
    return _kept[key]


def _stream():
    """The process's own stream: calls on one model share its scratch memory, so they share a stream too."""
    if not _streams:
        _streams.append(torch.cuda.Stream())
    return _streams[0]


def _csr(sets):
    off = np.zeros(len(sets) + 1, dtype=np.int32)
    off[1:] = np.cumsum([len(s) for s in sets])
    return off, np.asarray([a for s in sets for a in sorted(s)], dtype=np.int32)


def _draw_set(g, adapters):
    size = min(adapters, 1 + int(g.choice(3, p=(0.6, 0.3, 0.1))))
    return [int(a) for a in g.choice(adapters, size=size, replace=False)]


def _set_lists(g, draw_one, frames):
    """Slowly changing sets: from one list to the next every frame redraws its set with probability 0.1."""
    sets, lists = [draw_one() for _ in range(frames)], []
    for _ in range(SETS_IN_TURN):
        lists.append(_csr(sets))
        sets = [draw_one() if g.random() < 0.1 else s for s in sets]
    return lists


def _label_words(present):
    """bool [n, classes] -> int32 bit sets [n, ceil(classes / 32)]."""
    n, k = present.shape
    words = (k + 31) // 32
    padded = torch.zeros((n, 32 * words), dtype=torch.bool, device="cuda")
    padded[:, :k] = present
    value = (padded.view(n, words, 32).long() << torch.arange(32, device="cuda")).sum(-1)
    return torch.where(value >= 2 ** 31, value - 2 ** 32, value).int()


def _ints(a):
    return torch.from_numpy(np.ascontiguousarray(a, dtype=np.int32)).cuda()


def prepare(case, seed):
    gen, g = _generator(seed), np.random.default_rng(seed)
    state = {"path": case["path"], "turn": 0}
    F = case["frames"]
    if case["path"] == "contexts":
        # frames show a scene each (scenes are unevenly frequent); one to five of its labels, now and then a stray one
        K = case["classes"]
        scenes = max(2, K // 4)
        scene = (scenes * torch.rand(F, generator=gen, device="cuda") ** 2).long()
        present = torch.zeros((F, K), dtype=torch.bool, device="cuda")
        keep = 1 + torch.randint(5, (F,), generator=gen, device="cuda")
        for j in range(5):
            label = (scene * 4 + torch.randint(6, (F,), generator=gen, device="cuda")) % K
            present[torch.arange(F, device="cuda")[keep > j], label[keep > j]] = True
        stray = torch.rand(F, generator=gen, device="cuda") < 0.1
        present[stray.nonzero()[:, 0], torch.randint(K, (int(stray.sum()),), generator=gen, device="cuda")] = True
        state.update(labels=_label_words(present), co=torch.empty((K, K), device="cuda"), classes=K, size=case["size"],
                     contexts=case["contexts"], overlap=case["overlap"])
        return state
    if case["path"] == "linear":
        p = 1.0 / np.arange(1, LINEAR_ADAPTERS + 1) ** 1.2
        p = p / p.sum() if case["zipf"] else None
        one = lambda: [int(a) for a in g.choice(LINEAR_ADAPTERS, size=int(g.integers(1, LINEAR_MAX_SET + 1)),  # noqa: E731
                                                replace=False, p=p)]
        rows = F * 197
        x = torch.randn((rows, case["k_in"]), generator=gen, device="cuda").bfloat16()
        res = torch.randn((rows, case["n_out"]), generator=gen, device="cuda").bfloat16() if case["epilogue"] == 2 else None
        key = tuple(sorted((k, v) for k, v in case.items() if k not in ("name", "zipf")))
        state.update(lin=_keep(key, lambda: _build_linear(case)), x=x, residual=res, frames=F,
                     y=torch.empty((rows, case["n_out"]), device="cuda", dtype=torch.bfloat16), lists=_set_lists(g, one, F))
        return state
    if case["path"] == "select":
        case = dict(case, model="deit_tiny", img=224, rank=16, last_blocks=2)
    K, na = case["classes"], case["adapters"]
    max_frames = F * (1 + MAX_SET) if case["path"] == "branched" else F
    key = tuple(sorted((k, v) for k, v in case.items() if k not in ("name", "own_stream", "copy")))
    state["model"] = _keep(key, lambda: _build_model(case, max_frames))
    state["scores"] = torch.empty((F, K), device="cuda")
    one = lambda: _draw_set(g, na)  # noqa: E731
    if case["path"] in ("stream", "select"):
        # the sets of the step before and where the next ones go
        sets = [one() for _ in range(F)]
        off, ids = _csr(sets)
        state.update(off=_ints(off), ids=_ints(np.pad(ids, (0, F * na - len(ids)))), next_off=torch.zeros(F + 1, dtype=torch.int32, device="cuda"),
                     next_ids=torch.zeros(F * na, dtype=torch.int32, device="cuda"))
        seen = torch.zeros((F, K), dtype=torch.bool, device="cuda")
        groups = _groups(K, na)
        pairs = [(f, int(g.choice(groups[sets[f][0]]) if g.random() < 0.8 else g.integers(K))) for f in range(F) for _ in range(2)]
        at = torch.tensor(pairs, device="cuda")
        seen[at[:, 0], at[:, 1]] = True
        state["labels"] = _label_words(seen)
    if case["path"] == "select":
        # scores of a confident classifier: up to three labels well above the threshold, mostly of the set in use
        pairs = [(f, int(g.choice(groups[sets[f][0]]) if g.random() < 0.8 else g.integers(K)))
                 for f in range(F) for _ in range(int(g.integers(0, 4)))] or [(0, 0)]
        at = torch.tensor(pairs, device="cuda")
        state["scores"] = 0.3 * torch.rand((F, K), generator=gen, device="cuda")
        state["scores"][at[:, 0], at[:, 1]] = 0.6 + 0.4 * torch.rand(len(pairs), generator=gen, device="cuda")
        state["copy"] = case["copy"]
        return state
    # a clip's frame: a still picture under sensor noise
    picture = 2.0 * torch.rand((F, 3, case["img"], case["img"]), generator=gen, device="cuda") - 1.0
    state["frames"] = (picture + 0.05 * torch.randn(picture.shape, generator=gen, device="cuda")).bfloat16()
    state["base"] = torch.empty((F, K), device="cuda")
    state["stream"] = _stream() if case["own_stream"] else None
    if case["path"] != "stream":
        state["lists"] = _set_lists(g, one, F)
        state["trunk"] = LAYERS - case["last_blocks"]
    torch.cuda.synchronize()
    return state


# ---- one pass ---------------------------------------------------------------------------------------
def run(state):
    path = state["path"]
    if path == "contexts":
        binding.cooccurrence(state["labels"], state["classes"], state["co"])
        co = state["co"].cpu().numpy()
        found = binding.build_contexts(co, state["size"], state["contexts"], state["overlap"])
        return {"co": co, "sizes": np.asarray([len(c) for c in found], dtype=np.int32),
                "ids": np.asarray([k for c in found for k in c], dtype=np.int32)}
    if path == "select":
        state["model"].select(state["scores"], SCORE_THR, state["copy"], True, state["labels"], state["off"], state["ids"],
                              state["next_off"], state["next_ids"])
        return {k: state[k] for k in ("labels", "next_off", "next_ids")}
    if path == "stream":
        m, st = state["model"], state["stream"]
        m.forward_device_sets(state["frames"], state["off"], state["ids"], state["scores"], state["base"], stream=st)
        m.select(state["base"], SCORE_THR, False, True, state["labels"], state["off"], state["ids"], state["next_off"],
                 state["next_ids"], stream=st)
        return {k: state[k] for k in ("scores", "base", "labels", "next_off", "next_ids")}
    off, ids = state["lists"][state["turn"]]
    state["turn"] = (state["turn"] + 1) % SETS_IN_TURN
    if path == "linear":
        state["lin"].forward(state["x"], state["frames"], off, ids, state["y"], residual=state["residual"])
        return state["y"]
    if path == "branched":
        state["model"].forward_branched(state["frames"], off, ids, state["trunk"], state["scores"], state["base"],
                                        stream=state["stream"])
    else:
        state["model"].forward(state["frames"], off, ids, state["scores"], state["base"], stream=state["stream"])
    return {"scores": state["scores"], "base": state["base"]}


# ---- what a pass cannot do without ------------------------------------------------------------------
def work(case):
    F = case["frames"]
    if case["path"] == "contexts":
        K = case["classes"]
        return {"bytes": 4 * F * ((K + 31) // 32) + 4 * K * K, "flops": 0}
    if case["path"] == "select":
        K = case["classes"]
        return {"bytes": 4 * F * K + 2 * 4 * F * ((K + 31) // 32) + 2 * 4 * F * (1 + MEAN_SET), "flops": 0}
    if case["path"] == "linear":
        k, n, rows = case["k_in"], case["n_out"], F * 197
        mean = (1 + LINEAR_MAX_SET) / 2
        moved = rows * (k + n + (n if case["epilogue"] == 2 else 0)) + k * n + min(LINEAR_ADAPTERS, F * mean) * case["rank"] * (k + n)
        return {"bytes": 2 * moved, "flops": 2 * rows * (k * n + mean * case["rank"] * (k + n))}
    d, _, m = BACKBONES[case["model"]]
    T, K = (case["img"] // 16) ** 2 + 1, case["classes"]
    block = 2 * T * (4 * d * d + 2 * d * m) + 4 * T * T * d
    linears = _shapes(case["model"]) if case["last_blocks"] == LAYERS else _shapes(case["model"])[:1]
    ranks = case["rank"] * sum(k + n for k, n in linears)          # one adapter's parameters in a block
    lora = 2 * T * ranks * MEAN_SET
    tail = case["last_blocks"]
    mult = 1 + MEAN_SET if case["path"] == "branched" else 1       # branches of a frame in the adapted blocks
    flops = F * (2 * (T - 1) * PATCH_DIM * d + (LAYERS - tail) * block + tail * (mult * block + lora) + 2 * d * K)
    params = PATCH_DIM * d + LAYERS * (4 * d * d + 2 * d * m) + d * K + min(case["adapters"], MEAN_SET * F) * tail * ranks
    return {"bytes": 2 * params + 2 * F * 3 * case["img"] ** 2 + 2 * 4 * F * K, "flops": flops}


def tolerance(case):
    if case["path"] in ("contexts", "select"):
        return "exact"            # counts, bit sets and id lists
    # bf16 storage with 32-bit sums against the 32-bit build on the same inputs: the linear's rows differ by
    # 1.7e-3 (largest 6e-3), scores by up to 2.8e-3 (largest 1.7e-2); four times that
    return {"rel": 7e-3, "max": 0.025} if case["path"] == "linear" else {"rel": 1.1e-2, "max": 0.07}
