"""The renderer's measured workloads: single renders in every precision,
culled, tiling and batched renders, the learned level of detail, the network's
training step, word evaluation and the general-presentation scan.

A case is a plain dict; ``prepare`` makes what a user's program holds before
the call (parameters, image, workspace, a captured batch, a trainer),
``run`` makes one pass through the package's public entry points.  The seed
moves the view (a user pans and zooms a little between renders) or, where a
workload is drawn at random anyway, draws other groups and rows.

Renders return the hit image and the word counters (drawn, dropped, FP64
words).  The fourth counter, the number of image adds a kernel issued, says how
a kernel merges equal pixels; it is a diagnostic of the launch and differs
between two culled renders of one job, so it is not an output.
"""
import math

import numpy as np
import torch

import klsynth
import paper_1709_08018_gb300 as kl

PRECISIONS = {"fp64": kl.FP64, "mixed": kl.MIXED, "df64": kl.DF64}

# The indexed Cayley table of the once-punctured torus: states and symbols
# I, a, b, A, B = 0..4, 0 = crash.
TORUS_TABLE = [[0, 1, 2, 3, 4], [1, 1, 2, 0, 4], [2, 1, 2, 3, 0], [3, 0, 2, 3, 4],
               [4, 1, 0, 3, 4]]

GASKET = {"ta_re": 2.0, "ta_im": 0.0, "tb_re": 2.0, "tb_im": 0.0}
NEAR_CUSP = {"ta_re": 1.91, "ta_im": 0.05, "tb_re": 1.91, "tb_im": 0.05}


def _render(group, depth, width, height, half, precision, **more):
    return {"kind": "render", **group, "depth": depth, "width": width, "height": height,
            "half": half, "precision": precision, "cull": 0, "tiling": 0, **more}


def listed():
    return [
        # a thumbnail or an interactive preview: the smallest call, where
        # launches and latency are all there is
        {"name": "fp64-preview-d10", **_render(GASKET, 10, 1024, 1024, 1.5, "fp64")},
        # a picture for print in the paper's arithmetic
        {"name": "fp64-gasket-d18", **_render(GASKET, 18, 4096, 4096, 1.5, "fp64")},
        # the largest job of one call: all 4.6e9 words of a near-cusp group
        {"name": "fp64-nearcusp-d20", **_render(NEAR_CUSP, 20, 8192, 8192, 2.0, "fp64")},
        # the fast precision a production render takes
        {"name": "mixed-nearcusp-d20", **_render(NEAR_CUSP, 20, 8192, 8192, 2.0, "mixed")},
        # FP64-grade words on the FP32 pipe, a wide frame of odd size
        {"name": "df64-wide-d17", **_render({"ta_re": 2.2, "ta_im": 0.03, "tb_re": 2.6,
                                             "tb_im": -0.04}, 17, 3839, 2161, 1.5, "df64")},
        # certified blocks placed at once, for deep exact renders
        {"name": "cull-nearcusp-d20", **_render(NEAR_CUSP, 20, 8192, 8192, 2.0, "mixed", cull=1)},
        # every node of the word tree, a display-sized frame
        {"name": "tiling-gasket-d14", **_render(GASKET, 14, 1920, 1080, 1.5, "mixed", tiling=1)},
        # a parameter sweep: many groups of uneven depth, captured once, replayed
        {"name": "sweep-64-groups", "kind": "batch", "groups": 64, "depth_lo": 12,
         "depth_hi": 18, "side": 1024, "precision": "mixed", "cull": 0},
        # word values for plots and accuracy checks: a million sampled indices
        {"name": "eval-1e6-d20", "kind": "eval", **NEAR_CUSP, "depth": 20, "n": 1_000_000,
         "precision": "fp64"},
        # the paper's scan for a group given by its indexed Cayley table
        {"name": "scan-d13", "kind": "scan", **GASKET, "depth": 13, "width": 2000,
         "height": 1500},
        # a training step of the level-of-detail network at its usual batch
        {"name": "train-16384", "kind": "train", "rows": 16384},
        # the network-pruned render of a depth-22 group
        {"name": "lod-d22", "kind": "lod", "depth": 22, "side": 8192, "lo": 8, "hi": 13},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _draw_group(rng):
    pick = rng.random()
    if pick < 0.2:
        return dict(GASKET)
    if pick < 0.4:
        return dict(NEAR_CUSP)
    return {"ta_re": round(rng.uniform(2.0, 3.0), 4), "ta_im": round(rng.uniform(-0.05, 0.05), 4),
            "tb_re": round(rng.uniform(2.0, 3.0), 4), "tb_im": round(rng.uniform(-0.05, 0.05), 4)}


def draw(rng):
    kind = rng.choice(["render"] * 6 + ["batch", "eval", "scan", "train", "lod"])
    if kind == "render":
        tiling = rng.random() < 0.2
        cull = rng.random() < 0.3
        precision = rng.choice(["fp64", "mixed"] if cull else ["fp64", "mixed", "df64"])
        return _render(_draw_group(rng), rng.randint(6, 17 if tiling else 19),
                       _log_int(rng, 200, 8192), _log_int(rng, 200, 8192),
                       round(rng.uniform(0.6, 2.0), 3), precision, cull=int(cull),
                       tiling=int(tiling))
    if kind == "batch":
        return {"kind": "batch", "groups": _log_int(rng, 2, 64), "depth_lo": rng.randint(8, 12),
                "depth_hi": rng.randint(13, 18), "side": _log_int(rng, 200, 1024),
                "precision": rng.choice(["mixed", "fp64"]), "cull": int(rng.random() < 0.4)}
    if kind == "eval":
        return {"kind": "eval", **_draw_group(rng), "depth": rng.randint(5, 20),
                "n": _log_int(rng, 100, 1_000_000),
                "precision": rng.choice(["fp64", "mixed", "df64"])}
    if kind == "scan":
        return {"kind": "scan", **_draw_group(rng), "depth": rng.randint(6, 14),
                "width": _log_int(rng, 200, 4096), "height": _log_int(rng, 200, 4096)}
    if kind == "train":
        return {"kind": "train", "rows": _log_int(rng, 1000, 1_000_000)}
    lo = rng.randint(6, 8)
    depth = rng.randint(17, 22)
    return {"kind": "lod", "depth": depth, "side": _log_int(rng, 1000, 8192), "lo": lo,
            "hi": rng.randint(max(lo + 1, depth - 9), min(14, depth - 6))}


# ---------------------------------------------------------------------------
# inputs

def _view(seed, half, width=1, height=1):
    """The square view [-half, half]^2 (widened to the image's shape so that
    pixels stay square), panned and zoomed by up to a percent."""
    g = np.random.default_rng(seed)
    zoom = half * (1.0 + 0.01 * g.random())
    cx, cy = (0.01 * half * (2.0 * g.random(2) - 1.0)).tolist()
    hx = zoom * max(1.0, width / height)
    hy = zoom * max(1.0, height / width)
    return (cx - hx, cx + hx, cy - hy, cy + hy)


def _traces(c):
    return complex(c["ta_re"], c["ta_im"]), complex(c["tb_re"], c["tb_im"])


def _params(c, seed):
    kind = c["kind"]
    if kind == "render":
        return kl.params_init(*_traces(c), c["depth"], c["width"], c["height"],
                              _view(seed, c["half"], c["width"], c["height"]),
                              PRECISIONS[c["precision"]], cull=c["cull"], mode=c["tiling"])
    if kind == "eval":
        return kl.params_init(*_traces(c), c["depth"], 4096, 4096, _view(seed, 2.0),
                              PRECISIONS[c["precision"]])
    if kind == "scan":
        return kl.params_init(*_traces(c), c["depth"], c["width"], c["height"],
                              _view(seed, 1.5, c["width"], c["height"]), kl.FP64)
    if kind == "lod":
        g, _ = klsynth.draw_groups(klsynth.LOD_HELDOUT_SEED + seed, 1)[0]
        return kl.params_init(g.ta, g.tb, c["depth"], c["side"], c["side"],
                              (-2.0, 2.0, -2.0, 2.0), kl.MIXED)
    raise ValueError(kind)


def _batch_params(c, seed):
    groups = klsynth.draw_groups(klsynth.BATCH_SEED + seed, c["groups"], c["depth_lo"],
                                 c["depth_hi"])
    return [kl.params_init(g.ta, g.tb, d, c["side"], c["side"], (-1.5, 1.5, -1.5, 1.5),
                           PRECISIONS[c["precision"]], cull=c["cull"]) for g, d in groups]


def _network():
    """A network that scores a node as a trained one does: the image of a
    subtree shrinks with 1 / |r|^2 (r: the lower left entry of the node
    matrix), so the predicted label falls linearly in log |r| and crosses 1/2
    where a subtree of a [-2, 2]^2, 8192-pixel view falls under 1/32 pixel."""
    w = np.zeros(kl.KL_MLP_NPARAMS, dtype=np.float32)
    W1, W2 = w[0:512].reshape(8, 64), w[576:4672].reshape(64, 64)
    W1[4, 0], W1[4, 1], W1[5, 2], W1[5, 3] = 1.0, -1.0, 1.0, -1.0  # |re r|, |im r|
    W2[0:2, 0], W2[2:4, 0] = 1.0, -1.0                             # (|re r| - |im r|)+
    W2[2:4, 1] = 1.0                                               # |im r|
    w[4736:4738] = -2.0                                            # -2 max(...)
    w[4800] = 0.5 + 2.0 * 5.9
    return torch.from_numpy(w).cuda()


def _rows(c, seed):
    """Training rows: node features sign(v) log(1 + |v|) of matrices of levels
    8 .. 15, and clipped labels that fall with the size of the entries."""
    g = torch.Generator(device="cuda").manual_seed(seed)
    n = c["rows"]
    size = 1.0 + 7.0 * torch.rand((n, 1), device="cuda", generator=g)
    x = size + 0.4 * torch.randn((n, 8), device="cuda", generator=g)
    x *= torch.randint(0, 2, (n, 8), device="cuda", generator=g) * 2.0 - 1.0
    t = torch.clamp(torch.round(6.0 - size[:, 0] + 0.5 * torch.randn(n, device="cuda",
                                                                     generator=g)), 0.0, 3.0)
    p = np.random.default_rng(seed)
    w = np.zeros(kl.KL_MLP_NPARAMS, dtype=np.float32)  # He initialisation
    w[0:512] = p.normal(0.0, math.sqrt(2.0 / 8), 512)
    w[576:4672] = p.normal(0.0, math.sqrt(2.0 / 64), 4096)
    w[512:576] = w[4672:4736] = 0.01
    w[4736:4800] = p.normal(0.0, math.sqrt(1.0 / 64), 64)
    w[4800] = 1.0
    return torch.from_numpy(w).cuda(), x.contiguous(), t.contiguous()


def _indices(c, seed):
    idx = klsynth.index_sample(klsynth.SAMPLE_SEED + seed, c["n"], c["depth"])
    return torch.from_numpy(idx.astype(np.int64)).cuda()


# ---------------------------------------------------------------------------
# passes

LR, BETA1, BETA2, EPS, UNDER = 2e-3, 0.9, 0.999, 1e-8, 32.0


def prepare(case, seed):
    kind = case["kind"]
    if kind == "render":
        r = kl.Renderer(_params(case, seed))
        return {"kind": kind, "renderer": r}
    if kind == "batch":
        b = kl.Batch(_batch_params(case, seed))
        b.capture()
        return {"kind": kind, "batch": b}
    if kind == "eval":
        p = _params(case, seed)
        ws = torch.empty(kl.workspace_bytes(p), dtype=torch.uint8, device="cuda")
        return {"kind": kind, "p": p, "index": _indices(case, seed), "workspace": ws}
    if kind == "scan":
        p = _params(case, seed)
        return {"kind": kind, "p": p, "fsa": kl.fsa_from_params(TORUS_TABLE, p),
                "image": torch.empty((p.height, p.width), dtype=torch.int32, device="cuda"),
                "counters": torch.zeros(kl.KL_N_COUNTERS, dtype=torch.int64, device="cuda")}
    if kind == "train":
        w, x, t = _rows(case, seed)
        return {"kind": kind, "x": x, "t": t,
                "trainer": kl.MlpTrainer(w, lr=LR, beta1=BETA1, beta2=BETA2, eps=EPS,
                                         under_weight=UNDER)}
    return {"kind": kind, "mlp": _network(),
            "renderer": kl.LodRenderer(_params(case, seed), case["lo"], case["hi"])}


def run(state):
    kind = state["kind"]
    if kind == "render":
        image, counters = state["renderer"]()
        return {"image": image, "words": counters[:kl.KL_CNT_ATOMICS]}
    if kind == "batch":
        images, counters = state["batch"].replay()
        return {"images": images, "words": counters[:, :kl.KL_CNT_ATOMICS]}
    if kind == "eval":
        return {"uv": kl.eval_words(state["p"], state["index"], state["workspace"])}
    if kind == "scan":
        image, counters = kl.render_fsa(state["fsa"], state["p"], state["image"],
                                        state["counters"])
        return {"image": image, "words": counters[:kl.KL_CNT_ATOMICS]}
    if kind == "train":
        tr = state["trainer"]
        loss = tr.step(state["x"], state["t"])
        return {"loss": loss, "grad": tr.grad, "params": tr.params, "m": tr.m, "v": tr.v}
    image, counters, stats = state["renderer"](state["mlp"], -1.0, 1.0 / 128)
    return {"image": image, "words": counters[:kl.KL_CNT_ATOMICS], "stats": stats}


# ---------------------------------------------------------------------------
# work

def _words(depth):
    return 4 * 3 ** (depth - 1)


# One word's value in pole form with its pixel: two adds, |w|^2, a reciprocal,
# two numerators, two final multiply-adds.
WORD_FLOPS = 16
MLP_MACS = 8 * 64 + 64 * 64 + 64


def work(case):
    kind = case["kind"]
    if kind == "render":
        pixels = case["width"] * case["height"]
        words = 2 * (3 ** case["depth"] - 1) if case["tiling"] else _words(case["depth"])
        # a culled render need not look at every word: a few words per pixel hit
        if case["cull"]:
            words = min(words, 16 * pixels)
        return {"bytes": 4 * pixels + 32, "flops": WORD_FLOPS * words}
    if kind == "batch":
        pixels = case["groups"] * case["side"] ** 2
        mid = sum(_words(d) for d in range(case["depth_lo"], case["depth_hi"] + 1))
        words = case["groups"] * mid / (case["depth_hi"] - case["depth_lo"] + 1)
        if case["cull"]:
            words = min(words, 16 * pixels)
        return {"bytes": 4 * pixels, "flops": WORD_FLOPS * words}
    if kind == "eval":
        return {"bytes": 24 * case["n"], "flops": WORD_FLOPS * case["n"]}
    if kind == "scan":
        return {"bytes": 4 * case["width"] * case["height"],
                "flops": WORD_FLOPS * _words(case["depth"])}
    if kind == "train":
        n = case["rows"]
        return {"bytes": 36 * n + 7 * 4 * kl.KL_MLP_NPARAMS,
                "flops": 2 * n * (2 * MLP_MACS + 64 * 64 + 64)}
    # the level of detail: the image, and the nodes of its last level scored
    return {"bytes": 4 * case["side"] ** 2,
            "flops": 2 * MLP_MACS * _words(case["lo"] + 1)}


# ---------------------------------------------------------------------------
# the same outputs in 64 bits, in plain torch

def _maps(p):
    g = list(p.gens)
    return [[complex(g[8 * x + 2 * k], g[8 * x + 2 * k + 1]) for k in range(4)] for x in range(4)]


def _apply(M, z):
    return (M[0] * z + M[1]) / (M[2] * z + M[3])


def _exact_words(p, index, depth):
    """Pixel coordinates of the indexed words: the seed of the last letter,
    then the letters' maps from the last to the first."""
    letters = [index // 3 ** (depth - 1)]
    for k in range(1, depth):
        digit = index // 3 ** (depth - 1 - k) % 3
        letters.append(digit + (digit >= (letters[-1] + 2) % 4))
    M = torch.tensor(_maps(p), dtype=torch.complex128, device="cuda")
    s = list(p.seeds)
    z = torch.tensor([complex(s[2 * x], s[2 * x + 1]) for x in range(4)],
                     dtype=torch.complex128, device="cuda")[letters[-1]]
    for w in reversed(letters):
        m = M[w]
        z = (m[:, 0] * z + m[:, 1]) / (m[:, 2] * z + m[:, 3])
    sx, sy = p.width / (p.x1 - p.x0), p.height / (p.y1 - p.y0)
    return torch.stack([(z.real - p.x0) * sx, (p.y1 - z.imag) * sy], dim=1)


def _bin(p, z, image):
    """Counts the values z into the flat image."""
    for part in z.split(1 << 26):
        u = torch.floor((part.real - p.x0) * (p.width / (p.x1 - p.x0)))
        v = torch.floor((p.y1 - part.imag) * (p.height / (p.y1 - p.y0)))
        ok = (u >= 0) & (u < p.width) & (v >= 0) & (v < p.height)
        at = (v[ok].to(torch.int64) * p.width + u[ok].to(torch.int64))
        image += torch.bincount(at, minlength=image.numel())


def _exact_image(p, lengths):
    """The hit image of all words of the given lengths."""
    maps, s = _maps(p), list(p.seeds)
    image = torch.zeros(p.width * p.height, dtype=torch.int64, device="cuda")
    # by first letter: the values of all words of one length
    z = [_apply(maps[x], torch.tensor([complex(s[2 * x], s[2 * x + 1])],
                                      dtype=torch.complex128, device="cuda")) for x in range(4)]
    for k in range(1, max(lengths) + 1):
        if k > 1:
            z = [_apply(maps[x], torch.cat([z[y] for y in range(4) if y != (x + 2) % 4]))
                 for x in range(4)]
        if k in lengths:
            for x in range(4):
                _bin(p, z[x], image)
    return image.to(torch.int32).reshape(p.height, p.width)


def _exact_train(case, seed):
    """Loss, gradient and parameters after one Adam step, with FP64 sums."""
    w0, x, t = _rows(case, seed)
    w = w0.double().requires_grad_()
    h = torch.relu(x.double() @ w[0:512].reshape(8, 64) + w[512:576])
    h = torch.relu(h @ w[576:4672].reshape(64, 64) + w[4672:4736])
    e = h @ w[4736:4800] + w[4800] - t.double()
    loss = (torch.where(e < 0, UNDER, 1.0) * e * e).mean()
    loss.backward()
    g = w.grad
    m, v = (1 - BETA1) * g, (1 - BETA2) * g * g
    step = LR * (m / (1 - BETA1)) / (torch.sqrt(v / (1 - BETA2)) + EPS)
    return {"loss": loss.detach().reshape(1), "grad": g, "params": w.detach() - step, "m": m,
            "v": v}


def exact(case, seed):
    kind = case["kind"]
    if kind == "eval":
        return {"uv": _exact_words(_params(case, seed), _indices(case, seed), case["depth"])}
    if kind == "train":
        return _exact_train(case, seed)
    # images are whole numbers, compared value for value; where the words are
    # few enough the counts are made here too (a word on a pixel's edge may
    # fall to either side of it)
    if (kind == "render" and case["depth"] <= 14) or (kind == "scan" and case["depth"] <= 14):
        tiling = kind == "render" and case["tiling"]
        d = case["depth"]
        return {"image": _exact_image(_params(case, seed), range(1, d + 1) if tiling else [d]),
                "words": None}
    return None
