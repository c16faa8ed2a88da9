"""Performance cases: the work that a user of this framework has it do, through its public entry points.

A case is a dict of plain values; its "kind" names the entry point:

  chain        Pipeline.run: preprocess, registration, rotation fit, remap, ROI cross-correlation, F solve
  register     hrebsd_demons_register_batch on preprocessed patterns
  preprocess   hrebsd_preprocess_batch
  filters      the real-scan preprocessing of Pipeline: mean pattern, background division, band-pass
  second_pass  hrebsd_fit_rotation, hrebsd_remap, hrebsd_xcf_roi_batch, hrebsd_solve_F on a field in hand
  cnn_infer    hrebsd_cnn_infer_patterns
  cnn_train    eight hrebsd_cnn_train_step calls, then the weights and gradients read back

Patterns are kinematic Kikuchi patterns (25 FCC bands on a quadratic background, Poisson counts) of
random orientations, test patterns rotated by a misorientation drawn per pair and slightly strained.
"""
import itertools
import math

import numpy as np
import torch

import paper_1907_05993_gb300 as P
from paper_1907_05993_gb300.pipeline import Pipeline, PipelineConfig

F32, F64, I32 = torch.float32, torch.float64, torch.int32
PC = (0.5, 0.5, 0.6)          # pattern centre and detector distance, in pattern widths / heights
STOP = (1e-4, 5)              # the workloads' stop rule: relative SSD decrease over 5 iterations
CNN_LAYERS = (("e1a", 2, 16), ("e1b", 16, 16), ("e2a", 16, 32), ("e2b", 32, 32), ("e3a", 32, 64), ("e3b", 64, 64),
              ("ba", 64, 128), ("bb", 128, 128), ("d3a", 192, 64), ("d3b", 64, 64), ("d2a", 96, 32), ("d2b", 32, 32),
              ("d1a", 48, 16), ("d1b", 16, 16))
CNN_MFLOP = 9 * 2e-6 * (64 * 64 * (2 * 16 + 16 * 16 + 48 * 16 + 16 * 16) + 32 * 32 * (16 * 32 + 3 * 32 * 32 + 2 * 32 * 32) +
                        16 * 16 * (32 * 64 + 64 * 64 + 192 * 64 + 64 * 64) + 8 * 8 * (64 * 128 + 128 * 128))
TRAIN_STEPS, TRAIN_LR = 8, 5e-5   # the step size near the end of the training schedule


# ------------------------------------------------------------------ the cases
def listed():
    return [
        # a whole map: 100 x 100 points, 4 grains, uneven iteration counts (the repository's headline workload)
        dict(name="scan_256", kind="chain", n=10_000, refs=4, H=256, W=256, levels=4, cap=100, stop=True, S=64, rois=5,
             mis_lo=0.0, mis_hi=6.0, counts=500),
        # one pattern pair while the user waits (latency; launches count)
        dict(name="single_pair_128", kind="chain", n=1, refs=1, H=128, W=128, levels=3, cap=50, stop=False, S=32,
             rois=5, mis_lo=2.0, mis_hi=2.0, counts=500),
        # targets of a training set: every pair has a reference of its own
        dict(name="register_own_refs_128", kind="register", n=2048, refs=2048, H=128, W=128, levels=3, cap=100,
             stop=True, init=False, mis_lo=0.0, mis_hi=12.0, counts=500),
        # the paper's detector and settings: 1244 x 1024, 7 levels of 20 iterations
        dict(name="register_1244x1024", kind="register", n=16, refs=4, H=1024, W=1244, levels=7, cap=20, stop=False,
             init=False, mis_lo=0.0, mis_hi=6.0, counts=500),
        # a detector binned to a size that is no power of two
        dict(name="register_92x100", kind="register", n=150, refs=2, H=100, W=92, levels=3, cap=60, stop=True,
             init=False, mis_lo=0.0, mis_hi=3.0, counts=500),
        # started from a field at 64 x 64 with low caps at the fine levels, as after the learned initialiser
        dict(name="register_from_init_256", kind="register", n=2000, refs=8, H=256, W=256, levels=4, cap=25, stop=True,
             init=True, mis_lo=0.0, mis_hi=12.0, counts=500),
        # background fit, division and normalisation of a batch
        dict(name="preprocess_256", kind="preprocess", n=4096, H=256, W=256, counts=500),
        # experimental patterns: static and dynamic background, then a band-pass
        dict(name="filters_256", kind="filters", n=1000, H=256, W=256, dynamic=12.0, lp=0.7, hp=20.0, counts=200),
        # the second pass of a quarter of the map, 25 ROIs of 64 x 64
        dict(name="second_pass_256", kind="second_pass", n=2500, refs=4, H=256, W=256, S=64, rois=5, mis_lo=0.0,
             mis_hi=6.0, counts=500),
        # the second pass at the paper's scale, 100 ROIs of 256 x 256
        dict(name="second_pass_1244x1024", kind="second_pass", n=16, refs=4, H=1024, W=1244, S=256, rois=10,
             mis_lo=0.0, mis_hi=6.0, counts=500),
        # the learned initialiser's prediction for a batch of patterns
        dict(name="cnn_infer_256", kind="cnn_infer", n=4096, refs=8, H=256, W=256, mis_lo=0.0, mis_hi=12.0, counts=500),
        # training of the learned initialiser: eight batches, then the weights are read back for a checkpoint
        dict(name="cnn_train_256", kind="cnn_train", n=256, mis_lo=0.0, mis_hi=12.0, counts=500),
    ]


def _log_int(rng, lo, hi):
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    kind = rng.choice(["chain", "chain", "register", "register", "register", "preprocess", "filters", "second_pass",
                       "second_pass", "cnn_infer", "cnn_train"])
    counts = rng.randint(200, 500)
    mis = dict(mis_lo=0.0, mis_hi=round(rng.uniform(1.0, 12.0), 2))
    if kind == "chain":
        H = rng.choice([128, 256])
        return dict(kind=kind, n=_log_int(rng, 1, 4000 if H == 256 else 10_000), refs=rng.randint(1, 8), H=H, W=H,
                    levels=3 if H == 128 else 4, cap=rng.randint(20, 100), stop=rng.random() < 0.7, S=H // 4, rois=5,
                    counts=counts, **mis)
    if kind == "register":
        form = rng.choice(["square", "odd", "odd", "paper"])
        if form == "square":
            H = W = rng.choice([64, 128, 256])
            n, levels = _log_int(rng, 1, 2048), int(math.log2(H)) - 4
        elif form == "odd":
            H, W = rng.randint(64, 300), rng.randint(64, 300)
            n, levels = _log_int(rng, 1, 500), 3 if min(H, W) < 128 else 4
        else:
            H, W, n, levels = rng.randint(480, 1024), rng.randint(480, 1244), rng.randint(1, 16), 5
        refs = n if n <= 2048 and rng.random() < 0.3 else min(n, rng.randint(1, 8))
        return dict(kind=kind, n=n, refs=refs, H=H, W=W, levels=levels, cap=rng.randint(10, 60),
                    stop=rng.random() < 0.6, init=H == 256 and W == 256 and rng.random() < 0.5, counts=counts, **mis)
    if kind == "preprocess":
        H, W = rng.choice([(64, 64), (128, 128), (256, 256), (100, 92), (480, 640), (1024, 1244)])
        return dict(kind=kind, n=_log_int(rng, 1, 268_000_000 // (H * W)), H=H, W=W, counts=counts)
    if kind == "filters":
        H, W = rng.choice([(128, 128), (256, 256), (100, 92), (480, 640)])
        return dict(kind=kind, n=_log_int(rng, 1, 65_000_000 // (H * W)), H=H, W=W,
                    dynamic=round(rng.uniform(5.0, 20.0), 2), lp=round(rng.uniform(0.5, 1.5), 2),
                    hp=round(rng.uniform(8.0, 30.0), 2), counts=counts)
    if kind == "second_pass":
        S = rng.choice([32, 64, 64, 128, 256])
        H, W = {32: (128, 128), 64: (256, 256), 128: (1024, 1024), 256: (1024, 1244)}[S]
        return dict(kind=kind, n=_log_int(rng, 1, {32: 2500, 64: 2500, 128: 24, 256: 16}[S]), refs=rng.randint(1, 8),
                    H=H, W=W, S=S, rois=10 if S == 256 else 5, counts=counts, **mis)
    if kind == "cnn_infer":
        H = rng.choice([64, 128, 256])
        return dict(kind=kind, n=_log_int(rng, 1, 4096), refs=rng.randint(1, 8), H=H, W=H, counts=counts, **mis)
    return dict(kind=kind, n=_log_int(rng, 16, 256), counts=counts, **mis)


# ------------------------------------------------------------------ inputs
def _planes():
    """The 25 planes of {111}, {200}, {220}, {311}, one of each +- pair."""
    out = []
    for fam in ((1, 1, 1), (2, 0, 0), (2, 2, 0), (3, 1, 1)):
        for p in sorted(set(itertools.permutations(fam))):
            for s in itertools.product((1, -1), repeat=3):
                v = tuple(a * b for a, b in zip(p, s))
                if v > (0, 0, 0) and v not in out:
                    out.append(v)
    return np.array(out, dtype=np.float64)


def _rotations(axis, angle):
    """Rodrigues' formula for axes [n, 3] (any length) and angles [n]."""
    a = axis / np.linalg.norm(axis, axis=1, keepdims=True)
    K = np.zeros((len(a), 3, 3))
    K[:, 0, 1], K[:, 0, 2], K[:, 1, 2] = -a[:, 2], a[:, 1], -a[:, 0]
    K -= K.transpose(0, 2, 1)
    s, c = np.sin(angle)[:, None, None], np.cos(angle)[:, None, None]
    return np.eye(3) + s * K + (1 - c) * (K @ K)


def _render(g, F, H, W, counts, gen):
    """Patterns [n, H, W] of the orientations g [n, 3, 3] deformed by F [n, 3, 3]."""
    hkl = _planes()
    G = np.einsum("nba,nbc,pc->npa", np.linalg.inv(F), g, hkl / 3.6)
    gn = np.linalg.norm(G, axis=2)
    lam = 12.2643 / math.sqrt(20e3 * (1 + 0.978476e-6 * 20e3))
    tab = lambda a: torch.from_numpy(a.astype(np.float32)).cuda()
    normal, theta_b, amp = tab(G / gn[..., None]), tab(np.arcsin(lam * gn / 2)), 3.0 / np.sum(hkl * hkl, axis=1)
    x = (torch.arange(W, device="cuda", dtype=F32) + 0.5 - PC[0] * W)[None, :].expand(H, W)
    y = (torch.arange(H, device="cuda", dtype=F32) + 0.5 - PC[1] * H)[:, None].expand(H, W)
    d = torch.stack([x, y, torch.full((H, W), PC[2] * W, device="cuda")], -1).reshape(-1, 3)
    d = (d / d.norm(dim=1, keepdim=True)).T.contiguous()
    xd, yd = x / W * 2, y / H * 2
    bg = (1.0 - 0.3 * (xd * xd + yd * yd) + 0.05 * yd).reshape(-1)
    out = torch.empty((len(g), H, W), device="cuda", dtype=F32)
    step = max(1, (1 << 26) // (H * W))
    for a in range(0, len(g), step):
        nm, tb = normal[a:a + step], theta_b[a:a + step]
        bands = torch.zeros((len(nm), H * W), device="cuda")
        for p in range(len(hkl)):
            th = torch.asin((nm[:, p] @ d).clamp_(-1, 1)) / tb[:, p, None]
            bands += float(amp[p]) * torch.exp(-0.5 * th * th)
        img = bg * (1 + 0.5 * bands)
        img *= counts / img.mean(dim=1, keepdim=True)
        out[a:a + step] = torch.poisson(img, generator=gen).view(-1, H, W)
    return out


def _pairs(case, seed, H, W):
    """refs [R, H, W], tests [n, H, W], ref_idx [n], the deformations [n, 3, 3]."""
    rng, gen = np.random.default_rng(seed), torch.Generator("cuda").manual_seed(seed)
    n, R = case["n"], case.get("refs", case["n"])
    g = _rotations(rng.normal(size=(R, 3)), rng.uniform(0, math.pi, R))
    idx = np.arange(n) * R // n
    Rm = _rotations(rng.normal(size=(n, 3)), np.radians(rng.uniform(case["mis_lo"], case["mis_hi"], n)))
    E = rng.normal(size=(n, 3, 3)) * 5e-4
    F = Rm @ (np.eye(3) + 0.5 * (E + E.transpose(0, 2, 1)))
    refs = _render(g, np.tile(np.eye(3), (R, 1, 1)), H, W, case["counts"], gen)
    tests = _render(g[idx], F, H, W, case["counts"], gen)
    return refs, tests, torch.from_numpy(idx.astype(np.int32)).cuda(), F


def _normalised(x):
    """In place: zero mean, unit variance, the background's quadric divided out as rendered."""
    n, H, W = x.shape
    xd = (torch.arange(W, device="cuda", dtype=F32) + 0.5) / W * 2 - 1
    yd = (torch.arange(H, device="cuda", dtype=F32) + 0.5) / H * 2 - 1
    x /= 1.0 - 0.3 * (xd[None, :] ** 2 + yd[:, None] ** 2) + 0.05 * yd[:, None]
    for a in range(0, n, 256):
        v = x[a:a + 256]
        v -= v.mean(dim=(1, 2), keepdim=True)
        v /= v.std(dim=(1, 2), keepdim=True)
    return x


def _rotation_field(F, H, W, noise, gen):
    """The field [n, 2, H, W] of pairs deformed by F (test point = F reference point), with smooth noise."""
    n = len(F)
    Fi = torch.from_numpy(np.linalg.inv(F).astype(np.float32)).cuda()
    x = (torch.arange(W, device="cuda", dtype=F32) + 0.5 - PC[0] * W)[None, None, :]
    y = (torch.arange(H, device="cuda", dtype=F32) + 0.5 - PC[1] * H)[None, :, None]
    zs = PC[2] * W
    out = torch.empty((n, 2, H, W), device="cuda", dtype=F32)
    for a in range(0, n, 256):
        f = Fi[a:a + 256, :, :, None, None]
        v = [f[:, i, 0] * x + f[:, i, 1] * y + f[:, i, 2] * zs for i in range(3)]
        out[a:a + 256, 0] = x - zs * v[0] / v[2]
        out[a:a + 256, 1] = y - zs * v[1] / v[2]
        low = torch.randn((len(v[0]), 2, 9, 9), device="cuda", generator=gen) * noise
        out[a:a + 256] += torch.nn.functional.interpolate(low, size=(H, W), mode="bicubic", align_corners=False)
    return out


def _rois(case):
    """An even grid of rois x rois ROI centres with every ROI inside the pattern."""
    S, k = case["S"], case["rois"]
    inset = S // 2 if k == 10 else S // 2 + S // 4
    xs = np.rint(np.linspace(inset, case["W"] - inset, k)).astype(np.int32)
    ys = np.rint(np.linspace(inset, case["H"] - inset, k)).astype(np.int32)
    return np.array([(x, y) for y in ys for x in xs], dtype=np.int32)


class _Ctx:
    """A library handle, given back with its state."""

    def __init__(self):
        self.h = P.hrebsd_create(torch.cuda.current_device())

    def __del__(self):
        if self.h is not None:
            P.hrebsd_destroy(self.h)
            self.h = None


def _caps(case):
    """Iteration caps per level (finest first); started from a field, the levels coarser than it are skipped."""
    c = case["cap"]
    return [c, c, max(1, 2 * c // 5)] + [0] * (case["levels"] - 3) if case.get("init") else [c] * case["levels"]


def _cnn_vector(seed):
    """He-normal weights with small biases in the library's layout: per layer [co][9][ci padded to 16], then [co]."""
    rng, out = np.random.default_rng(seed), []
    for _, ci, co in CNN_LAYERS:
        w = np.zeros((co, 9, (ci + 15) // 16 * 16))
        w[:, :, :ci] = rng.normal(0, math.sqrt(2 / (9 * ci)), (co, 9, ci))
        out += [w.ravel(), rng.normal(0, 0.02, co)]
    out += [rng.normal(0, 0.25, 32), rng.normal(0, 0.02, 2)]
    return np.concatenate(out).astype(np.float32)


def _cnn_train_inputs(case, seed):
    """(inputs [8, n, 2, 64, 64] bf16, targets, weights, Adam moments as in the middle of a training)."""
    n = case["n"]
    gen, rng = torch.Generator("cuda").manual_seed(seed + 1), np.random.default_rng(seed + 1)
    refs, tests, _, F = _pairs(dict(case, n=n * TRAIN_STEPS, refs=n * TRAIN_STEPS), seed, 64, 64)
    x = torch.stack([_normalised(refs), _normalised(tests)], 1).to(torch.bfloat16)
    y = _rotation_field(F, 64, 64, 0.05, gen)
    vec = _cnn_vector(seed)
    used = vec != 0
    m = (rng.normal(0, 0.03, vec.size) * used).astype(np.float32)
    v = (rng.uniform(0.03, 0.3, vec.size) * used).astype(np.float32)
    return x.view(TRAIN_STEPS, n, 2, 64, 64), y.view(TRAIN_STEPS, n, 2, 64, 64), vec, m, v


def _inputs(case, seed):
    """The tensors of a case, from the seed alone."""
    kind = case["kind"]
    if kind == "cnn_train":
        return dict(zip(("x", "y", "vec", "m", "v"), _cnn_train_inputs(case, seed)))
    if kind in ("preprocess", "filters"):
        c = dict(case, mis_lo=0.0, mis_hi=12.0, refs=min(case["n"], 16))
        _, tests, _, _ = _pairs(c, seed, case["H"], case["W"])
        return dict(x=tests)
    refs, tests, idx, F = _pairs(case, seed, case["H"], case["W"])
    if kind == "chain":
        return dict(refs=refs, tests=tests, idx=idx)
    s = dict(refs=_normalised(refs), tests=_normalised(tests), idx=idx)
    gen = torch.Generator("cuda").manual_seed(seed + 1)
    if kind == "second_pass":
        s["field"] = _rotation_field(F, case["H"], case["W"], 0.1, gen)
    elif kind == "cnn_infer":
        s["vec"] = _cnn_vector(seed)
    elif case["init"]:
        s["init"] = _rotation_field(F, case["H"] // 4, case["W"] // 4, 0.2, gen)
    return s


def prepare(case, seed):
    s = _inputs(case, seed)
    s["case"], kind = case, case["kind"]
    dev = lambda shape, dtype: torch.empty(shape, dtype=dtype, device="cuda")
    n, H, W = case["n"], case.get("H"), case.get("W")
    if kind == "chain":
        tol, window = STOP if case["stop"] else (0.0, 0)
        s["pipe"] = Pipeline(PipelineConfig(H, W, _rois(case), case["S"], case["levels"], tuple(_caps(case)), 1.0, 1.0,
                                            tol, window, *PC))
        s["out"] = {}
        return s
    s["ctx"] = _Ctx()
    s["geom"] = P.hrebsd_geometry(*PC)
    if kind == "register":
        tol, window = STOP if case["stop"] else (0.0, 0)
        s["params"] = P.demons_params(case["levels"], _caps(case), 1.0, 1.0, 1.0, tol, window,
                                      2 if case["init"] else -1)
        s["out"] = dict(field=dev((n, 2, H, W), F32), iters=dev((n, case["levels"]), I32), status=dev((n,), I32))
    elif kind == "preprocess":
        s["out"] = dict(x=dev((n, H, W), F32))
    elif kind == "filters":
        s["out"] = dict(mean=dev((H, W), F32), flat=dev((n, H, W), F32), x=dev((n, H, W), F32))
    elif kind == "second_pass":
        s["roi"] = torch.from_numpy(_rois(case)).cuda()
        N = len(s["roi"])
        s["out"] = dict(F_first=dev((n, 9), F64), R_finite=dev((n, 9), F64), remapped=dev((n, H, W), F32),
                        q=dev((n, N, 2), F32), peak=dev((n, N, 2), I32), ph=dev((n, N), F32),
                        near_tie=dev((n, N), I32), F=dev((n, 9), F64), status=torch.zeros(n, dtype=I32, device="cuda"))
    elif kind == "cnn_infer":
        P.hrebsd_cnn_init(s["ctx"].h, s["vec"])
        s["out"] = dict(field=dev((n, 2, 64, 64), F32))
    else:
        P.hrebsd_cnn_init(s["ctx"].h, s["vec"])
        P.hrebsd_cnn_set_state(s["ctx"].h, s["m"], s["v"], 1000)
        s["out"] = dict(loss=torch.zeros(TRAIN_STEPS, device="cuda"))
    return s


# ------------------------------------------------------------------ one pass
def run(s):
    c, o = s["case"], s["out"]
    kind, n, H, W = c["kind"], c["n"], c.get("H"), c.get("W")
    if kind == "chain":
        return s["pipe"].run(s["refs"], s["tests"], s["idx"], out=o)
    ctx = s["ctx"].h
    if kind == "register":
        P.hrebsd_demons_register_batch(ctx, s["refs"], s["tests"], s["idx"], c["refs"], n, H, W, s["params"],
                                       s.get("init"), o["field"], o["iters"], o["status"])
    elif kind == "preprocess":
        P.hrebsd_preprocess_batch(ctx, s["x"], n, H, W, True, o["x"])
    elif kind == "filters":
        P.hrebsd_mean_pattern(ctx, s["x"], n, H, W, o["mean"])
        P.hrebsd_background_batch(ctx, s["x"], n, H, W, o["mean"], c["dynamic"], o["flat"])
        P.hrebsd_bandpass_batch(ctx, o["flat"], n, H, W, c["lp"], c["hp"], o["x"])
    elif kind == "second_pass":
        N, geom, roi = len(s["roi"]), s["geom"], s["roi"]
        P.hrebsd_fit_rotation(ctx, s["field"], n, H, W, roi, N, geom, o["F_first"], o["R_finite"], o["status"])
        P.hrebsd_remap(ctx, s["refs"], s["idx"], o["R_finite"], n, H, W, geom, o["remapped"])
        P.hrebsd_xcf_roi_batch(ctx, o["remapped"], s["tests"], n, H, W, roi, N, c["S"], True, o["q"], o["peak"],
                               o["ph"], o["near_tie"])
        P.hrebsd_solve_F(ctx, o["q"], roi, N, n, H, W, geom, o["R_finite"], o["F"], o["status"])
    elif kind == "cnn_infer":
        P.hrebsd_cnn_infer_patterns(ctx, s["refs"], s["tests"], s["idx"], n, H, W, o["field"])
    else:
        for k in range(TRAIN_STEPS):
            P.hrebsd_cnn_train_step(ctx, s["x"][k], s["y"][k], n, TRAIN_LR, o["loss"][k:k + 1])
        params, grads = P.hrebsd_cnn_get_params(ctx)
        return dict(loss=o["loss"], params=params, grads=grads)
    return o


# ------------------------------------------------------------------ what a pass cannot do without
def _demons_work(c):
    """Floating-point operations: per pixel and iteration four 7-tap passes over two components (112), the warp and
    the force (40); with the stop rule at least its window plus one iteration per level (at most the cap)."""
    its = [min(k, STOP[1] + 1) if c["stop"] else k for k in _caps(c)]
    return sum(152.0 * k * c["n"] * (c["H"] >> l) * (c["W"] >> l) for l, k in enumerate(its))


def _xcf_work(c):
    """Per ROI one complex forward and one inverse 2-D FFT of size S and about 20 S^2 around them."""
    S = c["S"]
    return c["n"] * c["rois"] ** 2 * (2 * 5 * S * S * math.log2(S * S) + 20 * S * S)


def work(case):
    kind, n = case["kind"], case["n"]
    if kind == "cnn_train":
        return dict(bytes=TRAIN_STEPS * n * 64 * 64 * (4 + 8) + 2 * 4 * _cnn_vector(0).size,
                    flops=TRAIN_STEPS * n * 3 * CNN_MFLOP * 1e6)
    px = case["H"] * case["W"]
    images = 4.0 * px * (n + case.get("refs", 0))
    if kind == "chain":
        # in: patterns; out: preprocessed patterns, field, remapped references (the ROI results are small)
        return dict(bytes=2 * images + 12.0 * n * px, flops=_demons_work(case) + _xcf_work(case))
    if kind == "register":
        return dict(bytes=images + 8.0 * n * px, flops=_demons_work(case))
    if kind == "preprocess":
        return dict(bytes=2 * images, flops=40.0 * n * px)
    if kind == "filters":
        # in: patterns; out: mean, corrected patterns, band-passed patterns; three separable blurs
        taps = sum(2 * math.ceil(3 * case[k]) + 1 for k in ("dynamic", "lp", "hp"))
        return dict(bytes=3 * images, flops=4.0 * taps * n * px)
    if kind == "second_pass":
        return dict(bytes=images + 4.0 * n * px, flops=_xcf_work(case) + 50.0 * n * px)
    return dict(bytes=images + 8.0 * n * 64 * 64, flops=n * CNN_MFLOP * 1e6)


# ------------------------------------------------------------------ the same in 64 bits (plain torch)
def _x_preprocess(x):
    n, H, W = x.shape
    xd = (torch.arange(W, device="cuda", dtype=F64) + 0.5) / W * 2 - 1
    yd = (torch.arange(H, device="cuda", dtype=F64) + 0.5) / H * 2 - 1
    X, Y = xd[None, :].expand(H, W), yd[:, None].expand(H, W)
    A = torch.stack([torch.ones_like(X), X, Y, X * X, X * Y, Y * Y]).reshape(6, -1)
    out = torch.empty((n, H, W), device="cuda", dtype=F64)
    for a in range(0, n, 256):
        v = x[a:a + 256].double().reshape(-1, H * W)
        v = v / (torch.linalg.solve(A @ A.T, A @ v.T).T @ A)
        v = v - v.mean(dim=1, keepdim=True)
        out[a:a + 256] = (v / v.square().mean(dim=1, keepdim=True).sqrt()).view(-1, H, W)
    return out


def _x_blur(x, sigma):
    """Separable Gaussian of radius ceil(3 sigma) over the last two axes, replicated borders."""
    r = math.ceil(3 * sigma)
    t = np.exp(-np.arange(-r, r + 1) ** 2 / (2.0 * sigma * sigma))
    t /= t.sum()
    for dim in (-1, -2):
        n = x.shape[dim]
        edge = lambda i: x.narrow(dim, i, 1).expand(*[r if d == x.dim() + dim else -1 for d in range(x.dim())])
        p = torch.cat([edge(0), x, edge(n - 1)], dim)
        x = sum(float(t[k]) * p.narrow(dim, k, n) for k in range(2 * r + 1))
    return x


def _x_bilinear(img, x, y):
    """Samples of img [n, ..., h, w] at index coordinates [n, ...] clamped to the image."""
    n, h, w = img.shape
    x, y = x.clamp(0, w - 1), y.clamp(0, h - 1)
    x0, y0 = x.floor().clamp(max=w - 2), y.floor().clamp(max=h - 2)
    fx, fy = x - x0, y - y0
    at = (y0 * w + x0).long().reshape(n, -1)
    flat = img.reshape(n, -1)
    g = lambda k: flat.gather(1, at + k).reshape(x.shape)
    return (1 - fy) * ((1 - fx) * g(0) + fx * g(1)) + fy * ((1 - fx) * g(w) + fx * g(w + 1))


def _x_gradient(f):
    g = []
    for dim in (2, 1):
        n = f.shape[dim]
        at = lambda i: f.narrow(dim, i, 1)
        inner = 0.5 * (f.narrow(dim, 2, n - 2) - f.narrow(dim, 0, n - 2))
        g.append(torch.cat([at(1) - at(0), inner, at(n - 1) - at(n - 2)], dim))
    return g


def _x_level(F, M, u, cap, stop):
    n, h, w = F.shape
    gx, gy = _x_gradient(F)
    X = torch.arange(w, device="cuda", dtype=F64)[None, None, :]
    Y = torch.arange(h, device="cuda", dtype=F64)[None, :, None]
    act, E = torch.arange(n, device="cuda"), []
    for k in range(cap):
        whole = len(act) == n
        ua, Fa, Ma, gxa, gya = (u, F, M, gx, gy) if whole else (u[act], F[act], M[act], gx[act], gy[act])
        d = _x_bilinear(Ma, X - ua[:, 0], Y - ua[:, 1]) - Fa
        E.append(torch.full((n,), math.inf, device="cuda", dtype=F64))
        E[k][act] = d.square().sum(dim=(1, 2))
        den = gxa * gxa + gya * gya + d * d
        t = torch.where(den > 1e-9, d / den, 0.0)
        new = _x_blur(ua + _x_blur(torch.stack([t * gxa, t * gya], 1), 1.0), 1.0)
        if stop and k >= STOP[1]:
            go = (E[k - STOP[1]][act] - E[k][act]) >= STOP[0] * E[k - STOP[1]][act]
            act, new = act[go], new[go]
            whole = len(act) == n
        u = new if whole else u.index_copy(0, act, new)
        if not len(act):
            break
    return u


def _x_register(refs, tests, idx, case, init):
    """The field [n, 2, H, W] in 64 bits, some pairs at a time."""
    H, W, caps, L = case["H"], case["W"], _caps(case), case["levels"]
    half = lambda v: torch.nn.functional.avg_pool2d(v[:, None], 2)[:, 0]
    out = torch.empty((len(tests), 2, H, W), device="cuda", dtype=F64)
    step = max(1, (1 << 25) // (H * W))
    for a in range(0, len(tests), step):
        Fp, Mp = [tests[a:a + step].double()], [refs[idx[a:a + step].long()].double()]
        for l in range(1, L):
            Fp.append(half(Fp[-1]))
            Mp.append(half(Mp[-1]))
        top = 2 if init is not None else L - 1
        u = init[a:a + step].double() if init is not None else torch.zeros((len(Fp[0]), 2, H >> top, W >> top),
                                                                           device="cuda", dtype=F64)
        for l in range(top, -1, -1):
            u = _x_level(Fp[l], Mp[l], u, caps[l], case["stop"])
            if l:
                h, w = H >> (l - 1), W >> (l - 1)
                X = ((torch.arange(w, device="cuda", dtype=F64) + 0.5) / 2 - 0.5)[None, None, :].expand(len(u), h, w)
                Y = ((torch.arange(h, device="cuda", dtype=F64) + 0.5) / 2 - 0.5)[None, :, None].expand(len(u), h, w)
                u = torch.stack([2 * _x_bilinear(u[:, i], X, Y) for i in range(2)], 1)
        out[a:a + step] = u
    return out


def _x_fit(r, t, H, W):
    """F [n, 3, 3] with det F = 1 minimising |Z* F r / (F r)_3 - r'|^2 over point pairs r, t [n, N, 2]."""
    pc, zs = torch.tensor([PC[0] * W, PC[1] * H], device="cuda", dtype=F64), PC[2] * W
    r, t = r - pc, t - pc
    r = torch.cat([r, torch.full_like(r[..., :1], zs)], -1)
    n = len(r)
    F = torch.eye(3, device="cuda", dtype=F64).repeat(n, 1, 1)
    for _ in range(12):
        v = torch.einsum("nab,nib->nia", F, r)
        res = zs * v[..., :2] / v[..., 2:] - t
        J = torch.zeros((n, r.shape[1], 2, 9), device="cuda", dtype=F64)
        for a in range(2):
            J[:, :, a, 3 * a:3 * a + 3] = zs * r / v[..., 2:]
            J[:, :, a, 6:] = -zs * v[..., a:a + 1] * r / v[..., 2:] ** 2
        J = J[..., :8].reshape(n, -1, 8)
        step = torch.linalg.solve(J.mT @ J, -(J.mT @ res.reshape(n, -1, 1)))[..., 0]
        F = (F.reshape(n, 9) + torch.nn.functional.pad(step, (0, 1))).view(n, 3, 3)
    d = torch.linalg.det(F)
    return F / (d.abs() ** (1 / 3) * d.sign())[:, None, None]


def _x_remap(refs, idx, R, H, W):
    """Keys cubic samples of the references at the projection of R^T r'."""
    out = torch.empty((len(idx), H, W), device="cuda", dtype=F64)
    X = (torch.arange(W, device="cuda", dtype=F64) + 0.5 - PC[0] * W)[None, None, :]
    Y = (torch.arange(H, device="cuda", dtype=F64) + 0.5 - PC[1] * H)[None, :, None]
    zs = PC[2] * W
    near = lambda s: 1.5 * s ** 3 - 2.5 * s ** 2 + 1
    far = lambda s: -0.5 * s ** 3 + 2.5 * s ** 2 - 4 * s + 2
    step = max(1, (1 << 24) // (H * W))
    for a in range(0, len(idx), step):
        Ra, img = R[a:a + step, :, :, None, None], refs[idx[a:a + step].long()].double().reshape(-1, H * W)
        v = [Ra[:, 0, i] * X + Ra[:, 1, i] * Y + Ra[:, 2, i] * zs for i in range(3)]
        x, y = PC[0] * W + zs * v[0] / v[2] - 0.5, PC[1] * H + zs * v[1] / v[2] - 0.5
        x0, y0 = x.floor(), y.floor()
        wts = lambda f: (far(1 + f), near(f), near(1 - f), far(2 - f))
        wx, wy = wts(x - x0), wts(y - y0)
        acc = 0.0
        for m in range(4):
            row = (y0 + m - 1).clamp(0, H - 1) * W
            for k in range(4):
                at = (row + (x0 + k - 1).clamp(0, W - 1)).long().reshape(len(img), -1)
                acc = acc + wy[m] * wx[k] * img.gather(1, at).view(x.shape)
        out[a:a + step] = acc
    return out


def _x_xcf(rem, tests, roi, S):
    """Shifts [n, N, 2] and peak heights [n, N] of the windowed ROIs' circular cross-correlation."""
    win = torch.from_numpy(np.hanning(S)).cuda()
    n, N = len(tests), len(roi)
    q, ph = torch.empty((n, N, 2), device="cuda", dtype=F64), torch.empty((n, N), device="cuda", dtype=F64)
    for i, (cx, cy) in enumerate(roi.tolist()):
        cut = lambda v: v[:, cy - S // 2:cy + S // 2, cx - S // 2:cx + S // 2].double()
        a, b = cut(rem), cut(tests)
        a, b = ((v - v.mean(dim=(1, 2), keepdim=True)) * win[:, None] * win for v in (a, b))
        c = torch.fft.ifft2(torch.fft.fft2(b) * torch.fft.fft2(a).conj()).real
        c0, at = c.reshape(n, -1).max(dim=1)
        py, px = at // S, at % S
        g = lambda dy, dx: c[torch.arange(n, device="cuda"), (py + dy) % S, (px + dx) % S]
        sub = lambda lo, hi: (lo - hi) / (2 * (lo - 2 * c0 + hi))
        wrap = lambda p: torch.where(p >= S // 2, p - S, p)
        q[:, i, 0] = wrap(px) + sub(g(0, -1), g(0, 1))
        q[:, i, 1] = wrap(py) + sub(g(-1, 0), g(1, 0))
        ph[:, i] = c0 / (a.square().sum(dim=(1, 2)) * b.square().sum(dim=(1, 2))).sqrt()
    return q, ph


def _x_second_pass(refs, tests, idx, field, case):
    n, H, W = case["n"], case["H"], case["W"]
    roi = torch.from_numpy(_rois(case)).cuda()
    c = roi.double()[None].expand(n, -1, 2)
    at = (c[..., 0] - 0.5, c[..., 1] - 0.5)
    u = torch.stack([_x_bilinear(field[:, i].double(), *at) for i in range(2)], -1)
    F1 = _x_fit(c - u, c, H, W)
    U, _, Vh = torch.linalg.svd(F1)
    R = U @ Vh
    rem = _x_remap(refs, idx, R, H, W)
    q, ph = _x_xcf(rem, tests, roi, case["S"])
    F = _x_fit(c, c + q, H, W) @ R
    return dict(F_first=F1.view(n, 9), R_finite=R.view(n, 9), remapped=rem, q=q, peak=None, ph=ph, near_tie=None,
                F=F.view(n, 9), status=None)


def _x_network(vec, x):
    """The U-Net on x [n, 2, 64, 64] in 64 bits, differentiable in the parameter vector."""
    p, at = {}, 0
    for name, ci, co in CNN_LAYERS:
        pad = (ci + 15) // 16 * 16
        w = vec[at:at + co * 9 * pad].view(co, 9, pad)[:, :, :ci]
        at += co * 9 * pad
        p[name] = (w.permute(0, 2, 1).reshape(co, ci, 3, 3), vec[at:at + co])
        at += co
    fn = torch.nn.functional

    def conv(name, v):   # nine shifted products: cuDNN has no fast 64-bit convolution
        w, b = p[name]
        n, ci, h, k = v.shape
        q = fn.pad(v, (1, 1, 1, 1))
        cols = torch.cat([q[:, :, i:i + h, j:j + k].reshape(n, ci, h * k) for i in range(3) for j in range(3)], 1)
        y = w.permute(0, 2, 3, 1).reshape(w.shape[0], -1) @ cols
        return torch.relu(y.view(n, -1, h, k) + b[None, :, None, None])

    pool = lambda v: fn.max_pool2d(v, 2)
    up = lambda v: fn.interpolate(v, scale_factor=2, mode="nearest")
    e1 = conv("e1b", conv("e1a", x))
    e2 = conv("e2b", conv("e2a", pool(e1)))
    e3 = conv("e3b", conv("e3a", pool(e2)))
    d3 = conv("d3b", conv("d3a", torch.cat([up(conv("bb", conv("ba", pool(e3)))), e3], 1)))
    d2 = conv("d2b", conv("d2a", torch.cat([up(d3), e2], 1)))
    d1 = conv("d1b", conv("d1a", torch.cat([up(d2), e1], 1)))
    return torch.einsum("oc,nchw->nohw", vec[at:at + 32].view(2, 16), d1) + vec[at + 32:at + 34][None, :, None, None]


def _x_train(s):
    vec, m, v = (torch.from_numpy(s[k]).cuda().double() for k in ("vec", "m", "v"))
    losses = []
    for k in range(TRAIN_STEPS):
        grad, loss, n = torch.zeros_like(vec), 0.0, s["x"].shape[1]
        for a in range(0, n, 64):
            w = vec.clone().requires_grad_(True)
            d = _x_network(w, s["x"][k, a:a + 64].double()) - s["y"][k, a:a + 64].double()
            part = d.square().sum() / (n * 2 * 64 * 64)
            part.backward()
            grad, loss = grad + w.grad, loss + part.item()
        losses.append(loss)
        t = 1001 + k
        m, v = 0.9 * m + 0.1 * grad, 0.999 * v + 0.001 * grad * grad
        vec = vec - TRAIN_LR * (m / (1 - 0.9 ** t)) / ((v / (1 - 0.999 ** t)).sqrt() + 1e-8)
    return dict(loss=torch.tensor(losses, dtype=F64), params=vec, grads=grad)


def exact(case, seed):
    kind, n = case["kind"], case["n"]
    if kind in ("chain", "register") and 1.0 * n * case["H"] * case["W"] * case["cap"] > 1.5e10:
        return None   # minutes in 64 bits
    s = _inputs(case, seed)
    with torch.no_grad():
        if kind == "preprocess":
            return dict(x=_x_preprocess(s["x"]))
        if kind == "filters":
            mean = s["x"].double().mean(dim=0)
            out = dict(mean=mean, flat=torch.empty(s["x"].shape, device="cuda", dtype=F64),
                       x=torch.empty(s["x"].shape, device="cuda", dtype=F64))
            step = max(1, (1 << 24) // (case["H"] * case["W"]))
            for a in range(0, n, step):
                v = s["x"][a:a + step].double()
                v = torch.where(mean.abs() >= 1e-12, v / mean, 0.0)
                b = _x_blur(v, case["dynamic"])
                v = torch.where(b.abs() >= 1e-12, v / b, 0.0)
                out["flat"][a:a + step] = v
                out["x"][a:a + step] = _x_blur(v, case["lp"]) - _x_blur(v, case["hp"])
            return out
        if kind == "second_pass":
            return _x_second_pass(s["refs"], s["tests"], s["idx"], s["field"], case)
        if kind == "register":
            return dict(field=_x_register(s["refs"], s["tests"], s["idx"], case, s.get("init")), iters=None, status=None)
        if kind == "chain":
            refs, tests = _x_preprocess(s["refs"]), _x_preprocess(s["tests"])
            field = _x_register(refs, tests, s["idx"], case, None)
            return dict(_x_second_pass(refs, tests, s["idx"], field, case), ref_pre=refs, test_pre=tests, field=field,
                        iters=None)
        if kind == "cnn_infer":
            vec, f = torch.from_numpy(s["vec"]).cuda().double(), case["H"] // 64
            out = torch.empty((n, 2, 64, 64), device="cuda", dtype=F64)
            small = lambda v: torch.nn.functional.avg_pool2d(v.double()[:, None], f)
            for a in range(0, n, 128):
                x = torch.cat([small(s["refs"][s["idx"][a:a + 128].long()]), small(s["tests"][a:a + 128])], 1)
                out[a:a + 128] = _x_network(vec, x)
            return dict(field=out)
    return _x_train(s)
