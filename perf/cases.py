"""The work that users of the registration library have it do, as timed cases.

A SLAM back end registers pairs of surface fragments, one at a time or a batch
of loop candidates at once; tools and tests run the stages on their own; a
training program steps through the robust objective or the refined pose. Sizes
are those of the repository's seeded configurations: 5,000-point object scenes,
150,000- and 200,000-point rooms, uneven batches of 10,000 to 120,000 points,
32 x 50,000-point objectives, maps of millions of surfels.

The fragments are made here, on the GPU, like the repository's generators make
theirs: furnished rooms on a 1 cm lattice snapped to a 1 cm voxel grid in each
fragment's own frame, 3 mm noise, a partial overlap along an oblique sweep;
or patches, spheres and boxes sampled by area.
"""
import ctypes
import math

import numpy as np
import torch

import paper_1801_01572_gb300 as lsr

DEV = "cuda:0"
R_NORMAL, R_FEATURE, EPS = 0.05, 0.125, 0.0375  # the library's default radii
LEVELS, ITERS = 3, 50                           # and refinement schedule
HYPOTHESES = 4_000_000                          # the paper's (and default) hypothesis count


# --------------------------------------------------------------------------- the cases
def listed():
    return [
        # a small object scan against another, as a tracker relocalises: many short launches
        dict(name="pair_objects_5k", kind="pair", scene="objects", n_p=5_000, n_q=5_000, overlap=0.7, precision="fp32"),
        # the headline registration: two room fragments with default parameters
        dict(name="pair_room_150k", kind="pair", scene="room", n_p=150_000, n_q=150_000, overlap=0.5, precision="fp32"),
        # the largest fragments of the repository, matched on the tensor cores
        dict(name="pair_room_200k_bf16", kind="pair", scene="room", n_p=200_000, n_q=200_000, overlap=0.5,
             precision="bf16"),
        # loop candidates of one keyframe, uneven sizes and overlaps, verified as a batch on concurrent streams
        dict(name="batch_rooms_8", kind="batch", pairs=8, n_lo=10_000, n_hi=120_000),
        # descriptors of one fragment for a place-recognition index: normals, SPFH, FPFH on device arrays
        dict(name="features_room_119999", kind="features", scene="room", n=119_999),
        # descriptor matching alone, exact on the FP32 cores, uneven sets
        dict(name="match_fp32_60k_90k", kind="match", n_p=60_001, n_q=90_000, precision="fp32"),
        # and on the tensor cores
        dict(name="match_bf16_40k", kind="match", n_p=40_000, n_q=40_001, precision="bf16"),
        # scoring of pose candidates that another module proposes
        dict(name="consensus_50k_256", kind="consensus", n_p=50_000, n_q=50_000, poses=256),
        # refinement of an odometry guess without a global search
        dict(name="refine_room_50k", kind="refine", n_p=50_000, n_q=50_000),
        # training through the refined pose: its gradient in the points
        dict(name="pose_grad_50k", kind="pose_grad", n_p=50_000, n_q=50_000),
        # training on the robust objective: forward and backward of a batch of pairs
        dict(name="objective_8x50k", kind="objective", pairs=8, n_p=50_000, n_q=50_000),
        # correction of a dense map after a loop closure
        dict(name="surfels_2m", kind="surfels", n=2_000_000, keyframes=300),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["pair", "pair", "batch", "features", "match", "consensus", "refine", "pose_grad", "objective",
                       "surfels"])
    if kind == "pair":
        if rng.random() < 0.3:
            return dict(kind="pair", scene="objects", n_p=_log_int(rng, 3_000, 8_000), n_q=_log_int(rng, 3_000, 8_000),
                        overlap=rng.uniform(0.6, 0.8), precision=rng.choice(["fp32", "bf16"]))
        return dict(kind="pair", scene="room", n_p=_log_int(rng, 20_000, 200_000), n_q=_log_int(rng, 20_000, 200_000),
                    overlap=rng.uniform(0.4, 0.8), precision=rng.choice(["fp32", "bf16"]))
    if kind == "batch":
        return dict(kind="batch", pairs=rng.randint(2, 8), n_lo=10_000, n_hi=_log_int(rng, 20_000, 120_000))
    if kind == "features":
        if rng.random() < 0.3:
            return dict(kind="features", scene="objects", n=_log_int(rng, 2_000, 20_000))
        return dict(kind="features", scene="room", n=_log_int(rng, 10_000, 200_000))
    if kind == "match":
        return dict(kind="match", n_p=_log_int(rng, 3_000, 90_000), n_q=_log_int(rng, 3_000, 90_000),
                    precision=rng.choice(["fp32", "bf16"]))
    if kind == "consensus":
        return dict(kind="consensus", n_p=_log_int(rng, 5_000, 60_000), n_q=_log_int(rng, 5_000, 60_000),
                    poses=_log_int(rng, 4, 512))
    if kind in ("refine", "pose_grad"):
        return dict(kind=kind, n_p=_log_int(rng, 5_000, 150_000), n_q=_log_int(rng, 5_000, 150_000))
    if kind == "objective":
        return dict(kind="objective", pairs=rng.randint(1, 16), n_p=_log_int(rng, 5_000, 60_000),
                    n_q=_log_int(rng, 5_000, 60_000))
    return dict(kind="surfels", n=_log_int(rng, 50_000, 4_000_000), keyframes=_log_int(rng, 20, 400))


def work(case):
    k = case["kind"]
    if k == "pair":
        return _pair_work(case["scene"], case["n_p"], case["n_q"], case["precision"])
    if k == "batch":
        mean = (case["n_lo"] + case["n_hi"]) // 2
        w = _pair_work("room", mean, mean, "bf16")
        return {x: case["pairs"] * w[x] for x in w}
    if k == "features":
        # xyz in; normal, curvature, count, SPFH, its count and FPFH out
        return {"bytes": case["n"] * (12 + 20 + 136 + 132), "flops": case["n"] * _feature_flops(case["scene"])}
    if k == "match":
        return {"bytes": 132 * (case["n_p"] + case["n_q"]) + 8 * case["n_p"],
                "flops": 66.0 * case["n_p"] * case["n_q"] if case["precision"] == "bf16" else 0.0}
    if k == "consensus":
        # a transform and at least one squared distance per point and pose
        return {"bytes": 12 * (case["n_p"] + case["n_q"]) + 60 * case["poses"],
                "flops": 26.0 * case["n_p"] * case["poses"]}
    if k == "refine":
        return {"bytes": 12 * (case["n_p"] + case["n_q"]), "flops": _refine_flops(case["n_p"])}
    if k == "pose_grad":
        return {"bytes": 24 * (case["n_p"] + case["n_q"]), "flops": 200.0 * case["n_p"]}
    if k == "objective":
        return {"bytes": case["pairs"] * 36 * (case["n_p"] + case["n_q"]), "flops": 160.0 * case["pairs"] * case["n_p"]}
    # position, normal and two stamps in; position, normal and keep flag out; ~20 keyframes tested per surfel
    return {"bytes": 57 * case["n"], "flops": 20.0 * 70 * case["n"]}


def _feature_flops(scene):
    k = 490 if scene == "room" else 60  # neighbours within 12.5 cm at the scenes' sampling
    return k * (30.0 + 66.0)            # half the pair features of 60 flop (each counts for both ends), 33 FMA


def _refine_flops(n):
    # a rigid transform, one distance and 17 weighted sums per point: ITERS steps over all points, and over a
    # quarter and a sixteenth of them on the coarser levels
    return 70.0 * ITERS * n * (1 + 1 / 4 + 1 / 16)


def _pair_work(scene, n_p, n_q, precision):
    flops = (n_p + n_q) * _feature_flops(scene) + 64.0 * HYPOTHESES + _refine_flops(n_p)
    if precision == "bf16":
        flops += 66.0 * n_p * n_q
    return {"bytes": 12 * (n_p + n_q) + 600, "flops": flops}


# --------------------------------------------------------------------------- what a program has in hand
_contexts = {}


def _context(**params):
    """The program's context for one set of parameters: one for its lifetime."""
    key = tuple(sorted(params.items()))
    if key not in _contexts:
        _contexts[key] = lsr.Context(0, **params)
    return _contexts[key]


_handle = None


def _abi():
    """A context of the C ABI, for the stages that a program runs on device arrays."""
    global _handle
    if _handle is None:
        _handle = ctypes.c_void_p()
        _ok(lsr.lib().lsr_create(ctypes.byref(_handle), None, 0, None))
    return _handle


def _ok(rc):
    if rc != 0:
        raise RuntimeError("lsr error %d" % rc)


def prepare(case, seed):
    state = {k: v for k, v in case.items() if k != "name"}
    rng = np.random.default_rng(seed)
    gen = torch.Generator(device=DEV).manual_seed(int(seed))
    k = case["kind"]
    if k == "pair":
        state["pair"] = _pair(case["scene"], case["n_p"], case["n_q"], case["overlap"], rng, gen)
        state["ctx"] = _context(**_precision(case["precision"]))
    elif k == "batch":
        sizes = rng.integers(case["n_lo"], case["n_hi"] + 1, (case["pairs"], 2))
        overlaps = rng.uniform(0.3, 0.8, case["pairs"])
        pairs = [_pair("room", int(a), int(b), float(o), rng, gen) for (a, b), o in zip(sizes, overlaps)]
        state["P"], state["Q"] = [p["P"] for p in pairs], [p["Q"] for p in pairs]
        state["vps"] = np.stack([np.concatenate([p["vpP"], p["vpQ"]]) for p in pairs]).astype(np.float32)
        # a deployment pins the streams and tile that the autotuner would time
        state["ctx"] = _context(batch_streams=4, **_precision("bf16"))
    elif k == "features":
        p = _pair(case["scene"], case["n"], 1_000, 0.5, rng, gen)
        state["P"], state["n"] = p["P"], case["n"]
        state["vp"] = (ctypes.c_float * 3)(*[float(x) for x in p["vpP"]])
        state["h"] = _abi()
    elif k == "match":
        p = _pair("room", case["n_p"], case["n_q"], 0.5, rng, gen)
        F = []
        for X, vp in ((p["P"], p["vpP"]), (p["Q"], p["vpQ"])):
            N = _normals(X.double(), vp)[0].float()
            F.append(_fpfh(X.double(), N.double())[2].float().contiguous())
        state["FP"], state["FQ"] = F
        state["mode"] = lsr.MATCH_BF16 if case["precision"] == "bf16" else lsr.MATCH_FP32
        state["ctx"] = _context(match_tile=1)
    elif k == "consensus":
        p = _pair("room", case["n_p"], case["n_q"], 0.6, rng, gen)
        state["P"], state["Q"] = p["P"], p["Q"]
        # proposals: a third within a few degrees and centimetres of the true pose, the others anywhere
        Rt = np.empty((case["poses"], 3, 4))
        for i in range(case["poses"]):
            T = _nudge(p["T"], rng, math.radians(4.0), 0.08) if i % 3 == 0 else _pose(rng) @ p["T"]
            Rt[i] = T[:3]
        state["Rt"] = torch.from_numpy(Rt.reshape(-1, 12).astype(np.float32)).to(DEV)
        state["ctx"] = _context()
    elif k == "refine":
        p = _pair("room", case["n_p"], case["n_q"], 0.6, rng, gen)
        state["P"], state["Q"] = p["P"], p["Q"]
        state["T"] = _nudge(p["T"], rng, math.radians(2.0), 0.03)
        state["ctx"] = _context()
    elif k == "pose_grad":
        p = _pair("room", case["n_p"], case["n_q"], 0.6, rng, gen)
        state["P"], state["Q"], state["T"] = p["P"], p["Q"], p["T"]
        state["G"] = rng.standard_normal((4, 4))  # the loss's gradient in the pose
        state["ctx"] = _context()
    elif k == "objective":
        clouds, T0, xi = [], [], []
        for _ in range(case["pairs"]):
            p = _pair("room", case["n_p"], case["n_q"], 0.5, rng, gen)
            clouds += [p["P"].requires_grad_(), p["Q"].requires_grad_()]
            T0.append(p["T"])
            xi.append(rng.standard_normal(6) * 2e-3)
        state["clouds"] = clouds
        state["T0"] = torch.from_numpy(np.stack(T0))
        state["xi"] = torch.from_numpy(np.stack(xi)).requires_grad_()
        state["w"] = torch.from_numpy(rng.uniform(0.5, 1.5, case["pairs"]))  # pair weights of the loss
        state["ctx"] = _context()
    else:
        _surfel_map(state, case["n"], case["keyframes"], rng, gen)
        state["ctx"] = _context()
    torch.cuda.synchronize()
    return state


def _precision(name):
    return dict(match_precision=lsr.MATCH_BF16, match_tile=1) if name == "bf16" else dict(match_precision=lsr.MATCH_FP32)


# --------------------------------------------------------------------------- one pass
def run(state):
    k = state["kind"]
    if k == "pair":
        p = state["pair"]
        return _registration(state["ctx"].register_pair(p["P"], p["Q"], p["vpP"], p["vpQ"]), len(p["P"]))
    if k == "batch":
        found = state["ctx"].register_batch(state["P"], state["Q"], state["vps"])
        return [_registration(r, len(P)) for r, P in zip(found, state["P"])]
    if k == "features":
        n, L, h, P, d = state["n"], lsr.lib(), state["h"], state["P"], state["P"].device
        N, curv = torch.empty((n, 3), device=d), torch.empty(n, device=d)
        S, F = torch.empty((n, 33), device=d), torch.empty((n, 33), device=d)
        near, used = torch.empty(n, dtype=torch.int32, device=d), torch.empty(n, dtype=torch.int32, device=d)
        _ok(L.lsr_stage_normals(h, P.data_ptr(), n, ctypes.cast(state["vp"], ctypes.c_void_p), R_NORMAL, N.data_ptr(),
                                near.data_ptr(), curv.data_ptr()))
        _ok(L.lsr_stage_spfh(h, P.data_ptr(), N.data_ptr(), n, R_FEATURE, S.data_ptr(), used.data_ptr()))
        _ok(L.lsr_stage_fpfh(h, P.data_ptr(), N.data_ptr(), S.data_ptr(), n, R_FEATURE, F.data_ptr()))
        return {"normals": N, "neighbours": near, "curvature": curv, "spfh": S, "pairs": used, "fpfh": F}
    if k == "match":
        nn, d1, _ = state["ctx"].stage_match(state["FP"], state["FQ"], state["mode"])
        return {"nn": nn, "d1": d1}
    if k == "consensus":
        count, sumd2 = state["ctx"].stage_consensus(state["P"], state["Q"], state["Rt"], EPS)
        return {"count": count, "sumd2": sumd2}
    if k == "refine":
        T, _ = state["ctx"].stage_refine(state["P"], state["Q"], state["T"], EPS, 1.0, LEVELS, ITERS)
        return _as_points(T)
    if k == "pose_grad":
        dP, dQ = torch.empty_like(state["P"]), torch.empty_like(state["Q"])
        _, _, g, H, lam, _ = state["ctx"].pose_implicit_grad(state["P"], state["Q"], state["T"], state["G"], EPS, None,
                                                             dP, dQ)
        return {"dP": dP, "dQ": dQ, "g": g, "H": H, "lambda": lam}
    if k == "objective":
        E = lsr.RobustAlignBatch.apply(state["xi"], state["T0"], EPS, EPS * EPS, state["ctx"], *state["clouds"])
        grads = torch.autograd.grad((E * state["w"]).sum(), [state["xi"], *state["clouds"]])
        return {"E": E.detach(), "dxi": grads[0], "dclouds": list(grads[1:])}
    s = state
    pos, nrm, keep, kept = s["ctx"].surfel_correct(s["pos"], s["nrm"], s["t0"], s["tu"], s["T_old"], s["T_new"],
                                                   s["t_kf"], s["cam"])
    return {"pos": pos, "nrm": nrm, "keep": keep, "kept": kept}


def _as_points(T):
    """A pose in the type of the points that it goes on to move."""
    return np.asarray(T, np.float32)


def _registration(r, n_p):
    """What a caller takes from a registration: the pose, the hypothesis behind it, how well it fits."""
    return {"T": _as_points(r.T), "T_hyp": _as_points(r.T_hyp), "status": r.status, "inlier_ratio": r.inliers / n_p,
            "fitness": r.fitness}


# --------------------------------------------------------------------------- inputs: poses and fragments
def _rotation(axis, angle):
    x, y, z = axis / np.linalg.norm(axis)
    K = np.array([[0, -z, y], [z, 0, -x], [-y, x, 0]])
    return np.eye(3) + math.sin(angle) * K + (1 - math.cos(angle)) * (K @ K)


def _pose(rng):
    """Any rotation, and a translation of up to a metre."""
    T = np.eye(4)
    q, r = np.linalg.qr(rng.standard_normal((3, 3)))
    q = q * np.sign(np.diag(r))
    T[:3, :3] = q if np.linalg.det(q) > 0 else -q
    d = rng.standard_normal(3)
    T[:3, 3] = d / np.linalg.norm(d) * rng.uniform() ** (1 / 3)
    return T


def _nudge(T, rng, angle, shift):
    D = np.eye(4)
    D[:3, :3] = _rotation(rng.standard_normal(3), angle * rng.uniform())
    d = rng.standard_normal(3)
    D[:3, 3] = d / np.linalg.norm(d) * shift * rng.uniform()
    out = T.copy()
    c = T[:3, 3] + T[:3, :3] @ np.array([2.0, 1.75, 0.75])  # about the scene's middle
    out[:3, :3] = D[:3, :3] @ T[:3, :3]
    out[:3, 3] = D[:3, :3] @ (T[:3, 3] - c) + c + D[:3, 3]
    return out


def _t(x):
    return torch.as_tensor(np.asarray(x, np.float64), device=DEV)


def _box(c, R, half):
    """Faces of a box as rectangles (centre, two axes, two half extents)."""
    for ax in range(3):
        a, b = (ax + 1) % 3, (ax + 2) % 3
        for s in (-1.0, 1.0):
            yield c + s * half[ax] * R[:, ax], R[:, a], R[:, b], half[a], half[b]


def _room(rng):
    """Floor, four walls and twenty boxes and cylinders: rectangles, cylinders (x, y, radius, height), the middle."""
    W, D, H = 4.0 * rng.uniform(0.85, 1.15), 3.5 * rng.uniform(0.85, 1.15), 1.5
    x, y, z = np.eye(3)
    rects = [(np.array([W / 2, D / 2, 0]), x, y, W / 2, D / 2), (np.array([W / 2, 0, H / 2]), x, z, W / 2, H / 2),
             (np.array([W / 2, D, H / 2]), x, z, W / 2, H / 2), (np.array([0, D / 2, H / 2]), y, z, D / 2, H / 2),
             (np.array([W, D / 2, H / 2]), y, z, D / 2, H / 2)]
    cyls = []
    for k in range(20):
        if k % 2:
            cyls.append((rng.uniform(0.4, W - 0.4), rng.uniform(0.4, D - 0.4), rng.uniform(0.1, 0.35),
                         rng.uniform(0.3, 1.4)))
            continue
        half = np.array([rng.uniform(0.2, 0.6), rng.uniform(0.15, 0.4), rng.uniform(0.2, 0.9)])
        c = np.array([rng.uniform(0.5, W - 0.5), rng.uniform(0.5, D - 0.5), half[2]])
        yaw = rng.uniform(0, 2 * math.pi)
        if k % 4 == 0:  # against a wall, some hung on it
            side = rng.integers(4)
            c[:2] = [(c[0], half[1]), (c[0], D - half[1]), (half[1], c[1]), (W - half[1], c[1])][side]
            yaw = 0.0 if side < 2 else math.pi / 2
            c[2] = half[2] if rng.uniform() < 0.6 else rng.uniform(0.8, 1.6)
        rects += list(_box(c, _rotation(z, yaw), half))
    return rects, cyls, np.array([W / 2, D / 2, 1.2])


def _lattice(rects, cyls, step, rng):
    out = []
    for c, a, b, h1, h2 in rects:
        u = torch.arange(-h1 + rng.uniform(0, step), h1, step, dtype=torch.float64, device=DEV)
        v = torch.arange(-h2 + rng.uniform(0, step), h2, step, dtype=torch.float64, device=DEV)
        out.append((_t(c) + u[:, None, None] * _t(a) + v[None, :, None] * _t(b)).reshape(-1, 3))
    for x, y, r, h in cyls:
        n = max(8, int(round(2 * math.pi * r / step)))
        th = (torch.arange(n, dtype=torch.float64, device=DEV) + rng.uniform()) * (2 * math.pi / n)
        z = torch.arange(rng.uniform(0, step), h, step, dtype=torch.float64, device=DEV)
        th, z = torch.meshgrid(th, z, indexing="ij")
        out.append(torch.stack([x + r * torch.cos(th), y + r * torch.sin(th), z], -1).reshape(-1, 3))
        u = torch.arange(-r + rng.uniform(0, step), r, step, dtype=torch.float64, device=DEV)
        u, v = torch.meshgrid(u, u, indexing="ij")
        top = torch.stack([x + u, y + v, torch.full_like(u, h)], -1).reshape(-1, 3)
        out.append(top[(u * u + v * v <= r * r).reshape(-1)])
    return torch.cat(out)


def _snap(X, step):
    """The centres of the occupied voxels of X."""
    k = torch.floor(X / step).long()
    lo = k.min(0).values
    ext = (k.max(0).values - lo + 1).tolist()
    k = k - lo
    key = torch.unique((k[:, 2] * ext[1] + k[:, 1]) * ext[0] + k[:, 0])
    k = torch.stack([key % ext[0], key // ext[0] % ext[1], key // (ext[0] * ext[1])], 1) + lo
    return (k.double() + 0.5) * step


def _moved(T, X):
    return X @ _t(T[:3, :3]).T + _t(T[:3, 3])


def _pair(scene, n_p, n_q, overlap, rng, gen):
    """Two fragments of one scene and the pose T that takes P into Q's frame."""
    T = _pose(rng)
    if scene == "objects":
        P, Q, vp = _objects_pair(n_p, n_q, overlap, T, rng, gen)
        sigma = 0.002
    else:
        rects, cyls, vp = _room(rng)
        ang = rng.integers(4) * math.pi / 2 + math.radians(rng.uniform(25.0, 65.0))
        d = _t([math.cos(ang), math.sin(ang), 0.0])
        P = _snap(_lattice(rects, cyls, 0.01, rng), 0.01)
        Q = _snap(_moved(T, _lattice(rects, cyls, 0.01, rng)), 0.01)
        back = np.linalg.inv(T)
        sP, iP = torch.sort(P @ d)
        sQ, iQ = torch.sort(_moved(back, Q) @ d)
        # P: n_p consecutive points along the sweep; Q: n_q from where the last overlap * n_p of them begin
        last = len(P) - max(n_p, int((1 - overlap) * n_p) + int(1.05 * n_q))
        if last < 0:
            raise ValueError("the room has too few points for %d and %d at overlap %.2f" % (n_p, n_q, overlap))
        i0 = int(rng.integers(0, last + 1))
        j0 = int(torch.searchsorted(sQ, sP[i0 + int((1 - overlap) * n_p)]))
        j0 = min(j0, len(Q) - n_q)
        P, Q = P[iP[i0:i0 + n_p]], Q[iQ[j0:j0 + n_q]]
        sigma = 0.003
    P, Q = (X[torch.randperm(len(X), generator=gen, device=DEV)] for X in (P, Q))
    P, Q = (X + sigma * torch.randn(X.shape, generator=gen, device=DEV, dtype=torch.float64) for X in (P, Q))
    return {"P": P.float().contiguous(), "Q": Q.float().contiguous(), "T": T, "vpP": vp.astype(np.float32),
            "vpQ": (T[:3, :3] @ vp + T[:3, 3]).astype(np.float32)}


def _objects_pair(n_p, n_q, overlap, T, rng, gen):
    """Six patches, three spheres and two boxes in a 2 m cube, sampled by area; a tenth of Q are outliers."""
    rects, balls = [], []
    for _ in range(6):
        R = _pose(rng)[:3, :3]
        rects.append((rng.uniform(-0.7, 0.7, 3), R[:, 0], R[:, 1], rng.uniform(0.2, 0.3), rng.uniform(0.2, 0.3)))
    for _ in range(3):
        balls.append((rng.uniform(-0.7, 0.7, 3), rng.uniform(0.12, 0.18)))
    for _ in range(2):
        rects += list(_box(rng.uniform(-0.6, 0.6, 3), _pose(rng)[:3, :3], rng.uniform(0.1, 0.15, 3)))
    area = np.array([4 * r[3] * r[4] for r in rects] + [4 * math.pi * b[1] ** 2 for b in balls])

    def sample(n):
        which = torch.multinomial(_t(area), n, True, generator=gen)
        uv = 2 * torch.rand((n, 2), generator=gen, device=DEV, dtype=torch.float64) - 1
        s = torch.randn((n, 3), generator=gen, device=DEV, dtype=torch.float64)
        s = s / s.norm(dim=1, keepdim=True)
        c = _t(np.array([r[0] for r in rects] + [b[0] for b in balls]))[which]
        a = _t(np.array([r[1] * r[3] for r in rects] + [np.zeros(3)] * len(balls)))[which]
        b = _t(np.array([r[2] * r[4] for r in rects] + [np.zeros(3)] * len(balls)))[which]
        rad = _t(np.array([0.0] * len(rects) + [x[1] for x in balls]))[which]
        return c + uv[:, :1] * a + uv[:, 1:] * b + rad[:, None] * s

    d = rng.standard_normal(3)
    d = _t(d / np.linalg.norm(d))
    P = sample(n_p)
    cut = torch.quantile(P @ d, 1.0 - overlap)
    Q = sample(int(4 * n_q / overlap))
    Q = _moved(T, Q[Q @ d >= cut][:n_q])
    lo, hi = Q.min(0).values, Q.max(0).values
    out = n_q // 10
    Q[:out] = lo + (hi - lo) * torch.rand((out, 3), generator=gen, device=DEV, dtype=torch.float64)
    return P, Q, np.array([0.0, -2.5, 1.0])


def _surfel_map(s, n, m, rng, gen):
    """Surfels of a room's surfaces and a loop of m keyframes whose corrected poses drift away along it."""
    W, D, H = 4.0, 3.5, 2.5
    u = torch.rand((n, 4), generator=gen, device=DEV, dtype=torch.float64)
    z = torch.zeros(n, dtype=torch.float64, device=DEV)
    x, y, h = u[:, 1] * W, u[:, 2] * D, u[:, 2] * H
    w = u[:, 0]
    pos = torch.where((w < 0.4)[:, None], torch.stack([x, y, z], 1), torch.stack([x, y, z + H], 1))
    for k, face in enumerate((torch.stack([x, z, h], 1), torch.stack([x, z + D, h], 1),
                              torch.stack([z, u[:, 1] * D, h], 1), torch.stack([z + W, u[:, 1] * D, h], 1))):
        on = (w >= 0.4 + 0.125 * k) & (w < 0.525 + 0.125 * k)
        pos = torch.where(on[:, None], face, pos)
    pos = pos + 0.003 * torch.randn((n, 3), generator=gen, device=DEV, dtype=torch.float64)
    nrm = torch.randn((n, 3), generator=gen, device=DEV, dtype=torch.float64)
    s["pos"], s["nrm"] = pos.float(), (nrm / nrm.norm(dim=1, keepdim=True)).float()
    s["t0"] = torch.randint(0, m, (n,), generator=gen, device=DEV).float() - 0.5
    s["tu"] = s["t0"] + torch.randint(2, 41, (n,), generator=gen, device=DEV).float()
    centre, axis = np.array([W / 2, D / 2, 1.4]), rng.standard_normal(3)
    s["T_old"], s["T_new"] = np.zeros((m, 4, 4)), np.zeros((m, 4, 4))
    for f in range(m):
        a = 2 * math.pi * f / m
        eye = centre + np.array([1.2 * math.cos(a), math.sin(a), 0.1 * math.sin(3 * a)])
        fwd = centre + np.array([-0.8 * math.cos(a + 0.3), -0.7 * math.sin(a + 0.3), -0.3]) - eye
        fwd /= np.linalg.norm(fwd)
        right = np.cross(fwd, [0.0, 0.0, 1.0])
        right /= np.linalg.norm(right)
        T = np.eye(4)
        T[:3, 0], T[:3, 1], T[:3, 2], T[:3, 3] = right, np.cross(fwd, right), fwd, eye
        C = np.eye(4)
        C[:3, :3] = _rotation(axis, math.radians(1.5) * f / max(m - 1, 1))
        C[:3, 3] = np.array([0.04, -0.03, 0.02]) * f / max(m - 1, 1)
        s["T_old"][f], s["T_new"][f] = T, C @ T
    s["t_kf"] = np.arange(m, dtype=np.float32)
    s["cam"] = np.array([525.0, 525.0, 319.5, 239.5, 640.0, 480.0, 4.0], np.float32)


# --------------------------------------------------------------------------- the same in 64 bits
def _f32(x):
    return float(np.float32(x))


def _near_pairs(X, r, chunk=4096):
    """(i, j, d2) of all ordered pairs within r, i == j included, a slab of i along the longest axis at a time."""
    ax = int((X.max(0).values - X.min(0).values).argmax())
    s, order = torch.sort(X[:, ax])
    Y, r2 = X[order], _f32(r) ** 2
    for a in range(0, len(X), chunk):
        b = min(len(X), a + chunk)
        lo = int(torch.searchsorted(s, s[a] - 1.001 * r))
        hi = int(torch.searchsorted(s, s[b - 1] + 1.001 * r, right=True))
        A, B = Y[a:b], Y[lo:hi]
        c = A.mean(0)
        A, B = A - c, B - c
        d2 = (A * A).sum(1)[:, None] + (B * B).sum(1)[None] - 2 * A @ B.T
        i, j = torch.nonzero(d2 <= r2 + 1e-9, as_tuple=True)
        e2 = ((A[i] - B[j]) ** 2).sum(1)
        keep = e2 <= r2
        i, j, e2 = i[keep], j[keep], e2[keep]
        yield order[a + i], order[lo + j], e2


def _sums(i, j, w, feat, out):
    """out[i] += w feat[j] over the pairs, as one product: the same order of sums on every run."""
    u, row = torch.unique(i, return_inverse=True)
    c, col = torch.unique(j, return_inverse=True)
    W = torch.zeros((len(u), len(c)), dtype=torch.float64, device=DEV)
    W[row, col] = w
    out[u] += W @ feat[c]


def _normals(X, vp):
    """Radius-PCA normals toward vp, curvature and neighbour count."""
    n = len(X)
    C = torch.zeros((n, 13), dtype=torch.float64, device=DEV)
    d = X - X.mean(0)
    feat = torch.cat([torch.ones((n, 1), dtype=torch.float64, device=DEV), d,
                      (d[:, :, None] * d[:, None, :]).reshape(n, 9)], 1)
    for i, j, d2 in _near_pairs(X, R_NORMAL):
        _sums(i, j, torch.ones_like(d2), feat, C)
    cnt, m, C = C[:, 0].round(), C[:, 1:4] / C[:, :1], C[:, 4:] / C[:, :1]
    w, V = torch.linalg.eigh((C - (m[:, :, None] * m[:, None, :]).reshape(n, 9)).reshape(n, 3, 3).cpu())
    w, V = w.to(DEV), V.to(DEV)
    N = V[:, :, 0]
    N = torch.where(((N * (_t(vp) - X)).sum(1) < 0)[:, None], -N, N)
    curv = w[:, 0].clamp(min=0) / w.sum(1).clamp(min=1e-300)
    bad = cnt < 3
    return torch.where(bad[:, None], torch.zeros_like(N), N), torch.where(bad, torch.full_like(curv, -1.0), curv)


def _fpfh(X, N):
    """SPFH, its pair counts and FPFH (Rusu et al. 2009) of points with normals (zero: invalid)."""
    n = len(X)
    valid = N.abs().sum(1) > 0
    H = torch.zeros(n * 33, dtype=torch.long, device=DEV)
    for i, j, d2 in _near_pairs(X, R_FEATURE):
        ok = (d2 > 0) & valid[i] & valid[j]
        i, j, d2 = i[ok], j[ok], d2[ok]
        e = (X[j] - X[i]) / d2.sqrt()[:, None]
        ni, nj = N[i], N[j]
        swap = ((ni * e).sum(1).abs() < (nj * e).sum(1).abs())[:, None]
        u, nt, e = torch.where(swap, nj, ni), torch.where(swap, ni, nj), torch.where(swap, -e, e)
        v = torch.linalg.cross(u, e)
        v2 = (v * v).sum(1)
        ok = v2 >= 1e-12
        i, u, nt, e, v = i[ok], u[ok], nt[ok], e[ok], v[ok] / v2[ok].sqrt()[:, None]
        w = torch.linalg.cross(u, v)
        th = torch.atan2((w * nt).sum(1), (u * nt).sum(1))
        for h, x in enumerate(((v * nt).sum(1), (u * e).sum(1), th / math.pi)):
            H.index_add_(0, i * 33 + 11 * h + ((x + 1) * 5.5).floor().clamp(0, 10).long(), torch.ones_like(i))
    H = H.reshape(n, 33)
    k = H[:, :11].sum(1)
    S = H.double() / k.clamp(min=1)[:, None]
    F, near = torch.zeros((n, 33), dtype=torch.float64, device=DEV), torch.zeros(n, dtype=torch.long, device=DEV)
    for i, j, d2 in _near_pairs(X, R_FEATURE):
        ok = (d2 > 0) & valid[i] & valid[j]
        i, j, d2 = i[ok], j[ok], d2[ok]
        _sums(i, j, d2.rsqrt(), S, F)
        near += torch.bincount(i, minlength=n)
    F = torch.where(valid[:, None], S + F / near.clamp(min=1)[:, None], torch.zeros_like(F))
    g = F.reshape(n, 3, 11).sum(2, keepdim=True)
    F = torch.where(g > 0, F.reshape(n, 3, 11) / g.clamp(min=1e-300), torch.zeros_like(g)).reshape(n, 33)
    return S, k, F


def _nearest(X, Q, chunk=2048):
    """Squared distance and index of the nearest Q row of every X row."""
    d, nn = [], []
    c = Q.mean(0)
    Q = Q - c
    q2 = (Q * Q).sum(1)
    for x in torch.split(X - c, chunk):
        j = (q2[None] - 2 * x @ Q.T).min(1).indices
        d.append(((x - Q[j]) ** 2).sum(1))
        nn.append(j)
    return torch.cat(d), torch.cat(nn)


def _refined(P, Q, T):
    """The graduated refinement: Geman-McClure weights on the nearest neighbours, three radii, every s-th point first."""
    T = _t(T).clone()
    for level in range(LEVELS):
        up = LEVELS - 1 - level
        r = _f32(EPS) * 2 ** up
        mu = r * r
        p, q = (X[::max(1, min(4 ** up, len(X) // 4096))].double() for X in (P, Q))
        c = T[:3, :3] @ p.mean(0) + T[:3, 3]
        for _ in range(ITERS):
            x = p @ T[:3, :3].T + T[:3, 3]
            d2, nn = _nearest(x, q)
            near = d2 < mu
            x, e, w = x[near] - c, x[near] - q[nn[near]], (mu / (mu + d2[near])) ** 2
            J = torch.zeros((len(x), 3, 6), dtype=torch.float64, device=DEV)
            J[:, 0, 1], J[:, 0, 2], J[:, 1, 0] = x[:, 2], -x[:, 1], -x[:, 2]
            J[:, 1, 2], J[:, 2, 0], J[:, 2, 1] = x[:, 0], x[:, 1], -x[:, 0]
            J[:, :, 3:] = torch.eye(3, dtype=torch.float64, device=DEV)
            A = torch.einsum("nia,n,nib->ab", J, w, J)
            delta = -torch.linalg.solve(A, torch.einsum("nia,n,ni->a", J, w, e))
            D = torch.eye(4, dtype=torch.float64, device=DEV)
            D[:3, :3] = torch.linalg.matrix_exp(_skew(delta[:3]))
            D[:3, 3] = c - D[:3, :3] @ c + delta[3:]
            c = c + (w[:, None] * x).sum(0) / w.sum()
            T = D @ T
            if float(delta.norm()) < 1e-6:
                break
    return T


def _skew(w):
    o = torch.zeros((), dtype=w.dtype, device=w.device)
    return torch.stack([torch.stack([o, -w[2], w[1]]), torch.stack([w[2], o, -w[0]]), torch.stack([-w[1], w[0], o])])


def _energy(p, q, xi, T, mu):
    """Pair terms rho(|Exp(xi) T p - q|^2), twice differentiable at xi = 0 too."""
    K = _skew(xi[:3])
    M = torch.linalg.matrix_exp(K)
    z = (p @ T[:3, :3].T + T[:3, 3]) @ M.T + xi[3:]
    s = ((z - q) ** 2).sum(1)
    return mu * s / (mu + s)


def exact(case, seed):
    k = case["kind"]
    if k in ("pair", "batch"):
        return None  # millions of hypotheses against every point: minutes in 64 bits
    s = prepare(case, seed)
    if k == "features":
        X = s["P"].double()
        N, curv = _normals(X, np.array(s["vp"], np.float64))
        S, _, F = _fpfh(X, N)
        return {"normals": N, "neighbours": None, "curvature": curv, "spfh": S, "pairs": None, "fpfh": F}
    if k == "match":
        return {"nn": None, "d1": _nearest(s["FP"].double(), s["FQ"].double())[0]}
    if k == "consensus":
        out, e2 = [], _f32(EPS) ** 2
        for Rt in s["Rt"].double().reshape(-1, 3, 4):
            x = s["P"].double() @ Rt[:, :3].T + Rt[:, 3]
            d2, _ = _nearest(x, s["Q"].double())
            out.append(torch.where(d2 < e2, d2, torch.zeros_like(d2)).sum())
        return {"count": None, "sumd2": torch.stack(out)}
    if k == "refine":
        return _refined(s["P"], s["Q"], s["T"])
    mu = _f32(EPS * EPS)
    if k == "pose_grad":
        P, Q, T, G = s["P"].double(), s["Q"].double(), _t(s["T"]), _t(s["G"])
        d2, nn = _nearest(P @ T[:3, :3].T + T[:3, 3], Q)
        held = torch.nonzero(d2 < _f32(EPS) ** 2).reshape(-1)
        p, q = P[held].requires_grad_(), Q[nn[held]].requires_grad_()
        xi = torch.zeros(6, dtype=torch.float64, device=DEV, requires_grad=True)
        g = torch.autograd.grad(_energy(p, q, xi, T, mu).sum(), xi, create_graph=True)[0]
        H = torch.stack([torch.autograd.grad(g[i], xi, retain_graph=True)[0] for i in range(6)])
        y = torch.zeros(6, dtype=torch.float64, device=DEV, requires_grad=True)
        D = torch.eye(4, dtype=torch.float64, device=DEV)[:3]
        moved = torch.cat([D[:, :3] + _skew(y[:3]), y[3:, None]], 1) @ T
        dl = torch.autograd.grad((moved * G[:3]).sum(), y)[0]
        lam = torch.linalg.solve(H, dl)
        dp, dq = torch.autograd.grad((g * lam).sum(), [p, q])
        dP, dQ = torch.zeros_like(P), torch.zeros_like(Q)
        dP[held] = -dp
        dQ.index_add_(0, nn[held], -dq)
        return {"dP": dP, "dQ": dQ, "g": g.detach(), "H": H, "lambda": lam}
    if k == "objective":
        E, dxi, dclouds = [], [], []
        e2 = _f32(EPS) ** 2
        for i in range(case["pairs"]):
            P, Q = (X.detach().double() for X in s["clouds"][2 * i:2 * i + 2])
            xi, T = s["xi"][i].detach().to(DEV).requires_grad_(), s["T0"][i].to(DEV)
            z = (P @ T[:3, :3].T + T[:3, 3]) @ torch.linalg.matrix_exp(_skew(xi.detach()[:3])).T + xi.detach()[3:]
            d2, nn = _nearest(z, Q)
            held = torch.nonzero(d2 < e2).reshape(-1)
            p, q = P[held].requires_grad_(), Q[nn[held]].requires_grad_()
            e = (_energy(p, q, xi, T, mu) - mu * e2 / (mu + e2)).sum()
            gx, gp, gq = torch.autograd.grad(e * s["w"][i].to(DEV), [xi, p, q])
            dP, dQ = torch.zeros_like(P), torch.zeros_like(Q)
            dP[held] = gp
            dQ.index_add_(0, nn[held], gq)
            E.append(e.detach())
            dxi.append(gx)
            dclouds += [dP, dQ]
        return {"E": torch.stack(E), "dxi": torch.stack(dxi), "dclouds": dclouds}
    return _surfels_exact(s)


def _surfels_exact(s):
    pos, nrm, t0, tu = (s[x].double() for x in ("pos", "nrm", "t0", "tu"))
    fx, fy, cx, cy, w, h, far = (float(x) for x in s["cam"])
    n = len(pos)
    sp, sn = torch.zeros_like(pos), torch.zeros_like(pos)
    cnt = torch.zeros(n, dtype=torch.float64, device=DEV)
    for f in range(len(s["t_kf"])):
        t = float(s["t_kf"][f])
        A = np.linalg.inv(s["T_old"][f])
        M = s["T_new"][f] @ A
        c = _moved(A, pos)
        u, v = fx * c[:, 0] / c[:, 2] + cx, fy * c[:, 1] / c[:, 2] + cy
        see = (t > t0) & (t < tu) & (c[:, 2] > 0) & (c[:, 2] <= far) & (u >= 0) & (u < w) & (v >= 0) & (v < h)
        see = see.double()[:, None]
        sp += see * _moved(M, pos)
        sn += see * (nrm @ _t(M[:3, :3]).T)
        cnt += see[:, 0]
    kept = (cnt > 0)[:, None]
    return {"pos": torch.where(kept, sp / cnt.clamp(min=1)[:, None], pos),
            "nrm": torch.where(kept, sn / sn.norm(dim=1, keepdim=True).clamp(min=1e-300), nrm), "keep": None,
            "kept": None}
