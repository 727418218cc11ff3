"""Performance cases of the RPBA library: the calls a user's program makes,
through the public binding (paper_1910_08138_gb300.rpba), at the sizes of the
repository's benchmark blocks and below.

Four kinds of case:

* "adjust": the library's main path on a block whose context exists: set the
  initial poses and points, the first intersection, and a number of outer
  iterations (rpba_set_cameras, rpba_set_points, rpba_intersect, rpba_iterate),
  then read the poses, the points and their active flags back. Blocks: an
  aerial grid (nadir, or nadir and oblique views), many independent blocks in
  one context, and a ring of cameras around an object with per-camera
  intrinsics. Forms: the library's defaults (all FP64, FP64 Cholesky), and the
  FP32 bulk form with the automatic or the direct solver. The default form
  starts from rough initial values and runs the default number of LM
  iterations; the FP32 form takes an outer iteration of an already adjusted
  block (initial values good to a few millimetres), one LM iteration as in
  bench.py's step, or a few on the smallest block.
* "covariance": the covariances of all points of a block.
* "train": loss and gradient of the learned preconditioner's network.
* "sigma0": sigma_0 and RMS of a block in caller-owned device memory.

Inputs are synthetic, from the seed alone (synth.py's generators for the
blocks). `exact` evaluates the same calls in 64 bits with plain torch and
numpy, without the library.
"""

from __future__ import annotations

import math

import numpy as np
import torch

from paper_1910_08138_gb300 import rpba, synth

# ---------------------------------------------------------------------------
# cases
# ---------------------------------------------------------------------------


def _adjust(name, rig, form, nx, ny, points, per_point, subs, outer, **more):
    case = dict(name=name, kind="adjust", rig=rig, form=form, nx=nx, ny=ny, points=points, per_point=per_point,
                subs=subs, outer=outer, oblique=0, spacing=4.0, noise=0.5, outliers=0.02, weighted=False,
                start=1.0 if form == "default" else 0.02, inner=20 if form == "default" else 1)
    case.update(more)
    return case


def listed():
    return [
        # a small survey in the default form: 50 cameras, 8k observations; the
        # call is bound by the latency of its chain of small launches
        _adjust("default_50", "grid", "default", 10, 5, 2000, 4, 2, 2),
        # a mid-sized survey in the default form: 1,000 cameras, 600k observations
        _adjust("default_1000", "grid", "default", 25, 40, 100_000, 6, 8, 1, oblique=30),
        # the small survey in the FP32 form: the smallest adjustment
        _adjust("chosen_50", "grid", "chosen", 10, 5, 2000, 4, 2, 1, oblique=30, inner=4),
        # the mid-sized survey in the FP32 form, block-Jacobi PCG
        _adjust("chosen_1000", "grid", "chosen", 25, 40, 100_000, 6, 8, 1, oblique=30),
        # a wide-baseline block of 10,000 cameras, 2M observations, 64 sub-blocks
        _adjust("chosen_10000", "grid", "chosen", 100, 100, 400_000, 5, 64, 1, oblique=45, spacing=8.0, noise=1.0,
                outliers=0.05),
        # a nadir survey with weighted observations and the direct solver
        # (weakly connected sub-blocks, on which CG takes many steps)
        _adjust("direct_4900", "grid", "direct", 70, 70, 150_001, 5, 32, 1, spacing=15.0, outliers=0.05, oblique=30,
                weighted=True),
        # many independent blocks of 20 to 400 cameras in one context
        _adjust("blocks_32", "blocks", "chosen", 32, 1, 60_000, 5, 4, 1, oblique=30),
        # a photo collection with focal length and radial parameter per camera,
        # direct solver
        _adjust("ring_961", "ring", "direct", 961, 1, 20_000, 18, 12, 1, noise=1.0),
        # the covariances of all points, for quality reports and as weights
        dict(name="covariance_100k", kind="covariance", nx=25, ny=40, points=100_000, per_point=6, subs=8,
             oblique=30, spacing=4.0, noise=0.5, outliers=0.02, weighted=False),
        # one training pass of the preconditioner's network over 40 systems
        dict(name="train_40", kind="train", systems=40, cams=60, probes=4),
        # the smallest call: sigma_0 of a small block held by the caller
        dict(name="sigma0_8k", kind="sigma0", cams=50, points=2000, obs=8000, weighted=True),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    pick = rng.choice(["default", "chosen", "chosen", "wide", "direct", "blocks", "ring", "covariance", "train",
                       "sigma0"])
    if pick in ("default", "chosen", "wide", "direct"):
        cams = _log_int(rng, 40, {"default": 700, "chosen": 1200, "wide": 8000, "direct": 4000}[pick])
        nx = max(5, int(round(math.sqrt(cams) * rng.uniform(0.7, 1.2))))
        ny = max(5, cams // nx)
        per_cam = rng.uniform(35, 100) if pick != "wide" else rng.uniform(20, 45)
        default = pick == "default"
        return _drop_name(_adjust("", "grid", "chosen" if pick == "wide" else pick, nx, ny,
                                  int(nx * ny * per_cam) | 1, rng.randint(4, 7),
                                  max(1, min(64, nx * ny // rng.randint(40, 160))),
                                  rng.randint(1, 3) if default else 1, oblique=rng.choice([0, 30] if default else [30, 45]),
                                  spacing=rng.choice([4.0, 6.0, 10.0]), noise=rng.choice([0.5, 1.0]),
                                  outliers=rng.choice([0.0, 0.02, 0.05]), weighted=rng.random() < 0.3,
                                  inner=20 if default else rng.choice([1, 2, 4]) if nx * ny < 200 else 1))
    if pick == "blocks":
        n = rng.randint(4, 32)
        return _drop_name(_adjust("", "blocks", "chosen", n, 1, n * rng.randint(700, 1900), rng.randint(4, 6),
                                  rng.randint(2, 6), 1, oblique=30))
    if pick == "ring":
        cams = _log_int(rng, 60, 960)
        return _drop_name(_adjust("", "ring", "direct", cams, 1,
                                  cams * rng.randint(12, 21), rng.randint(8, 18), max(1, cams // 80), 1, noise=1.0))
    if pick == "covariance":
        cams = _log_int(rng, 60, 1000)
        nx = max(6, int(math.sqrt(cams)))
        ny = max(6, cams // nx)
        return dict(kind="covariance", nx=nx, ny=ny, points=nx * ny * rng.randint(20, 99) | 1,
                    per_point=rng.randint(3, 7), subs=max(1, nx * ny // 125), oblique=rng.choice([0, 30]),
                    spacing=4.0, noise=0.5, outliers=0.02, weighted=rng.random() < 0.5)
    if pick == "train":
        return dict(kind="train", systems=rng.randint(2, 40), cams=rng.randint(8, 60), probes=rng.randint(1, 4))
    cams = _log_int(rng, 10, 500)
    points = cams * rng.randint(20, 100)
    return dict(kind="sigma0", cams=cams, points=points, obs=points * rng.randint(3, 6) | 1,
                weighted=rng.random() < 0.5)


def _drop_name(case):
    del case["name"]
    return case


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------


def _cells(nx, ny, subs):
    """Sub-block of every camera of an nx x ny grid: `subs` rectangular cells."""
    cx = max(c for c in range(1, subs + 1) if subs % c == 0 and c <= max(1, math.sqrt(subs * nx / ny) + 0.5))
    cy = subs // cx
    cx, cy = min(cx, nx), min(cy, ny)
    ix, iy = np.meshgrid(np.arange(nx), np.arange(ny), indexing="ij")
    return ((ix * cx // nx) * cy + iy * cy // ny).reshape(-1).astype(np.int32)


def _grid(rng, case, nx, ny, points):
    far = case.get("start", 1.0)
    blk = synth.grid_block(rng, nx, ny, case["spacing"], 30.0, points, case["per_point"], case["noise"],
                           case["outliers"], oblique_deg=float(case["oblique"]),
                           nadir_every=5 if case["oblique"] else 1, rot_sigma=0.01 * far, pos_sigma=0.1 * far,
                           pt_sigma=0.1 * far)
    blk["cam_subblock"] = _cells(nx, ny, case["subs"])
    return blk


def _problem(case, seed):
    rng = np.random.Generator(np.random.PCG64(seed))
    rig = case.get("rig", "grid")
    if rig == "grid":
        prob = _grid(rng, case, case["nx"], case["ny"], case["points"])
    elif rig == "blocks":  # case["nx"] blocks, sizes spread over 20 to 400 cameras
        sizes = np.exp(np.linspace(math.log(20.0), math.log(400.0), case["nx"]))
        per_cam = case["points"] / sizes.sum()
        members = []
        for size in sizes:
            side = int(math.sqrt(size))
            ny = int(size) // side
            members.append(_grid(rng, case, side, ny, int(side * ny * per_cam) + 8))
        prob = synth.merge_blocks(members)
    else:
        prob = synth.ring_block(rng, case["nx"], case["points"], float(case["per_point"]), case["subs"],
                                sigma_px=case["noise"], outlier_frac=case["outliers"], f_sigma_rel=0.01 * case["start"],
                                rot_sigma=0.002 * case["start"], pos_sigma=0.03 * case["start"],
                                pt_sigma=0.03 * case["start"])
    if case["weighted"]:  # C^-1 of every observation: anisotropic, about one
        K = prob["obs_cam"].size
        a, c = rng.uniform(0.5, 2.0, K), rng.uniform(0.5, 2.0, K)
        b = rng.uniform(-0.4, 0.4, K) * np.sqrt(a * c)
        prob["obs_winv"] = np.stack([a, b, c], axis=1)
    return prob


def _options(case):
    options = dict(robust=1, robust_from_start=1)
    if case["form"] != "default":
        options.update(precision=1, solver=2 if case["form"] == "direct" else 4, max_inner=case["inner"])
    return options


def _pinned(array):
    t = torch.empty(array.shape, dtype=torch.from_numpy(array[:0]).dtype, pin_memory=True)
    out = t.numpy()
    out[...] = array
    return out


def _systems(case, seed):
    """SPD matrices with the block structure of a reduced camera system and
    their probe vectors: cameras on a strip, every point couples up to four
    neighbouring cameras."""
    rng = np.random.Generator(np.random.PCG64(seed))
    out = []
    for s in range(case["systems"]):
        n = max(4, case["cams"] - (7 * s) % max(1, case["cams"] // 2))
        scale = np.repeat(np.exp(rng.uniform(0.0, 4.0, n)), 6) * rng.uniform(0.5, 2.0, 6 * n)
        pts = 8 * n
        first = rng.integers(0, n, pts)
        rows = np.zeros((pts, 3, n, 6))
        for off in (0, 1, 2, 3):
            cam = first + off
            hit = np.nonzero((cam < n) & ((off < 2) | (rng.random(pts) < 0.5)))[0]
            rows[hit, :, cam[hit], :] = rng.normal(size=(hit.size, 3, 6))
        G = rows.reshape(3 * pts, 6 * n) * np.sqrt(scale)
        S = G.T @ G
        S += np.diag(1e-2 * np.diag(S) + 1e-3 * np.diag(S).mean())
        out.append((S, rng.normal(size=(case["probes"], 6 * n))))
    return out


def _network_weights(seed):
    rng = np.random.Generator(np.random.PCG64(seed + 1))
    return (0.1 * rng.normal(size=rpba.gnn_param_count())).astype(np.float32)


def _sigma0_arrays(case, seed):
    rng = np.random.Generator(np.random.PCG64(seed))
    M, N, K = case["cams"], case["points"], case["obs"]
    q, _ = np.linalg.qr(np.eye(3) + 0.05 * rng.normal(size=(M, 3, 3)))
    R = q * np.sign(np.einsum("mii->mi", q))[:, None, :]
    t = np.stack([rng.normal(0, 2, M), rng.normal(0, 2, M), rng.uniform(25, 35, M)], axis=1)
    intr = np.tile([1000.0, 1000.0, 750.0], (M, 1))
    X = rng.normal(0, 3, (N, 3))
    cam, pt = rng.integers(0, M, K), rng.integers(0, N, K)
    xc = np.einsum("kab,kb->ka", R[cam], X[pt]) + t[cam]
    xy = 1000.0 * xc[:, :2] / xc[:, 2:] + intr[cam, 1:] + rng.normal(0, 0.5, (K, 2))
    a, c = rng.uniform(0.5, 2.0, K), rng.uniform(0.5, 2.0, K)
    return dict(R=R, t=t, intr=intr, X=X, active=(rng.random(N) < 0.97).astype(np.uint8),
                obs_cam=cam.astype(np.int32), obs_point=pt.astype(np.int32), obs_xy=xy,
                obs_winv=np.stack([a, 0.2 * np.sqrt(a * c), c], axis=1) if case["weighted"] else None,
                obs_w=np.where(rng.random(K) < 0.05, 1e-4, 1.0))


def prepare(case, seed):
    if case["kind"] == "train":
        net = rpba.Gnn(seed=0)
        net.set_weights(_network_weights(seed))
        for S, z in _systems(case, seed):
            net.add_system(S, z)
        return dict(kind="train", net=net)
    if case["kind"] == "sigma0":
        arrays = {k: None if v is None else torch.from_numpy(np.ascontiguousarray(v)).cuda()
                  for k, v in _sigma0_arrays(case, seed).items()}
        return dict(kind="sigma0", sizes=(case["cams"], case["points"], case["obs"]), arrays=arrays)
    prob = _problem(case, seed)
    N = prob["points"].shape[0]
    if case["kind"] == "covariance":
        ids = np.random.Generator(np.random.PCG64(seed + 1)).permutation(N).astype(np.int32)
        return dict(kind="covariance", ctx=rpba.Rpba(prob), ids=ids)
    ctx = rpba.Rpba(prob, **_options(case))
    state = dict(kind="adjust", ctx=ctx, outer=case["outer"], pose=_pinned(prob["cam_pose"]),
                 points=_pinned(prob["points"]), all_active=_pinned(np.ones(N, np.uint8)), fk=None,
                 out_pose=_pinned(np.zeros_like(prob["cam_pose"])), out_points=_pinned(np.zeros((N, 3))),
                 out_active=_pinned(np.zeros(N, np.uint8)))
    if prob.get("intrinsics"):
        state["fk"] = np.stack([prob["cam_intr"][:, 0], prob["cam_k1"]], axis=1)
    return state


# ---------------------------------------------------------------------------
# one pass
# ---------------------------------------------------------------------------


def run(state):
    if state["kind"] == "train":
        loss, grad = state["net"].loss_grad()
        return dict(loss=loss, grad=grad)
    if state["kind"] == "sigma0":
        a = {k: None if v is None else v.data_ptr() for k, v in state["arrays"].items()}
        s0, rms, sums = rpba.rpba_sigma0_noalloc(*state["sizes"], **a, stream=torch.cuda.current_stream())
        return dict(sigma0=s0, rms=rms, sums=sums)
    ctx = state["ctx"]
    if state["kind"] == "covariance":
        return dict(cov=ctx.covariance(state["ids"]))
    ctx.set_cameras(state["pose"])
    if state["fk"] is not None:
        ctx.set_intrinsics(state["fk"])
    ctx.set_points(state["points"], state["all_active"])
    ctx.intersect()
    report = ctx.iterate(state["outer"])
    pose = ctx.cameras(out=state["out_pose"])
    X, active = ctx.points(out=(state["out_points"], state["out_active"]))
    dropped = torch.from_numpy(active).eq(0).unsqueeze(1)  # a dropped point has no position
    X = torch.from_numpy(X).masked_fill_(dropped, 0.0)
    out = dict(pose=pose, points=X, active=active, sigma0=report["sigma0"], rms=report["rms"],
               outer=report["outer"])
    if state["fk"] is not None:
        out["intrinsics"] = ctx.intrinsics()
    return out


# ---------------------------------------------------------------------------
# work
# ---------------------------------------------------------------------------


def work(case):
    """Inputs read once and outputs written once; the operations of one LM
    iteration per outer iteration (about 1,000 per observation for the
    residuals, Jacobians, normal equations and the intersections, and the
    triangular factorisations or 20 CG products of the camera systems)."""
    if case["kind"] == "train":
        n = [max(4, case["cams"] - (7 * s) % max(1, case["cams"] // 2)) for s in range(case["systems"])]
        nodes = sum(n)
        edges = 6 * nodes  # three neighbours on each side
        macs = nodes * (21 * 64 + 6 * 64 * 64 + 64 * 21) + edges * 4 * 64
        factor = edges / 2 * 36 * 2 * case["probes"] * 2 * 4
        return {"bytes": 8 * edges * 36 + 8 * nodes * 6 * case["probes"] + 8 * rpba.gnn_param_count(),
                "flops": 3 * 2 * macs + factor}
    if case["kind"] == "sigma0":
        K = case["obs"]
        return {"bytes": K * (8 + 16 + 8 + (24 if case["weighted"] else 0)) + 25 * case["points"] + 120 * case["cams"],
                "flops": 45 * K}
    rig = case.get("rig", "grid")
    cams = case["nx"] * case["ny"] if rig != "blocks" else float(
        np.exp(np.linspace(math.log(20.0), math.log(400.0), case["nx"])).sum())
    K, N = case["points"] * case["per_point"], case["points"]
    inputs = K * (8 + 16 + (24 if case["weighted"] else 0))
    if case["kind"] == "covariance":
        return {"bytes": inputs + N * (24 + 4 + 72) + 120 * cams, "flops": 80 * K + 50 * N}
    cd = 8 if rig == "ring" else 6
    n = cd * cams / case["subs"] if rig != "blocks" else cd * cams / (case["subs"] * case["nx"])
    subs = case["subs"] * (case["nx"] if rig == "blocks" else 1)
    solve = n ** 3 / 3 if case["form"] != "chosen" or subs > 64 else 20 * 2 * n * n
    return {"bytes": inputs + 2 * (8 * cd * cams + 25 * N), "flops": case["outer"] * (1000 * K + subs * solve)}


# ---------------------------------------------------------------------------
# the same in 64 bits, with torch and numpy alone
# ---------------------------------------------------------------------------


def exact(case, seed):
    if case["kind"] == "train":
        return _exact_train(case, seed)
    if case["kind"] == "sigma0":
        return _exact_sigma0(case, seed)
    prob = _problem(case, seed)
    ref = _Reference(prob)
    if case["kind"] == "covariance":
        ids = np.random.Generator(np.random.PCG64(seed + 1)).permutation(prob["points"].shape[0])
        N, _, _, behind, _, _ = ref.point_normals(ref.X, ref.w)
        C = torch.linalg.inv(N)
        C[behind | (ref.count < 2)] = float("nan")
        return dict(cov=C[torch.from_numpy(ids).to(C.device)].cpu().numpy())
    ref.intersect(ref.active.clone())
    outer, s0, rms = ref.iterate(case["outer"], case["inner"])
    X, act = ref.X.clone(), ref.active
    X[~act] = 0.0
    out = dict(pose=ref.poses().cpu().numpy(), points=X.cpu().numpy(), active=act.to(torch.uint8).cpu().numpy(),
               sigma0=s0, rms=rms, outer=outer)
    if prob.get("intrinsics"):
        out["intrinsics"] = torch.stack([ref.f, ref.k1], 1).cpu().numpy()
    return out


def _exact_sigma0(case, seed):
    a = _sigma0_arrays(case, seed)
    cam, pt = a["obs_cam"], a["obs_point"]
    xc = np.einsum("kab,kb->ka", a["R"][cam], a["X"][pt]) + a["t"][cam]
    v = a["intr"][cam, :1] * xc[:, :2] / xc[:, 2:] + a["intr"][cam, 1:] - a["obs_xy"]
    W = a["obs_winv"] if a["obs_winv"] is not None else np.tile([1.0, 0.0, 1.0], (v.shape[0], 1))
    e = a["obs_w"] * (W[:, 0] * v[:, 0] ** 2 + 2 * W[:, 1] * v[:, 0] * v[:, 1] + W[:, 2] * v[:, 1] ** 2)
    on = a["active"][pt] == 1
    good = on & (a["obs_w"] == 1.0)
    sums = np.array([e[on].sum(), on.sum(), (v[good] ** 2).sum(), good.sum(), (a["active"] == 1).sum()], float)
    red = max(1.0, 2 * sums[1] - 6 * case["cams"] - 3 * sums[4] + 7)
    return dict(sigma0=math.sqrt(sums[0] / red), rms=math.sqrt(sums[2] / (2 * sums[3])), sums=sums)


def _exact_train(case, seed):
    """Loss and gradient by automatic differentiation of the definition in
    include/rpba.h; the network's matrices are applied in BF16."""
    H, F = 64, 21
    shapes = [("W0", (H, F)), ("b0", (H,))]
    for t in "123":
        shapes += [("A" + t, (H, H)), ("B" + t, (H, H)), ("c" + t, (H,))]
    shapes += [("Wo", (F, H)), ("bo", (F,)), ("ws", (H,)), ("wp", (H,)), ("we", (1,)), ("bq", (1,))]
    w = torch.from_numpy(_network_weights(seed)).double().requires_grad_(True)
    p, at = {}, 0
    for name, shape in shapes:
        size = math.prod(shape)
        v = w[at:at + size].view(shape)
        if name[0] in "WAB":  # rounded to BF16, the gradient passed through
            v = v + (v.detach().float().bfloat16().double() - v.detach())
        p[name], at = v, at + size
    tril = torch.tril_indices(6, 6)
    total = 0.0
    systems = _systems(case, seed)
    for S, z in systems:
        n = S.shape[0] // 6
        S, z = torch.from_numpy(S), torch.from_numpy(z)
        blocks = S.view(n, 6, n, 6).permute(0, 2, 1, 3)
        B = torch.diagonal(blocks, dim1=0, dim2=1).permute(2, 0, 1)
        d = torch.diagonal(B, dim1=1, dim2=2)
        norm = torch.linalg.matrix_norm(blocks)
        edge = torch.any(blocks.flatten(2) != 0, dim=2) & ~torch.eye(n, dtype=torch.bool)
        e = torch.where(edge, norm / torch.sqrt(torch.outer(norm.diagonal(), norm.diagonal())), 0.0)
        strict = torch.tril_indices(6, 6, -1)
        corr = (B / torch.sqrt(d[:, :, None] * d[:, None, :]))[:, strict[0], strict[1]]
        x = torch.cat([torch.log(d) - torch.log(d).mean(0), corr], 1)
        h = torch.relu(x @ p["W0"].T + p["b0"])
        for t in "123":
            h = torch.relu(h @ p["A" + t].T + (e @ h) @ p["B" + t].T + p["c" + t])
        C = torch.zeros(n, 6, 6, dtype=torch.float64)
        C[:, tril[0], tril[1]] = h @ p["Wo"].T + p["bo"]
        M = torch.eye(6, dtype=torch.float64) + 0.5 * torch.tanh(C)
        s = h @ p["ws"]
        q = s[:, None] + s[None, :] + (h * p["wp"]) @ h.T + p["we"] * e + p["bq"]
        gamma = torch.where(edge & (torch.arange(n)[:, None] > torch.arange(n)), torch.tanh(q), 0.0)
        L = torch.linalg.cholesky(B)
        Li = torch.block_diag(*torch.linalg.inv(L))
        N = gamma.repeat_interleave(6, 0).repeat_interleave(6, 1) * (Li @ S @ Li.T)
        G = torch.block_diag(*torch.linalg.inv(M)) @ (torch.eye(6 * n, dtype=torch.float64) - N) @ Li
        V = z @ G
        T = ((V @ S) * V).sum(1).mean()
        logdet = torch.log(torch.diagonal(M, dim1=1, dim2=2)).sum() + torch.log(torch.diagonal(L, dim1=1, dim2=2)).sum()
        total = total + (torch.log(T / (6 * n)) + 2.0 * logdet / (6 * n)) / len(systems)
    total.backward()
    return dict(loss=float(total.detach()), grad=w.grad.numpy())


def _rotations(w):
    th = torch.linalg.vector_norm(w, dim=1)
    a = torch.sinc(th / math.pi)
    b = 0.5 * torch.sinc(th / (2 * math.pi)) ** 2
    K = torch.zeros(w.shape[0], 3, 3, dtype=w.dtype, device=w.device)
    K[:, 0, 1], K[:, 0, 2], K[:, 1, 2] = -w[:, 2], w[:, 1], -w[:, 0]
    K = K - K.transpose(1, 2)
    return torch.eye(3, dtype=w.dtype, device=w.device) + a[:, None, None] * K + b[:, None, None] * (K @ K)


class _Reference:
    """The method on one block in plain torch, 64 bits (see include/rpba.h for
    the statement of every step)."""

    def __init__(self, prob):
        dev = "cuda" if torch.cuda.is_available() else "cpu"
        put = lambda a: torch.from_numpy(np.ascontiguousarray(a)).to(dev)  # noqa: E731
        self.dev = dev
        self.cd = 8 if prob.get("intrinsics") else 6
        pose = put(prob["cam_pose"])
        self.R, self.t = _rotations(pose[:, :3]), pose[:, 3:].clone()
        intr = put(prob["cam_intr"])
        self.f, self.pp = intr[:, 0].clone(), intr[:, 1:]
        self.k1 = put(prob["cam_k1"]) if self.cd == 8 else torch.zeros_like(self.f)
        self.X = put(prob["points"]).clone()
        self.M, self.N = pose.shape[0], self.X.shape[0]
        sub_of = put(prob["cam_subblock"]).long()
        cam, pt = put(prob["obs_cam"]).long(), put(prob["obs_point"]).long()
        self.L = int(sub_of.max()) + 1
        key, order = torch.sort(sub_of[cam] * self.N + pt, stable=True)  # by (sub-block, point)
        self.cam, self.pt = cam[order], pt[order]
        uniq, self.inst, self.inst_n = torch.unique_consecutive(key, return_inverse=True, return_counts=True)
        self.P = uniq.numel()
        self.inst_pt, self.inst_sub = uniq % self.N, uniq // self.N
        self.inst_start = torch.cumsum(self.inst_n, 0) - self.inst_n
        self.xy = put(prob["obs_xy"])[order] - self.pp[self.cam]
        K = self.cam.numel()
        W = torch.tensor([1.0, 0.0, 1.0], dtype=torch.float64, device=dev).expand(K, 3)
        if prob.get("obs_winv") is not None:
            W = put(prob["obs_winv"])[order]
        self.W = torch.stack([W[:, 0], W[:, 1], W[:, 1], W[:, 2]], 1).view(K, 2, 2)
        self.w = torch.ones(K, dtype=torch.float64, device=dev)
        self.count = torch.bincount(self.pt, minlength=self.N)
        self.active = self.count >= 2
        self.tie = torch.bincount(self.inst_pt, minlength=self.N) >= 2
        self.Xl = self.X[self.inst_pt]
        self.Wl = torch.zeros(self.P, 3, 3, dtype=torch.float64, device=dev)
        self.sub_of = sub_of
        n_sub = torch.bincount(sub_of, minlength=self.L)
        first = torch.cumsum(n_sub, 0) - n_sub
        rank = torch.argsort(torch.argsort(sub_of, stable=True), stable=True)  # cameras by (sub-block, id)
        self.local, self.n_sub = rank - first[sub_of], n_sub.tolist()
        self.block0 = torch.cumsum(n_sub * n_sub, 0) - n_sub * n_sub
        # every ordered pair of observations of one instance
        n = self.inst_n[self.inst]
        self.pa = torch.repeat_interleave(torch.arange(K, device=dev), n)
        local = torch.arange(self.pa.numel(), device=dev) - torch.repeat_interleave(torch.cumsum(n, 0) - n, n)
        self.pb = self.inst_start[self.inst[self.pa]] + local

    def poses(self):
        R = self.R
        v = torch.stack([R[:, 2, 1] - R[:, 1, 2], R[:, 0, 2] - R[:, 2, 0], R[:, 1, 0] - R[:, 0, 1]], 1)
        s, c = 0.5 * torch.linalg.vector_norm(v, dim=1), 0.5 * (R.diagonal(dim1=1, dim2=2).sum(1) - 1.0)
        th = torch.atan2(s, c)
        # the axis: from the skew part, or near half a turn from the symmetric part
        near = th > math.pi - 1e-3
        w = v * (0.5 * th / torch.where(s > 1e-12, s, 1.0))[:, None]
        B = 0.5 * (R + R.transpose(1, 2))
        eye = torch.eye(3, dtype=R.dtype, device=R.device)
        A = (B - c[:, None, None] * eye) / (1.0 - c)[:, None, None].clamp_min(1e-3)
        k = A.diagonal(dim1=1, dim2=2).argmax(1)
        axis = A[torch.arange(A.shape[0], device=R.device), k]
        axis = axis / torch.linalg.vector_norm(axis, dim=1, keepdim=True).clamp_min(1e-300)
        axis = axis * torch.where((axis * v).sum(1) < 0, -1.0, 1.0)[:, None]
        return torch.cat([torch.where(near[:, None], axis * th[:, None], w), self.t], 1)

    def project(self, R, t, f, k1, X, jac=False):
        """Residual-free projection (relative to the principal point), depth,
        and with jac the Jacobians for the point and the camera."""
        i = self.cam
        RX = (R[i] @ X[:, :, None])[:, :, 0]
        xc = RX + t[i]
        z = xc[:, 2]
        p = xc[:, :2] / z[:, None]
        r2 = (p * p).sum(1)
        g = 1.0 + k1[i] * r2
        uv = (f[i] * g)[:, None] * p
        if not jac:
            return uv, z
        D = (f[i] * g)[:, None, None] * torch.eye(2, dtype=p.dtype, device=p.device)
        D = D + (2.0 * f[i] * k1[i])[:, None, None] * p[:, :, None] * p[:, None, :]
        dp = torch.zeros(p.shape[0], 2, 3, dtype=p.dtype, device=p.device)
        dp[:, 0, 0] = dp[:, 1, 1] = 1.0 / z
        dp[:, :, 2] = -p / z[:, None]
        Pm = D @ dp
        a = torch.zeros(p.shape[0], 3, 3, dtype=p.dtype, device=p.device)  # -[RX]x
        a[:, 0, 1], a[:, 0, 2], a[:, 1, 2] = RX[:, 2], -RX[:, 1], RX[:, 0]
        a = a - a.transpose(1, 2)
        Jc = [Pm @ a, Pm]
        if self.cd == 8:
            Jc.append(torch.stack([g[:, None] * p, (f[i] * r2)[:, None] * p], 2))
        return uv, z, Pm @ R[i], torch.cat(Jc, 2)

    def state(self):
        return self.R, self.t, self.f, self.k1

    def residuals(self):
        return self.project(*self.state(), self.X[self.pt])[0] - self.xy

    def point_normals(self, X, w):
        """Per point N and g over its observations, per instance N, whether an
        observation lies behind its camera."""
        uv, z, Jx, _ = self.project(*self.state(), X[self.pt], jac=True)
        A = w[:, None, None] * (Jx.transpose(1, 2) @ self.W)
        Nk, gk = A @ Jx, (A @ (uv - self.xy)[:, :, None])[:, :, 0]
        zeros = lambda n, *s: torch.zeros(n, *s, dtype=torch.float64, device=self.dev)  # noqa: E731
        Nq = zeros(self.P, 3, 3).index_add_(0, self.inst, Nk)
        Nj = zeros(self.N, 3, 3).index_add_(0, self.inst_pt, Nq)
        gj = zeros(self.N, 3).index_add_(0, self.pt, gk)
        behind = torch.zeros(self.N, dtype=torch.bool, device=self.dev)
        behind[self.pt[z <= 0]] = True
        return Nj, gj, Nq, behind, uv, z

    def intersect(self, running, px_tol=1e-3, tol=1e-10, cond_max=1e12, max_iter=10):
        run = running.clone()
        for it in range(max_iter):
            if not bool(run.any()):
                break
            Nj, gj, Nq, behind, _, _ = self.point_normals(self.X, self.w)
            det = torch.linalg.det(Nj)
            safe = torch.where((det > 0)[:, None, None], Nj, torch.eye(3, dtype=Nj.dtype, device=Nj.device))
            inv = torch.linalg.inv_ex(safe)[0]
            cond = torch.linalg.matrix_norm(Nj) * torch.linalg.matrix_norm(inv)
            ok = run & ~behind & (det > 0) & (cond <= cond_max)
            d = (inv @ gj[:, :, None])[:, :, 0]
            self.X = torch.where(ok[:, None], self.X - d, self.X)
            conv = torch.linalg.vector_norm(d, dim=1) <= tol * (1 + torch.linalg.vector_norm(self.X, dim=1))
            moved = (d[:, None, :] @ Nj @ d[:, :, None])[:, 0, 0]
            conv = ok & (conv | (moved <= px_tol ** 2 * self.count))
            failed = run & (~ok | (~conv if it == max_iter - 1 else torch.zeros_like(conv)))
            self.active &= ~failed
            q = conv[self.inst_pt] & self.tie[self.inst_pt]
            self.Wl = torch.where(q[:, None, None], Nj[self.inst_pt] - Nq, self.Wl)
            off = failed[self.inst_pt] | (conv & ~self.tie)[self.inst_pt]
            self.Wl[off] = 0.0
            run = run & ~conv & ~failed
        q = running[self.inst_pt]
        self.Xl = torch.where(q[:, None], self.X[self.inst_pt], self.Xl)

    def costs(self, R, t, f, k1, Xl):
        uv, z = self.project(R, t, f, k1, Xl[self.inst])
        v = (uv - self.xy)[:, :, None]
        e = self.w * (v.transpose(1, 2) @ self.W @ v)[:, 0, 0]
        e = torch.where(z > 0, e, float("inf"))
        e = torch.where(self.active[self.pt], e, 0.0)
        F = torch.zeros(self.L, dtype=torch.float64, device=self.dev).index_add_(0, self.inst_sub[self.inst], e)
        d = (Xl - self.X[self.inst_pt])[:, :, None]
        tp = (d.transpose(1, 2) @ self.Wl @ d)[:, 0, 0]
        return F.index_add_(0, self.inst_sub, torch.where(self.active[self.inst_pt], tp, 0.0))

    def solve_step(self, lam, run):
        """Camera updates (M x cd), instance updates and failures at damping lam."""
        cd, dev = self.cd, self.dev
        uv, _, Jx, Jc = self.project(*self.state(), self.Xl[self.inst], jac=True)
        on = self.active[self.pt]
        w = torch.where(on, self.w, 0.0)
        r = (uv - self.xy)[:, :, None]
        A = w[:, None, None] * (Jx.transpose(1, 2) @ self.W)
        Bc = w[:, None, None] * (Jc.transpose(1, 2) @ self.W)
        zeros = lambda n, *s: torch.zeros(n, *s, dtype=torch.float64, device=dev)  # noqa: E731
        Nq = zeros(self.P, 3, 3).index_add_(0, self.inst, A @ Jx) + self.Wl
        gq = zeros(self.P, 3).index_add_(0, self.inst, (A @ r)[:, :, 0])
        gq = gq + (self.Wl @ (self.Xl - self.X[self.inst_pt])[:, :, None])[:, :, 0]
        diag = torch.diagonal(Nq, dim1=1, dim2=2)
        diag += lam[self.inst_sub][:, None] * diag.clone()
        act = self.active[self.inst_pt]
        Nq[~act] = torch.eye(3, dtype=torch.float64, device=dev)
        gq[~act] = 0.0
        Ni = torch.linalg.inv_ex(Nq)[0]
        Nxc = A @ Jc
        Z = Ni[self.inst] @ Nxc
        U = zeros(self.M, cd, cd).index_add_(0, self.cam, Bc @ Jc)
        y = zeros(self.M, cd).index_add_(0, self.cam, (-(Bc @ r) + Z.transpose(1, 2) @ gq[self.inst][:, :, None])[:, :, 0])
        ncam = torch.tensor(self.n_sub, device=dev)
        S = zeros(int((ncam * ncam).sum()), cd * cd)
        step = 1 << 21
        for s in range(0, self.pa.numel(), step):
            a, b = self.pa[s:s + step], self.pb[s:s + step]
            l = self.sub_of[self.cam[a]]
            at = self.block0[l] + self.local[self.cam[a]] * ncam[l] + self.local[self.cam[b]]
            S.index_add_(0, at, -(Nxc[a].transpose(1, 2) @ Z[b]).reshape(-1, cd * cd))
        Ud = torch.diagonal(U, dim1=1, dim2=2)
        Ud += lam[self.sub_of][:, None] * Ud.clone()
        l = self.sub_of
        S.index_add_(0, self.block0[l] + self.local * (ncam[l] + 1), U.reshape(-1, cd * cd))
        dC, fail = zeros(self.M, cd), torch.zeros(self.L, dtype=torch.bool, device=dev)
        cams = torch.argsort(self.sub_of * self.M + self.local)
        c0 = 0
        for l, n in enumerate(self.n_sub):
            mine = cams[c0:c0 + n]
            c0 += n
            if not run[l] or n == 0:
                continue
            b0 = int(self.block0[l])
            Sl = S[b0:b0 + n * n].view(n, n, cd, cd).permute(0, 2, 1, 3).reshape(n * cd, n * cd)
            Lc, info = torch.linalg.cholesky_ex(Sl)
            if int(info):
                fail[l] = True
                continue
            dC[mine] = torch.cholesky_solve(y[mine].reshape(-1, 1), Lc).view(n, cd)
        rhs = -gq - zeros(self.P, 3).index_add_(0, self.inst, (Nxc @ dC[self.cam][:, :, None])[:, :, 0])
        dX = (Ni @ rhs[:, :, None])[:, :, 0]
        dX[~act] = 0.0
        return dC, dX, fail

    def adjust_sub_blocks(self, max_inner, lambda0=1e-4, ratio_min=1.01, max_reject=6):
        F = self.costs(*self.state(), self.Xl)
        best, lam = F.clone(), torch.full_like(F, lambda0)
        grace, rejected, its = [1] * self.L, [0] * self.L, [0] * self.L
        run = [n > 0 for n in self.n_sub]
        while any(run):
            dC, dX, fail = self.solve_step(lam, run)
            runs = torch.tensor(run, device=self.dev)
            dC[~runs[self.sub_of]] = 0.0
            dX[~runs[self.inst_sub]] = 0.0
            R, t = _rotations(dC[:, :3]) @ self.R, self.t + dC[:, 3:6]
            f, k1 = (self.f + dC[:, 6], self.k1 + dC[:, 7]) if self.cd == 8 else (self.f, self.k1)
            Xl = self.Xl + dX
            Ft = self.costs(R, t, f, k1, Xl)
            take = runs & ~fail & torch.isfinite(Ft) & (Ft < F)
            for l in range(self.L):
                if not run[l]:
                    continue
                its[l] += 1
                stop = its[l] >= max_inner
                if not bool(take[l]):
                    lam[l] *= 10.0
                    rejected[l] += 1
                    stop |= rejected[l] > max_reject
                else:
                    rejected[l] = 0
                    ratio = float(best[l] / Ft[l].clamp_min(1e-300))
                    lam[l] = max(float(lam[l]) / 10.0, lambda0)
                    best[l] = torch.minimum(best[l], Ft[l])
                    if ratio < ratio_min:
                        stop |= grace[l] == 0
                        grace[l] = max(0, grace[l] - 1)
                run[l] = not stop
            c, q = take[self.sub_of], take[self.inst_sub]
            self.R, self.t = torch.where(c[:, None, None], R, self.R), torch.where(c[:, None], t, self.t)
            self.f, self.k1 = torch.where(c, f, self.f), torch.where(c, k1, self.k1)
            self.Xl = torch.where(q[:, None], Xl, self.Xl)
            F = torch.where(take, Ft, F)

    def camera_median(self, value, cam):
        """Median of `value` per camera (mean of the middle pair; 0 without values)."""
        v, o = torch.sort(value)
        c, o2 = torch.sort(cam[o], stable=True)
        v = v[o2]
        n = torch.bincount(c, minlength=self.M)
        s = torch.cumsum(n, 0) - n
        last = max(v.numel() - 1, 0)
        mid = 0.5 * (v[(s + (n - 1).clamp_min(0) // 2).clamp_max(last)] + v[(s + n // 2).clamp_max(last)])
        return torch.where(n > 0, mid, 0.0)

    def robust_weights(self, t_v=4.0, down=1e-4):
        v, on = self.residuals(), self.active[self.pt]
        a = torch.sqrt(self.W[:, 0, 0])
        b = self.W[:, 0, 1] / a
        c = torch.sqrt(self.W[:, 1, 1] - b * b)
        e = torch.cat([a * v[:, 0] + b * v[:, 1], c * v[:, 1]])
        cam = torch.cat([self.cam, self.cam])
        both = torch.cat([on, on])
        e, cam = e[both], cam[both]
        sigma = 1.4826 * self.camera_median((e - self.camera_median(e, cam)[cam]).abs(), cam)
        s = sigma[self.cam]
        out = (s > 0) & (torch.sqrt((v[:, None, :] @ self.W @ v[:, :, None])[:, 0, 0]) > t_v * s)
        self.w = torch.where(on, torch.where(out, down, 1.0), self.w)

    def sigma0(self):
        v, on = self.residuals(), self.active[self.pt] & (self.w != 0)
        e = self.w * (v[:, None, :] @ self.W @ v[:, :, None])[:, 0, 0]
        good = on & (self.w == 1.0)
        red = 2.0 * int(on.sum()) - self.cd * self.M - 3.0 * int(self.active.sum()) + 7.0
        rms = torch.sqrt((v[good] ** 2).sum() / (2.0 * max(int(good.sum()), 1)))
        return float(torch.sqrt(e[on].sum() / max(red, 1.0))), float(rms)

    def iterate(self, max_outer, max_inner, ratio_min=1.01):
        best, grace, done = self.sigma0()[0], 1, 0
        for _ in range(max_outer):
            self.adjust_sub_blocks(max_inner)
            single = self.active[self.inst_pt] & ~self.tie[self.inst_pt]
            self.X[self.inst_pt[single]] = self.Xl[single]
            self.robust_weights()
            self.intersect(self.active & self.tie)
            s = self.sigma0()[0]
            done += 1
            ratio, best = best / max(s, 1e-300), min(best, s)
            if ratio < ratio_min:
                if grace == 0:
                    break
                grace -= 1
        self.active[self.pt[self.w != 1.0]] = False
        return (done, *self.sigma0())
