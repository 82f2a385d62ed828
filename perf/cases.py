"""Performance cases: the calls a user of the filter library makes, over the sizes they make them at.

A tracking case is a whole scene: the filter is reset and stepped frame by frame through ``Filter.step`` (or
``step_batch``), with the estimates read after every frame, as a tracker does; after the last frame the retained
children and the clutter probabilities of its detections are read as well.  Detections are host arrays or tensors that
a detector left on the GPU.  The other cases are the calls that stand on their own: scoring pairs with the learned
gate's network, one step of its training, and the top-H selection without device allocation.

The worlds follow the repository's own workloads: 2-D and 3-D constant velocity, the convoy of the paper's Section 4.1
(Gaussian tracks, and the paper's particles), vehicles with constant turn rate, and batches of independent 2-D scenes.
"""
from __future__ import annotations

import ctypes
import math

import numpy as np
import torch

import paper_2512_06230_gb300 as glmb
from paper_2512_06230_gb300.gate import init_params

# Mahalanobis gates: chi-square quantiles at 1 - 1e-4 and 1 - 1e-12 (2 and 3 degrees of freedom)
GATE = {2: 18.420680743952364, 3: 21.10751346616021}
GATE_LOOSE = {2: 55.262042231857095, 3: 58.919755683202155}
H_UP = 100
DEV = "cuda"


def listed():
    return [
        # the paper's convoy, few objects and hypotheses, detections from the host: a real-time loop on small
        # frames, where a frame is launches, copies and one wait
        dict(name="convoy_n5_h25", kind="convoy", n=5, h_max=25, frames=50, particles=0, score_mode=0),
        # the same world with the paper's own particle track model
        dict(name="convoy_particles_n10_h100", kind="convoy", n=10, h_max=100, frames=40, particles=256, score_mode=1),
        # a dense 2-D scene of ordinary size, detections already on the GPU
        dict(name="cv2d_n100_h1000", kind="cv", dim=2, n=100, h_max=1000, frames=60, device=True),
        # the 3-D sweep: few objects with a generous cap, detections from the host
        dict(name="cv3d_n50_h5000", kind="cv", dim=3, n=50, h_max=5000, frames=40, device=False),
        # the 3-D sweep where the cap binds: a million children a frame, the largest ordinary load
        dict(name="cv3d_n200_h20000", kind="cv", dim=3, n=200, h_max=20000, frames=30, device=True),
        # the 3-D sweep with many objects: few hypotheses of thousands of tracks and detections
        dict(name="cv3d_n1000_h5000", kind="cv", dim=3, n=1000, h_max=5000, frames=30, device=True),
        # a server's frame: independent scenes of uneven size stepped together
        dict(name="batch_16", kind="batch", scenes=16, n=300, h_max=5000, frames=20, device=True),
        # vehicles with the particle track model (256 particles each)
        dict(name="ctrv_n200_h1000", kind="ctrv", n=200, h_max=1000, frames=30, particles=256, device=True),
        # a loose base gate whose surplus pairs the learned gate removes
        dict(name="gated_n300_h5000", kind="gated", dim=3, n=300, h_max=5000, frames=20, device=True),
        # scoring a data set of pairs with the gate's network (choosing a threshold)
        dict(name="gate_score_4m", kind="score", rows=1 << 22),
        # one training step of the gate on a mini-batch of the default size
        dict(name="gate_train_32k", kind="train", rows=32768),
        # truncation of a million children on its own
        dict(name="select_1m", kind="select", n=1_000_000, h_max=20000, tau=1e-9),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["cv"] * 5 + ["convoy"] * 2 + ["ctrv"] * 2 + ["batch", "gated", "score", "train", "select"])
    if kind == "cv":
        dim = rng.choice([2, 3])
        return dict(kind=kind, dim=dim, n=_log_int(rng, 5, 300 if dim == 2 else 1000), h_max=_log_int(rng, 20, 10000),
                    frames=rng.randint(15, 20), device=rng.random() < 0.5)
    if kind == "convoy":
        particles = rng.choice([0, 0, 64, 256])
        return dict(kind=kind, n=rng.randint(1, 20), h_max=_log_int(rng, 5, 100), frames=rng.randint(20, 50),
                    particles=particles, score_mode=1 if particles else rng.choice([0, 1]))
    if kind == "ctrv":
        return dict(kind=kind, n=_log_int(rng, 5, 500), h_max=_log_int(rng, 50, 2000), frames=rng.randint(15, 25),
                    particles=rng.choice([32, 100, 256, 300, 512]), device=rng.random() < 0.5)
    if kind == "batch":
        return dict(kind=kind, scenes=rng.randint(2, 16), n=_log_int(rng, 20, 300), h_max=_log_int(rng, 100, 5000),
                    frames=rng.randint(10, 20), device=rng.random() < 0.5)
    if kind == "gated":
        return dict(kind=kind, dim=rng.choice([2, 3]), n=_log_int(rng, 20, 300), h_max=_log_int(rng, 100, 5000),
                    frames=rng.randint(10, 20), device=rng.random() < 0.5)
    if kind == "score":
        return dict(kind=kind, rows=_log_int(rng, 1000, 1 << 22))
    if kind == "train":
        return dict(kind=kind, rows=_log_int(rng, 200, 1 << 18))
    return dict(kind=kind, n=_log_int(rng, 1000, 4_000_000), h_max=_log_int(rng, 100, 20000),
                tau=rng.choice([1e-5, 1e-9]))


# ---------------------------------------------------------------------------
# worlds: (births, Z) per frame
# ---------------------------------------------------------------------------
def _cluster(rng, positions, p_d, lam, sigma):
    """1 + Poisson(lam) detections of each detected position."""
    seen = positions[rng.random(len(positions)) < p_d]
    rep = np.repeat(seen, 1 + rng.poisson(lam, len(seen)), axis=0)
    return rep + sigma * rng.normal(size=rep.shape)


def _cv_frames(rng, dim, n, frames, clutter=None):
    """Constant-velocity objects: 2-D in [0, 1000]^2, appearing over the first half hundred frames; 3-D in
    [0, 5000]^3, alive from the start with Poisson(0.01 n) appearances a frame."""
    extent, p_d, lam = (1000.0, 0.9, 1.5) if dim == 2 else (5000.0, 0.85, 2.0)
    if clutter is None:
        clutter = 20.0 if dim == 2 else 50.0
    sigma, q, dt, p_s = 5.0, 1.0, 1.0, 0.99
    start = np.sort(rng.integers(0, min(50, frames), n)) if dim == 2 else np.zeros(n, np.int64)
    L = np.linalg.cholesky(q * np.array([[dt ** 3 / 3, dt ** 2 / 2], [dt ** 2 / 2, dt]]))
    pos, vel = np.zeros((0, dim)), np.zeros((0, dim))
    cov = np.diag([(2 * sigma) ** 2] * dim + [10.0 ** 2] * dim)
    out = []
    for k in range(frames):
        keep = rng.random(len(pos)) < p_s
        a, b = rng.normal(size=(2, int(keep.sum()), dim))
        pos, vel = pos[keep] + dt * vel[keep] + L[0, 0] * a, vel[keep] + L[1, 0] * a + L[1, 1] * b
        new = int(np.sum(start == k)) + (int(rng.poisson(0.01 * n)) if dim == 3 and k else 0)
        p = rng.uniform(0, extent, (new, dim))
        v = rng.normal(size=(new, dim))
        v *= rng.uniform(0, 10, (new, 1)) / np.linalg.norm(v, axis=1, keepdims=True)
        pos, vel = np.concatenate([pos, p]), np.concatenate([vel, v])
        zero = np.zeros(dim)
        births = [(0.5, np.concatenate([m, zero]), cov) for m in p + 2 * sigma * rng.normal(size=p.shape)]
        births += [(0.05, np.concatenate([m, zero]), cov)
                   for m in rng.uniform(0, extent, (int(rng.poisson(1.0)), dim))]
        Z = np.concatenate([_cluster(rng, pos, p_d, lam, sigma),
                            rng.uniform(0, extent, (int(rng.poisson(clutter)), dim))])
        out.append((births, Z[rng.permutation(len(Z))]))
    model = dict(dim_x=2 * dim, dim_z=dim, dt=dt, q=q, R=sigma ** 2 * np.eye(dim), p_s=p_s, p_d=p_d, lambda_d=lam,
                 clutter_rate=clutter, volume=extent ** dim, gate=GATE[dim], score_mode=0)
    return out, model


def _ctrv_step(x, dt, acc, yaw):
    """Vehicles (px, py, v, heading, turn rate) along their arcs, with accelerations."""
    px, py, v, psi, om = x.T
    half = 0.5 * om * dt
    chord = v * dt * np.sinc(half / math.pi)
    return np.stack([px + chord * np.cos(psi + half) + 0.5 * dt * dt * np.cos(psi) * acc,
                     py + chord * np.sin(psi + half) + 0.5 * dt * dt * np.sin(psi) * acc,
                     v + dt * acc, psi + om * dt + 0.5 * dt * dt * yaw, om + dt * yaw], 1)


def _ctrv_frames(rng, n, frames):
    """Vehicles in a 1 km square with 10 clutter detections a frame, appearing over the first 20 frames."""
    sigma, off, extent = 3.0, 200.0, 1000.0
    start = np.sort(rng.integers(0, min(20, frames), n))
    cov = np.diag([(2 * sigma) ** 2, (2 * sigma) ** 2, 25.0, 0.09, 0.0025])
    cov_false = np.diag([(2 * sigma) ** 2, (2 * sigma) ** 2, 25.0, 2.25, 0.0025])
    x = np.zeros((0, 5))
    out = []
    for k in range(frames):
        x = x[rng.random(len(x)) < 0.99]
        x = _ctrv_step(x, 1.0, 0.5 * rng.normal(size=len(x)), 0.02 * rng.normal(size=len(x)))
        new = int(np.sum(start == k))
        b = np.concatenate([off + rng.uniform(0, extent, (new, 2)), rng.uniform(5, 15, (new, 1)),
                            rng.uniform(-math.pi, math.pi, (new, 1)), rng.uniform(-0.05, 0.05, (new, 1))], 1)
        x = np.concatenate([x, b])
        m = np.stack([b[:, 0] + 2 * sigma * rng.normal(size=new), b[:, 1] + 2 * sigma * rng.normal(size=new),
                      np.full(new, 10.0), b[:, 3] + 0.3 * rng.normal(size=new), np.zeros(new)], 1)
        births = [(0.5, r, cov) for r in m]
        births += [(0.05, np.array([*(off + rng.uniform(0, extent, 2)), 10.0, rng.uniform(-math.pi, math.pi), 0.0]),
                    cov_false) for _ in range(int(rng.poisson(1.0)))]
        Z = np.concatenate([_cluster(rng, x[:, :2], 0.9, 1.0, sigma),
                            off + rng.uniform(0, extent, (int(rng.poisson(10.0)), 2))])
        out.append((births, Z[rng.permutation(len(Z))]))
    model = dict(dim_x=5, dim_z=2, dt=1.0, q=0.0, R=sigma ** 2 * np.eye(2), p_s=0.99, p_d=0.9, lambda_d=1.0,
                 clutter_rate=10.0, volume=extent ** 2, gate=GATE[2], score_mode=1, model=1, sigma_a=0.5,
                 sigma_w=0.05, ess_frac=0.5)
    return out, model


def _convoy_frames(rng, n, frames, particles, score_mode):
    """Copies of one closed ground track, two samples apart, five detections each, no clutter."""
    steps, extent, dt, sigma, det = 548, 80.0, 0.1, 0.25, 5
    u = 2 * math.pi * 3 * np.arange(steps) / steps
    xy = np.stack([np.cos(u), rng.uniform(0.6, 1.0) * np.sin(u)], 1) * 0.4 * extent + 0.5 * extent
    vel = (np.roll(xy, -1, 0) - np.roll(xy, 1, 0)) / (2 * dt)
    sb = 2 * sigma
    out = []
    for k in range(frames):
        at = (k + 2 * np.arange(n)) % steps
        births = []
        if k == 0 and particles:
            mean = np.stack([*xy[at].T, np.hypot(*vel[at].T), np.arctan2(vel[at, 1], vel[at, 0]), np.zeros(n)], 1)
            mean += rng.normal(size=(n, 5)) * np.array([sb, sb, 1.0, 0.1, 0.1])
            births = [(0.5, m, np.diag([sb * sb, sb * sb, 1.0, 0.01, 0.01])) for m in mean]
        elif k == 0:
            mean = np.concatenate([xy[at], vel[at]], 1) + rng.normal(size=(n, 4)) * np.array([sb, sb, 1.0, 1.0])
            births = [(0.5, m, np.diag([sb * sb, sb * sb, 1.0, 1.0])) for m in mean]
        for _ in range(int(rng.poisson(1.0))):
            p = rng.uniform(0, extent, 2)
            if particles:
                births.append((0.05, np.array([*p, 10.0, rng.uniform(-math.pi, math.pi), 0.0]),
                               np.diag([sb * sb, sb * sb, 36.0, 3.24, 0.09])))
            else:
                births.append((0.05, np.array([*p, 0.0, 0.0]), np.diag([sb * sb, sb * sb, 36.0, 36.0])))
        out.append((births, np.repeat(xy[at], det, 0) + sigma * rng.normal(size=(n * det, 2))))
    model = dict(dim_x=4, dim_z=2, dt=dt, q=10.0, R=sigma ** 2 * np.eye(2), p_s=0.999, p_d=0.999,
                 lambda_d=det - 1.0, clutter_rate=0.5, volume=extent ** 2, gate=GATE_LOOSE[2], score_mode=score_mode)
    if particles:
        model.update(dim_x=5, q=0.0, model=1, sigma_a=3.0, sigma_w=3.0, ess_frac=0.5)
    return out, model


def _gate_network(rng):
    """Gate parameters with one path through the network that falls with d^2, as training finds, among others that
    hardly weigh; with the threshold below, pairs of d^2 over about 25 leave the table."""
    p = init_params(int(rng.integers(1 << 30)), [0.0, 6.0, 0.8, 8.0, 12.0], [1.0, 8.0, 0.3, 8.0, 3.0])
    W1, b1, W2, b2 = p[:320].reshape(64, 5), p[320:384], p[384:4480].reshape(64, 64), p[4480:4544]
    W3, w4 = p[4544:8640].reshape(64, 64), p[8704:8768]
    W1[:, 0] *= 0.1
    W1[0] = [-0.125, 0, 0, 0, 0]
    b1[0] = 6.0
    W2[0], W3[0] = 0, 0
    W2[0, 0] = W3[0, 0] = w4[0] = 1.0
    w4[1:] *= 0.02
    return p, 2.9


# ---------------------------------------------------------------------------
def _capacities(case):
    """Filter capacities as a user sets them: from the scene's size, before its detections are known."""
    kind, n = case["kind"], case["n"]
    if kind == "batch":
        return dict(max_births=64, max_tracks=n + 48, max_meas=int(n * 0.9 * 6 + 4 * 40.0 + 64))
    if kind == "convoy":
        births, meas = n + 16, 5 * n + 16
    elif kind == "ctrv":
        births, meas = 2 * n // min(20, case["frames"]) + 24, 4 * n + 104
    elif case["dim"] == 2:
        births, meas = 2 * n // min(50, case["frames"]) + 24, int(n * 0.9 * 6 + 4 * 20.0 + 64)
    else:
        births, meas = n + 16, 4 * n + 164
    return dict(max_births=births, max_tracks=2 * n + births + 64, max_meas=max(64, meas))


def _log(case, dim_x, scenes=1):
    """Where a tracker keeps a scene's results: rows after a frame's tracks (and a scene's hypotheses) stay zero."""
    c = _capacities(case)
    lead, cap = (scenes, case["frames"]), c["max_tracks"]
    return dict(n=np.zeros(lead, np.int64), labels=np.zeros((*lead, cap, 2), np.int64), r=np.zeros((*lead, cap)),
                mean=np.zeros((*lead, cap, dim_x)), cov=np.zeros((*lead, cap, dim_x, dim_x)),
                pmf=np.zeros((*lead, cap + 1)), retained=np.zeros((scenes, case["h_max"]), np.int64),
                logw=np.zeros((scenes, case["h_max"])), r_clutter=np.zeros((scenes, c["max_meas"])))


def _filter(frames, model, seed, device, **sizes):
    cfg = dict(model, h_up=H_UP, tau=1e-5, seed=seed ^ 0x5EED)
    cfg.update(sizes)
    f = glmb.Filter(cfg)
    work = []
    for births, Z in frames:
        Z = np.ascontiguousarray(Z, np.float32)
        work.append((glmb.births_array(births, cfg["dim_x"]), torch.from_numpy(Z).to(DEV) if device else Z))
    return f, work


def prepare(case, seed):
    rng = np.random.default_rng(seed)
    kind = case["kind"]
    if kind == "score" or kind == "train":
        return _prepare_gate(case, rng)
    if kind == "select":
        # children of a frame: parents' weights times the factors of a few deviating associations
        lw = 3.0 * rng.normal(size=case["n"]) - rng.exponential(4.0, case["n"])
        lw[rng.random(case["n"]) < 0.3] = -np.inf          # duplicates
        fn = glmb.load().glmb_select_top_static
        p = ctypes.c_void_p
        fn.argtypes, fn.restype = [p, ctypes.c_int64, ctypes.c_int32, ctypes.c_double, p, p, p, p], ctypes.c_int
        h = case["h_max"]
        return dict(case=case, fn=fn, logw=torch.from_numpy(lw).to(DEV),
                    idx=torch.full((h,), -1, dtype=torch.int64, device=DEV),
                    out=torch.zeros(h, dtype=torch.float64, device=DEV),
                    n=torch.zeros(1, dtype=torch.int32, device=DEV))
    device = bool(case.get("device", False))
    if kind == "batch":
        filters, frames = [], []
        for j in range(case["scenes"]):
            n = int(rng.integers(5, case["n"] + 1))
            lam = float(rng.uniform(5, 40))
            world, model = _cv_frames(rng, 2, n, case["frames"], lam)
            h = int(rng.integers(min(100, case["h_max"]), case["h_max"] + 1))
            f, work = _filter(world, model, seed + j, device, h_max=h, max_components=400 * (n + 48),
                              max_pairs=1 << 20, **_capacities(dict(case, n=n)))
            filters.append(f)
            frames.append(work)
        torch.cuda.synchronize()
        return dict(case=case, filters=filters, frames=[list(w) for w in zip(*frames)],
                    log=_log(case, 4, case["scenes"]))
    n, h = case["n"], case["h_max"]
    sizes = dict(h_max=h, **_capacities(case))
    if kind == "cv" or kind == "gated":
        world, model = _cv_frames(rng, case["dim"], n, case["frames"])
    elif kind == "ctrv":
        world, model = _ctrv_frames(rng, n, case["frames"])
        sizes.update(n_particles=case["particles"], max_components=100 * (n + 64))
    else:
        world, model = _convoy_frames(rng, n, case["frames"], case["particles"], case["score_mode"])
        if case["particles"]:
            sizes.update(n_particles=case["particles"], max_components=h * (2 * n + 64) + 64)
    if kind == "gated":
        model["gate"] = GATE_LOOSE[case["dim"]]
        sizes["max_pairs"] = 1 << 22
    f, work = _filter(world, model, seed, device, **sizes)
    if kind == "gated":
        params, threshold = _gate_network(rng)
        f.set_gate(params, threshold, glmb.Filter.GATE_PRUNE)
    torch.cuda.synchronize()
    return dict(case=case, filter=f, frames=work, log=_log(case, model["dim_x"]))


def _prepare_gate(case, rng):
    n = case["rows"]
    gen = torch.Generator(device=DEV)
    gen.manual_seed(int(rng.integers(1 << 40)))

    def uniform():
        return torch.rand(n, device=DEV, generator=gen)

    # features as the table gives them: d^2, |e|, existence, age, log det S
    X = torch.stack([-6.0 * torch.log1p(-uniform()), -4.0 * torch.log1p(-uniform()) - 4.0 * torch.log1p(-uniform()),
                     uniform(), torch.floor(40 * uniform()),
                     5.0 + 1.5 * torch.randn(n, device=DEV, generator=gen)], 1).contiguous()
    P = torch.from_numpy(init_params(int(rng.integers(1 << 30)), [6.0, 8.0, 0.5, 20.0, 5.0],
                                     [6.0, 5.7, 0.3, 11.5, 1.5])).to(DEV)
    state = dict(case=case, X=X, P=P, err=torch.zeros(1, dtype=torch.int32, device=DEV))
    if case["kind"] == "train":
        y = ((X[:, 0] < 9.0) & (uniform() < 0.8)).float()
        npos = y.sum().clamp(min=1.0)
        # parameters and Adam moments of a run in progress, in one buffer
        m = 1e-3 * torch.randn(glmb.GATE_NTRAIN, device=DEV, generator=gen)
        v = 1e-6 * (0.1 + torch.rand(glmb.GATE_NTRAIN, device=DEV, generator=gen))
        saved = torch.cat([P, m, v])
        live = saved.clone()
        a, b = glmb.GATE_NPARAM, glmb.GATE_NPARAM + glmb.GATE_NTRAIN
        state.update(y=y, wt=torch.where(y > 0.5, 0.5 / npos, 0.5 / (n - npos).clamp(min=1.0)).contiguous(),
                     saved=saved, live=live, P=live[:a], m=live[a:b], v=live[b:],
                     grad=torch.zeros(glmb.GATE_NPARAM, device=DEV),
                     loss=torch.zeros(1, dtype=torch.float64, device=DEV))
    return state


def _keep_frame(log, scene, frame, f):
    cap = f.cfg["max_tracks"]
    est = f.estimates(cap=cap, pmf_cap=cap + 1)
    n = log["n"][scene, frame] = est["n"]
    for k in ("labels", "r", "mean", "cov"):
        log[k][scene, frame, :n] = est[k]
    log["pmf"][scene, frame, : cap + 1] = est["pmf"]


def _keep_end(log, scene, f):
    idx, logw = f.retained()
    log["retained"][scene, : len(idx)], log["logw"][scene, : len(idx)] = idx, logw
    r = f.meas_assoc()
    log["r_clutter"][scene, : len(r)] = r


def run(state):
    kind = state["case"]["kind"]
    if kind == "score":
        return glmb.mlp_forward(state["P"], state["X"], state["err"])
    if kind == "train":
        state["live"].copy_(state["saved"])                # the checkpoint the step starts from
        glmb.mlp_backward(state["P"], state["X"], state["y"], state["wt"], state["grad"], state["loss"], state["err"])
        glmb.mlp_adam(state["P"], state["grad"], state["m"], state["v"], 100, 2e-3)
        return dict(grad=state["grad"], loss=state["loss"], params=state["P"], m=state["m"], v=state["v"])
    if kind == "select":
        c = state["case"]
        st = state["fn"](state["logw"].data_ptr(), c["n"], c["h_max"], c["tau"], state["idx"].data_ptr(),
                         state["out"].data_ptr(), state["n"].data_ptr(), torch.cuda.current_stream().cuda_stream)
        if st:
            raise glmb.GlmbError(st, "glmb_select_top_static")
        return dict(idx=state["idx"], logw=state["out"], n=state["n"])
    device, log = bool(state["case"].get("device", False)), state["log"]
    fs = state["filters"] if kind == "batch" else [state["filter"]]
    for f in fs:
        f.reset()
    for k, frame in enumerate(state["frames"]):
        if kind == "batch":
            glmb.step_batch(fs, frame, device=device)
        else:
            births, Z = frame
            fs[0].step(births, Z, device=device)
        for j, f in enumerate(fs):
            _keep_frame(log, j, k, f)
    for j, f in enumerate(fs):
        _keep_end(log, j, f)
    return log


# ---------------------------------------------------------------------------
def _parents(case, h_max=None):
    """Hypotheses per frame: the cap, or what the posterior holds above tau (measured on these worlds)."""
    n, h = case["n"], h_max or case["h_max"]
    if case["kind"] == "convoy" or case["kind"] == "ctrv":
        return min(h, 30 * n)
    if case.get("dim", 2) == 2:
        return min(h, 40 * n)
    at = np.interp(math.log(n), np.log([5, 50, 200, 300, 500, 1000]), np.log([50, 1900, 9000, 1000, 42, 9]))
    return min(h, int(math.exp(at)))


def work(case):
    """What a pass cannot do without.  Tracking: detections and births read, estimates written; for each child one
    random number per track and per detection, 25 integer operations each (Philox4x32-10, four numbers a call)."""
    kind = case["kind"]
    if kind == "score":
        n = case["rows"]
        return dict(bytes=24.0 * n, flops=2.0 * n * (5 * 64 + 64 * 64 * 2 + 64))
    if kind == "train":
        n = case["rows"]
        return dict(bytes=28.0 * n + 4 * 6 * glmb.GATE_NTRAIN,
                    flops=2.0 * n * (3 * (5 * 64 + 64 * 64 * 2 + 64) - 5 * 64))
    if kind == "select":
        return dict(bytes=8.0 * case["n"] + 16.0 * case["h_max"], flops=2.0 * case["n"])
    n, frames = case["n"], case["frames"]
    scenes = 1
    h = case["h_max"]
    if kind == "batch":
        scenes, n, h = case["scenes"], 0.5 * case["n"], 0.5 * case["h_max"]
    if kind == "convoy":
        tracks, meas, dx = n + 1.0, 5.0 * n, 4
    elif kind == "ctrv":
        tracks, meas, dx = 0.9 * n, 1.8 * n + 10, 5
    elif case.get("dim", 2) == 2:
        tracks, meas, dx = 0.5 * n, 0.5 * n * 2.25 + 20, 4
    else:
        tracks, meas, dx = 1.0 * n, 2.55 * n + 50, 6
    parents = _parents(dict(case, n=max(n, 1)), max(1, int(h)))
    ops = 25.0 * H_UP * parents * (tracks + meas)
    if kind == "ctrv" or (kind == "convoy" and case["particles"]):
        ops += 200.0 * case["particles"] * tracks * 2
    return dict(bytes=frames * scenes * (4.0 * meas * 3 + 8.0 * tracks * (dx * dx + dx + 2) + 700.0),
                flops=frames * scenes * ops)


# ---------------------------------------------------------------------------
def exact(case, seed):
    """The network's calls and the selection in 64 bits.  None for tracking: a pass is a chain of frames of sampled
    hypotheses, and restating the filter without the library takes minutes a scene."""
    kind = case["kind"]
    if kind == "select":
        lw = prepare(case, seed)["logw"].cpu().numpy()
        ok = np.nonzero(np.isfinite(lw))[0]
        w = lw[ok]
        lse = w.max() + math.log(np.sum(np.exp(w - w.max())))
        ok = ok[w - lse >= math.log(case["tau"])]
        ok = np.sort(ok[np.lexsort((ok, -lw[ok]))[: case["h_max"]]])
        w = lw[ok]
        w = w - (w.max() + math.log(np.sum(np.exp(w - w.max()))))
        out = np.zeros(case["h_max"])
        out[: len(ok)] = w
        return dict(idx=None, logw=out, n=None)
    if kind != "score" and kind != "train":
        return None
    s = prepare(case, seed)

    def rounded(t):
        return t.to(torch.bfloat16).double()

    P = s["P"].double()
    W1, b1 = rounded(P[:320].float()).view(64, 5), P[320:384]
    W2, b2 = rounded(P[384:4480].float()).view(64, 64), P[4480:4544]
    W3, b3 = rounded(P[4544:8640].float()).view(64, 64), P[8640:8704]
    w4, b4, mu, sd = rounded(P[8704:8768].float()), P[8768], P[8769:8774], P[8774:8779]
    step = 1 << 18
    logits, loss = [], 0.0
    g = {k: 0.0 for k in ("W1", "b1", "W2", "b2", "W3", "b3", "w4", "b4")}

    def slope(z):
        return 0.5 * (1 + torch.erf(z / math.sqrt(2))) + z * torch.exp(-0.5 * z * z) / math.sqrt(2 * math.pi)

    for i in range(0, case["rows"], step):
        x = rounded((s["X"][i:i + step].double() - mu) / sd)
        z1 = x @ W1.T + b1
        h1 = rounded(torch.nn.functional.gelu(z1))
        z2 = h1 @ W2.T + b2
        h2 = rounded(torch.nn.functional.gelu(z2))
        z3 = h2 @ W3.T + b3
        h3 = rounded(torch.nn.functional.gelu(z3))
        z = h3 @ w4 + b4
        logits.append(z)
        if kind == "train":
            y, wt = s["y"][i:i + step].double(), s["wt"][i:i + step].double()
            loss = loss + (wt * (torch.nn.functional.softplus(z) - y * z)).sum()
            d = wt * (torch.sigmoid(z) - y)
            d3 = d[:, None] * w4 * slope(z3)
            d2 = (d3 @ W3) * slope(z2)
            d1 = (d2 @ W2) * slope(z1)
            for k, t in (("W1", d1.T @ x), ("b1", d1.sum(0)), ("W2", d2.T @ h1), ("b2", d2.sum(0)),
                         ("W3", d3.T @ h2), ("b3", d3.sum(0)), ("w4", h3.T @ d), ("b4", d.sum())):
                g[k] = g[k] + t
    if kind == "score":
        return torch.cat(logits)
    grad = torch.cat([g[k].reshape(-1) for k in ("W1", "b1", "W2", "b2", "W3", "b3", "w4", "b4")])
    m = 0.9 * s["m"].double() + 0.1 * grad
    v = 0.999 * s["v"].double() + 0.001 * grad * grad
    params = P.clone()
    params[: glmb.GATE_NTRAIN] -= 2e-3 * (m / (1 - 0.9 ** 100)) / (torch.sqrt(v / (1 - 0.999 ** 100)) + 1e-8)
    return dict(grad=torch.cat([grad, torch.zeros(10, dtype=torch.float64, device=DEV)]), loss=loss.reshape(1),
                params=params, m=m, v=v)
