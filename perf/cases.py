"""The work a user of the localizer has it do, as measurable cases.

Every case goes through the public calls of ``paper_1910_00572_gb300``: odometry steps of one
session, steps with a scan, batched ticks, pose readouts, and a served mix.  The sizes are those of
the repository's own workloads and of the paper's tensor, and ragged ones between them.

A session's device memory comes from torch through ``loc_set_allocator``, as in a program that
keeps the belief on the GPU for its own torch code: the two [K][H][W] belief buffers are the first
two allocations of a session, and every propagation writes the one that is not current.  So a pass
returns the whole updated belief without copying it to the host.  The stored tensor is the belief
up to a positive factor (times 2^14 for FP16 storage).
"""
import math
import time

import numpy as np
import torch

import paper_1910_00572_gb300 as loc

CELL = 0.05                                     # metres
R_MAX, N_BEAMS, STRIDE, SIGMA_R = 10.0, 360, 4, 0.1
DENSE_SIGMA_R = 1.0                             # wide, as where furniture moves: every state is scored
TORCH = {"f32": torch.float32, "bf16": torch.bfloat16, "f16": torch.float16}
MULT = {"f32": 1.0, "bf16": 1.0, "f16": 16384.0}


def listed():
    return [
        # one robot, one odometry message at a time (Algorithm 1): the smallest map, where the
        # launch and the latency of one plane after the other count
        {"name": "step_64x64x16_f32", "kind": "step", "H": 64, "W": 64, "K": 16, "storage": "f32"},
        # the paper's own tensor (500 x 500 cells of a floor plan, 128 bins)
        {"name": "step_500x500x128_f32", "kind": "step", "H": 500, "W": 500, "K": 128, "storage": "f32"},
        # the office plan of the single-session benchmark
        {"name": "step_512x512x64_f32", "kind": "step", "H": 512, "W": 512, "K": 64, "storage": "f32"},
        # a map as a mapping run leaves it: an odd width, no row aligned to 16 bytes
        {"name": "step_613x797x48_f32", "kind": "step", "H": 613, "W": 797, "K": 48, "storage": "f32"},
        # a large site in 16-bit storage, FP16 and BF16 (the largest belief in common use here)
        {"name": "step_1816x1816x36_f16", "kind": "step", "H": 1816, "W": 1816, "K": 36, "storage": "f16"},
        {"name": "step_2048x2048x72_bf16", "kind": "step", "H": 2048, "W": 2048, "K": 72, "storage": "bf16"},
        # differential-drive noise: wider along the heading than across it (Eq. 6)
        {"name": "aniso_512x512x64_f32", "kind": "aniso", "H": 512, "W": 512, "K": 64, "storage": "f32"},
        # a step and a sampled scan update (dithering, ray casts, Eq. 9 on the samples)
        {"name": "scan_2048x2048x72_bf16", "kind": "scan", "H": 2048, "W": 2048, "K": 72, "storage": "bf16",
         "n_samples": 4096},
        # a step and a dense scan update (Eq. 9 on every state from the range table)
        {"name": "dense_512x512x64_f32", "kind": "dense", "H": 512, "W": 512, "K": 64, "storage": "f32",
         "n_angles": 384},
        # a step and what a planner reads after it: the pose with its second hypothesis, the belief map
        {"name": "pose_512x512x64_f32", "kind": "pose", "H": 512, "W": 512, "K": 64, "storage": "f32"},
        # a fleet on one GPU: one tick of 32 robots on maps of uneven size, BF16
        {"name": "batch_32_bf16", "kind": "batch", "n": 32, "lo": 128, "hi": 1024, "storage": "bf16", "mix": 3},
        # the serving loop: 100 ms of messages of 12 robots (ten odometry messages each, a scan of
        # every second robot), until all of it is done
        {"name": "serve_12_bf16", "kind": "serve", "n": 12, "lo": 256, "hi": 1024, "storage": "bf16", "mix": 4,
         "n_samples": 1024},
    ]


def _side(rng, lo, hi, odd):
    s = int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))
    return s if odd else max(8, s // 8 * 8)


def draw(rng):
    kind = rng.choice(["step"] * 5 + ["aniso", "scan", "dense", "pose", "batch", "serve"])
    storage = rng.choice(["f32", "bf16", "f16"] if kind == "step" else ["f32", "bf16"])
    if kind in ("batch", "serve"):
        c = {"kind": kind, "n": rng.randint(2, 32 if kind == "batch" else 12), "lo": 128, "hi": rng.choice([256, 512, 1024]),
             "storage": storage, "mix": rng.randrange(1 << 20)}
        if kind == "serve":
            c["n_samples"] = rng.choice([512, 1024, 4096])
        return c
    odd = rng.random() < 0.4
    hi = {"step": 2048, "scan": 2048, "pose": 1024}.get(kind, 768)
    while True:
        c = {"kind": kind, "H": _side(rng, 64, hi, odd), "W": _side(rng, 64, hi, odd), "storage": storage}
        c["K"] = rng.choice([24, 36, 48, 64]) if kind == "dense" else rng.randint(16, 128)
        # no dearer than the largest listed case of its kind
        if c["H"] * c["W"] * c["K"] <= {"step": 120e6, "scan": 120e6, "pose": 60e6}.get(kind, 16.7e6):
            break
    if kind == "scan":
        c["n_samples"] = rng.choice([512, 1024, 4096])
    if kind == "dense":
        c["n_angles"] = c["K"] * rng.randint(2, 6)
    return c


# ------------------------------------------------------------------ inputs, made from the seed

def office(rng, H, W):
    """Rooms of 3 to 8 m with 0.1 m walls and one 0.9 m door each, between corridors of 1.5 to 2.5 m
    (uint8, 1 = occupied)."""
    occ = np.zeros((H, W), np.uint8)

    def bands(n):
        out, pos = [], int(rng.integers(30, 50))
        while pos + 30 < n:
            end = min(pos + int(rng.integers(60, 160)), n - 2)
            out.append((pos, end))
            pos = end + (int(rng.integers(30, 50)) if len(out) % 2 == 0 else 0)
        return out

    for y0, y1 in bands(H):
        for x0, x1 in bands(W):
            occ[y0:y1, x0:x1] = 1
            occ[y0 + 2:y1 - 2, x0 + 2:x1 - 2] = 0
            d = int(rng.integers(2, max(3, x1 - x0 - 20)))
            if rng.random() < 0.5:
                occ[y0:y0 + 2, x0 + d:x0 + d + 18] = 0
            else:
                occ[y1 - 2:y1, x0 + d:x0 + d + 18] = 0
    for _ in range(H * W // 4000):                   # furniture
        y, x, s = int(rng.integers(2, H)), int(rng.integers(2, W)), int(rng.integers(1, 4))
        occ[y:y + s, x:x + s] = 1
    occ[:2] = occ[-2:] = occ[:, :2] = occ[:, -2:] = 1
    return occ


def drive(rng, occ):
    """A loop of 16 odometry messages, eight out and the same way back, about one cell each, from a
    free place; and the eight true poses out.  A little odometry noise (2 % and 0.01 rad)."""
    H, W = occ.shape
    free = np.argwhere(occ == 0)
    for _ in range(300):
        j, i = free[int(rng.integers(len(free)))]
        pose = np.array([(i + 0.5) * CELL, (j + 0.5) * CELL, rng.uniform(-math.pi, math.pi)])
        out, poses, ok = [], [pose], True
        for _ in range(8):
            u, w = rng.uniform(0.6, 1.3) * CELL, rng.uniform(-0.06, 0.06)
            x, y, th = poses[-1]
            x, y = x + u * math.cos(th), y + u * math.sin(th)
            ok &= 0 <= y / CELL < H and 0 <= x / CELL < W and occ[int(y / CELL) % H, int(x / CELL) % W] == 0
            out.append((u, 0.0, w))
            poses.append(np.array([x, y, th + w]))
        if ok:
            break
    back = [(-u * math.cos(w), u * math.sin(w), -w) for u, _, w in reversed(out)]
    odom = np.array(out + back)
    odom[:, :2] *= 1.0 + 0.02 * rng.standard_normal((16, 2))
    odom[:, 2] += 0.01 * rng.standard_normal(16)
    return odom, poses


def scan_at(rng, occ, pose):
    """360 beams from the pose (a quarter-cell march), 5 cm of noise and 5 % dropouts."""
    H, W = occ.shape
    a = pose[2] - math.pi + math.radians(1) * np.arange(N_BEAMS)
    t = np.arange(1, int(R_MAX / CELL) * 4 + 1) * 0.25
    x, y = pose[0] / CELL + np.cos(a)[:, None] * t, pose[1] / CELL + np.sin(a)[:, None] * t
    i, j = np.floor(x).astype(int), np.floor(y).astype(int)
    hit = (i < 0) | (j < 0) | (i >= W) | (j >= H) | (occ[j.clip(0, H - 1), i.clip(0, W - 1)] != 0)
    r = np.where(hit.any(1), t[hit.argmax(1)] * CELL, R_MAX) + 0.05 * rng.standard_normal(N_BEAMS)
    r[rng.random(N_BEAMS) < 0.05] = R_MAX
    return r.clip(0.0, R_MAX).astype(np.float32)


def prior(rng, occ, K, pose, storage):
    """A belief in the middle of localization, on the GPU in FP32: a background over the free cells,
    a dozen hypotheses and the true pose.  Its values are exact in the storage type."""
    H, W = occ.shape
    free = torch.from_numpy((occ == 0).astype(np.float32)).cuda()
    g = torch.Generator("cuda").manual_seed(int(rng.integers(1 << 40)))
    b = torch.rand((K, H, W), generator=g, device="cuda").mul_(free)
    b.mul_(0.02 / (0.5 * K * float(free.sum())))
    cells = np.argwhere(occ == 0)
    spots = [(int(pose[1] / CELL), int(pose[0] / CELL), int(round(pose[2] / (2 * math.pi / K))) % K)]
    spots += [(*map(int, cells[int(rng.integers(len(cells)))]), int(rng.integers(K))) for _ in range(12)]
    for j, i, k in spots:
        s, R = float(rng.uniform(1.0, 3.0)), 12
        j0, j1, i0, i1 = max(0, j - R), min(H, j + R + 1), max(0, i - R), min(W, i + R + 1)
        jj = torch.arange(j0, j1, device="cuda")[:, None] - j
        ii = torch.arange(i0, i1, device="cuda")[None] - i
        blob = torch.exp(-(jj * jj + ii * ii) / (2 * s * s)) * free[j0:j1, i0:i1]
        wgt = float(rng.uniform(0.3, 1.0)) / (2 * math.pi * s * s * 4)
        for d in range(-4, 5):
            b[(k + d) % K, j0:j1, i0:i1] += blob * (wgt * math.exp(-d * d / 4.0))
    b.div_(b.sum(dtype=torch.float64).float())
    if storage != "f32":
        b = (b * MULT[storage]).to(TORCH[storage]).float() / MULT[storage]
    return b


# ------------------------------------------------------------------ sessions on torch's memory

_memory = {}                                    # device pointer -> the tensor that holds it
_taken = []                                     # pointers in the order they were handed out


def _alloc(nbytes, stream):
    t = torch.empty(max(nbytes, 1), dtype=torch.uint8, device="cuda")
    _memory[t.data_ptr()] = t
    _taken.append(t.data_ptr())
    return t.data_ptr()


def _use_torch_memory():
    if not _taken:
        loc.loc_set_allocator(_alloc, lambda p, stream: _memory.pop(p, None))


class Belief:
    """The two belief buffers of a session: the first two allocations since `mark`."""

    def __init__(self, mark, K, H, W, storage):
        e = torch.empty((), dtype=TORCH[storage]).element_size()
        self.both = [_memory[p][:K * H * W * e].view(TORCH[storage]).view(K, H, W) for p in _taken[mark:mark + 2]]
        self.cur = 0

    def stepped(self, n=1):
        self.cur ^= n & 1
        return self.both[self.cur]


def inputs(seed, H, W, K, storage, scans=0):
    """Everything of one robot that comes from the seed: map, odometry loop, prior belief, scans."""
    rng = np.random.default_rng(seed)
    occ = office(rng, H, W)
    odom, poses = drive(rng, occ)
    b0 = prior(rng, occ, K, poses[0], storage)
    return occ, odom, b0, [scan_at(rng, occ, poses[1 + n]) for n in range(scans)]


def loop_scan(scans, t):
    """The scan for where the loop is after t messages: on the way out, or back at the same place."""
    n = t % 16
    return scans[max((n if n <= 8 else 16 - n) - 1, 0)]


SCAN = dict(angle_min=-math.pi, angle_inc=math.radians(1))


class Robot:
    """One session on an office plan, its loop of odometry messages and, where asked for, scans."""

    def __init__(self, seed, H, W, K, storage, scans=0, **kw):
        _use_torch_memory()
        occ, self.odom, b0, self.scans = inputs(seed, H, W, K, storage, scans)
        self.t = 0
        mark = len(_taken)
        self.h = loc.loc_create(occ, loc.loc_params_default(H=H, W=W, K=K, cell_m=CELL, storage=storage,
                                                            stream=loc.torch_stream(), **kw))
        self.belief = Belief(mark, K, H, W, storage)
        loc.loc_set_belief(self.h, b0.cpu().numpy())

    def step(self):
        loc.loc_step(self.h, *self.odom[self.t % 16])
        self.t += 1
        return self.belief.stepped()

    def scan(self):
        return loop_scan(self.scans, self.t)

    def __del__(self):
        if getattr(self, "h", None) is not None:
            loc.loc_destroy(self.h)
            self.h = None


def mix(case):
    """The sizes of a fleet's maps: sides log-uniform, multiples of 8, K of the batched workload."""
    rng = np.random.default_rng(case["mix"])
    out = []
    for _ in range(case["n"]):
        s = int(round(math.exp(rng.uniform(math.log(case["lo"]), math.log(case["hi"]))) / 8)) * 8
        out.append((s, s, int(rng.choice([36, 48, 64, 72]))))
    return out


class Fleet:
    """Sessions of uneven size in one batch."""

    def __init__(self, case, seed):
        self.robots = [Robot(seed * 1000 + n, H, W, K, case["storage"]) for n, (H, W, K) in enumerate(mix(case))]
        self.batch = loc.loc_batch_create([r.h for r in self.robots], tile=3)
        self.odom = np.stack([r.odom for r in self.robots])
        self.t = 0

    def tick(self):
        o = self.odom[:, self.t % 16]
        self.t += 1
        loc.loc_batch_step(self.batch, o[:, 0], o[:, 1], o[:, 2])
        return [r.belief.stepped() for r in self.robots]

    def __del__(self):
        if getattr(self, "batch", None) is not None:
            loc.loc_batch_destroy(self.batch)
            self.batch = None
        self.robots = []


class Served:
    """Sessions of a server; odometry at 100 Hz, a tenth of a loop message each."""

    def __init__(self, case, seed):
        _use_torch_memory()
        sizes = mix(case)
        seen = [inputs(seed * 1000 + n, H, W, K, case["storage"], 8 if n % 2 == 0 else 0) for n, (H, W, K) in enumerate(sizes)]
        priors = [b0.cpu().numpy() for _, _, b0, _ in seen]
        odom = [np.repeat(o, 10, axis=0) / 10.0 for _, o, _, _ in seen]
        self.scans = [scans for _, _, _, scans in seen]
        self.server = loc.loc_server_create(loc.loc_server_params_default(
            hbm_budget_bytes=100e9, storage=case["storage"], tile=3))
        self.ids, self.beliefs = [], []
        for (H, W, K), (occ, _, _, _), b0 in zip(sizes, seen, priors):
            mark = len(_taken)
            sid = loc.loc_server_open(self.server, occ, loc.loc_params_default(
                H=H, W=W, K=K, cell_m=CELL, storage=case["storage"], n_samples=case["n_samples"], min_shift_cells=1.0))
            while loc.loc_server_session(self.server, sid)[0] == loc.LOC_SESSION_PENDING:
                time.sleep(0.0005)
            loc.loc_set_belief(loc.loc_server_session(self.server, sid)[1], b0)
            self.ids.append(sid)
            self.beliefs.append(Belief(mark, K, H, W, case["storage"]))
        loc.loc_server_odometry(self.server, self.ids, 0.0, 0.0, 0.0)      # every robot reports in
        loc.loc_server_drain(self.server)
        self.odom = np.stack(odom)
        self.moved = np.zeros((len(self.ids), 3))          # Algorithm 1's gate: |p| so far, theta
        self.t = 0

    def window(self):
        """100 ms of messages, and their end."""
        for sid, scans in zip(self.ids, self.scans):
            if scans:
                loc.loc_server_scan(self.server, sid, loop_scan(scans, self.t), **SCAN, r_max=R_MAX, beam_stride=STRIDE,
                                    sigma_r=SIGMA_R)
        o = self.odom[:, 10 * (self.t % 16):10 * (self.t % 16) + 10]
        loc.loc_server_odometry(self.server, np.repeat(self.ids, 10), *(o[..., c].ravel() for c in range(3)))
        loc.loc_server_drain(self.server)
        self.t += 1
        return [b.stepped(self.gate(m, msgs)) for b, m, msgs in zip(self.beliefs, self.moved, o)]

    def gate(self, m, msgs):
        """How many of the messages made the session propagate."""
        n = 0
        for u, v, w in msgs:
            c, s = math.cos(m[2]), math.sin(m[2])
            m += (c * u - s * v, s * u + c * v, w)
            if math.hypot(m[0], m[1]) / CELL >= 1.0:
                m[:2] = 0.0
                n += 1
        return n

    def __del__(self):
        if getattr(self, "server", None) is not None:
            loc.loc_server_destroy(self.server)
            self.server = None


# ------------------------------------------------------------------ the cases

ANISO = dict(sigma_xy_cells=1.0, sigma_cross_cells=0.5)


def prepare(case, seed):
    kind = case["kind"]
    if kind == "batch":
        return kind, Fleet(case, seed)
    if kind == "serve":
        return kind, Served(case, seed)
    kw = {"n_samples": case["n_samples"]} if kind == "scan" else ANISO if kind == "aniso" else {}
    r = Robot(seed, case["H"], case["W"], case["K"], case["storage"], scans=8 if kind in ("scan", "dense") else 0, **kw)
    if kind == "dense":
        loc.loc_range_table(r.h, case["n_angles"], R_MAX)
    return kind, r


def run(state):
    kind, s = state
    if kind == "batch":
        return s.tick()
    if kind == "serve":
        return s.window()
    b = s.step()
    if kind == "scan":
        loc.loc_lidar_update(s.h, s.scan(), **SCAN, r_max=R_MAX, beam_stride=STRIDE, sigma_r=SIGMA_R)
    elif kind == "dense":
        loc.loc_lidar_update_dense(s.h, s.scan(), **SCAN, beam_stride=STRIDE, sigma_r=DENSE_SIGMA_R)
    elif kind == "pose":
        e = loc.loc_estimate(s.h, 0.5, 2)
        return {"belief": b, "map": loc.loc_marginal(s.h, loc.LOC_MAP_MAX),
                "state": np.array([e[n] for n in ("k", "j", "i", "second_j", "second_i")], np.int32),
                "pose": np.array([e[n] for n in ("x", "y", "theta")], np.float32),
                "mass": np.array([e[n] for n in ("p", "mass_near", "second_p", "second_ratio")], np.float32)}
    return b


def work(case):
    """Bytes: a belief is read once and written once by a propagation (and by a dense update), read
    once by a sampled scan and by a readout; the map and its correction are 5 bytes a cell."""
    kind = case["kind"]
    e = 4 if case["storage"] == "f32" else 2
    sizes = mix(case) if kind in ("batch", "serve") else [(case["H"], case["W"], case["K"])]
    hw, n = sum(H * W for H, W, _ in sizes), sum(H * W * K for H, W, K in sizes)
    bytes_, flops = 2 * e * n + 5 * hw, 46 * n
    if kind == "aniso":
        flops = 218 * n
    elif kind == "scan":
        bytes_ += e * n
    elif kind == "serve":
        bytes_ += e * sum(H * W * K for H, W, K in sizes[::2])
    elif kind == "dense":
        bytes_ += 2 * e * n + case["n_angles"] * hw
        flops += 3 * 85 * n
    elif kind == "pose":
        bytes_ += e * n + 4 * hw
    return {"bytes": bytes_, "flops": flops}


# ------------------------------------------------------------------ the same in 64 bits

def taps(sigma, r):
    g = [math.exp(-0.5 * (d / sigma) ** 2) for d in range(-r, r + 1)]
    return [x / sum(g) for x in g]


def blur(x, g, dim):
    """1-D convolution with zero boundary."""
    r, n = len(g) // 2, x.shape[dim]
    out = x * g[r]
    for d in range(1, min(r, n - 1) + 1):
        out.narrow(dim, d, n - d).add_(x.narrow(dim, 0, n - d), alpha=g[r + d])
        out.narrow(dim, 0, n - d).add_(x.narrow(dim, d, n - d), alpha=g[r - d])
    return out


def pull(plane, oy, ox):
    """plane[j + oy, i + ox], zero outside the grid."""
    H, W = plane.shape
    out = torch.zeros_like(plane)
    j0, j1, i0, i1 = max(0, -oy), min(H, H - oy), max(0, -ox), min(W, W - ox)
    if j0 < j1 and i0 < i1:
        out[j0:j1, i0:i1] = plane[j0 + oy:j1 + oy, i0 + ox:i1 + ox]
    return out


def propagate(b, M, msg, aniso=False):
    """Algorithm 1 for a first message (theta_t = 0 before it), unnormalised."""
    K = b.shape[0]
    u, v, w = msg
    S = torch.empty_like(b)
    for k in range(K):
        c, s = math.cos(2 * math.pi * k / K), math.sin(2 * math.pi * k / K)
        x, y = -(c * u - s * v) / CELL, -(s * u + c * v) / CELL
        ox, oy = math.floor(x), math.floor(y)
        fx, fy = x - ox, y - oy
        S[k] = (1 - fy) * ((1 - fx) * pull(b[k], oy, ox) + fx * pull(b[k], oy, ox + 1)) \
            + fy * ((1 - fx) * pull(b[k], oy + 1, ox) + fx * pull(b[k], oy + 1, ox + 1))
    S *= M
    gt = taps(1.0, 3)
    C = S * gt[3]
    for d in range(1, 4):
        C += gt[3 + d] * (torch.roll(S, d, 0) + torch.roll(S, -d, 0))
    del S
    if not aniso:
        g = taps(0.5, 2)
        C = blur(blur(C, g, 2), g, 1)
        G = blur(blur(M, g, 1), g, 0)
        return C * torch.where(M > 0, 1.0 / G.clamp_min(1e-300), torch.zeros_like(G))
    d = torch.arange(-3, 4, device="cuda", dtype=torch.float64)
    for k in range(K):
        c, s = math.cos(2 * math.pi * k / K + w), math.sin(2 * math.pi * k / K + w)
        along, across = d[None] * c + d[:, None] * s, d[:, None] * c - d[None] * s
        g = torch.exp(-0.5 * ((along / ANISO["sigma_xy_cells"]) ** 2 + (across / ANISO["sigma_cross_cells"]) ** 2))[None, None]
        T, G = (torch.nn.functional.conv2d(x[None, None], g, padding=3)[0, 0] for x in (C[k], M))
        C[k] = torch.where(M > 0, T / G.clamp_min(1e-300), torch.zeros_like(G))
    return C


def range_codes(M, dirs):
    """The 8-bit expected ranges of every cell along each direction: the grid walk from the cell
    centre, in FP32 as it is defined, to the first occupied cell or the edge."""
    H, W = M.shape
    rmax = np.float32(R_MAX / CELL)
    inv = float(np.float32(255.0) / rmax)
    flat = (M > 0).reshape(-1)
    cell = torch.arange(H * W, device="cuda", dtype=torch.int32)
    out = torch.empty((len(dirs), H * W), dtype=torch.uint8, device="cuda")
    for n in range(0, len(dirs), 32):
        dx, dy = (torch.from_numpy(np.ascontiguousarray(dirs[n:n + 32, c])).cuda()[:, None] for c in (0, 1))
        tdx, tdy = (torch.where(x != 0, 1.0 / x.abs(), torch.full_like(x, math.inf)) for x in (dx, dy))
        sx, sy = (torch.where(x > 0, 1, -1).to(torch.int32) for x in (dx, dy))
        j, i = ((cell // W).expand(len(dx), -1).clone(), (cell % W).expand(len(dx), -1).clone())
        ax, ay = torch.full(j.shape, 0.5, device="cuda"), torch.full(j.shape, 0.5, device="cuda")
        t = torch.zeros(j.shape, device="cuda")
        live = flat[None].expand(len(dx), -1).clone()
        while bool(live.any()):
            tx, ty = ax * tdx, ay * tdy
            in_x = tx <= ty
            i += torch.where(in_x & live, sx, 0)
            j += torch.where(in_x | ~live, 0, sy)
            now = torch.minimum(tx, ty).clamp_max(float(rmax))
            t = torch.where(live, now, t)
            ax += (in_x & live).float()
            ay += (~in_x & live).float()
            inside = (i >= 0) & (i < W) & (j >= 0) & (j < H)
            live &= inside & (now < float(rmax)) & flat[(j.clamp(0, H - 1) * W + i.clamp(0, W - 1)).long()]
        out[n:n + 32] = torch.floor(t * inv + 0.5).clamp_max(255.0).to(torch.uint8)
    return out.view(len(dirs), H, W)


def dense(X, M, z, theta, A):
    """Eq. 9 on every state from the table of A directions; the most probable state becomes 1."""
    K = X.shape[0]
    a = 2 * math.pi / A * np.arange(A)
    codes = range_codes(M, np.stack([np.cos(a), np.sin(a)], 1).astype(np.float32))
    step = float(np.float32(R_MAX / 255.0))
    k = torch.arange(K, device="cuda") * (A // K)
    L = torch.zeros_like(X)
    for b in range(0, N_BEAMS, STRIDE):
        if z[b] < R_MAX:
            m = math.floor((theta + (SCAN["angle_min"] + SCAN["angle_inc"] * b)) / (2 * math.pi / A) + 0.5)
            L -= (float(z[b]) - codes[(k + m) % A].double() * step) ** 2 / (2 * DENSE_SIGMA_R ** 2)
    L += X.log()
    L -= L.masked_fill(M.expand_as(L) == 0, -math.inf).max()
    return L.exp() * M


def exact_robot(seed, case, H, W, K):
    storage = case["storage"]
    occ, odom, b0, scans = inputs(seed, H, W, K, storage, 8 if case["kind"] == "dense" else 0)
    M = torch.from_numpy((occ == 0).astype(np.float64)).cuda()
    b = b0.double()
    del b0
    X = propagate(b.div_(b.sum()), M, odom[0], case["kind"] == "aniso")
    if case["kind"] == "dense":
        X = dense(X, M, loop_scan(scans, 1), odom[0][2], case["n_angles"])
    return X.mul_(MULT[storage])


def exact(case, seed):
    """None where a dithering decides: which cells are sampled hangs on the last bit of every value."""
    if case["kind"] in ("scan", "serve"):
        return None
    if case["kind"] == "batch":
        return [exact_robot(seed * 1000 + n, case, H, W, K) for n, (H, W, K) in enumerate(mix(case))]
    X = exact_robot(seed, case, case["H"], case["W"], case["K"])
    if case["kind"] != "pose":
        return X
    K, H, W = X.shape
    b = X / X.sum()
    a = int(b.argmax())
    k, j, i = a // (H * W), a // W % H, a % W
    p = float(b[k, j, i])
    jj, ii = torch.arange(H, device="cuda")[:, None] - j, torch.arange(W, device="cuda")[None] - i
    disk = jj * jj + ii * ii <= int(0.5 ** 2 / CELL ** 2 + 1e-9)
    near = [(k + d) % K for d in range(-2, 3)]
    second = float(b.amax(0).masked_fill(disk, 0.0).max())
    return {"belief": X, "map": b.amax(0), "state": None, "pose": None,
            "mass": np.array([p, float((b[near] * disk).sum()), second, second / p])}
