"""The work that users of the tracking library have it do, as measurable cases.

Each case is one pass through the public entry points of
`paper_2207_10940_gb300.dri`: a camera frame (or one frame of each of many
cameras) goes in with its IMU samples and the new state comes out.  `listed`
names the cases, `draw` gives more of the same ranges, `prepare` is what a
program has in hand before the call, `run` is the call, `work` its unavoidable
bytes and operations, `exact` the same results in plain 64-bit numpy / torch.

Inputs are looped sequences: a camera moves along a one-second sinusoidal path
(30 frames; peak 1.5 m/s and 90 deg/s, the serving benchmark's motion) through
a box room with spheres and a value-noise texture, with the sensors' noise.
Every pass takes the next frame.

Results are returned in FP32, the precision of the images and of the pixel
arithmetic they come from; the states' FP64 fields carry no more than that.
"""
from __future__ import annotations

import ctypes
import math

import numpy as np
import torch

from paper_2207_10940_gb300 import dri, synth

PERIOD = 30                     # frames of one loop (1 s at 30 frames/s)
FPS = 30.0
RATE = 400                      # IMU samples per second

# Levels and Gauss-Newton iterations per level, finest first: the frame-pair
# and the sequence configurations of the benchmark.
SCHEDULES = {2: (10, 5), 3: (10, 5, 4)}

# First-frame prior of a calibrated rig: pose, velocity, gyro and accelerometer bias, gravity.
PRIOR = (1e-6, 0.05, 1e-3, 5e-3, 2e-3)


# ---------------------------------------------------------------------------
# cases
# ---------------------------------------------------------------------------

def _case(kind, **kw):
    c = dict(kind=kind, sizes="640x480", count=1, levels=3, flags=0, mode="inertial", gravity=2,
             first_order=0, occlusion=0.0, depth_weight=0, pinned=0, rows="")
    c.update(kw)
    return c


def listed():
    return [
        # one linearisation of a small pair inside a real-time callback that may not allocate
        _case("pair", name="pair 160x120", sizes="160x120", levels=1),
        # the same at that entry's size limit, with its optional terms
        _case("pair", name="pair 320x240 options", sizes="320x240", levels=1, occlusion=0.05, depth_weight=1),
        # one low-resolution camera, the frame-pair schedule: the smallest tracked frame
        _case("track", name="track 320x240", sizes="320x240", levels=2),
        # the benchmark's single camera, frames arriving in pinned host memory
        _case("track", name="track 640x480 host", sizes="640x480", pinned=1),
        # one large camera of ragged size (no row is aligned beyond 4 bytes)
        _case("track", name="track 1277x717", sizes="1277x717"),
        # the vision-only baseline with the occlusion test and depth-dependent weight
        _case("track", name="track rgbd 501x377", sizes="501x377", mode="rgbd", occlusion=0.05, depth_weight=1),
        # frame-to-model tracking: every frame against a prediction rendered by a map
        _case("model", name="model 640x480", sizes="640x480"),
        # a small rig of odd cameras with first-order biases and reduced-precision maps
        _case("batch", name="batch 6 odd fp16", sizes="333x251,417x313", count=6, flags=3, first_order=1, rows="16,4,2"),
        # a dozen ordinary cameras, too few to fill the chip, in a program that wants the
        # same bits on every run: it fixes the rows per thread that the tuner once chose
        _case("batch", name="batch 12x 320x240", sizes="320x240", count=12, rows="16,8,4"),
        # the benchmark's headline batch
        _case("batch", name="batch 64x 640x480", sizes="640x480", count=64),
        # the benchmark's uneven batch: 24 small, 32 middle, 8 large
        _case("batch", name="batch mixed 64", sizes="320x240*3,640x480*4,1280x720*1", count=64),
        # the serving loop with cameras of three resolutions, one request each per pass
        _case("serve", name="serve 96 mixed", sizes="320x240,640x480,1280x720", count=96),
    ]


def _size(rng, lo, hi):
    """A camera size of lo .. hi pixels (log-uniform), aspect 4:3 to 16:9; half of them odd."""
    n = math.exp(rng.uniform(math.log(lo), math.log(hi)))
    a = rng.uniform(4 / 3, 16 / 9)
    w, h = int(math.sqrt(n * a)), int(math.sqrt(n / a))
    if rng.random() < 0.5:
        w, h = w // 16 * 16, h // 16 * 16
    return w, h


def draw(rng):
    kind = rng.choice(["pair", "track", "track", "model", "batch", "batch", "serve"])
    kw = dict(levels=rng.choice([2, 3]), flags=rng.choice([0, 0, 0, 1, 2, 3]))
    if rng.random() < 0.3:
        kw.update(occlusion=round(rng.uniform(0.03, 0.1), 3), depth_weight=rng.choice([0, 1]))
    if kind == "pair":
        w, h = _size(rng, 96 * 72, 320 * 239)
        return _case(kind, sizes="%dx%d" % (min(w, 320), min(h, 240)), **dict(kw, levels=1))
    if rng.random() < 0.25:
        kw.update(first_order=1)
    if kind in ("track", "model"):
        mode = rng.choice(["inertial", "inertial", "gyro", "rgbd"])
        kw.update(mode=mode, gravity=3 if mode == "inertial" and rng.random() < 0.2 else 2, pinned=rng.choice([0, 1]))
        return _case(kind, sizes="%dx%d" % _size(rng, 160 * 120, 1280 * 720), **kw)
    sizes = [_size(rng, 160 * 120, 1280 * 720) for _ in range(rng.choice([1, 2, 3]))]
    px = sum(w * h for w, h in sizes) / len(sizes)
    most = max(4, min(96, int(48 * 640 * 480 / px)))
    n = int(math.exp(rng.uniform(math.log(4), math.log(most + 0.99))))
    if kind == "batch" and n * px < 24 * 640 * 480:
        kw.update(rows="16,8,4")
    return _case(kind, sizes=",".join("%dx%d" % s for s in sizes), count=n, **kw)


def _sizes(case):
    """Size of each camera: the listed sizes in turn, each as often as its '*k' says."""
    turn = []
    for s in case["sizes"].split(","):
        wh, _, k = s.partition("*")
        w, h = wh.split("x")
        turn += [(int(w), int(h))] * int(k or 1)
    return [turn[i % len(turn)] for i in range(case["count"])]


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------

class _Scene:
    """One camera's looped sequence: images, IMU samples and the path's states."""

    def __init__(self, seed, w, h, want_model, pinned, n_frames):
        self.w, self.h = w, h
        self.cam = synth.scaled_camera(w, h)
        seq = synth.sinusoid_sequence(seed=seed, cam=self.cam, n_frames=PERIOD, fps=FPS, rate=RATE,
                                      period_frames=PERIOD, render_frames=False)
        self.seq = seq
        dev = torch.device("cuda")
        gen = torch.Generator(dev).manual_seed(1000003 * (seed % 1000003) + w * 4096 + h)
        sc = seq.scene
        lo = torch.tensor(sc.lo, device=dev, dtype=torch.float64)
        hi = torch.tensor(sc.hi, device=dev, dtype=torch.float64)
        texture = []
        for octave in range(4):
            n = [max(2, int(math.ceil(float(e) * 4 * 2 ** octave))) for e in (sc.hi - sc.lo)]
            texture.append(torch.rand((1, 1, n[2], n[1], n[0]), device=dev, generator=gen))
        u = (torch.arange(w, device=dev, dtype=torch.float64) - self.cam.cx) / self.cam.fx
        v = (torch.arange(h, device=dev, dtype=torch.float64) - self.cam.cy) / self.cam.fy
        ray = torch.stack([u.expand(h, w), v[:, None].expand(h, w), torch.ones(h, w, device=dev, dtype=torch.float64)], -1)
        self.depth, self.inten, self.model = [], [], []
        for k in range(n_frames):
            g = seq.gt[k]
            R = torch.tensor(seq.R_IW @ g["R_WC"], device=dev)
            o = torch.tensor(seq.R_IW @ g["r_WC"], device=dev)
            d = ray @ R.T
            wall = torch.where(d > 0, (hi - o) / d, (lo - o) / d)
            t, axis = wall.min(-1)
            normal = -torch.sign(d) * torch.nn.functional.one_hot(axis, 3)
            a = (d * d).sum(-1)
            for cen, r in zip(sc.centers, sc.radii):
                c = torch.tensor(cen, device=dev)
                b = d @ (o - c)
                disc = b * b - a * (float((o - c) @ (o - c)) - float(r) ** 2)
                ts = (-b - disc.clamp(min=0).sqrt()) / a
                hit = (disc >= 0) & (ts > 1e-9) & (ts < t)
                t = torch.where(hit, ts, t)
                normal = torch.where(hit[..., None], (o + d * t[..., None] - c) / float(r), normal)
            pts = o + d * t[..., None]
            grid = ((pts - lo) / (hi - lo) * 2 - 1).float()[None, None]
            tex, norm = 0.0, 0.0
            for octave, vol in enumerate(texture):
                tex = tex + 0.5 ** octave * torch.nn.functional.grid_sample(vol, grid, padding_mode="border", align_corners=False)[0, 0, 0]
                norm += 0.5 ** octave
            clean = 0.1 + 0.8 * tex / norm
            noise = torch.randn((2, h, w), device=dev, generator=gen)
            self.depth.append((t.float() + 0.002 * noise[0]).contiguous())
            self.inten.append((clean + 0.01 * noise[1]).clamp(0, 1).contiguous())
            if want_model:                     # the same view as a map's prediction, in W
                RW = torch.tensor(seq.R_IW, device=dev)
                self.model.append(((pts @ RW).float().contiguous(), (normal @ RW).float().contiguous(),
                                   clean.contiguous(), np.concatenate([g["r_WC"], g["q_WC"]])))
        if pinned:
            self.depth = [d.cpu().pin_memory() for d in self.depth]
            self.inten = [i.cpu().pin_memory() for i in self.inten]
        # one period of samples; sample j of any later period repeats sample j % RATE
        rng = np.random.default_rng([seed, 7])
        rows = synth.imu_samples(seq.traj, RATE, 0.0, 1.0, seq.bg, seq.ba, rng)
        j = np.rint(rows[:, 0] * RATE).astype(int)
        self.imu = np.zeros((RATE, 7))
        self.imu[j[(j >= 0) & (j < RATE)]] = rows[(j >= 0) & (j < RATE)]

    def samples(self, a, b):
        """IMU samples with indices a .. b - 1 (time j / RATE)."""
        j = np.arange(a, b)
        s = self.imu[j % RATE]
        s[:, 0] = j / RATE
        return s

    def start_state(self, k0):
        """What a program whose rig was calibrated at a standstill knows when the camera
        starts at frame k0: identity pose, the velocity, and the biases and gravity
        direction to within PRIOR."""
        g = self.seq.gt[k0]
        return dict(t=k0 / FPS, r_WC=np.zeros(3), q_WC=np.array([1.0, 0, 0, 0]), v_I=g["v_I"], bg=0.9 * self.seq.bg,
                    ba=0.95 * self.seq.ba, q_IW=synth.matrix_to_quat(self.seq.R_IW @ g["R_WC"]))


def _cameras(case, seed, n_frames=PERIOD):
    """(scene, first frame) of each camera; cameras of one size share a scene and
    start at different places of its loop."""
    scenes, out = {}, []
    for i, (w, h) in enumerate(_sizes(case)):
        if (w, h) not in scenes:
            scenes[w, h] = _Scene(seed + 17 * len(scenes), w, h, case["kind"] == "model", case["pinned"], n_frames)
        out.append((scenes[w, h], 0 if case["count"] == 1 else (7 * i) % PERIOD))
    return out


def _config(case, scene):
    c = scene.cam
    modes = dict(inertial=dri.DRI_TRACK_INERTIAL, rgbd=dri.DRI_TRACK_RGBD_ONLY, gyro=dri.DRI_TRACK_GYRO_ONLY)
    return dri.config_for(c.width, c.height, c.fx, c.fy, c.cx, c.cy, case["levels"],
                          SCHEDULES.get(case["levels"], (10,)), q_CS=synth.matrix_to_quat(scene.seq.R_CS),
                          r_CS=scene.seq.r_CS, prior_sigma=PRIOR, precision_flags=case["flags"], track_mode=modes[case["mode"]],
                          gravity_dof=dri.DRI_GRAVITY_3D if case["gravity"] == 3 else dri.DRI_GRAVITY_2DOF,
                          imu_mode=dri.DRI_IMU_FIRST_ORDER if case["first_order"] else dri.DRI_IMU_REINTEGRATE,
                          occlusion_thr=case["occlusion"], icp_depth_weight=case["depth_weight"])


RESULT = np.dtype([("x1", "f8", 20), ("t1", "f8"), ("x0", "f8", 20), ("t0", "f8"), ("n_icp", "i4", 4),
                   ("n_rgb", "i4", 4), ("n_margin", "i4", 4), ("cost", "f8"), ("status", "i4"), ("initialised", "i4")])


class _State:
    """Open streams (or a server) and where each is in its loop."""

    def __init__(self, case, seed):
        self.case = case
        self.server = self.streams = None
        self.cams = _cameras(case, seed)
        self.pixels = np.array([[max(1, (s.w >> l) * (s.h >> l)) for l in range(4)] for s, _ in self.cams], dtype=np.float64)
        self.cuda_stream = torch.cuda.Stream()
        torch.cuda.synchronize()
        inits = [dri.state_from_dict(s.start_state(k)) for s, k in self.cams]
        if case["kind"] == "serve":
            self.server = dri.dri_server_create(120 << 30, 256, self.cuda_stream)
            self.handles = [dri.dri_server_open_stream(self.server, _config(case, s), x) for (s, _), x in zip(self.cams, inits)]
        else:
            self.streams = [dri.Stream(_config(case, s), x, self.cuda_stream) for (s, _), x in zip(self.cams, inits)]
            self.handles = [s.handle for s in self.streams]
        if case["rows"]:
            dri.dri_batch_set_options(self.streams, rows_per_thread=[int(r) for r in case["rows"].split(",")][:case["levels"]])
        self.frame = [k for _, k in self.cams]
        self.pushed = [max(0, k * RATE // int(FPS) - 1) for _, k in self.cams]

    def imu_ahead(self, i):
        """Samples not yet handed over when camera i's next frame needs them: the
        recorded sequence is played back a second at a time."""
        need = self.frame[i] * RATE // int(FPS) + 2
        if need < self.pushed[i]:
            return None
        a, self.pushed[i] = self.pushed[i], need + RATE
        return dri.imu_array(self.cams[i][0].samples(a, self.pushed[i]))

    def step(self):
        case, cams = self.case, self.cams
        if self.server is not None:
            tickets = []
            for i, h in enumerate(self.handles):
                scene, k = cams[i][0], self.frame[i]
                imu = self.imu_ahead(i)
                tickets.append(dri.dri_server_submit(self.server, h, k / FPS, scene.depth[k % PERIOD], scene.inten[k % PERIOD], () if imu is None else imu))
                self.frame[i] = k + 1
            results = [dri.dri_server_poll(self.server, t)[1] for t in tickets]
        else:
            for i, h in enumerate(self.handles):
                scene, k = cams[i][0], self.frame[i]
                imu = self.imu_ahead(i)
                if imu is not None:
                    dri.dri_push_imu(h, imu)
                if case["kind"] == "model" and k > cams[i][1]:
                    V, N, I, T = scene.model[(k - 1) % PERIOD]
                    dri.dri_upload_reference(h, V, N, I, T)
                dri.dri_upload_frame(h, k / FPS, scene.depth[k % PERIOD], scene.inten[k % PERIOD])
                self.frame[i] = k + 1
            results = [dri.dri_track(self.handles[0])] if case["kind"] != "batch" else dri.dri_track_batch(self.streams)
        r = np.frombuffer(b"".join(results), dtype=RESULT)
        L = case["levels"]
        # per level the share of the pixels that took part, as a program watches it
        return dict(x1=r["x1"].astype(np.float32), x0=r["x0"].astype(np.float32), cost=r["cost"].astype(np.float32),
                    inliers=np.stack([r["n_icp"][:, :L] / self.pixels[:, :L], r["n_rgb"][:, :L] / self.pixels[:, :L]], -1).astype(np.float32),
                    status=r["status"].copy())

    def __del__(self):
        try:
            if self.server is not None:
                dri.dri_server_destroy(self.server)
            for s in self.streams or ():
                s.close()
        except Exception:
            pass


def _warm_frames(case):
    """Frames a long-running program has tracked before the measured one, beyond the
    first: a batch's plan times its launch options on the first two unless they are fixed."""
    return 2 if case["kind"] in ("batch", "serve") and not case["rows"] else 0


def _pair_states(case, scene):
    """Where the pair is linearised: the reference at the first pose, the live frame a
    little beside the second."""
    g0, g1 = scene.seq.gt[0], scene.seq.gt[1]
    x = []
    for g, dr, da in ((g0, 0.0, 0.0), (g0, 2e-4, 1e-4), (g1, -3e-3, 2e-3)):
        q = _quat_mul(_quat_exp(np.array([da, -da, 0.5 * da])), g["q_WC"])
        x.append(dict(t=0.0, r_WC=g["r_WC"] + dr, q_WC=q, v_I=g["v_I"], bg=np.zeros(3), ba=np.zeros(3), q_IW=g["q_IW"]))
    return x


def prepare(case, seed):
    if case["kind"] != "pair":
        st = _State(case, seed)
        for _ in range(1 + _warm_frames(case)):
            st.step()
        return st
    (scene, _), = _cameras(case, seed, 2)
    out = torch.zeros(ctypes.sizeof(dri.dri_linearisation), dtype=torch.uint8, device="cuda")
    return dict(case=case, cfg=_config(case, scene), scene=scene, out=out, x=[dri.state_from_dict(x) for x in _pair_states(case, scene)],
                cuda_stream=torch.cuda.current_stream())


def run(state):
    if isinstance(state, _State):
        return state.step()
    s, out = state["scene"], state["out"]
    dri.dri_linearise_pair_noalloc(state["cfg"], s.depth[0], s.inten[0], s.depth[1], s.inten[1], *state["x"], out, None, state["cuda_stream"])
    f = out.view(torch.float64)
    o = 34 * 34 + 34
    r = f[o:o + 86].float()
    return dict(systems=r[:84], cost=r[84:], n=out.view(torch.int64)[-4:-2])


# ---------------------------------------------------------------------------
# unavoidable work
# ---------------------------------------------------------------------------

def work(case):
    """Bytes: the live and the reference depth and intensity read once (what a model
    prediction holds instead: 28 bytes per pixel) and the result.  Operations: the two
    terms' residuals, Jacobians and 29 sums each, about 2 x 130 per pixel and
    iteration, the normals and gradients (60 per pixel), and per Gauss-Newton step the
    joint system's assembly and factorisation (about 40 thousand)."""
    b = f = 0
    iters = SCHEDULES.get(case["levels"], (10,)) if case["kind"] != "pair" else (1,)
    for w, h in _sizes(case):
        b += w * h * (8 + (28 if case["kind"] == "model" else 8)) + 400
        for l, it in enumerate(iters):
            f += (w >> l) * (h >> l) * (260 * it + 60)
        f += 0 if case["kind"] == "pair" else 40000 * sum(iters)
    return {"bytes": b, "flops": f}


# ---------------------------------------------------------------------------
# the same results in 64 bits
# ---------------------------------------------------------------------------

def _hat(w):
    return np.array([[0, -w[2], w[1]], [w[2], 0, -w[0]], [-w[1], w[0], 0]], dtype=np.float64)


def _exp(w):
    t = np.linalg.norm(w)
    K = _hat(w)
    if t < 1e-4:
        return np.eye(3) + (1 - t * t / 6) * K + (0.5 - t * t / 24) * (K @ K)
    return np.eye(3) + math.sin(t) / t * K + (1 - math.cos(t)) / t ** 2 * (K @ K)


def _log(R):
    v = 0.5 * np.array([R[2, 1] - R[1, 2], R[0, 2] - R[2, 0], R[1, 0] - R[0, 1]])
    s = np.linalg.norm(v)
    return v * (1 + s * s / 6) if s < 1e-4 else v * (math.atan2(s, 0.5 * (np.trace(R) - 1)) / s)


def _jr(w):
    t = np.linalg.norm(w)
    K = _hat(w)
    if t < 1e-3:
        return np.eye(3) - (0.5 - t * t / 24) * K + (1 / 6 - t * t / 120) * (K @ K)
    return np.eye(3) - (1 - math.cos(t)) / t ** 2 * K + (t - math.sin(t)) / t ** 3 * (K @ K)


def _quat_exp(w):
    t = np.linalg.norm(w)
    s = 0.5 - t * t / 48 if t < 1e-4 else math.sin(t / 2) / t
    return np.concatenate([[math.cos(t / 2)], s * w])


def _quat_mul(a, b):
    return np.concatenate([[a[0] * b[0] - a[1:] @ b[1:]], a[0] * b[1:] + b[0] * a[1:] + np.cross(a[1:], b[1:])])


def _rot(q):
    w, v = q[0], q[1:]
    return (w * w - v @ v) * np.eye(3) + 2 * np.outer(v, v) + 2 * w * _hat(v)


class _X:
    """A state of Eq. 1; d has 18 entries (position, rotation, velocity, biases, gravity)."""

    def __init__(self, r, q, v, bg, ba, qg):
        self.r, self.q, self.v, self.bg, self.ba, self.qg = (np.array(a, dtype=np.float64) for a in (r, q, v, bg, ba, qg))
        self.q /= np.linalg.norm(self.q)
        self.qg /= np.linalg.norm(self.qg)
        self.R, self.G = _rot(self.q), _rot(self.qg)

    def plus(self, d):
        return _X(self.r + d[:3], _quat_mul(_quat_exp(d[3:6]), self.q), self.v + d[6:9], self.bg + d[9:12], self.ba + d[12:15],
                  _quat_mul(_quat_exp(d[15:18]), self.qg))

    def minus(self, o):
        return np.concatenate([self.r - o.r, _log(self.R @ o.R.T), self.v - o.v, self.bg - o.bg, self.ba - o.ba, _log(self.G @ o.G.T)])

    def vector(self):
        return np.concatenate([self.r, self.q, self.v, self.bg, self.ba, self.qg])


class _Level:
    """Maps of one image at one pyramid level, 64-bit values of the stored FP32 ones."""

    def __init__(self, cfg, l, depth, inten, normals=None):
        s = 2.0 ** l
        self.fx, self.fy = cfg.fx / s, cfg.fy / s
        self.cx, self.cy = (cfg.cx + 0.5) / s - 0.5, (cfg.cy + 0.5) / s - 0.5
        self.h, self.w = depth.shape
        d = self.d = depth.double()
        self.I = inten.double()
        dev = d.device
        self.rx = (torch.arange(self.w, device=dev, dtype=torch.float64) - self.cx) / self.fx
        self.ry = ((torch.arange(self.h, device=dev, dtype=torch.float64) - self.cy) / self.fy)[:, None]
        self.V = torch.stack([d * self.rx, d * self.ry, d], -1)
        self.ok = (d >= cfg.depth_min) & (d <= cfg.depth_max)
        if normals is None:
            N = torch.zeros_like(self.V)
            c = torch.linalg.cross(self.V[:-1, 1:] - self.V[:-1, :-1], self.V[1:, :-1] - self.V[:-1, :-1])
            n = c.norm(dim=-1, keepdim=True)
            good = self.ok[:-1, :-1] & self.ok[:-1, 1:] & self.ok[1:, :-1] & (n[..., 0] > 0)
            c = c / n.clamp(min=1e-300)
            c = torch.where((c * self.V[:-1, :-1]).sum(-1, keepdim=True) > 0, -c, c)
            N[:-1, :-1] = torch.where(good[..., None], c, torch.zeros_like(c))
            normals = N
        self.N = normals
        g = torch.zeros((self.h, self.w, 2), device=dev, dtype=torch.float64)
        g[1:-1, 1:-1, 0] = 0.5 * (self.I[1:-1, 2:] - self.I[1:-1, :-2])
        g[1:-1, 1:-1, 1] = 0.5 * (self.I[2:, 1:-1] - self.I[:-2, 1:-1])
        self.IG = torch.cat([self.I[..., None], g], -1)


def _half_size(cfg, d, I, N=None):
    """The next level's stored FP32 images (and, for a prediction, normals)."""
    h, w = d.shape[0] // 2, d.shape[1] // 2
    s, n = torch.zeros((h, w), device=d.device), torch.zeros((h, w), device=d.device)
    for y in (0, 1):
        for x in (0, 1):
            v = d[y:2 * h:2, x:2 * w:2]
            s, n = torch.where(v > 0, s + v, s), n + (v > 0)
    d2 = torch.where(n > 0, s / n.clamp(min=1), torch.zeros_like(s))
    I2 = ((I[0:2 * h:2, 0:2 * w:2] + I[0:2 * h:2, 1:2 * w:2]) + (I[1:2 * h:2, 0:2 * w:2] + I[1:2 * h:2, 1:2 * w:2])) * 0.25
    if N is not None:
        N = N[:2 * h, :2 * w].reshape(h, 2, w, 2, 3).sum((1, 3))
        N = N / N.norm(dim=-1, keepdim=True).clamp(min=1e-300)
        N = N * ((d2 >= cfg.depth_min) & (d2 <= cfg.depth_max))[..., None]
    return d2, I2, N


def _levels(cfg, depth, inten, normals=None):
    d, I, N = depth.float().cuda(), inten.float().cuda(), normals
    out = []
    for l in range(cfg.levels):
        if l:
            d, I, N = _half_size(cfg, d, I, N)
        out.append(_Level(cfg, l, d, I, N))
    return out


def _project(c, p, R, r):
    """Points p (live camera) in the reference camera by p_ref = R p + r, and their pixels."""
    q = p @ torch.as_tensor(R, device=p.device).T + torch.as_tensor(r, device=p.device)
    z = torch.where(q[..., 2] > 0, q[..., 2], torch.ones_like(q[..., 2]))
    return q, z, c.fx * q[..., 0] / z + c.cx, c.fy * q[..., 1] / z + c.cy


def _sums(J, e, ok):
    J, e = J[ok], e[ok]
    return (J.T @ J).cpu().numpy(), -(J.T @ e).cpu().numpy(), float(e @ e), int(ok.sum())


def _pixel_terms(cfg, cur, ref, T, x0, x1):
    """Both terms at (x0, x1) in world coordinates: 6x6 systems on x1's pose (unweighted
    sums), the photometric one also on x0's."""
    R_ref, r_ref = T
    live = cur.ok
    q, z, xr, yr = _project(ref, cur.V, R_ref.T @ x1.R, R_ref.T @ (x1.r - r_ref))
    xi, yi = torch.floor(xr + 0.5), torch.floor(yr + 0.5)
    ok = live & (q[..., 2] > 0) & (xi >= 0) & (xi < ref.w) & (yi >= 0) & (yi < ref.h)
    at = (yi.clamp(0, ref.h - 1).long(), xi.clamp(0, ref.w - 1).long())
    N, V = ref.N[at], ref.V[at]
    n1 = cur.N @ torch.as_tensor(R_ref.T @ x1.R, device=q.device).T
    diff = q - V
    ok = ok & ref.ok[at] & (N.abs().sum(-1) > 0) & (cur.N.abs().sum(-1) > 0) & (diff.norm(dim=-1) < cfg.icp_dist_thr)
    ok = ok & ((n1 * N).sum(-1) > math.cos(math.radians(cfg.icp_angle_thr_deg)))
    R = torch.as_tensor(R_ref, device=q.device)
    s1 = cur.V @ torch.as_tensor(x1.R, device=q.device).T
    NW = N @ R.T
    J, e = torch.cat([NW, torch.linalg.cross(s1, NW)], -1), (N * diff).sum(-1)
    if cfg.icp_depth_weight:
        wgt = 1 / cur.d.clamp(min=1e-6) ** 2
        J, e = J * wgt[..., None], e * wgt
    icp = _sums(J, e, ok)
    q, z, x, y = _project(ref, cur.V, x0.R.T @ x1.R, x0.R.T @ (x1.r - x0.r))
    ok = live & (q[..., 2] > 0) & (x >= 0) & (x < ref.w - 1) & (y >= 0) & (y < ref.h - 1)
    if cfg.occlusion_thr > 0:
        dr = ref.d[torch.floor(y + 0.5).clamp(0, ref.h - 1).long(), torch.floor(x + 0.5).clamp(0, ref.w - 1).long()]
        ok = ok & ~((dr > 0) & ((z - dr).abs() > cfg.occlusion_thr))
    ix, iy = x.floor().clamp(0, ref.w - 2).long(), y.floor().clamp(0, ref.h - 2).long()
    ax, ay = (x - ix)[..., None], (y - iy)[..., None]
    tap = (1 - ax) * (1 - ay) * ref.IG[iy, ix] + ax * (1 - ay) * ref.IG[iy, ix + 1] \
        + (1 - ax) * ay * ref.IG[iy + 1, ix] + ax * ay * ref.IG[iy + 1, ix + 1]
    gx, gy = ref.fx * tap[..., 1], ref.fy * tap[..., 2]
    a = torch.stack([gx / z, gy / z, -(gx * q[..., 0] + gy * q[..., 1]) / z ** 2], -1)
    aW = a @ torch.as_tensor(x0.R, device=q.device).T
    J1 = torch.cat([aW, torch.linalg.cross(s1, aW)], -1)
    rgb = _sums(J1, tap[..., 0] - cur.I, ok)
    return icp, rgb


def _preintegrate(samples, t0, t1, bg, ba, nd=None):
    dR, dv, dp = np.eye(3), np.zeros(3), np.zeros(3)
    Fg, Vg, Pg, Va, Pa = (np.zeros((3, 3)) for _ in range(5))
    S = np.zeros((9, 9))
    ts = samples[:, 0]
    for k in range(len(ts)):
        a, b = max(ts[k], t0), min(ts[k + 1], t1) if k + 1 < len(ts) else t1
        dt = b - a
        if dt <= 0:
            continue
        w, f = samples[k, 1:4] - bg, samples[k, 4:7] - ba
        E, J, A = _exp(w * dt), _jr(w * dt), dR @ _hat(f)
        if nd:
            F = np.eye(9)
            F[:3, :3], F[3:6, :3], F[6:, :3], F[6:, 3:6] = E.T, -A * dt, -0.5 * A * dt * dt, np.eye(3) * dt
            Bg, Ba = np.zeros((9, 3)), np.zeros((9, 3))
            Bg[:3], Ba[3:6], Ba[6:] = J * dt, dR * dt, 0.5 * dR * dt * dt
            S = F @ S @ F.T + nd[0] ** 2 / dt * Bg @ Bg.T + nd[1] ** 2 / dt * Ba @ Ba.T
        Pg, Pa = Pg + Vg * dt - 0.5 * A @ Fg * dt * dt, Pa + Va * dt - 0.5 * dR * dt * dt
        Vg, Va = Vg - A @ Fg * dt, Va - dR * dt
        Fg = E.T @ Fg - J * dt
        dp, dv, dR = dp + dv * dt + 0.5 * dR @ f * dt * dt, dv + dR @ f * dt, dR @ E
    return dR, dv, dp, Fg, Vg, Pg, Va, Pa, S


class _Tracker:
    """The tracker of the library's header in 64 bits: one call of track per frame."""

    def __init__(self, cfg, x):
        self.cfg, self.x, self.xbar = cfg, x, x
        self.Rc, self.rc = _rot(np.array(cfg.T_CS[3:7])), np.array(cfg.T_CS[:3])
        self.g3 = cfg.gravity_dof == dri.DRI_GRAVITY_3D
        self.gyro, self.rgbd = cfg.track_mode == dri.DRI_TRACK_GYRO_ONLY, cfg.track_mode == dri.DRI_TRACK_RGBD_ONLY
        n = 18 if self.g3 else 17
        self.keep = np.r_[0:n, 18:18 + n]      # estimated components of the 2 x 18
        sig = np.repeat(np.array(cfg.prior_sigma[:]), [6, 3, 3, 3, n - 15])
        self.Hs, self.bs, self.n = np.diag(sig ** -2.0), np.zeros(n), n
        self.ref = None

    def predict(self, x, pre, T):
        dR, dv, dp = pre[:3]
        g = np.array([0, 0, -self.cfg.g])
        c = x.v * T + 0.5 * g * T * T
        Rh = x.R @ self.Rc @ dR @ self.Rc.T
        return x.r + x.R @ self.rc + x.G.T @ c + x.R @ self.Rc @ dp - Rh @ self.rc, Rh, x.v + g * T + x.G @ x.R @ self.Rc @ dv, c

    def imu(self, x0, x1, pre, T):
        """e = x^1(x0) boxminus x1 and its 18 x 36 Jacobian."""
        dR, dv, dp, Fg, Vg, Pg, Va, Pa, _ = pre
        r, Rh, v, c = self.predict(x0, pre, T)
        e = np.concatenate([r - x1.r, _log(Rh @ x1.R.T), v - x1.v, x0.bg - x1.bg, x0.ba - x1.ba, _log(x0.G @ x1.G.T)])
        A, I = x0.R @ self.Rc, np.eye(3)
        W = A @ dR
        li, ri = np.linalg.inv(_jr(-e[3:6])), np.linalg.inv(_jr(e[3:6]))
        J = np.zeros((18, 36))
        J[0:3, 0:3], J[0:3, 3:6], J[0:3, 6:9] = I, -_hat(r - x0.r - x0.G.T @ c), x0.G.T * T
        J[0:3, 9:12], J[0:3, 12:15], J[0:3, 15:18] = A @ Pg + _hat(Rh @ self.rc) @ W @ Fg, A @ Pa, x0.G.T @ _hat(c)
        J[3:6, 3:6], J[3:6, 9:12] = li, li @ W @ Fg
        J[6:9, 3:6], J[6:9, 6:9], J[6:9, 9:12] = -x0.G @ _hat(A @ dv), I, x0.G @ A @ Vg
        J[6:9, 12:15], J[6:9, 15:18] = x0.G @ A @ Va, -_hat(x0.G @ A @ dv)
        J[9:12, 9:12], J[12:15, 12:15], J[15:18, 15:18] = I, I, np.linalg.inv(_jr(-e[15:18]))
        J[0:3, 18:21], J[3:6, 21:24], J[6:9, 24:27], J[9:12, 27:30], J[12:15, 30:33] = -I, -ri, -I, -I, -I
        J[15:18, 33:36] = -np.linalg.inv(_jr(e[15:18]))
        return e, J

    def weight(self, x0, imu, t0, t1):
        c, T = self.cfg, t1 - t0
        pre = _preintegrate(imu, t0, t1, x0.bg, x0.ba, (c.gyr_nd, c.acc_nd))
        W = x0.R @ self.Rc @ pre[0]
        G = np.zeros((9, 9))
        G[0:3, 0:3], G[0:3, 6:9], G[3:6, 0:3], G[6:9, 3:6] = _hat(W @ self.Rc.T @ self.rc) @ W, x0.R @ self.Rc, W, x0.G @ x0.R @ self.Rc
        S = np.zeros((18, 18))
        S[:9, :9] = G @ pre[8] @ G.T
        S[9:, 9:] = np.diag(np.repeat([c.gyr_rw ** 2 * T, c.acc_rw ** 2 * T, c.sigma_grav_rw ** 2], 3))
        if not self.gyro:
            return pre, np.linalg.inv(S)
        rows = np.r_[3:6, 9:12]
        out = np.zeros((18, 18))
        out[np.ix_(rows, rows)] = np.linalg.inv(S[np.ix_(rows, rows)])
        return pre, out

    def track(self, levels, imu, t0, t1):
        c, T = self.cfg, t1 - t0
        Wi, Wr = c.sigma_d ** -2.0, c.sigma_I ** -2.0
        x0 = x1 = self.x
        if not self.rgbd:
            pre, W = self.weight(x0, imu, t0, t1)
            r, Rh, v, _ = self.predict(x0, pre, T)
            x1 = _X(x0.r if self.gyro else r, synth.matrix_to_quat(Rh), x0.v if self.gyro else v, x0.bg, x0.ba, x0.qg)
        held = np.r_[6:9, 12:17]
        held = np.concatenate([held, 17 + held])
        for l in reversed(range(c.levels)):
            for _ in range(c.iters[l]):
                icp, rgb = _pixel_terms(c, levels[l], self.ref[l], self.T, x0, x1)
                counts = (icp[3], rgb[3])
                if self.rgbd:
                    d = np.zeros(18)
                    d[:6] = np.linalg.solve(Wi * icp[0] + c.rgbd_lambda * Wr * rgb[0], Wi * icp[1] + c.rgbd_lambda * Wr * rgb[1])
                    x1, cost = x1.plus(d), Wi * icp[2] + c.rgbd_lambda * Wr * rgb[2]
                    continue
                pre = _preintegrate(imu, t0, t1, x0.bg, x0.ba)
                e, J = self.imu(x0, x1, pre, T)
                H, b = np.zeros((36, 36)), np.zeros(36)
                M = np.eye(6)
                M[3:, :3] = _hat(x1.r - x0.r)
                B = np.zeros((6, 36))
                B[:, 0:6], B[:, 18:24] = -M.T, np.eye(6)
                H += B.T @ (Wr * rgb[0]) @ B + J.T @ W @ J
                b += B.T @ (Wr * rgb[1]) - J.T @ W @ e
                H[18:24, 18:24] += Wi * icp[0]
                b[18:24] += Wi * icp[1]
                H, b, n = H[np.ix_(self.keep, self.keep)], b[self.keep], self.n
                H[:n, :n] += self.Hs
                b[:n] += self.bs - self.Hs @ x0.minus(self.xbar)[:n]
                if self.gyro:
                    H[held], H[:, held], b[held] = 0, 0, 0
                    H[held, held] = 1
                D = np.zeros(2 * n)
                if self.g3:
                    D[15:18] = D[33:36] = 1
                s = 1 / np.sqrt(np.diag(H) + D)
                dd = s * np.linalg.solve((H + np.diag(D)) * s[:, None] * s, s * b)
                d = np.zeros(36)
                d[self.keep] = dd
                x0, x1 = x0.plus(d[:18]), x1.plus(d[18:])
                cost = Wi * icp[2] + Wr * rgb[2] + e @ W @ e
        if not self.rgbd:
            b = b - H @ dd
            X = np.linalg.solve(H[:n, :n], np.column_stack([H[:n, n:], b[:n]]))
            self.Hs, self.bs = H[n:, n:] - H[n:, :n] @ X[:, :n], b[n:] - H[n:, :n] @ X[:, n]
            self.Hs = 0.5 * (self.Hs + self.Hs.T)
            if self.gyro:
                h = held[held < 17]
                self.Hs[h], self.Hs[:, h], self.bs[h] = 0, 0, 0
        self.x = self.xbar = x1
        return x1.vector(), x0.vector(), cost

    def reference(self, levels):
        self.ref, self.T = levels, (self.x.R, self.x.r)


def exact(case, seed):
    if case["kind"] == "pair":
        (scene, _), = _cameras(case, seed, 2)
        cfg = _config(case, scene)
        xr, x0, x1 = (_X(*(x[k] for k in ("r_WC", "q_WC", "v_I", "bg", "ba", "q_IW"))) for x in _pair_states(case, scene))
        icp, rgb = _pixel_terms(cfg, _levels(cfg, scene.depth[1], scene.inten[1])[0], _levels(cfg, scene.depth[0], scene.inten[0])[0], (xr.R, xr.r), x0, x1)
        Wi, Wr = cfg.sigma_d ** -2.0, cfg.sigma_I ** -2.0
        return dict(systems=np.concatenate([Wi * icp[0].ravel(), Wi * icp[1], Wr * rgb[0].ravel(), Wr * rgb[1]]),
                    cost=np.array([Wi * icp[2], Wr * rgb[2]]), n=None)
    warm = _warm_frames(case)
    if case["count"] * (warm + 1) * sum(w * h for w, h in _sizes(case)) / case["count"] > 60 * 640 * 480 or case["count"] > 16:
        return None                            # minutes
    rows = []
    for scene, k0 in _cameras(case, seed):
        cfg = _config(case, scene)
        s = scene.start_state(k0)
        tr = _Tracker(cfg, _X(*(s[k] for k in ("r_WC", "q_WC", "v_I", "bg", "ba", "q_IW"))))
        tr.reference(_levels(cfg, scene.depth[k0 % PERIOD], scene.inten[k0 % PERIOD]))
        for k in range(k0 + 1, k0 + 2 + warm):
            if case["kind"] == "model":
                V, N, I, pose = scene.model[(k - 1) % PERIOD]
                R, r = _rot(pose[3:]), pose[:3]
                d = ((V.double() - torch.as_tensor(r, device=V.device)) @ torch.as_tensor(R, device=V.device))[..., 2].float()
                n = N.double() @ torch.as_tensor(R, device=V.device)
                n = n * ((d >= cfg.depth_min) & (d <= cfg.depth_max))[..., None]
                tr.ref, tr.T = _levels(cfg, d, I, n), (R, r)
            levels = _levels(cfg, scene.depth[k % PERIOD], scene.inten[k % PERIOD])
            a, b = (k - 1) * RATE // int(FPS), k * RATE // int(FPS) + 2
            res = tr.track(levels, scene.samples(max(0, a), b), (k - 1) / FPS, k / FPS)
            tr.reference(levels)
        rows.append(res)
    return dict(x1=np.array([r[0] for r in rows]), x0=np.array([r[1] for r in rows]), cost=np.array([r[2] for r in rows]), inliers=None, status=None)
