"""The work a user of this framework has it do, as cases that can be timed.

Each case goes through the package's public entry points over seeded synthetic
inputs made on the GPU: a closed room with boxes and spheres, a smooth periodic
camera motion, its IMU readings and noisy RGB-D frames.  Sizes are those of
this repository's configurations, tests and benchmark (64^3 / 80x60, 128^3 /
320x240, 256^3 / 640x480, the serving mix), the 200^3 grid of the paper, and
odd sizes between them.

Kinds:
  step       tracking and mapping, frame by frame, the posterior read back
             after each frame (device frames); a view of the map at the end
  step_host  the same from frames in pinned host memory
  adam       the same with the paper's Adam pose optimiser
  serve      one request of every stream of a multi-stream server, and one
             stream's map read out
  mapping    closed-form fusion of frames with known poses, then a view
  descent    one step of gradient-descent mapping over several frames
  render     novel views of a map at given poses
  rollout    predicted states and images of candidate control sequences
  adjoint    a differentiable-rendering training step through torch.autograd
  map_io     a map exported to and imported from the caller's layout
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2212_02988_gb300 import Filter, config, make_state, state_arrays
from paper_2212_02988_gb300.autograd import render as autograd_render
from paper_2212_02988_gb300.serve import Server

DEV = "cuda"
G = np.array([0.0, 0.0, -9.81])
BODY_CAM = np.array([[0.0, 0.0, 1.0], [-1.0, 0.0, 0.0], [0.0, -1.0, 0.0]])
SD, SC = 0.02, 0.1            # loss scales of the descent and the training step
LR_OCC, LR_RGB = 1e-8, 5e-8   # the benchmark's descent steps


def listed():
    room64 = dict(n=64, extent=4.0, W=80, H=60, rate=10.0, imu=200.0, vmax=1.0, wmax=60.0, prims=12)
    room128 = dict(n=128, extent=6.4, W=320, H=240, rate=20.0, imu=200.0, vmax=1.5, wmax=120.0, prims=40)
    room256 = dict(n=256, extent=6.4, W=640, H=480, rate=30.0, imu=1000.0, vmax=5.0, wmax=300.0, prims=40)
    room200 = dict(n=200, extent=6.0, W=251, H=189, rate=15.0, imu=200.0, vmax=1.5, wmax=90.0, prims=30)
    return [
        # a small robot's filter: every call is a few microseconds of work
        dict(room64, name="step_64_80x60", kind="step", storage="f32", frames=8),
        # a handheld sensor's filter
        dict(room128, name="step_128_320x240", kind="step", storage="f32", frames=8),
        # the headline workload: a fast vehicle at full resolution
        dict(room256, name="step_256_640x480", kind="step", storage="f32", frames=8),
        # the same end to end: frames arrive in pinned host memory, the map in bf16
        dict(room256, name="step_host_256_bf16", kind="step_host", storage="bf16", frames=8),
        # many cameras on one GPU: ten streams of the serving mix, bf16 maps
        dict(room128, name="serve_10_streams", kind="serve", storage="bf16", frames=8, streams=10),
        # the paper's own pose optimiser: 1000 steps of 200 pixels
        dict(room128, name="adam_128_320x240", kind="adam", storage="f32", frames=2),
        # offline mapping of a recorded trajectory at the paper's grid, an odd frame size
        dict(room200, name="mapping_200_251x189", kind="mapping", storage="f32", frames=16),
        # the alternative mapper: a descent step over eight frames
        dict(room128, name="descent_128_8x320x240", kind="descent", storage="f32", frames=8),
        # novel views of a finished map, an odd grid stride and frame size
        dict(room200, name="render_200_251x189", kind="render", storage="bf16", frames=4),
        # a planner's candidates, states and images: 32 sequences of 10 frames
        dict(room256, name="rollout_256_32x10", kind="rollout", storage="f32", frames=10, seqs=32),
        # a training step through the renderer: map and pose gradients, the map updated in place
        dict(room256, name="adjoint_256_640x480", kind="adjoint", storage="f32", frames=1),
        # a session saved and restored: the whole map out of the filter and in again
        dict(room256, name="map_io_256", kind="map_io", storage="f32", frames=1),
    ]


def draw(rng):
    lu = lambda a, b: int(round(math.exp(rng.uniform(math.log(a), math.log(b)))))
    kind = rng.choice(["step", "step", "step_host", "serve", "mapping", "descent", "render", "rollout", "adjoint",
                       "map_io", "adam"])
    n = 8 * lu(8, 32)
    W = lu(80, 640)
    c = dict(kind=kind, n=n, extent=round(rng.uniform(4.0, 6.4), 2), W=W, H=max(48, int(W * rng.uniform(0.7, 0.8))),
             rate=round(rng.uniform(10.0, 30.0), 1), imu=rng.choice([200.0, 500.0, 1000.0]),
             vmax=round(rng.uniform(0.5, 2.0), 2), wmax=float(rng.randrange(30, 150)), prims=rng.randrange(12, 41),
             storage=rng.choice(["f32", "bf16"]), frames=rng.randrange(3, 9))
    if kind == "adam":
        c["frames"] = rng.randrange(1, 3)
    if kind in ("adjoint", "map_io"):
        c["frames"] = 1
    if kind == "rollout":
        c["seqs"] = rng.randrange(1, 33)
    if kind == "serve":
        c["streams"] = rng.randrange(2, 13)
        c["storage"] = "bf16"
    return c


# ------------------------------------------------------------------ inputs
class World:
    """A seeded room, a periodic camera motion of `frames` frames, the IMU
    readings along it, and what a camera there sees."""

    def __init__(self, c, seed):
        self.c, self.seed = c, seed
        r = np.random.default_rng([seed, 17])
        e, vs, P = c["extent"], c["extent"] / c["n"], max(c["frames"], 8)
        self.P, self.dt, self.vs = P, 1.0 / c["rate"], vs
        self.T = P * self.dt
        half = 0.5 * e - 3.0 * vs
        self.half = half
        h = np.array([1, 1, 1, 2, 2, 2]) * r.integers(1, 3, 6)
        self.freq = h / self.T
        self.phase = r.uniform(0, 2 * np.pi, 6)
        self.centre = r.uniform(-0.25, 0.25, 3) * np.array([e, e, 0.5 * e])
        self.yaw0 = r.uniform(-np.pi, np.pi)
        amp = np.concatenate([r.uniform(0.4, 1, 3) * [1, 1, 0.4], r.uniform(0.5, 1, 3) * [1, 0.3, 0.2]])
        v = np.linalg.norm(2 * np.pi * self.freq[:3] * amp[:3])
        w = np.linalg.norm(2 * np.pi * self.freq[3:] * amp[3:])
        amp[:3] *= min(0.8 * c["vmax"] / v, 0.2 * e / amp[:3].max())
        amp[3:] *= min(0.8 * np.radians(c["wmax"]) / w, 1.0)
        self.amp = amp
        keep = np.stack([self.at(t)[0] for t in np.linspace(0, self.T, 40)])
        prims = []
        for _ in range(20000):
            if len(prims) >= c["prims"]:
                break
            q, s, box = r.uniform(-half, half, 3), 0.5 * r.uniform(0.2, 1.0, 3), r.uniform() < 0.5
            s = s if box else np.full(3, s[0])
            d = np.linalg.norm(np.maximum(np.abs(keep - q) - s, 0), axis=1) if box else np.linalg.norm(keep - q, axis=1) - s[0]
            if d.min() > 0.35:
                prims.append((box, q, s, r.uniform(0.05, 0.95, 3)))
        self.prims = prims
        g = torch.Generator().manual_seed(seed)
        self.cells = torch.rand((24, 24, 24, 3), generator=g).mul_(0.8).add_(0.1).to(DEV)   # wall checker colours

    def at(self, t):
        """(position, velocity, acceleration, camera rotation) at time t."""
        a, f = self.amp, 2 * np.pi * self.freq
        s, co = np.sin(f * t + self.phase), np.cos(f * t + self.phase)
        return (self.centre + a[:3] * s[:3], a[:3] * f[:3] * co[:3], -a[:3] * f[:3] ** 2 * s[:3], self._rot(a[3:] * s[3:]))

    def _rot(self, ang):
        (cy, cp, cr), (sy, sp, sr) = np.cos(ang + [self.yaw0, 0, 0]), np.sin(ang + [self.yaw0, 0, 0])
        Rz = np.array([[cy, -sy, 0], [sy, cy, 0], [0, 0, 1]])
        Ry = np.array([[cp, 0, sp], [0, 1, 0], [-sp, 0, cp]])
        Rx = np.array([[1, 0, 0], [0, cr, -sr], [0, sr, cr]])
        return Rz @ Ry @ Rx @ BODY_CAM

    def omega(self, t, h=1e-5):
        W = (self.at(t + h)[3] @ self.at(t - h)[3].T - np.eye(3)) / (2 * h)
        return 0.5 * np.array([W[2, 1] - W[1, 2], W[0, 2] - W[2, 0], W[1, 0] - W[0, 1]])

    def pose(self, i):
        p, _, _, R = self.at((i % self.P) * self.dt)
        return np.concatenate([p, quat_of(R)])

    def velocity(self, i):
        t = (i % self.P) * self.dt
        return np.concatenate([self.at(t)[1], self.omega(t)])

    def imu(self, i):
        """Readings in (t_{i-1}, t_i], i in 1 .. P: rows of time, specific force, angular rate."""
        r = np.random.default_rng([self.seed, 18, i])
        k = max(1, int(round(self.c["imu"] * self.dt)))
        rows = []
        for j in range(1, k + 1):
            t = (i - 1 + j / k) * self.dt
            _, _, a, R = self.at(t)
            rows.append(np.concatenate([[t], R.T @ (a - G) + r.normal(0, 0.02, 3),
                                        R.T @ self.omega(t) + r.normal(0, 0.002, 3)]))
        return np.array(rows)

    def wall_colour(self, p, axis):
        """The checker colour of points on the room's walls (the wall's normal along `axis`)."""
        q = torch.floor((p + 0.5 * self.c["extent"]) / 0.27).long().remainder_(24)
        return self.cells[q[..., 0], q[..., 1], (q[..., 2] + 5 * axis) % 24]

    def frame(self, i):
        """Noisy (depth, colour) of frame i: exact intersections plus Gaussian noise."""
        c, f64 = self.c, torch.float64
        p, _, _, R = self.at((i % self.P) * self.dt)
        W, H = c["W"], c["H"]
        u = (torch.arange(W, device=DEV, dtype=f64) - 0.5 * (W - 1)) / (70.0 * W / 80.0)
        v = (torch.arange(H, device=DEV, dtype=f64) - 0.5 * (H - 1)) / (70.0 * W / 80.0)
        d = torch.stack([u.expand(H, W), v[:, None].expand(H, W), torch.ones(H, W, device=DEV, dtype=f64)], -1)
        d = d @ torch.tensor(R.T.copy(), device=DEV)
        o = torch.tensor(p, device=DEV)
        best, axis = (torch.where(d > 0, self.half - o, -self.half - o) / d).nan_to_num(nan=math.inf).abs().min(-1)
        col = self.wall_colour((o + best[..., None] * d).float(), axis)
        for box, q, s, alb in self.prims:
            q, s = torch.tensor(q, device=DEV), torch.tensor(s, device=DEV)
            if box:
                a, b = (q - s - o) / d, (q + s - o) / d
                tn, tf = torch.minimum(a, b).amax(-1), torch.maximum(a, b).amin(-1)
                hit = (tn <= tf) & (tn > 0) & (tn < best)
            else:
                oc = o - q
                A, B, C = (d * d).sum(-1), 2 * (d @ oc), oc @ oc - s[0] ** 2
                D = B * B - 4 * A * C
                tn = (-B - D.clamp(min=0).sqrt()) / (2 * A)
                hit = (D >= 0) & (tn > 0) & (tn < best)
            best = torch.where(hit, tn, best)
            col = torch.where(hit[..., None], torch.tensor(alb, device=DEV, dtype=torch.float32), col)
        g = torch.Generator(device=DEV).manual_seed(self.seed * 1009 + i)
        depth = best.float() + 0.01 * torch.randn((H, W), generator=g, device=DEV)
        return depth.contiguous(), (col + 0.02 * torch.randn((H, W, 3), generator=g, device=DEV)).contiguous()

    def settled(self):
        """The map a long run leaves: truncated signed distances, surface colours, variances."""
        n, vs = self.c["n"], self.vs
        x = (torch.arange(n, device=DEV, dtype=torch.float32) + 0.5) * vs - 0.5 * self.c["extent"]
        p = torch.stack(torch.meshgrid(x, x, x, indexing="ij"), -1).flip(-1)   # [k, j, i] -> (x, y, z)
        wall = self.half - p.abs()
        sdf, axis = wall.min(-1)
        out = wall.clamp(max=0).square().sum(-1).sqrt()
        sdf = torch.where(out > 0, -out, sdf)
        col = self.wall_colour(p.clamp(-self.half, self.half), axis)
        for box, q, s, alb in self.prims:
            q, s = torch.tensor(q, device=DEV, dtype=torch.float32), torch.tensor(s, device=DEV, dtype=torch.float32)
            if box:
                a = (p - q).abs() - s
                d = a.clamp(min=0).square().sum(-1).sqrt() + a.amax(-1).clamp(max=0)
            else:
                d = (p - q).square().sum(-1).sqrt() - s[0]
            near = d < sdf
            sdf = torch.where(near, d, sdf)
            col = torch.where(near[..., None], torch.tensor(alb, device=DEV, dtype=torch.float32), col)
        tr = 2.0 * vs
        seen, band = sdf >= -tr, sdf.abs() <= tr
        far = torch.tensor(1e4, device=DEV)
        return (torch.where(seen, -sdf.clamp(-tr, tr), torch.tensor(-0.001, device=DEV)).contiguous(),
                (col * band[..., None]).contiguous(), torch.where(seen, torch.tensor(0.1, device=DEV), far).contiguous(),
                torch.where(band, torch.tensor(0.1, device=DEV), far).contiguous())


def quat_of(R):
    m = np.array([1 + R[0, 0] + R[1, 1] + R[2, 2], 1 + R[0, 0] - R[1, 1] - R[2, 2], 1 - R[0, 0] + R[1, 1] - R[2, 2],
                  1 - R[0, 0] - R[1, 1] + R[2, 2]])
    k = int(m.argmax())
    s = 0.5 / math.sqrt(m[k])
    q = [[m[0], R[2, 1] - R[1, 2], R[0, 2] - R[2, 0], R[1, 0] - R[0, 1]],
         [R[2, 1] - R[1, 2], m[1], R[1, 0] + R[0, 1], R[0, 2] + R[2, 0]],
         [R[0, 2] - R[2, 0], R[1, 0] + R[0, 1], m[2], R[2, 1] + R[1, 2]],
         [R[1, 0] - R[0, 1], R[0, 2] + R[2, 0], R[2, 1] + R[1, 2], m[3]]][k]
    return np.array(q) * s


def belief(w):
    """A filter state in mid-flight: frame 0's pose, a velocity estimate, its covariance."""
    cov = np.diag([4e-4] * 3 + [1e-4] * 3 + [2e-3] * 3 + [3e-3] * 3)
    return w.pose(0), w.velocity(0) + np.array([0.05, -0.02, 0.01, 0.1, -0.2, 0.05]), cov


def streams_of(c, seed):
    """The serving mix: maps of 64^3, 128^3 and 256^3, frames of 160x120, 320x240 and 640x480."""
    r = np.random.default_rng([seed, 4])
    out = []
    for k in range(c["streams"]):
        n, e = [(64, 4.0), (128, 6.4), (256, 6.4)][(k + 1) % 3 if k < 3 else int(r.integers(3))]
        W, H = [(160, 120), (320, 240), (640, 480)][k % 3 if k < 3 else int(r.integers(3))]
        out.append(dict(c, kind="step", n=n, extent=e, W=W, H=H, rate=float(r.uniform(10, 30)), imu=200.0, vmax=1.5,
                        wmax=120.0))
    return out


def candidates(c, w, seed):
    r = np.random.default_rng([seed, 5])
    base = [w.imu(1 + i % w.P) for i in range(c["frames"])]
    out = []
    for s in range(c["seqs"]):
        off = np.concatenate([[0.0], r.normal(0, 0.5, 3), r.normal(0, 0.2, 3)])
        out.append([b + off for b in base] if s < c["seqs"] - 1 or c["seqs"] == 1 else [None] * c["frames"])
    return out


# ----------------------------------------------------------------- the cases
def make_filter(c, w, state=None, **over):
    F = Filter(config(c["n"], c["extent"], c["W"], c["H"], storage=c["storage"], **over),
               make_state(*(state or (w.pose(0), w.velocity(0)))))
    F.map_load(*w.settled())
    return F


def prepare(case, seed):
    c, kind = case, case["kind"]
    if kind == "serve":
        sub = streams_of(c, seed)
        worlds = [World(s, seed + 100 * k) for k, s in enumerate(sub)]
        srv = Server(24 << 30, max_slots=len(sub), storage=c["storage"])
        st = dict(c=c, srv=srv, at=0, streams=[])
        for s, w in zip(sub, worlds):
            sid = srv.open(config(s["n"], s["extent"], s["W"], s["H"]), make_state(w.pose(0), w.velocity(0)), w.settled())
            fr = [tuple(x.cpu().pin_memory() for x in w.frame(i)) for i in range(w.P)]
            st["streams"].append(dict(sid=sid, n=s["n"], dt=w.dt, frames=fr, imu=[w.imu(i) for i in range(1, w.P + 1)]))
            srv.submit(sid, None, w.dt, *fr[0])
        srv.drain()
        srv.poll()
        return st
    w = World(c, seed)
    st = dict(c=c, w=w)
    if kind in ("step", "step_host", "adam"):
        over = dict(optimiser=1) if kind == "adam" else {}
        F = make_filter(c, w, **over)
        fr = [w.frame(i) for i in range(w.P)]
        if kind == "step_host":
            fr = [tuple(x.cpu().pin_memory() for x in f) for f in fr]
        (F.step_host if kind == "step_host" else F.step)(None, w.dt, *fr[0])
        st.update(F=F, at=0, frames=fr, imu=[w.imu(i) for i in range(1, w.P + 1)], view=w.pose(0))
    elif kind == "mapping":
        F = make_filter(c, w)
        st.update(F=F, frames=[w.frame(i) for i in range(c["frames"])], view=w.pose(1),
                  states=[make_state(w.pose(i), w.velocity(i)) for i in range(c["frames"])])
    elif kind == "descent":
        fr = [w.frame(i) for i in range(c["frames"])]
        st.update(F=make_filter(c, w), poses=np.stack([w.pose(i) for i in range(c["frames"])]),
                  depth=torch.stack([f[0] for f in fr]), rgb=torch.stack([f[1] for f in fr]))
    elif kind == "render":
        st.update(F=make_filter(c, w), poses=[w.pose(i) for i in range(c["frames"])])
    elif kind == "rollout":
        st.update(F=make_filter(c, w, belief(w)), windows=candidates(c, w, seed))
    elif kind == "adjoint":
        occ, rgb, vo, vr = w.settled()
        F = Filter(config(c["n"], c["extent"], c["W"], c["H"], storage=c["storage"]))
        F.map_load(occ, rgb, vo, vr)
        st.update(F=F, occ=occ.requires_grad_(True), rgb=rgb.requires_grad_(True),
                  pose=torch.tensor(w.pose(0), requires_grad=True), frame=w.frame(1))
    else:
        st.update(F=make_filter(c, w), map=w.settled())
    return st


def run(state):
    st, kind = state, state["c"]["kind"]
    if kind == "serve":
        i = st["at"]
        st["at"] += 1
        for s in st["streams"]:
            P = len(s["frames"])
            st["srv"].submit(s["sid"], s["imu"][i % P], s["dt"], *s["frames"][(i + 1) % P])
        got = []
        while len(got) < len(st["streams"]):
            got += st["srv"].poll(timeout_ms=1000)
        got.sort(key=lambda r: r["stream"])
        first = st["streams"][0]   # a session's map is read out while the others go on
        return {**{k: np.stack([r[k] for r in got]) for k in ("pose", "vel", "cov")},
                "map": st["srv"].map_store(first["sid"], (first["n"],) * 3)}
    F, c = st["F"], st["c"]
    if kind in ("step", "step_host", "adam"):
        step, P, out = F.step_host if kind == "step_host" else F.step, len(st["frames"]), []
        for i in range(st["at"], st["at"] + c["frames"]):
            out.append(state_arrays(step(st["imu"][i % P], st["w"].dt, *st["frames"][(i + 1) % P], want_state=True)))
        st["at"] += c["frames"]
        return {**{k: np.stack([o[k] for o in out]) for k in ("pose", "vel", "cov")}, "view": F.render(st["view"])}
    if kind == "mapping":
        for s, (d, r) in zip(st["states"], st["frames"]):
            F.set_state(s)
            F.update_map(d, r)
        return {"map": F.map_store(), "view": F.render(st["view"])}
    if kind == "descent":
        loss = F.map_descent(st["poses"], st["depth"], st["rgb"], SD, SC, LR_OCC, LR_RGB)
        return {"loss": loss, "map": F.map_store()}
    if kind == "render":
        return [F.render(p) for p in st["poses"]]
    if kind == "rollout":
        out = F.rollout(st["windows"], st["w"].dt)
        rec = np.stack([np.frombuffer(s, np.float64, 157) for seq in out.pop("states") for s in seq])
        return {**out, "pose": rec[:, :7], "vel": rec[:, 7:13], "cov": rec[:, 13:].reshape(-1, 12, 12)}
    if kind == "adjoint":
        occ, rgb, pose = st["occ"], st["rgb"], st["pose"]
        pose.grad = occ.grad = rgb.grad = None
        d, r = autograd_render(pose, occ, rgb, F)
        D, C = st["frame"]
        hit = d.detach() > 0
        loss = (0.5 / SD ** 2) * ((d - D) * hit).square().sum() + (0.5 / SC ** 2) * ((r - C) * hit[..., None]).square().sum()
        loss.backward()
        with torch.no_grad():
            occ.sub_(occ.grad, alpha=LR_OCC)
            rgb.sub_(rgb.grad, alpha=LR_RGB)
        return {"depth": d.detach(), "rgb": r.detach(), "g_pose": pose.grad, "g_occ": occ.grad, "g_rgb": rgb.grad}
    out = F.map_store()
    F.map_load(*st["map"])
    return {"before": out, "after": F.map_store()}


def work(case):
    """Bytes: frames and controls in, images and states out, every map value
    that an update must read and write (about a thirtieth of the voxels a
    frame) or an import or export moves.  Operations: about 600 for each
    observed pixel and localisation pass, 300 for each ray (its hit's
    interpolation and a handful of samples), 30 for each updated voxel."""
    c, kind = case, case["kind"]
    if kind == "serve":
        px, vox = c["streams"] * 320 * 240, c["streams"] * 128 ** 3 / 30
        return {"bytes": px * 16 + vox * 18 + 36 * 128 ** 3, "flops": px * (11 * 600 + 300) + vox * 30}
    px, N = c["W"] * c["H"], c["n"] ** 3
    vox, f = N / 30, c["frames"]
    if kind in ("step", "step_host"):
        return {"bytes": f * (px * 16 + vox * 18) + px * 21, "flops": f * (px * (11 * 600 + 300) + vox * 30)}
    if kind == "adam":
        return {"bytes": f * (px * 16 + vox * 18) + px * 21, "flops": f * (1000 * 200 * 400 + px * 900 + vox * 30)}
    if kind == "mapping":
        return {"bytes": f * (px * 16 + vox * 18) + 48 * N + px * 21, "flops": f * vox * 30 + px * 300}
    if kind == "descent":
        return {"bytes": f * px * 16 + 16 * 2 * N + 48 * N, "flops": f * px * 900 + N * 20}
    if kind == "render":
        return {"bytes": f * px * 21 + vox * 4, "flops": f * px * 300}
    if kind == "rollout":
        return {"bytes": c["seqs"] * f * px * 16 + vox * 16, "flops": c["seqs"] * f * px * 300}
    if kind == "adjoint":   # the map in, its gradients out, the map updated; images in and out
        return {"bytes": 16 * 5 * N + px * 48, "flops": px * 900 + 8 * N}
    return {"bytes": 3 * 48 * N, "flops": N}


# ------------------------------------------------- the same in 64 bits, plainly
def rot_of(q):
    w, x, y, z = q / np.linalg.norm(q)
    return np.array([[1 - 2 * (y * y + z * z), 2 * (x * y - w * z), 2 * (x * z + w * y)],
                     [2 * (x * y + w * z), 1 - 2 * (x * x + z * z), 2 * (y * z - w * x)],
                     [2 * (x * z - w * y), 2 * (y * z + w * x), 1 - 2 * (x * x + y * y)]])


def skew(a):
    return np.array([[0, -a[2], a[1]], [a[2], 0, -a[0]], [-a[1], a[0], 0]])


def so3(a):
    """(Exp(a), left Jacobian of SO(3) at a)."""
    t, K = np.linalg.norm(a), skew(a)
    if t < 1e-4:
        return np.eye(3) + K + K @ K / 2 + K @ K @ K / 6, np.eye(3) + K / 2 + K @ K / 6
    return (np.eye(3) + np.sin(t) / t * K + (1 - np.cos(t)) / t ** 2 * K @ K,
            np.eye(3) + (1 - np.cos(t)) / t ** 2 * K + (t - np.sin(t)) / t ** 3 * K @ K)


def blk(A, B):
    M = np.zeros((6, 6))
    M[:3, :3], M[3:, 3:] = A, B
    return M


class Plain:
    """The filter in plain 64-bit numpy and torch."""

    def __init__(self, c, maps, pose, vel, cov=None, adam=False):
        self.c, self.adam, self.vs = c, adam, c["extent"] / c["n"]
        self.fx, self.cx, self.cy = 70.0 * c["W"] / 80.0, 0.5 * (c["W"] - 1), 0.5 * (c["H"] - 1)
        self.occ, self.rgb, self.vo, self.vr = (m.detach().double() for m in maps)
        self.t, self.R, self.v = pose[:3].copy(), rot_of(pose[3:]), vel.copy()
        self.q = pose[3:] / np.linalg.norm(pose[3:])
        self.cov, self.nloc = (np.eye(12) * 1e-8 if cov is None else cov), 0
        u = (torch.arange(c["W"], device=DEV, dtype=torch.float64) - self.cx) / self.fx
        v = (torch.arange(c["H"], device=DEV, dtype=torch.float64) - self.cy) / self.fx
        self.dc = torch.stack([u.expand(c["H"], c["W"]), v[:, None].expand(c["H"], c["W"]),
                               torch.ones(c["H"], c["W"], device=DEV, dtype=torch.float64)], -1)

    # ---- the render: first sample above zero, interpolated with the one before
    def tri(self, A, g):
        n = self.c["n"]
        f0 = g.detach().floor()
        w = g - f0
        i0 = f0.long()
        lo, hi = i0.clamp(0, n - 1), (i0 + 1).clamp(0, n - 1)
        out = 0.0
        for k in range(8):
            b = [(k >> a) & 1 for a in range(3)]
            x, y, z = ((hi if b[a] else lo)[..., a] for a in range(3))
            wt = 1.0
            for a in range(3):
                wt = wt * (w[..., a] if b[a] else 1 - w[..., a])
            v = A[z, y, x]
            out = out + (wt[..., None] if v.dim() > wt.dim() else wt) * v
        return out

    def rays(self, t, R):
        d = (self.dc.reshape(-1, 3) @ R.T)
        r = d / d.norm(dim=1, keepdim=True)
        return (t + 0.5 * self.c["extent"]) / self.vs - 0.5, r / self.vs, 1.0 / self.dc.reshape(-1, 3).norm(dim=1)

    def march(self, t, R):
        """Index of each ray's first sample above zero (0: none, -1: the first sample)."""
        n, eps = self.c["n"], 0.4 * self.vs
        c, r, _ = self.rays(t, R)
        hk = torch.zeros(len(r), dtype=torch.long, device=DEV)
        live = torch.arange(len(r), device=DEV)
        for k in range(1, int(6 * n / 0.4) + 2):
            g = c + (k * eps) * r[live]
            ok = ((g >= -0.5) & (g < n - 0.5)).all(1)
            live, g = live[ok], g[ok]
            if not len(live):
                break
            hit = self.tri(self.occ, g) > 0
            hk[live[hit]] = -1 if k == 1 else k
            live = live[~hit]
        return hk

    def shade(self, t, R, hk, occ=None, rgb=None):
        c, r, zs = self.rays(t, R)
        m = (hk >= 2).nonzero()[:, 0]
        eps = 0.4 * self.vs
        d0, d1 = (hk[m] - 1).double() * eps, hk[m].double() * eps
        occ, rgb = self.occ if occ is None else occ, self.rgb if rgb is None else rgb
        p0, p1 = c + d0[:, None] * r[m], c + d1[:, None] * r[m]
        f0, f1 = self.tri(occ, p0), self.tri(occ, p1)
        a = -f0 / (f1 - f0)
        D = torch.zeros(len(r), device=DEV, dtype=torch.float64).index_put((m,), (d0 + a * (d1 - d0)) * zs[m])
        c0, c1 = self.tri(rgb, p0), self.tri(rgb, p1)
        C = torch.zeros((len(r), 3), device=DEV, dtype=torch.float64).index_put((m,), c0 + a[:, None] * (c1 - c0))
        s = self.dc.shape[:2]
        return D.reshape(s), C.reshape(*s, 3)

    def render(self, pose):
        t, R = torch.tensor(pose[:3], device=DEV), torch.tensor(rot_of(pose[3:]), device=DEV)
        D, C = self.shade(t, R, self.march(t, R))
        return {"depth": D, "rgb": C, "mask": None, "hitk": None}

    # ---- the map update
    def valid(self, D):
        ok = (D > 0) & torch.isfinite(D)
        for ax in (0, 1):
            e = (D.diff(dim=ax).abs() <= 0.1)
            pad = torch.ones_like(e.narrow(ax, 0, 1))
            ok = ok & torch.cat([e, pad], ax) & torch.cat([pad, e], ax)
        return ok

    def fuse(self, D, C):
        D, C = D.to(DEV).double(), C.to(DEV).double()
        n, W, H, tr = self.c["n"], self.c["W"], self.c["H"], 2 * self.vs
        R, t, ok_px = torch.tensor(self.R, device=DEV), torch.tensor(self.t, device=DEV), self.valid(D)
        x = (torch.arange(n, device=DEV, dtype=torch.float64) + 0.5) * self.vs - 0.5 * self.c["extent"]
        for k0 in range(0, n, 32):   # slabs of z
            p = torch.stack(torch.meshgrid(x[k0:k0 + 32], x, x, indexing="ij"), -1).flip(-1)
            X = (p - t) @ R
            z = X[..., 2]
            u = torch.floor(self.fx * X[..., 0] / z + self.cx + 0.5)
            v = torch.floor(self.fx * X[..., 1] / z + self.cy + 0.5)
            ok = (z > 0) & (u >= 0) & (u < W) & (v >= 0) & (v < H)
            ui, vi = torch.where(ok, u, 0).long(), torch.where(ok, v, 0).long()
            sdf = D[vi, ui] - z
            ok = ok & ok_px[vi, ui] & (sdf >= -tr)
            band = ok & (sdf.abs() <= tr)
            s = slice(k0, k0 + 32)
            w = self.vo[s] / 1.0
            self.occ[s] = torch.where(ok, (self.occ[s] + w * -sdf.clamp(-tr, tr)) / (1 + w), self.occ[s])
            self.vo[s] = torch.where(ok, w / (1 + w), w)
            w = self.vr[s]
            self.rgb[s] = torch.where(band[..., None], (self.rgb[s] + w[..., None] * C[vi, ui]) / (1 + w[..., None]), self.rgb[s])
            self.vr[s] = torch.where(band, w / (1 + w), w)

    # ---- the state
    def predict(self, imu, dt):
        R, u = self.R, np.zeros(6)
        if imu is not None and len(imu):
            m = imu.mean(0)
            d = imu[:, 0] - m[0]
            gend = m[4:] + ((d[:, None] * (imu[:, 4:] - m[4:])).sum(0) / max((d * d).sum(), 1e-300)) * (imu[-1, 0] - m[0])
            wm = R @ m[4:]
            u[:3] = so3(0.5 * dt * wm)[0] @ R @ m[1:4] + G
            u[3:] = (so3(dt * wm)[0] @ R @ gend - self.v[3:]) / dt
        self.pv = self.v + u * dt
        self.pt = self.t + self.pv[:3] * dt
        E, J = so3(self.pv[3:] * dt)
        self.pR = E @ R
        a = self.pv[3:] * dt
        th = np.linalg.norm(a)
        s = 0.5 * np.sinc(0.5 * th / np.pi)
        dq, q = np.concatenate([[np.cos(0.5 * th)], s * a]), self.q
        self.pq = np.concatenate([[dq[0] * q[0] - dq[1:] @ q[1:]], dq[0] * q[1:] + q[0] * dq[1:] + np.cross(dq[1:], q[1:])])
        self.pq /= math.copysign(np.linalg.norm(self.pq), self.pq[0])   # w >= 0
        A, B = blk(np.eye(3), E), blk(np.eye(3) * dt, J * dt)
        F = np.block([[A, B], [np.zeros((6, 6)), np.eye(6)]])
        Qv, Qp = np.diag([0.03 ** 2] * 6), np.diag([0.05 ** 2] * 3 + [0.02 ** 2] * 3)
        S = F @ self.cov @ F.T + np.block([[B @ Qv @ B.T + Qp, B @ Qv], [Qv @ B.T, Qv]])
        self.pcov = S = 0.5 * (S + S.T)
        self.L = np.linalg.inv(S[:6, :6])
        self.D = S[6:, :6] @ self.L
        self.Sv = S[6:, 6:] - self.D @ S[:6, 6:]

    def anchor(self):
        self.aR, self.at = self.R, self.t
        r = self.render(np.concatenate([self.t, self.q]))
        D, self.aC = r["depth"], r["rgb"]
        self.ok1 = ok = self.valid(D)
        P = D[..., None] * self.dc
        N, ok0 = torch.zeros_like(P), torch.zeros_like(ok)
        N[1:-1, 1:-1] = torch.cross(P[1:-1, 2:] - P[1:-1, :-2], P[2:, 1:-1] - P[:-2, 1:-1], dim=-1)
        ok0[1:-1, 1:-1] = ok[1:-1, 1:-1] & ok[1:-1, 2:] & ok[1:-1, :-2] & ok[2:, 1:-1] & ok[:-2, 1:-1]
        nn = N.norm(dim=-1)
        ok0 &= nn > 0
        N = N / nn.clamp(min=1e-300)[..., None]
        self.aN = torch.where((N * P).sum(-1, keepdim=True) > 0, -N, N)
        self.ok0, self.aP = ok0, P

    def residuals(self, R, t, P, C, m):
        """Kept residuals r (K, 4) and Jacobians (K, 4, 6) of points P (camera frame), colours C, validity m."""
        W, H = self.c["W"], self.c["H"]
        M, b = torch.tensor(self.aR.T @ R, device=DEV), torch.tensor(self.aR.T @ (t - self.at), device=DEV)
        y = P @ M.T
        X = y + b
        z = X[:, 2]
        u, v = self.fx * X[:, 0] / z + self.cx, self.fx * X[:, 1] / z + self.cy
        nu, nv, bu, bv = torch.floor(u + 0.5), torch.floor(v + 0.5), torch.floor(u), torch.floor(v)
        keep = m & (z > 0) & (nu >= 0) & (nu <= W - 1) & (nv >= 0) & (nv <= H - 1) & (bu >= 0) & (bu <= W - 2) & (bv >= 0) & (bv <= H - 2)
        X, y, z, u, v, C = X[keep], y[keep], z[keep], u[keep], v[keep], C[keep]
        nu, nv, bu, bv = (a[keep].long() for a in (nu, nv, bu, bv))
        a, c = (u - bu)[:, None], (v - bv)[:, None]
        n = self.aN[nv, nu]
        I00, I10, I01, I11 = self.aC[bv, bu], self.aC[bv, bu + 1], self.aC[bv + 1, bu], self.aC[bv + 1, bu + 1]
        rg = (n * (self.aP[nv, nu] - X)).sum(1, keepdim=True)
        rc = (1 - c) * (I00 + a * (I10 - I00)) + c * (I01 + a * (I11 - I01)) - C
        ok = self.ok0[nv, nu] & self.ok1[bv, bu] & self.ok1[bv, bu + 1] & self.ok1[bv + 1, bu] & self.ok1[bv + 1, bu + 1]
        ok = ok & (rg.abs() <= 0.45)[:, 0] & (rc.abs() <= 0.15).all(1)
        gu, gv = (1 - c) * (I10 - I00) + c * (I11 - I01), (1 - a) * (I01 - I00) + a * (I11 - I10)
        f, iz = self.fx, (1 / z)[:, None]
        ac = torch.stack([gu * f * iz, gv * f * iz, -(gu * X[:, :1] + gv * X[:, 1:2]) * f * iz * iz], -1)
        A = torch.cat([-n[:, None], ac], 1)
        J = torch.cat([A, torch.cross(y[:, None].expand_as(A), A, dim=-1)], -1)
        return torch.cat([rg, rc], 1)[ok], J[ok]

    def localise(self, D, C):
        D, C = D.to(DEV).double(), C.to(DEV).double()
        P, C, m = (D[..., None] * self.dc).reshape(-1, 3), C.reshape(-1, 3), self.valid(D).reshape(-1)
        b = torch.tensor([0.02, 0.1, 0.1, 0.1], device=DEV, dtype=torch.float64)
        fl = torch.tensor([1e-3, 1e-2, 1e-2, 1e-2], device=DEV, dtype=torch.float64)
        T, xi = blk(self.aR, self.aR), np.zeros(6)
        at = lambda: (so3(xi[3:])[0] @ self.pR, self.pt + xi[:3])
        if self.adam:
            v2, b2, NP, k = np.zeros(6), 1.0, len(P), 200
            lr = np.array([1e-3] * 3 + [3.6e-4] * 3)
            base = self.nloc * 1000 * k
            for s in range(1000):
                i = np.arange(base + s * k + 1, base + (s + 1) * k + 1, dtype=np.uint64)
                with np.errstate(over="ignore"):
                    h = np.uint64(0x5EED2212) + i * np.uint64(0x9E3779B97F4A7C15)
                    h = (h ^ (h >> np.uint64(30))) * np.uint64(0xBF58476D1CE4E5B9)
                    h = (h ^ (h >> np.uint64(27))) * np.uint64(0x94D049BB133111EB)
                    h = h ^ (h >> np.uint64(31))
                p = torch.from_numpy((((h >> np.uint64(32)) * np.uint64(NP)) >> np.uint64(32)).astype(np.int64)).to(DEV)
                r, J = self.residuals(*at(), P[p], C[p], m[p])
                g = T @ ((torch.sign(r) / b)[..., None] * J).sum((0, 1)).cpu().numpy()
                g = NP / k * blk(np.eye(3), so3(xi[3:])[1]).T @ g + self.L @ xi
                b2 *= 0.999
                v2 = 0.999 * v2 + 0.001 * g * g
                xi = xi - lr * g / (np.sqrt(v2 / (1 - b2)) + 1e-8)
        else:
            for _ in range(10):
                r, J = self.residuals(*at(), P, C, m)
                w = 1 / (b * torch.maximum(r.abs(), fl))
                Jw = J * w[..., None]
                H = T @ torch.einsum("kri,krj->ij", Jw, J).cpu().numpy() @ T.T
                g = T @ torch.einsum("kri,kr->i", Jw, r).cpu().numpy()
                M = blk(np.eye(3), so3(xi[3:])[1])
                xi = xi - np.linalg.solve(M.T @ H @ M + self.L, M.T @ g + self.L @ xi)
        R, t = at()
        r, J = self.residuals(R, t, P, C, m)
        J = J / b[:, None]
        Ht = T @ torch.einsum("kri,krj->ij", J, J).cpu().numpy() @ T.T
        Mi = np.linalg.inv(blk(np.eye(3), so3(xi[3:])[1]))
        S = np.linalg.inv(2 * Ht + Mi.T @ self.L @ Mi)
        S = S if self.nloc == 0 else 0.8 * self.cov[:6, :6] + 0.2 * S
        Dm = self.D @ Mi
        th = np.linalg.norm(xi[3:])
        dq, q = np.concatenate([[np.cos(0.5 * th)], 0.5 * np.sinc(0.5 * th / np.pi) * xi[3:]]), self.pq
        self.q = np.concatenate([[dq[0] * q[0] - dq[1:] @ q[1:]], dq[0] * q[1:] + q[0] * dq[1:] + np.cross(dq[1:], q[1:])])
        self.q /= math.copysign(np.linalg.norm(self.q), self.q[0])
        self.R, self.t, self.v = R, t, self.pv + self.D @ xi
        self.cov = np.block([[S, S @ Dm.T], [Dm @ S, Dm @ S @ Dm.T + self.Sv]])
        self.cov = 0.5 * (self.cov + self.cov.T)
        self.nloc += 1

    def step(self, imu, dt, D, C):
        if imu is not None:
            self.predict(imu, dt)
            self.localise(D, C)
        self.fuse(D, C)
        self.anchor()
        return {"pose": np.concatenate([self.t, self.q]), "vel": self.v, "cov": self.cov}


def exact(case, seed):
    c, kind = case, case["kind"]
    if kind == "serve":
        out = []
        for k, s in enumerate(streams_of(c, seed)):
            w = World(s, seed + 100 * k)
            ref = Plain(s, w.settled(), w.pose(0), w.velocity(0))
            ref.step(None, w.dt, *w.frame(0))
            out.append(ref.step(w.imu(1), w.dt, *w.frame(1)))
            if k == 0:
                m = {"occ": ref.occ, "rgb": ref.rgb, "var_occ": ref.vo, "var_rgb": ref.vr}
        return {**{k: np.stack([o[k] for o in out]) for k in ("pose", "vel", "cov")}, "map": m}
    w = World(c, seed)
    if kind == "map_io":
        m = {k: v.double() for k, v in zip(("occ", "rgb", "var_occ", "var_rgb"), w.settled())}
        return {"before": m, "after": m}
    ref = Plain(c, w.settled(), w.pose(0), w.velocity(0), adam=kind == "adam")
    if kind in ("step", "step_host", "adam"):
        ref.step(None, w.dt, *w.frame(0))
        out = [ref.step(w.imu(i), w.dt, *w.frame(i)) for i in range(1, c["frames"] + 1)]
        return {**{k: np.stack([o[k] for o in out]) for k in ("pose", "vel", "cov")}, "view": ref.render(w.pose(0))}
    if kind == "mapping":
        for i in range(c["frames"]):
            ref.t, ref.R = w.pose(i)[:3], rot_of(w.pose(i)[3:])
            ref.fuse(*w.frame(i))
        return {"map": {"occ": ref.occ, "rgb": ref.rgb, "var_occ": ref.vo, "var_rgb": ref.vr}, "view": ref.render(w.pose(1))}
    if kind == "render":
        return [ref.render(w.pose(i)) for i in range(c["frames"])]
    if kind == "rollout":   # the states; the images would take too long
        out = []
        for seq in candidates(c, w, seed):
            f = Plain(c, (ref.occ[:1], ) * 4, *belief(w))
            for imu in seq:
                f.predict(imu, w.dt)
                f.t, f.R, f.q, f.v, f.cov = f.pt, f.pR, f.pq, f.pv, f.pcov
                out.append({"pose": np.concatenate([f.t, f.q]), "vel": f.v, "cov": f.cov})
        return {"depth": None, "rgb": None, **{k: np.stack([o[k] for o in out]) for k in ("pose", "vel", "cov")}}
    occ, rgb = (x.clone().requires_grad_(True) for x in (ref.occ, ref.rgb))
    if kind == "descent":
        loss = 0.5 / 1e4 * ((occ + 0.001).square().sum() + rgb.square().sum())
        for i in range(c["frames"]):
            t, R = torch.tensor(w.pose(i)[:3], device=DEV), torch.tensor(rot_of(w.pose(i)[3:]), device=DEV)
            hk = ref.march(t, R)
            d, r = ref.shade(t, R, hk, occ, rgb)
            D, C = w.frame(i)
            m = (hk >= 2).reshape(D.shape) & (D > 0)
            loss = loss + 0.5 / SD ** 2 * ((d - D)[m]).square().sum() + 0.5 / SC ** 2 * ((r - C)[m]).square().sum()
        loss.backward()
        return {"loss": float(loss.detach()), "map": {"occ": occ.detach() - LR_OCC * occ.grad,
                                                      "rgb": rgb.detach() - LR_RGB * rgb.grad, "var_occ": ref.vo, "var_rgb": ref.vr}}
    pose = torch.tensor(w.pose(0), device=DEV, requires_grad=True)
    x = pose[3:] / pose[3:].norm()
    a, b, cc, d = x[0], x[1], x[2], x[3]
    R = torch.stack([1 - 2 * (cc * cc + d * d), 2 * (b * cc - a * d), 2 * (b * d + a * cc), 2 * (b * cc + a * d),
                     1 - 2 * (b * b + d * d), 2 * (cc * d - a * b), 2 * (b * d - a * cc), 2 * (cc * d + a * b),
                     1 - 2 * (b * b + cc * cc)]).reshape(3, 3)
    hk = ref.march(pose[:3].detach(), R.detach())
    dd, rr = ref.shade(pose[:3], R, hk, occ, rgb)
    D, C = w.frame(1)
    hit = (hk >= 2).reshape(D.shape)
    (0.5 / SD ** 2 * (dd - D)[hit].square().sum() + 0.5 / SC ** 2 * (rr - C)[hit].square().sum()).backward()
    return {"depth": dd.detach(), "rgb": rr.detach(), "g_pose": pose.grad, "g_occ": occ.grad, "g_rgb": rgb.grad}
