"""The work that users of this framework have it do, as cases that can be timed.

A case is a dict of plain values.  `kind` says which entry point it goes
through:

  frames  BP.reconstruct on device tensors (one frame, or a batch of frames)
  host    BP.reconstruct_host on page-locked host buffers (the paper's timed
          on-line path: signals from the host, image to the host)
  plan    Plan.execute: uneven instances in one tuned, graph-replayed plan
  serve   Server.submit / wait: a burst of requests for several subjects
  times   fmm_gpu: arrival times of many sources (the off-line step)

2-D geometries follow the package's synthetic workloads: a skull ring around
the imaged disc, sensors on a circle of 0.469 grid widths, a record of 1.6
crossings.  3-D ones are the hemisphere and shell skull of the serving
subjects, scaled.  Every number that a user would measure (speed maps,
absorbers, noise) comes from the seed.
"""
import math

import numpy as np
import torch

from paper_1501_03869_gb300 import BP, Plan, Server, fmm_gpu, synth
from paper_1501_03869_gb300._lib import PAT_FLAG_GPU_TABLE, PAT_FLAG_TILE_128, PAT_FLAG_TILE_256

RING = 120.0 / 256.0     # ring radius over the grid width
CROSSINGS = 1.6          # record length over the ring's crossing time in water
DTYPES = {"f32": torch.float32, "bf16": torch.bfloat16, "f16": torch.float16}


def listed():
    return [
        # one small live frame: launch and latency bound
        dict(name="frame_128_f32", kind="frames", n=128, dx_mm=0.2, sensors=64, samples=1024,
             pixels=6092, frames=1, dtype="f32", delays="table", solid_angle=False, tile=128),
        # the paper-shaped live frame, device to device
        dict(name="frame_256_f32", kind="frames", n=256, dx_mm=0.1, sensors=512, samples=2048,
             pixels=21323, frames=1, dtype="f32", delays="table", solid_angle=False, tile=128),
        # the same frame as the paper times it: host signals in, host image out
        dict(name="host_256_f32", kind="host", n=256, dx_mm=0.1, sensors=512, samples=2048,
             pixels=21323, frames=1, dtype="f32", delays="table", solid_angle=False, tile=128),
        # the conventional back projection that the method is compared with
        dict(name="frame_256_constant_f32", kind="frames", n=256, dx_mm=0.1, sensors=512,
             samples=2048, pixels=21323, frames=1, dtype="f32", delays="constant",
             solid_angle=False, tile=128),
        # a short ragged sequence through the exact back projection
        dict(name="frames_256_solid_f16_12", kind="frames", n=250, dx_mm=0.1, sensors=500,
             samples=2000, pixels=20011, frames=12, dtype="f16", delays="table", solid_angle=True,
             tile=128),
        # precision form: many small 16-bit frames that share one table
        dict(name="batch_128_bf16_64", kind="frames", n=128, dx_mm=0.2, sensors=64, samples=1024,
             pixels=6092, frames=64, dtype="bf16", delays="table", solid_angle=False, tile=128),
        # a recorded sequence of paper-shaped frames reconstructed in one call
        dict(name="batch_256_f32_64", kind="frames", n=256, dx_mm=0.1, sensors=512, samples=2048,
             pixels=21323, frames=64, dtype="f32", delays="table", solid_angle=False, tile=256),
        # several subjects' pending frames, uneven in every size, in one plan
        dict(name="plan_uneven_f32_8", kind="plan", instances=8, n_lo=96, n_hi=384, sensors_lo=128,
             sensors_hi=1024, samples_lo=1024, samples_hi=4096, frames_lo=1, frames_hi=16,
             dtype="f32", tile=256, layout=4),
        # a burst of paper-shaped requests for two subjects at a server
        dict(name="serve_256_f32_24", kind="serve", n=256, dx_mm=0.1, sensors=512, samples=2048,
             pixels=21323, frames=24, subjects=2, dtype="f32"),
        # one live 3-D frame: the table stream from HBM
        dict(name="volume_f32_1", kind="frames", n=100, dx_mm=0.25, sensors=512, samples=2048,
             pixels=600000, depth=60, frames=1, dtype="f32", delays="table", solid_angle=False,
             tile=128),
        # a serving batch of 3-D frames of one subject
        dict(name="volume_bf16_8", kind="frames", n=120, dx_mm=0.25, sensors=640, samples=2048,
             pixels=1036800, depth=72, frames=8, dtype="bf16", delays="table", solid_angle=False,
             tile=128),
        # the off-line step: arrival times of one subject's sensors on the GPU
        dict(name="times_volume_32", kind="times", n=80, depth=48, dx_mm=0.25, sources=32),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["frames", "frames", "frames", "frames", "volume", "host", "plan", "serve",
                       "times"])
    dtype = rng.choice(["f32", "f32", "bf16", "f16"])
    if kind == "times":
        if rng.random() < 0.5:
            return dict(kind="times", n=_log_int(rng, 96, 384), depth=0, dx_mm=0.1,
                        sources=_log_int(rng, 16, 128))
        n = _log_int(rng, 48, 80)
        return dict(kind="times", n=n, depth=max(16, int(0.6 * n)), dx_mm=0.25,
                    sources=_log_int(rng, 4, 32))
    if kind == "plan":
        return dict(kind="plan", instances=rng.randint(3, 8), n_lo=96, n_hi=384, sensors_lo=128,
                    sensors_hi=1024, samples_lo=1024, samples_hi=4096, frames_lo=1, frames_hi=16,
                    dtype=dtype, tile=rng.choice([128, 256]), layout=rng.randint(0, 1 << 20))
    if kind == "volume":
        n, sensors = _log_int(rng, 48, 100), _log_int(rng, 96, 512)
        depth = max(24, int(0.6 * n))
        return dict(kind="frames", n=n, dx_mm=0.25, sensors=sensors, samples=_log_int(rng, 1024, 2048),
                    pixels=n * n * depth, depth=depth, frames=rng.choice([1, 2, 4, 8, 11, 16]),
                    dtype=dtype, delays="table", solid_angle=False, tile=128)
    n = _log_int(rng, 96, 320)
    sensors = _log_int(rng, 64, 1024)
    samples = _log_int(rng, 1000, 4096)
    pixels = int(rng.uniform(0.22, 0.34) * n * n)
    common = dict(n=n, dx_mm=round(rng.uniform(0.1, 0.2), 3), sensors=sensors, samples=samples,
                  pixels=pixels, dtype=dtype)
    most = max(1, int(7e8 / (pixels * sensors)))
    if kind == "serve":
        return dict(kind="serve", frames=min(rng.randint(4, 24), most), subjects=rng.randint(1, 3), **common)
    frames = 1 if rng.random() < 0.3 else min(_log_int(rng, 1, 64), most)
    if kind == "host":
        frames = min(frames, 8)
    return dict(kind=kind, frames=frames, delays=rng.choice(["table", "table", "constant"]),
                solid_angle=rng.random() < 0.25, tile=rng.choice([128, 256]), **common)


# --------------------------------------------------------------- geometry --
class _Subject:
    """One speed map with its sensors, mask and sampling (host arrays)."""

    def __init__(self, case, seed, salt=0):
        rng = np.random.default_rng([int(seed), int(salt), 11])
        n, depth = int(case["n"]), int(case.get("depth", 0))
        self.dx = case["dx_mm"] * 1e-3
        ns = int(case.get("sensors", case.get("sources", 0)))
        if depth:
            self.shape = (depth, n, n)
            s = n / 160.0
            centre = np.array([79.5 * s, 79.5 * s, 8.0 * s])
            self.origin = np.zeros(3)
            self.speed = synth.shell_skull_3d(self.shape, self.dx, tuple(centre), 56.0 * s, 5.0 * s,
                                              8.0 * s, rng, smooth_px=5.0 * s)
            self.centre = centre * self.dx
            self.sensors = synth.fibonacci_hemisphere(ns, 76.0 * s * self.dx, self.centre)
            self.sensors = np.minimum(self.sensors, (np.array(self.shape[::-1]) - 1) * self.dx)
            self.extent = 45.0 * s * self.dx
            self.crossing = 2 * 76.0 * s * self.dx / synth.C_WATER
            self.mask = None
            # as the serving subjects: 2048 samples at 20 ns for 160 nodes
            self.record = 2048 * 20e-9 * s
        else:
            self.shape = (n, n)
            s = n / 256.0
            self.origin = synth.centred_origin(self.shape, self.dx)
            self.speed = synth.skull_ring_2d(self.shape, 86.0 * s, 25.0 * s, rng, r_in_var=2.0 * s,
                                             thick_var=5.0 * s, smooth_px=6.0 * s)
            self.sensors = synth.ring_sensors(ns, RING * n * self.dx)
            self.centre = np.zeros(3)
            self.extent = 80.0 * s * self.dx
            self.record = CROSSINGS * 2 * RING * n * self.dx / synth.C_WATER
            self.mask = synth.nearest_nodes_mask(self.shape, int(case["pixels"])) if "pixels" in case else None
        self.nt = int(case.get("samples", 0))
        self.dt = self.record / self.nt if self.nt else 0.0

    def handle(self, case):
        flags = PAT_FLAG_TILE_256 if case.get("tile") == 256 else PAT_FLAG_TILE_128
        if case.get("delays") == "constant":
            bp = BP.constant(1560.0, self.shape, self.dx, self.origin, self.sensors, self.dt, self.nt,
                             mask=self.mask, flags=flags)
        else:
            bp = BP(self.speed, self.dx, self.origin, self.sensors, self.dt, self.nt, mask=self.mask,
                    flags=flags | PAT_FLAG_GPU_TABLE)
        if case.get("solid_angle"):
            bp.set_solid_angle(*self.elements())
        return bp

    def elements(self):
        """Inward normals and element lengths of the closed ring, full angle."""
        r = np.linalg.norm(self.sensors, axis=1)
        ns = len(r)
        return -self.sensors / r[:, None], np.full(ns, 2 * np.pi * r[0] / ns), 2 * np.pi


def _signals(sub, frames, dtype, seed, salt=0):
    """Seeded sensor records on the GPU: N-shaped pulses of small absorbers at
    about their arrival times plus 1 % noise, and the per-row scales of 16-bit
    records (None for float32)."""
    g = torch.Generator("cuda").manual_seed(int(seed) * 1000003 + int(salt) * 7919 + 5)
    nd = len(sub.shape)
    sens = torch.from_numpy(sub.sensors[:, :nd]).cuda()
    centre = torch.from_numpy(np.asarray(sub.centre[:nd], dtype=np.float64)).cuda()
    t = torch.arange(sub.nt, device="cuda", dtype=torch.float32) * sub.dt
    out = torch.zeros(frames, sens.shape[0], sub.nt, device="cuda")
    for f in range(frames):
        for _ in range(6):
            d = torch.randn(nd, generator=g, device="cuda", dtype=torch.float64)
            if nd == 3:
                d[2] = d[2].abs()
            r, amp, size = torch.rand(3, generator=g, device="cuda", dtype=torch.float64)
            pos = centre + d / d.norm() * r.sqrt() * sub.extent
            t0 = ((sens - pos).norm(dim=1) / 1600.0).float()[:, None]
            tau = ((1.0 + 2.0 * size) * sub.dx / 1540.0).float()
            out[f] += torch.where((t - t0).abs() <= tau, (0.5 + 0.5 * amp).float() * (t0 - t) / (2.0 * t0), 0.0)
        out[f] += 0.01 * out[f].abs().max() * torch.randn(out[f].shape, generator=g, device="cuda")
    if dtype == "f32":
        return out, None
    scale = out.abs().amax(dim=2).clamp_min(1e-30)
    return (out / scale[..., None]).to(DTYPES[dtype]).contiguous(), scale.contiguous()


def _pinned(t):
    return None if t is None else t.cpu().pin_memory()


def _codes(t):
    """numpy view of a host tensor: float32, or uint16 codes of 16-bit values."""
    return None if t is None else (t if t.dtype == torch.float32 else t.view(torch.int16)).numpy().view(
        np.float32 if t.dtype == torch.float32 else np.uint16)


def _instances(case):
    """Sizes of a plan's instances (the `layout` number names the mix)."""
    rng = np.random.default_rng([int(case["layout"]), 4])
    out = []
    for _ in range(case["instances"]):
        n = int(rng.integers(case["n_lo"], case["n_hi"] + 1))
        out.append(dict(n=n, dx_mm=float(rng.uniform(0.1, 0.2)), pixels=int(0.32 * n * n),
                        sensors=int(rng.integers(case["sensors_lo"], case["sensors_hi"] + 1)),
                        samples=int(rng.integers(case["samples_lo"], case["samples_hi"] + 1)),
                        frames=int(rng.integers(case["frames_lo"], case["frames_hi"] + 1)),
                        delays="table", tile=case["tile"]))
    return out


# ---------------------------------------------------------------- prepare --
def prepare(case, seed):
    kind = case["kind"]
    if kind == "times":
        return dict(kind=kind, sub=_Subject(case, seed))
    if kind == "plan":
        subs, bps, sigs, scales, outs, frames = [], [], [], [], [], []
        for k, c in enumerate(_instances(case)):
            sub = _Subject(c, seed, k)
            bp = sub.handle(c)
            sig, sc = _signals(sub, c["frames"], case["dtype"], seed, k)
            bps.append(bp)
            sigs.append(sig)
            scales.append(sc)
            frames.append(c["frames"])
            outs.append(torch.empty(bp.out_shape(c["frames"]), device="cuda"))
        plan = Plan(bps, frames, dtype=case["dtype"], autotune=True, graph=True)
        scales = None if case["dtype"] == "f32" else scales
        plan.execute(sigs, outs, scales)  # a plan's first execution tunes and captures it
        plan.sync()
        return dict(kind=kind, plan=plan, sig=sigs, scales=scales, out=outs)
    if kind == "serve":
        srv = Server(hbm_budget=16 << 30)
        per = _serve_frames(case)
        jobs = []
        for k, frames in enumerate(per):
            sub = _Subject(case, seed, k)
            sid = srv.register(sub.speed, sub.dx, sub.origin, sub.sensors, sub.dt, sub.nt, mask=sub.mask,
                               flags=PAT_FLAG_GPU_TABLE)
            sig, sc = _signals(sub, frames, case["dtype"], seed, k)
            sig, sc = _pinned(sig), _pinned(sc)
            out = torch.empty((frames,) + sub.shape, pin_memory=True)
            jobs.append((sid, sig, sc, out))
        # requests alternate between the subjects, as they would arrive
        order = sorted(((f / per[k], k, f) for k in range(len(per)) for f in range(per[k])))
        reqs = []
        for _, k, f in order:
            sid, sig, sc, out = jobs[k]
            reqs.append((sid, _codes(sig[f]), None if sc is None else sc[f].numpy(), out[f].numpy()))
        return dict(kind=kind, srv=srv, reqs=reqs, jobs=jobs, dtype=case["dtype"])
    sub = _Subject(case, seed)
    bp = sub.handle(case)
    sig, sc = _signals(sub, case["frames"], case["dtype"], seed)
    if kind == "host":
        sig, sc = _pinned(sig), _pinned(sc)
        out = torch.empty(bp.out_shape(case["frames"]), pin_memory=True)
        return dict(kind=kind, bp=bp, keep=(sig, sc, out), sig=_codes(sig), dtype=case["dtype"],
                    scales=None if sc is None else sc.numpy(), out=out.numpy())
    out = torch.empty(bp.out_shape(case["frames"]), device="cuda")
    return dict(kind=kind, bp=bp, sig=sig, scales=sc, out=out)


def _serve_frames(case):
    k = max(1, min(case["subjects"], case["frames"]))
    return [case["frames"] // k + (1 if i < case["frames"] % k else 0) for i in range(k)]


# -------------------------------------------------------------------- run --
def run(state):
    kind = state["kind"]
    if kind == "frames":
        return state["bp"].reconstruct(state["sig"], scales=state["scales"], out=state["out"])
    if kind == "host":
        return state["bp"].reconstruct_host(state["sig"], state["dtype"], scales=state["scales"],
                                            out=state["out"])
    if kind == "plan":
        return state["plan"].execute(state["sig"], state["out"], state["scales"])
    if kind == "serve":
        srv = state["srv"]
        tickets = [srv.submit(sid, sig, out, state["dtype"], scales) for sid, sig, scales, out in state["reqs"]]
        for t in tickets:
            srv.wait(t)
        return [job[3] for job in state["jobs"]]
    sub = state["sub"]
    return fmm_gpu(sub.speed, sub.dx, sub.origin, sub.sensors)


# ------------------------------------------------------------------- work --
def _frames_work(c, frames, dtype):
    pairs = float(c["pixels"]) * c["sensors"]
    word = 4 if dtype == "f32" else 2
    nodes = c["n"] ** 2 * (c.get("depth", 0) or 1)
    table = 0.0 if c.get("delays") == "constant" else 4.0 * pairs
    per_pair = (12.0 if c.get("delays") == "constant" else 0.0) + (12.0 if c.get("solid_angle") else 0.0)
    samples = float(frames) * c["sensors"] * c["samples"]
    return {"bytes": table + word * samples + 4.0 * frames * nodes,
            "flops": 5.0 * pairs * frames + per_pair * pairs + 4.0 * samples}


def work(case):
    if case["kind"] == "times":
        values = float(case["n"] ** 2 * (case["depth"] or 1)) * case["sources"]
        return {"bytes": 8.0 * values + 4.0 * values / case["sources"], "flops": 15.0 * values}
    if case["kind"] == "plan":
        parts = [_frames_work(c, c["frames"], case["dtype"]) for c in _instances(case)]
    elif case["kind"] == "serve":
        parts = [_frames_work(case, f, case["dtype"]) for f in _serve_frames(case)]
    else:
        parts = [_frames_work(case, case["frames"], case["dtype"])]
    return {k: sum(p[k] for p in parts) for k in ("bytes", "flops")}


# ------------------------------------------------------------------ exact --
def _arrivals(sub):
    """[sensors, *shape] first-order upwind arrival times in 64 bits: the
    Godunov system iterated to its fixed point over the whole grid."""
    inf = math.inf
    dims = len(sub.shape)
    speed = torch.from_numpy(sub.speed.astype(np.float64)).cuda()
    hf = sub.dx / speed
    ns = len(sub.sensors)
    T = torch.full((ns,) + tuple(m + 2 for m in sub.shape), inf, dtype=torch.float64, device="cuda")
    inner = (slice(None),) + (slice(1, -1),) * dims
    seeds, values = [], []
    for s, xyz in enumerate(sub.sensors):
        g = (xyz[:dims] - np.asarray(sub.origin)[:dims]) / sub.dx
        cell = np.minimum(np.floor(g).astype(int), np.array(sub.shape[::-1]) - 2)
        for corner in np.ndindex(*(2,) * dims):
            node = cell + np.array(corner)
            at = tuple(int(v) for v in node[::-1])
            seeds.append((s,) + tuple(v + 1 for v in at))
            values.append(float(np.linalg.norm((g - node) * sub.dx)) / float(sub.speed[at]))
    index = tuple(torch.tensor(v, device="cuda") for v in zip(*seeds))
    values = torch.tensor(values, dtype=torch.float64, device="cuda")
    T[index] = values
    for it in range(4 * sum(sub.shape)):
        a = []
        for d in range(dims):
            lo, hi = list(inner), list(inner)
            lo[1 + d], hi[1 + d] = slice(0, -2), slice(2, None)
            a.append(torch.minimum(T[tuple(lo)], T[tuple(hi)]))
        if dims == 3:
            low = torch.minimum(a[0], a[1])
            high = torch.maximum(a[0], a[1])
            a0, mid = torch.minimum(low, a[2]), torch.maximum(low, a[2])
            a1, a2 = torch.minimum(mid, high), torch.maximum(mid, high)
        else:
            a0, a1, a2 = torch.minimum(a[0], a[1]), torch.maximum(a[0], a[1]), None
        new = a0 + hf
        d01 = a1 - a0
        two = 0.5 * (a0 + a1 + torch.sqrt(2 * hf * hf - d01 * d01))
        new = torch.where(a1 < new, two, new)
        if a2 is not None:
            d02, d12 = a2 - a0, a2 - a1
            three = (a0 + a1 + a2 + torch.sqrt((3 * hf * hf - d01 * d01 - d02 * d02 - d12 * d12).clamp_min(0))) / 3
            new = torch.where(a2 < new, three, new)
        old = T[inner]
        new = torch.minimum(old, new)
        done = it % 16 == 15 and bool((old - new <= 1e-13 * new).all())
        T[inner] = new
        T[index] = values
        if done:
            break
    return T[inner]


def _image(sub, case, sig, scales):
    """Eq. (BP) in 64 bits: [frames, *shape], zero outside the mask."""
    dims = len(sub.shape)
    p = sig.cuda().double()
    if scales is not None:
        p = p * scales.cuda().double()[..., None]
    frames, ns, nt = p.shape
    b = 2 * p
    k = torch.arange(nt, device="cuda", dtype=torch.float64)
    b[..., 1:-1] -= k[1:-1] * (p[..., 2:] - p[..., :-2])
    b[..., -1] -= 2 * k[-1] * (p[..., -1] - p[..., -2])  # b_0 has t = 0
    where = torch.arange(int(np.prod(sub.shape)), device="cuda") if sub.mask is None else torch.from_numpy(
        np.flatnonzero(sub.mask)).cuda()
    left = where
    node = []
    for m in sub.shape[::-1]:  # x first
        node.append(left % m)
        left = left // m
    xyz = torch.stack(node, 1).double() * sub.dx + torch.from_numpy(np.asarray(sub.origin[:dims])).cuda()
    times = None if case.get("delays") == "constant" else _arrivals(sub).reshape(ns, -1)
    out = torch.zeros(frames, int(np.prod(sub.shape)), dtype=torch.float64, device="cuda")
    acc = torch.zeros(frames, where.numel(), dtype=torch.float64, device="cuda")
    normals, elem, omega = sub.elements() if case.get("solid_angle") else (None, None, None)
    for s in range(ns):
        v = xyz - torch.from_numpy(sub.sensors[s, :dims].copy()).cuda()
        r = v.norm(dim=1)
        u = (r / 1560.0 if times is None else times[s, where]) / sub.dt
        i = u.clamp(0, nt - 2).long()
        phase = u - i
        row = b[:, s]
        term = row[:, i] + phase * (row[:, i + 1] - row[:, i])
        w = 1.0 / ns
        if normals is not None:
            w = elem[s] * (v @ torch.from_numpy(normals[s, :dims].copy()).cuda()) / r ** dims / omega
        acc += torch.where(u <= nt - 1, w * term, 0.0)
    out[:, where] = acc
    return out.reshape((frames,) + sub.shape)


def _solve_cost(sub_sizes):
    return sum(nodes * ns * steps for nodes, ns, steps in sub_sizes)


def exact(case, seed):
    kind = case["kind"]
    parts = [c for c in _instances(case)] if kind == "plan" else [case] * (len(_serve_frames(case)) if kind == "serve" else 1)
    cost = 0.0
    for c in parts:
        depth = c.get("depth", 0)
        cost += c["n"] ** 2 * (depth or 1) * c.get("sensors", c.get("sources", 0)) * (2 * c["n"] + depth)
    if cost > 1.2e11 and case.get("delays") != "constant":
        return None  # the plain solver would take too long
    if kind == "times":
        return _arrivals(_Subject(case, seed))
    if kind in ("plan", "serve"):
        frames = [c["frames"] for c in parts] if kind == "plan" else _serve_frames(case)
        outs = []
        for k, (c, f) in enumerate(zip(parts, frames)):
            sub = _Subject(c, seed, k)
            outs.append(_image(sub, c, *_signals(sub, f, case["dtype"], seed, k)))
        return outs
    sub = _Subject(case, seed)
    return _image(sub, case, *_signals(sub, case["frames"], case["dtype"], seed))
