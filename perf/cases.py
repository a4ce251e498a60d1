"""Timed cases of the differentiable CT operators: what a user's program asks of this framework, from one
small 2D slice to a 512^3 scan.

Every case is a dict of plain values. `op` says which public entry points a pass goes through:

  fbp          filtered back-projection of a scan (operators.fbp), the analytic reconstruction
  train        a projection layer and its gradient: forward projection, then the matched adjoint through
               autograd, as in every step of a network that holds the projector
  step         one data-consistency step x - alpha A^T (A x - p) (operators.gradient_step)
  learned_fbp  FBP with a trained back-projection layer: filter, back-projection layer, and the gradient with
               respect to the filtered sinogram
  simulate     simulated acquisition: forward projection, gantry motion blur, detector noise
  plan         volumes of uneven sizes, each with its own geometry: forward projection, matched adjoint and
               back-projection of a batched plan
  unrolled     the unrolled, checkpointed gradient-descent network, forward and backward

`beam` is parallel or fan (2D), or circle, helix or free (cone beam; free: one projection matrix per view, from
a jittered orbit). Sizes are voxels and detector pixels, lengths millimetres, `arc` the angular range in units
of pi. The scans and phantoms are random ellipsoids (for scans their exact chord lengths plus noise), the
incoming gradients a residual: the difference of two scans plus noise.
"""
import math

import numpy as np
import torch

from paper_2511_08427_gb300 import artifacts, operators as ops, unrolled

DTYPES = {"float32": torch.float32, "bfloat16": torch.bfloat16, "float16": torch.float16}


def listed():
    return [
        # the smallest call: FBP of one 2D parallel-beam slice (128^2, 183 bins, 180 views), as in an
        # interactive or per-slice loop; launches and latency count
        dict(name="fbp_parallel128", op="fbp", beam="parallel", nz=1, ny=128, nx=128, voxel=1.0, nv=1, nu=183,
             pitch=1.0, views=180, arc=1.0, sid=0.0, sdd=0.0, batch=1, dtype="float32"),
        # one 2D fan-beam slice (256^2, 512 bins, 360 views) inside a network: projection and its gradient
        dict(name="train_fan256", op="train", beam="fan", nz=1, ny=256, nx=256, voxel=0.5, nv=1, nu=512,
             pitch=1.0, views=360, arc=2.0, sid=1000.0, sdd=1500.0, batch=1, dtype="float32"),
        # a training batch of larger 2D slices of odd size
        dict(name="train_parallel_batch", op="train", beam="parallel", nz=1, ny=362, nx=362, voxel=0.8, nv=1, nu=513,
             pitch=0.8, views=300, arc=1.0, sid=0.0, sdd=0.0, batch=8, dtype="float32"),
        # a small cone-beam scan whose sizes are multiples of nothing: projection and its gradient
        dict(name="train_cone_ragged", op="train", beam="circle", nz=75, ny=97, nx=101, voxel=0.5, nv=109, nu=157,
             pitch=0.77, views=90, arc=2.0, sid=750.0, sdd=1200.0, batch=1, dtype="float32"),
        # a batch of two volumes in 16-bit storage (mixed-precision training): projection and its gradient
        dict(name="train_cone_bf16", op="train", beam="circle", nz=128, ny=192, nx=192, voxel=0.5, nv=256, nu=320,
             pitch=0.7, views=120, arc=2.0, sid=750.0, sdd=1200.0, batch=2, dtype="bfloat16"),
        # the standard cone-beam configuration (256^3, 512^2 detector, 360 views): one gradient step
        dict(name="step_cone256", op="step", beam="circle", nz=256, ny=256, nx=256, voxel=0.5, nv=512, nu=512,
             pitch=0.6, views=360, arc=2.0, sid=750.0, sdd=1200.0, batch=1, dtype="float32"),
        # the paper's FDK listing (256^3, 400 x 600 detector) with a trained back-projection layer
        dict(name="learned_fdk256", op="learned_fbp", beam="circle", nz=256, ny=256, nx=256, voxel=0.5, nv=400,
             nu=600, pitch=1.0, views=360, arc=2.0, sid=750.0, sdd=1200.0, batch=1, dtype="float32"),
        # simulated half-precision data of a helical scan, for a training set
        dict(name="simulate_helix_f16", op="simulate", beam="helix", nz=160, ny=192, nx=192, voxel=0.5, nv=192,
             nu=384, pitch=0.6, views=360, arc=2.0, sid=750.0, sdd=1200.0, batch=1, dtype="float16", blur=7),
        # eight volumes of 64^3 to 160^3, each with its own scan, in one plan
        dict(name="plan_uneven", op="plan", beam="circle", volumes=8, side_lo=64, side_hi=160, views_lo=60,
             views_hi=180, det_lo=128, det_hi=256, voxel=0.5, sid=750.0, sdd=1200.0, dtype="float32"),
        # an unrolled network of ten checkpointed iterations on a small cone-beam scan
        dict(name="unrolled_cone96", op="unrolled", beam="circle", nz=64, ny=96, nx=96, voxel=0.5, nv=96, nu=144,
             pitch=0.8, views=60, arc=2.0, sid=750.0, sdd=1200.0, batch=1, dtype="float32", iterations=10),
        # an ordered subset (48 views) of the 512^3 scan on a free trajectory: projection and its gradient
        dict(name="train_free512_subset", op="train", beam="free", nz=512, ny=512, nx=512, voxel=0.4, nv=1024,
             nu=1024, pitch=0.4, views=48, arc=2.0, sid=750.0, sdd=1200.0, batch=1, dtype="float32"),
        # FDK of a whole 512^3 scan on a free trajectory (720 views of 1024^2)
        dict(name="fbp_free512", op="fbp", beam="free", nz=512, ny=512, nx=512, voxel=0.4, nv=1024, nu=1024,
             pitch=0.4, views=720, arc=2.0, sid=750.0, sdd=1200.0, batch=1, dtype="float32"),
    ]


def draw(rng):
    def size(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    def fitted(c):
        """The detector pitch at which the volume's shadow fills about nine tenths of the detector."""
        mag = c["sdd"] / c["sid"] if c["sid"] else 1.0
        wide = mag * c["voxel"] * math.hypot(c["nx"], c["ny"]) / (0.9 * c["nu"])
        tall = mag * c["voxel"] * c["nz"] / (0.9 * c["nv"]) if c["nz"] > 1 else 0.0
        c["pitch"] = round(max(wide, tall), 3)
        return c

    op = rng.choice(["fbp2", "train2", "fbp3", "train3", "train3", "step3", "learned_fbp3", "simulate3", "plan",
                     "unrolled3"])
    dtype = rng.choice(["float32", "float32", "bfloat16", "float16"])
    if op == "plan":
        lo = 8 * size(6, 12)
        return dict(op="plan", beam="circle", volumes=rng.randint(3, 10), side_lo=lo, side_hi=lo + 8 * rng.randint(2, 9),
                    views_lo=size(40, 80), views_hi=size(80, 200), det_lo=16 * size(6, 10), det_hi=16 * size(10, 18),
                    voxel=0.5, sid=750.0, sdd=1200.0, dtype=rng.choice(["float32", "bfloat16"]))
    if op.endswith("2"):
        beam = rng.choice(["parallel", "fan"])
        n = size(100, 512)
        c = dict(op=op[:-1], beam=beam, nz=1, ny=n, nx=max(64, int(n * rng.uniform(0.8, 1.25))),
                 voxel=rng.choice([0.5, 0.8, 1.0]), nv=1, nu=max(64, int(n * rng.uniform(1.3, 2.0))), pitch=1.0,
                 views=size(90, 500), arc=1.0 if beam == "parallel" else 2.0, sid=0.0 if beam == "parallel" else 1000.0,
                 sdd=0.0 if beam == "parallel" else 1500.0, batch=size(1, 12), dtype="float32")
        return fitted(c)
    op = op[:-1]
    big = {"fbp": 320, "train": 224, "step": 224, "learned_fbp": 224, "simulate": 224, "unrolled": 96}[op]
    n = size(48, big)
    c = dict(op=op, beam=rng.choice(["circle", "helix", "free"]), nz=max(24, int(n * rng.uniform(0.5, 1.0))),
             ny=max(32, int(n * rng.uniform(0.8, 1.0))), nx=n, voxel=rng.choice([0.4, 0.5, 0.7]),
             nv=max(32, int(n * rng.uniform(0.8, 1.6))), nu=max(48, int(n * rng.uniform(1.2, 2.0))), pitch=1.0,
             views=size(30, 240), arc=2.0, sid=750.0, sdd=1200.0, batch=1, dtype=dtype)
    if rng.random() < 0.6:   # most programs take round sizes, many do not
        for k in ("nz", "ny", "nx", "nv", "nu"):
            c[k] = 8 * max(4, round(c[k] / 8))
    if op == "simulate":
        c["blur"] = rng.choice([3, 5, 7, 9])
    if op == "unrolled":
        c["dtype"], c["iterations"], c["views"] = "float32", rng.randint(3, 10), size(30, 90)
    if op == "fbp" and c["beam"] == "helix":
        c["beam"] = "circle"
    if op in ("fbp", "learned_fbp") and c["dtype"] == "float16":
        c["dtype"] = "float32"   # the plain sum over the views can exceed the range of 16-bit floats
    return fitted(c)


# -- geometry: the frame of every view, in plain numpy ---------------------------------------------------------


def frames(c):
    """Source (or, for parallel beams, ray direction), detector centre and detector axes of every view, in mm."""
    n = c["views"]
    t = np.arange(n) * (c["arc"] * math.pi / n)
    cos, sin, zero = np.cos(t), np.sin(t), np.zeros(n)
    eu, ev = np.stack([-sin, cos, zero], 1), np.tile([0.0, 0.0, 1.0], (n, 1))
    if c["beam"] == "parallel":
        return np.stack([-cos, -sin, zero], 1), np.zeros((n, 3)), eu, ev
    z = pitch_of(c) * (np.arange(n) - 0.5 * (n - 1)) * (c["arc"] / n) / 2.0
    src = np.stack([c["sid"] * cos, c["sid"] * sin, z], 1)
    det = np.stack([-(c["sdd"] - c["sid"]) * cos, -(c["sdd"] - c["sid"]) * sin, z], 1)
    if c["beam"] == "free":
        r = np.random.default_rng(n)
        src, det = src + r.normal(0.0, 0.5, (n, 3)), det + r.normal(0.0, 0.5, (n, 3))
        for k, turn in enumerate(np.deg2rad(r.normal(0.0, 0.2, (n, 3)))):
            a, b, g = turn
            rz = lambda x: np.array([[math.cos(x), -math.sin(x), 0], [math.sin(x), math.cos(x), 0], [0, 0, 1]])  # noqa: E731
            ry = np.array([[math.cos(b), 0, math.sin(b)], [0, 1, 0], [-math.sin(b), 0, math.cos(b)]])
            rot = rz(a) @ ry @ rz(g)
            eu[k], ev[k] = rot @ eu[k], rot @ ev[k]
    return src, det, eu, ev


def pitch_of(c):
    """Helical pitch: half the detector's height at the isocentre."""
    return 0.5 * c["nv"] * c["pitch"] * c["sid"] / c["sdd"] if c["beam"] == "helix" else 0.0


def corner(c):
    """Source -> pixel (0, 0) and the steps per pixel (perspective beams)."""
    src, det, eu, ev = frames(c)
    d0 = det - src - 0.5 * (c["nu"] - 1) * c["pitch"] * eu - 0.5 * (c["nv"] - 1) * c["pitch"] * ev
    return src, d0, c["pitch"] * eu, c["pitch"] * ev


def matrices(c):
    src, d0, du, dv = corner(c)
    inv = np.linalg.inv(np.stack([du, dv, d0], 2))
    return np.concatenate([inv, -np.einsum("nij,nj->ni", inv, src)[:, :, None]], 2)


def geometry(c):
    arc = c["arc"] * math.pi
    if c["beam"] == "parallel":
        return ops.Geometry.parallel2d((c["ny"], c["nx"]), (c["voxel"],) * 2, c["nu"], c["pitch"], c["views"], arc)
    if c["beam"] == "fan":
        return ops.Geometry.fan2d((c["ny"], c["nx"]), (c["voxel"],) * 2, c["nu"], c["pitch"], c["views"], arc,
                                  c["sid"], c["sdd"])
    size = ((c["nz"], c["ny"], c["nx"]), (c["voxel"],) * 3, (c["nv"], c["nu"]), (c["pitch"],) * 2)
    if c["beam"] == "free":
        return ops.Geometry.cone_from_matrices(*size, matrices(c))
    return ops.Geometry.cone_circular(*size, c["views"], arc, c["sid"], c["sdd"], helical_pitch=pitch_of(c))


# -- inputs ----------------------------------------------------------------------------------------------------


def ellipsoids(c, seed, count=8):
    """(maps to the unit ball [count, 3, 3], centres, densities) of random ellipsoids inside the volume."""
    r = np.random.default_rng(seed)
    half = 0.5 * c["voxel"] * np.array([c["nx"], c["ny"], max(c["nz"], min(c["nx"], c["ny"])) if c["nz"] == 1 else c["nz"]])
    got = []
    for _ in range(count):
        q, _ = np.linalg.qr(r.normal(size=(3, 3)))
        axes = r.uniform(0.1, 0.45, 3) * half.min()
        centre = r.uniform(-0.5, 0.5, 3) * half * (1.0, 1.0, 0.0 if c["nz"] == 1 else 1.0)
        got.append((q.T / axes[:, None], centre, r.uniform(0.1, 1.0)))
    return got


def axis(n, step, **kw):
    return (torch.arange(n, device="cuda", **kw) - 0.5 * (n - 1)) * step


def phantom(c, seed, batch):
    x, y, z = (axis(c[k], c["voxel"], dtype=torch.float32) for k in ("nx", "ny", "nz"))
    out = torch.zeros((batch, c["nz"], c["ny"], c["nx"]), device="cuda")
    for b in range(batch):
        for m, o, rho in ellipsoids(c, seed * 64 + b):
            far = 0.0
            for i in range(3):
                far = far + ((x - o[0]) * m[i, 0] + ((y - o[1]) * m[i, 1])[:, None] + ((z - o[2]) * m[i, 2])[:, None, None]) ** 2
            out[b] += rho * (far <= 1.0)
    return out


def scan(c, seed, batch, count=6):
    """Chord lengths of random ellipsoids along every ray, [batch, views, nv, nu], in FP32."""
    src, det, eu, ev = frames(c)
    u, v = axis(c["nu"], c["pitch"], dtype=torch.float32), axis(c["nv"], c["pitch"], dtype=torch.float32)[:, None]
    out = torch.zeros((batch, c["views"], c["nv"], c["nu"]), device="cuda")
    put = lambda a: torch.tensor(a, dtype=torch.float32, device="cuda")[:, None, None]  # noqa: E731
    for n0 in range(0, c["views"], 40):
        k = slice(n0, n0 + 40)
        for b in range(batch):
            for m, o, rho in ellipsoids(c, seed * 64 + b, count):
                if c["beam"] == "parallel":   # from a point of the detector along the ray's direction
                    way, start = [put((src[k] @ m.T)[:, i]) for i in range(3)], ((det[k] - o) @ m.T)
                    at = [put(start[:, i]) + put((eu[k] @ m.T)[:, i]) * u for i in range(3)]
                    long = 1.0
                else:
                    p0, pu, pv = ((a[k] @ m.T) for a in (det - src, eu, ev))
                    way = [put(p0[:, i]) + put(pu[:, i]) * u + put(pv[:, i]) * v for i in range(3)]
                    at = [put(((src[k] - o) @ m.T)[:, i]) for i in range(3)]
                    long = (c["sdd"] ** 2 + u * u + v * v).sqrt()
                aa = sum(w * w for w in way)
                ab = sum(w * s for w, s in zip(way, at))
                cc = sum(s * s for s in at) - 1.0
                out[b, k] += (rho * 2.0) * long * (ab * ab - aa * cc).clamp_(min=0.0).sqrt_() / aa
    return out


def normal(shape, seed):
    return torch.randn(shape, device="cuda", generator=torch.Generator("cuda").manual_seed(int(seed)))


def noisy_scan(c, seed, batch):
    p = scan(c, seed, batch)
    return p.add_(normal(p.shape, seed), alpha=0.01 * float(p.max()))


def residual(c, seed, batch):
    p = scan(c, seed, batch, 4) - scan(c, seed + 7, batch, 4)
    return p.add_(normal(p.shape, seed + 1), alpha=0.1 * float(p.abs().max()))


def shaped(c, t):
    """In the layout and type of the case's tensors (2D: no z or v axis; no batch axis for one)."""
    t = t[:, 0] if c["nz"] == 1 and t.shape[1] == 1 and t.shape[-2:] == (c["ny"], c["nx"]) else t
    t = t[:, :, 0] if c["nv"] == 1 and t.dim() == 4 else t
    t = t[0] if c["batch"] == 1 else t
    return t.to(DTYPES[c["dtype"]]).contiguous()


def members(c):
    """The geometries of a plan, as cases of their own."""
    out, last = [], max(c["volumes"] - 1, 1)
    for i in range(c["volumes"]):
        part = lambda lo, hi, q: int(q * round((lo + (hi - lo) * i / last) / q))  # noqa: B023,E731
        side, det = part(c["side_lo"], c["side_hi"], 8), part(c["det_lo"], c["det_hi"], 16)
        out.append(dict(c, op="train", beam="helix" if i % 2 else "circle", nz=side, ny=side, nx=side, nv=det, nu=det,
                        views=part(c["views_lo"], c["views_hi"], 1), arc=2.0, batch=1,
                        pitch=round(c["sdd"] / c["sid"] * side * c["voxel"] * math.sqrt(2.0) / (0.9 * det), 3)))
    return out


def prepare(case, seed):
    op, s = case["op"], {"case": case}
    if op == "plan":
        parts = members(case)
        s["geometries"] = [geometry(m) for m in parts]
        s["plan"] = ops.Plan(s["geometries"], DTYPES[case["dtype"]])
        s["vols"] = [shaped(m, phantom(m, seed * 32 + i, 1)) for i, m in enumerate(parts)]
        s["cots"] = [shaped(m, residual(m, seed * 32 + i, 1)) for i, m in enumerate(parts)]
        return s
    g, batch = geometry(case), case["batch"]
    s["g"] = g
    if op in ("train", "step", "simulate"):
        s["x"] = shaped(case, phantom(case, seed, batch))
    if op == "train":
        s["x"].requires_grad_(True)
        s["cot"] = shaped(case, residual(case, seed, batch))
    if op in ("fbp", "learned_fbp", "step", "unrolled"):
        s["p"] = shaped(case, noisy_scan(case, seed, batch))
    if op == "learned_fbp":
        s["layer"] = (ops.ConeBackProjectionFor3D(ops.BP_INV_W2))
        s["cot"] = shaped(case, phantom(case, seed + 3, batch) - phantom(case, seed + 5, batch)
                          + 0.05 * normal((batch, case["nz"], case["ny"], case["nx"]), seed))
    if op == "step":
        s["alpha"] = step_size(case)
    if op == "simulate":
        s["noise"] = normal(g.sinogram_shape, seed)
        s["angles"] = torch.linspace(0.0, math.pi, case["views"], device="cuda")
    if op == "unrolled":
        s["net"] = unrolled.UnrolledGD(g, case["iterations"], alpha0=step_size(case), checkpoint=True)
        s["p"].requires_grad_(True)
        s["cot"] = normal(g.volume_shape, seed)
    return s


def step_size(c):
    """A step at which gradient descent converges: 1 / (longest path x views x samples' mean weight)."""
    side = c["voxel"] * max(c["nx"], c["ny"], c["nz"])
    mag = c["sdd"] / c["sid"]
    return 1.0 / (1.5 * side * c["views"] * c["voxel"] * max(1.0, (mag * c["voxel"] / c["pitch"]) ** 2))


# -- one pass --------------------------------------------------------------------------------------------------


def run(state):
    c = state["case"]
    op = c["op"]
    if op == "plan":
        plan = state["plan"]
        sinos = [torch.empty_like(t) for t in state["cots"]]
        grads = [torch.empty_like(t) for t in state["vols"]]
        backs = [torch.empty_like(t) for t in state["vols"]]
        plan.forward_project(state["vols"], sinos)
        plan.adjoint(state["cots"], grads)
        plan.back_project(state["cots"], backs, ops.BP_INV_W2)
        return {"projections": sinos, "gradients": grads, "back_projections": backs}
    g = state["g"]
    if op == "fbp":
        return ops.fbp(state["p"], g)
    if op == "train":
        p = ops.project(state["x"], g)
        grad, = torch.autograd.grad(p, state["x"], state["cot"])
        return {"projection": p.detach(), "gradient": grad}
    if op == "step":
        return ops.gradient_step(state["x"], state["p"], state["alpha"], g)
    if op == "learned_fbp":
        q = ops.fbp_filter(state["p"], g).requires_grad_(True)
        x = state["layer"](q, g)
        grad, = torch.autograd.grad(x, q, state["cot"])
        return {"volume": x.detach(), "gradient": grad}
    if op == "simulate":
        p = ops.project(state["x"], g)
        p = artifacts.motion_blur(p, g, state["angles"], c["blur"])
        return artifacts.gaussian_noise(p, g, state["noise"], 0.0, 0.05)
    x = state["net"](state["p"])
    grads = torch.autograd.grad(x, [state["net"].alpha, state["p"]], state["cot"])
    return {"volume": x.detach(), "alpha_gradient": grads[0], "scan_gradient": grads[1]}


# -- the work that a pass cannot do without ----------------------------------------------------------------------


def work(case):
    if case["op"] == "plan":
        parts = [work(dict(m, op=o)) for m in members(case) for o in ("project", "adjoint", "back")]
        return {k: sum(w[k] for w in parts) for k in ("bytes", "flops")}
    c, op, size = case, case["op"], 4 if case["dtype"] == "float32" else 2
    vox = c["batch"] * c["nx"] * c["ny"] * c["nz"]
    pix = c["batch"] * c["views"] * c["nv"] * c["nu"]
    mag = c["sdd"] / c["sid"] if c["sid"] else 1.0
    # samples in the volume: its extent over the area of a ray's cell at the centre times the step (half a voxel)
    rays = mag * c["voxel"] / c["pitch"]
    samples = 2.0 * vox * c["views"] * (rays * rays if c["nz"] > 1 else rays)
    line = {True: 34.0, False: 16.0}[c["nz"] > 1] * samples   # interpolation along the rays, or its transpose
    cast = 18.0 * vox * c["views"]                             # bilinear taps of every voxel in every view
    ramp = 10.0 * pix * math.log2(2 * c["nu"])
    moved, flops = {"project": (vox + pix, line), "adjoint": (vox + pix, line), "back": (vox + pix, cast),
                    "fbp": (vox + pix, cast + ramp), "train": (2 * (vox + pix), 2 * line),
                    "step": (2 * vox + pix, 2 * line), "learned_fbp": (2 * (vox + pix), 2 * cast + ramp),
                    "simulate": (vox + pix + 2 * pix, line + 10.0 * c.get("blur", 0) * pix),
                    "unrolled": (vox + 2 * pix, 8 * c.get("iterations", 0) * line)}[op]
    return {"bytes": size * moved, "flops": flops}


# -- the same in 64 bits, by plain torch -------------------------------------------------------------------------


def exact(case, seed):
    c = case
    if c["op"] == "plan":
        parts, out = members(c), {"projections": [], "gradients": [], "back_projections": []}
        s = prepare(c, seed)
        for m, x, y in zip(parts, s["vols"], s["cots"]):
            out["projections"].append(exact_project(m, x))
            out["gradients"].append(exact_adjoint(m, y))
            out["back_projections"].append(exact_back(m, y, True))
        return out
    s = prepare(c, seed)
    op = c["op"]
    if op == "fbp":
        return exact_back(c, exact_ramp(c, s["p"]), c["beam"] != "parallel")
    if op == "train":
        return {"projection": exact_project(c, s["x"].detach()), "gradient": exact_adjoint(c, s["cot"])}
    if op == "step":
        return exact_step(c, s["x"].double(), s["p"].double(), s["alpha"])
    if op == "learned_fbp":
        q = exact_ramp(c, s["p"])
        return {"volume": exact_back(c, q, True), "gradient": exact_spread(c, s["cot"])}
    if op == "simulate":
        p = exact_project(c, s["x"])
        p = exact_blur(p, s["angles"].double(), c["blur"])
        return p + 0.05 * s["noise"].double()
    with torch.enable_grad():
        p = s["p"].detach().double().requires_grad_(True)
        alpha = s["net"].alpha.detach().double().requires_grad_(True)
        x = torch.zeros(s["g"].volume_shape, device="cuda", dtype=torch.float64)
        for k in range(c["iterations"]):
            x = x - alpha[k] * Adjoint64.apply(Project64.apply(x, c) - p, c)
        grads = torch.autograd.grad(x, [alpha, p], s["cot"].double())
    return {"volume": x.detach(), "alpha_gradient": grads[0], "scan_gradient": grads[1]}


class Project64(torch.autograd.Function):
    @staticmethod
    def forward(ctx, x, c):
        ctx.c = c
        return exact_project(c, x)

    @staticmethod
    def backward(ctx, y):
        return exact_adjoint(ctx.c, y), None


class Adjoint64(torch.autograd.Function):
    @staticmethod
    def forward(ctx, y, c):
        ctx.c = c
        return exact_adjoint(c, y)

    @staticmethod
    def backward(ctx, x):
        return exact_project(ctx.c, x), None


def exact_step(c, x, p, alpha):
    return x - alpha * exact_adjoint(c, exact_project(c, x) - p)


def rays64(c, k):
    """Closest point to the volume's centre and unit direction of the rays of views k, [rays, 3] each."""
    put = lambda a: torch.tensor(a, dtype=torch.float64, device="cuda")[:, None, None, :]  # noqa: E731
    src, det, eu, ev = (put(a[k]) for a in frames(c))
    u, v = axis(c["nu"], c["pitch"], dtype=torch.float64)[:, None], axis(c["nv"], c["pitch"], dtype=torch.float64)[:, None, None]
    pix = det + u * eu + v * ev
    way = src.expand_as(pix) if c["beam"] == "parallel" else pix - src
    way = (way / way.norm(dim=-1, keepdim=True)).reshape(-1, 3)
    pix = pix.reshape(-1, 3)
    return pix - (pix * way).sum(-1, keepdim=True) * way, way


def samples64(c):
    """Chunks of the rays' samples: (flat ray indices, grid_sample positions [1, rays, samples, 1, 3])."""
    n = torch.tensor([c["nx"], c["ny"], c["nz"]], dtype=torch.float64, device="cuda")
    dt = 0.5 * c["voxel"]
    per = c["nv"] * c["nu"]
    group = max(1, (1 << 21) // per)
    for n0 in range(0, c["views"], group):
        at, way = rays64(c, slice(n0, min(n0 + group, c["views"])))
        q, d = at / c["voxel"] + 0.5 * (n - 1), way / c["voxel"]
        d = torch.where(d.abs() < 1e-14, torch.full_like(d, 1e-14), d)
        ends = torch.stack([(-1.0 - q) / d, (n - q) / d])
        lo, hi = ends.amin(0).amax(-1), ends.amax(0).amin(-1)
        k0 = torch.floor(lo / dt - 0.5)
        count = torch.ceil(hi / dt - 0.5) - k0 + 1
        rays = torch.nonzero(hi > lo).reshape(-1)
        if not len(rays):
            continue
        rays = rays[torch.argsort(count[rays], descending=True)]
        counts = count[rays].cpu()
        step = 64
        for s0 in range(0, int(counts[0]), step):
            live = rays[:int((counts > s0).sum())]
            some = max(1, (1 << 25) // step)
            for r0 in range(0, len(live), some):
                r = live[r0:r0 + some]
                t = (k0[r, None] + (s0 + 0.5) + torch.arange(step, dtype=torch.float64, device="cuda")) * dt
                pos = q[r, None, :] + t[..., None] * d[r, None, :]
                yield n0 * per + r, ((2.0 * pos + 1.0) / n - 1.0)[None, :, :, None, :]


def out64(c, got, sino):
    if sino:
        got = got.reshape((-1, c["views"], c["nv"], c["nu"]) if c["nz"] > 1 else (-1, c["views"], c["nu"]))
    else:
        got = got.reshape((-1, c["nz"], c["ny"], c["nx"]) if c["nz"] > 1 else (-1, c["ny"], c["nx"]))
    return got[0] if c["batch"] == 1 else got


def exact_project(c, x):
    x = x.detach().double().reshape(-1, 1, c["nz"], c["ny"], c["nx"])
    out = torch.zeros((x.shape[0], c["views"] * c["nv"] * c["nu"]), dtype=torch.float64, device="cuda")
    for r, grid in samples64(c):
        for b in range(x.shape[0]):
            got = torch.nn.functional.grid_sample(x[b:b + 1], grid, "bilinear", "zeros", align_corners=False)
            out[b].index_add_(0, r, got.reshape(len(r), -1).sum(1))
    return out64(c, out * (0.5 * c["voxel"]), True)


def exact_adjoint(c, y):
    y = y.detach().double().reshape(-1, c["views"] * c["nv"] * c["nu"]) * (0.5 * c["voxel"])
    out = torch.zeros((y.shape[0], 1, c["nz"], c["ny"], c["nx"]), dtype=torch.float64, device="cuda")
    for r, grid in samples64(c):
        for b in range(y.shape[0]):
            w = y[b, r].reshape(1, 1, -1, 1, 1).expand((1, 1) + tuple(grid.shape[1:4]))
            out[b:b + 1] += torch.ops.aten.grid_sampler_3d_backward(w, out[b:b + 1], grid, 0, 0, False, [True, False])[0]
    return out64(c, out, False)


def views64(c):
    """For every view: grid_sample positions [1, voxels, 1, 2] of the voxels on the detector, and their 1 / w."""
    x, y, z = (axis(c[k], c["voxel"], dtype=torch.float64) for k in ("nx", "ny", "nz"))
    size = torch.tensor([c["nu"], c["nv"]], dtype=torch.float64, device="cuda")
    if c["beam"] == "parallel":
        _, det, eu, ev = frames(c)
    else:
        mats = matrices(c)
    for n in range(c["views"]):
        if c["beam"] == "parallel":
            u = (x * eu[n, 0] + (y * eu[n, 1])[:, None]) / c["pitch"] + 0.5 * (c["nu"] - 1)
            pos, iw = torch.stack([u, torch.zeros_like(u)], -1), None
        else:
            a, b, w = (x * m[0] + (y * m[1])[:, None] + (z * m[2])[:, None, None] + m[3] for m in mats[n].tolist())
            iw = 1.0 / w
            pos = torch.stack([a * iw, b * iw], -1)
            pos = torch.where((w > 0.0)[..., None], pos, torch.full_like(pos, -1e6))
            iw = iw.reshape(-1)
        yield n, ((2.0 * pos + 1.0) / size - 1.0).reshape(1, -1, 1, 2), iw


def exact_back(c, p, weighted):
    """Voxel-driven back-projection (weighted: by 1 / w^2)."""
    p = p.detach().double().reshape(-1, c["views"], c["nv"], c["nu"])
    out = torch.zeros((p.shape[0], c["nz"] * c["ny"] * c["nx"]), dtype=torch.float64, device="cuda")
    for n, grid, iw in views64(c):
        for b in range(p.shape[0]):
            got = torch.nn.functional.grid_sample(p[b:b + 1, n:n + 1], grid, "bilinear", "zeros", align_corners=False).reshape(-1)
            out[b] += got * iw * iw if weighted and iw is not None else got
    return out64(c, out, False)


def exact_spread(c, x):
    """The transpose of exact_back(weighted)."""
    x = x.detach().double().reshape(-1, 1, 1, c["nz"] * c["ny"] * c["nx"], 1)
    out = torch.zeros((x.shape[0], c["views"], c["nv"], c["nu"]), dtype=torch.float64, device="cuda")
    for n, grid, iw in views64(c):
        for b in range(x.shape[0]):
            w = x[b] * (iw * iw).reshape(1, 1, -1, 1)
            out[b, n] = torch.ops.aten.grid_sampler_2d_backward(w, out[b:b + 1, n:n + 1], grid, 0, 0, False, [True, False])[0][0, 0]
    return out64(c, out, True)


def exact_ramp(c, p):
    """Cosine weight (diverging beams), band-limited ramp and FBP scale."""
    nu, p = c["nu"], p.detach().double().reshape(-1, c["views"], c["nv"], c["nu"])
    if c["beam"] == "parallel":
        scale = torch.full((c["views"],), math.pi / c["views"] / c["pitch"], dtype=torch.float64, device="cuda")
    else:
        src, d0, du, dv = (torch.tensor(a, dtype=torch.float64, device="cuda") for a in corner(c))
        out = torch.linalg.cross(du, dv)
        depth = (d0 * out).sum(1)
        r = -(src * out).sum(1) / depth
        scale = math.pi / c["views"] * r / c["pitch"]
        sdd = (depth / out.norm(dim=1)).abs()
        v, u = (torch.arange(n, dtype=torch.float64, device="cuda") for n in (c["nv"], nu))
        p = p.clone()
        for n in range(c["views"]):
            far = d0[n] + u[None, :, None] * du[n] + v[:, None, None] * dv[n]
            p[:, n] *= sdd[n] / far.norm(dim=-1)
    k = torch.arange(-nu + 1, nu, dtype=torch.float64, device="cuda")
    taps = torch.where(k % 2 == 0, torch.zeros_like(k), -1.0 / (math.pi * k) ** 2)
    taps[nu - 1] = 0.25
    length = 1 << (3 * nu).bit_length()
    f = torch.fft.rfft(taps, length)
    for n in range(c["views"]):
        p[:, n] = scale[n] * torch.fft.irfft(torch.fft.rfft(p[:, n], length) * f, length)[..., nu - 1:2 * nu - 1]
    return out64(c, p, True)


def exact_blur(p, angles, length):
    """Each view convolved with a line of `length` samples at its angle."""
    out = torch.zeros_like(p)
    nv, nu = p.shape[-2:]
    v, u = (torch.arange(n, dtype=torch.float64, device="cuda") for n in (nv, nu))
    size = torch.tensor([nu, nv], dtype=torch.float64, device="cuda")
    for n in range(p.shape[0]):
        for j in range(length):
            t = j - 0.5 * (length - 1)
            pos = torch.stack(torch.broadcast_tensors(u + t * torch.cos(angles[n]), (v + t * torch.sin(angles[n]))[:, None]), -1)
            out[n] += torch.nn.functional.grid_sample(p[None, n:n + 1], ((2 * pos + 1) / size - 1)[None], "bilinear", "zeros",
                                                      align_corners=False)[0, 0] / length
    return out
