"""The calls that users of the forward model make, as measurable cases.

A case is one pass through the public entry points (``Forward``, ``Server``,
``autograd.detector_curves`` and the C call that allocates nothing).  ``listed`` gives the
named ones, ``draw`` others of the same ranges, ``prepare`` builds what a program holds
before the call, ``run`` makes the call, ``work`` says what it cannot do without and
``exact`` gives the same outputs in 64 bits from the method's equations (its own code).

Kinds of case:
  solve    a whole forward solve from the pulse: reset, steps, detector curves and fields;
  window   further steps of a developed state (a run that is read out as it goes);
  grad     detector curves and their gradient with respect to both optical maps;
  layer    the per-voxel source iteration on caller-owned buffers;
  serve    a batch of requests of different sizes through the server.

Detector curves and gradients are sums of 32-bit radiances; they are handed on as 32-bit
tensors, as a misfit against measured curves takes them.
"""
import ctypes
import math

import numpy as np
import torch

import paper_2105_01028_gb300 as T
from paper_2105_01028_gb300.autograd import detector_curves

C0 = 299.792458  # mm / ns


# ---- the cases

def listed():
    return [
        # the small forward solve: 16^3 voxels, 48 directions, 100 steps (launches and latency count)
        dict(name="solve16_fp32", kind="solve", nx=16, ny=16, nz=16, nside=2, precision="fp32", optics="uniform",
             mua=0.01, mus=10.0, steps=100),
        dict(name="solve16_bf16", kind="solve", nx=16, ny=16, nz=16, nside=2, precision="bf16", optics="uniform",
             mua=0.01, mus=10.0, steps=100),
        # the phantom-scale homogeneous slab in each form of the scattering sum
        dict(name="slab_fp32", kind="window", nx=96, ny=96, nz=64, nside=4, precision="fp32", optics="uniform",
             mua=0.008, mus=8.0, steps=2),
        dict(name="slab_bf16", kind="window", nx=96, ny=96, nz=64, nside=4, precision="bf16", optics="uniform",
             mua=0.008, mus=8.0, steps=8),
        dict(name="slab_exact", kind="window", nx=96, ny=96, nz=64, nside=4, precision="fp32", optics="uniform",
             mua=0.008, mus=8.0, steps=8, exact=True),
        # the heterogeneous phantom with refraction at an air cylinder
        dict(name="phantom_bf16", kind="window", nx=128, ny=128, nz=96, nside=4, precision="bf16", optics="phantom",
             mua=0.008, mus=8.0, steps=4),
        # random-field optics of the served and gradient workloads, on odd grids
        dict(name="field_fp32", kind="window", nx=61, ny=47, nz=53, nside=4, precision="fp32", optics="field",
             mua=0.01, mus=10.0, steps=2),
        dict(name="field_bf16", kind="window", nx=77, ny=77, nz=77, nside=4, precision="bf16", optics="field",
             mua=0.01, mus=10.0, steps=4),
        # transport on 3072 directions, source function on 192 (the paper's fiducial angular grids)
        dict(name="twolevel_fp32", kind="window", nx=32, ny=32, nz=24, nside=16, nside_scatter=4, precision="fp32",
             optics="uniform", mua=0.008, mus=8.0, steps=2),
        # sensitivity of the detector curves to both optical maps, one call of an inversion
        dict(name="grad_fp32", kind="grad", nx=32, ny=32, nz=32, nside=4, precision="fp32", optics="field",
             mua=0.01, mus=10.0, steps=40, every=16),
        # the source iteration inside another program's memory pool
        dict(name="layer_fp32", kind="layer", na=192, nvox=110592, mua=0.01, mus=10.0),
        # a burst of requests of different sizes
        dict(name="serve_bf16", kind="serve", requests=6, nmin=32, nmax=56, precision="bf16", mua=0.01, mus=10.0,
             steps=64),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["solve", "window", "window", "window", "grad", "layer", "serve"])
    mua, mus = round(rng.uniform(0.005, 0.02), 5), round(rng.uniform(4.0, 12.0), 3)
    prec = rng.choice(["fp32", "bf16"])
    if kind == "solve":
        return dict(kind=kind, nx=_log(rng, 8, 40), ny=_log(rng, 8, 40), nz=_log(rng, 8, 40), nside=2,
                    precision=prec, optics=rng.choice(["uniform", "field"]), mua=mua, mus=mus, steps=_log(rng, 20, 120))
    if kind == "window":
        c = dict(kind=kind, nx=_log(rng, 24, 96), ny=_log(rng, 24, 96), nz=_log(rng, 24, 64),
                 nside=rng.choice([2, 4, 4]), precision=prec, optics=rng.choice(["uniform", "field"]), mua=mua,
                 mus=mus, steps=rng.randint(1, 2) if prec == "fp32" else rng.randint(1, 8))
        if c["optics"] == "uniform" and rng.random() < 0.33:
            c.update(exact=True, precision="fp32")
        elif rng.random() < 0.2:
            c.update(nx=_log(rng, 8, 32), ny=_log(rng, 8, 32), nz=_log(rng, 8, 24), nside=rng.choice([8, 16]),
                     nside_scatter=4)
        return c
    if kind == "grad":
        return dict(kind=kind, nx=_log(rng, 10, 32), ny=_log(rng, 10, 32), nz=_log(rng, 10, 32),
                    nside=rng.choice([2, 4]), precision="fp32", optics="field", mua=mua, mus=mus,
                    steps=_log(rng, 12, 40), every=_log(rng, 4, 16))
    if kind == "layer":
        return dict(kind=kind, na=rng.choice([48, 192, 192]), nvox=_log(rng, 1000, 200000), mua=mua, mus=mus)
    return dict(kind=kind, requests=rng.randint(2, 6), nmin=_log(rng, 16, 32), nmax=_log(rng, 33, 56), precision=prec,
                mua=mua, mus=mus, steps=_log(rng, 32, 64))


# ---- inputs

def _gen(seed):
    return torch.Generator(device="cuda").manual_seed(int(seed))


def _uniform01(seed, n):
    return np.random.default_rng(int(seed)).random(n)


def _smooth_field(shape, corr, gen):
    """Unit-variance Gaussian random field of correlation length ``corr`` voxels."""
    noise = torch.randn(shape, generator=gen, device="cuda", dtype=torch.float32)
    k2 = 0.0
    for a, n in enumerate(shape):
        k = torch.fft.fftfreq(n, device="cuda").reshape([-1 if b == a else 1 for b in range(3)])
        k2 = k2 + k * k
    f = torch.fft.ifftn(torch.fft.fftn(noise) * torch.exp(-2.0 * (math.pi * corr) ** 2 * k2)).real
    return (f - f.mean()) / f.std()


def _optics(c, seed):
    """mu_a, mu_s, n maps [nz, ny, nx], float32 on the GPU."""
    shape = (c["nz"], c["ny"], c["nx"])
    u = _uniform01(seed, 2)
    mua, mus = c["mua"] * (0.95 + 0.1 * u[0]), c["mus"] * (0.95 + 0.1 * u[1])
    ones = torch.ones(shape, device="cuda", dtype=torch.float32)
    if c["optics"] == "field":
        gen = _gen(seed)
        return (mua * torch.exp(0.3 * _smooth_field(shape, 5.0, gen)), mus * torch.exp(0.3 * _smooth_field(shape, 5.0, gen)),
                1.4 * ones)
    a, s, n = mua * ones, mus * ones, 1.4 * ones
    if c["optics"] == "phantom":
        z, y, x = torch.meshgrid(*(torch.arange(m, device="cuda") + 0.5 for m in shape), indexing="ij")
        sc = c["nx"] / 128.0
        v = _uniform01(seed + 1, 9).reshape(3, 3)
        for k, (r, f) in enumerate(((4.0, 2.0), (6.0, 3.5), (8.0, 5.0))):  # absorbing spheres
            cx, cy, cz = (0.5 + 0.35 * v[k, 0]) * c["nx"], (0.2 + 0.6 * v[k, 1]) * c["ny"], (0.2 + 0.6 * v[k, 2]) * c["nz"]
            a[(x - cx) ** 2 + (y - cy) ** 2 + (z - cz) ** 2 <= (r * sc) ** 2] = mua * f
        cyl = (x - 32.0 * sc) ** 2 + (y - 64.0 * sc) ** 2 <= (5.0 * sc) ** 2  # air cylinder
        a[cyl], s[cyl], n[cyl] = 0.0, 0.0, 1.0
    return a.contiguous(), s.contiguous(), n.contiguous()


def _problem(c, seed):
    """The problem dict that ``Forward`` and ``Server`` take."""
    mua, mus, nidx = _optics(c, seed)
    face = 0 if c["optics"] == "phantom" else 4
    nu, nv = (c["ny"], c["nz"]) if face == 0 else (c["nx"], c["ny"])
    cu, cv = float(nu // 2), float(nv // 2)
    dets = [dict(face=face, u_mm=min(cu + 0.5 + s * nu / 96.0, nu - 0.5), v_mm=cv + 0.5, radius_mm=0.5, half_angle_deg=15.0)
            for s in np.linspace(10.0, 40.0, 8)]
    return dict(nx=c["nx"], ny=c["ny"], nz=c["nz"], h=1.0, nside=c["nside"], nside_scatter=c.get("nside_scatter", 0),
                courant=0.5, n_ref=1.4, mua=mua, mus=mus, nidx=nidx, g=0.9, precision=c["precision"], tol=1e-6,
                max_iters=2000, exact=c.get("exact", False), fresnel=c["optics"] == "phantom", steps=c["steps"],
                source=dict(face=face, u_mm=cu, v_mm=cv, half_angle_deg=15.0, pulse_steps=1, energy=1.0),
                detectors=dets, bin_ps=10.0, nbins=600 if c["kind"] == "window" else c["steps"] // 4 + 2)


def _glow(c, seed, dtype=torch.float32):
    """A developed state: a glow around the source spot (std a quarter of the box, at most
    15 mm) that leans outward, with the source function that goes with it."""
    shape = (c["nz"], c["ny"], c["nx"])
    dirs = torch.as_tensor(T.healpix_dirs(c["nside"]), device="cuda", dtype=torch.float32)
    z, y, x = (t.reshape(1, -1) for t in torch.meshgrid(*(torch.arange(m, device="cuda") + 0.5 for m in shape), indexing="ij"))
    u = _uniform01(seed + 2, 2)
    x, y = x - c["nx"] * (0.45 + 0.1 * u[0]), y - c["ny"] * (0.45 + 0.1 * u[1])
    std = min(15.0, 0.25 * max(shape))
    r2 = x * x + y * y + z * z
    glow = torch.exp(-r2 / (2 * std * std)).float() + 1e-4
    r = torch.sqrt(r2).float()
    lean = 0.1 * torch.clamp(r / std, max=1.0) / r
    I = dirs[:, :1] * (x.float() * lean) + dirs[:, 1:2] * (y.float() * lean) + dirs[:, 2:] * (z.float() * lean)
    I = glow * (1.0 + I)
    if c.get("nside_scatter"):
        S = (0.999 * glow).expand(12 * c["nside_scatter"] ** 2, -1).contiguous()
    else:
        S = 0.998 * glow + 0.9 * (I - glow)
    return I, S


def prepare(case, seed):
    c = case
    if c["kind"] == "layer":
        return _prepare_layer(c, seed)
    if c["kind"] == "serve":
        return _prepare_serve(c, seed)
    prob = _problem(c, seed)
    if c["kind"] == "grad":
        w = torch.as_tensor(0.5 + _uniform01(seed + 3, 8 * prob["nbins"]).reshape(8, -1), device="cuda")
        prob["nidx"] = prob["nidx"].cpu().numpy()
        return dict(case=c, prob=prob, mua=prob["mua"].requires_grad_(), mus=prob["mus"].requires_grad_(), weights=w)
    fw = T.Forward(prob, stream=torch.cuda.current_stream().cuda_stream)
    nv, na = c["nx"] * c["ny"] * c["nz"], 12 * c["nside"] ** 2
    ns = 12 * (c.get("nside_scatter") or c["nside"]) ** 2
    st = dict(case=c, fw=fw, I=torch.empty(na, nv, device="cuda"), S=torch.empty(ns, nv, device="cuda"))
    if c["kind"] == "window":
        if c["optics"] == "phantom":
            fw.run(120)  # the pulse has crossed half the box
            fw.sync()
        else:
            I0, S0 = _glow(c, seed)
            torch.cuda.synchronize()
            fw.set_initial_state(I0, S0)
    return st


_LAYER_ARGS = [ctypes.c_int, ctypes.c_int] + [ctypes.c_void_p] * 7 + [ctypes.c_double, ctypes.c_int,
                                                                      ctypes.POINTER(ctypes.c_int), ctypes.c_void_p]


def _prepare_layer(c, seed):
    na, nv = c["na"], c["nvox"]
    nside = int(round(math.sqrt(na / 12)))
    gen = _gen(seed)
    P = torch.as_tensor(T.phase_matrix(nside, 0.9)[0], device="cuda").float().contiguous()
    dirs = torch.as_tensor(T.healpix_dirs(nside), device="cuda")
    ds = 1.0 / dirs.abs().max(dim=1).values
    mus = c["mus"] * torch.exp(0.3 * torch.randn(nv, generator=gen, device="cuda"))
    mua = c["mua"] * torch.exp(0.3 * torch.randn(nv, generator=gen, device="cuda"))
    mut = (mua + mus).double()
    x = ds[:, None] * mut[None, :]
    b1 = ((x - 1 + torch.exp(-x)) / x).float()
    bright = torch.exp(1.5 * torch.randn(nv, generator=gen, device="cuda"))
    lean = torch.randn(3, nv, generator=gen, device="cuda") * 0.1
    shape = 1.0 + dirs.float() @ lean
    Sp = (bright * shape).contiguous()
    Q = (Sp * (1 - b1) * (0.98 + 0.02 * torch.rand(na, nv, generator=gen, device="cuda"))).contiguous()
    fn = T.lib().trinity_source_iteration_noalloc
    fn.restype, fn.argtypes = ctypes.c_int, _LAYER_ARGS
    return dict(case=c, fn=fn, P=P, Q=Q, b1=b1.contiguous(), eps=(mua.double() / mut).float().contiguous(), Sp=Sp,
                S=torch.empty_like(Q), I=torch.empty_like(Q))


def _prepare_serve(c, seed):
    u = _uniform01(seed + 4, c["requests"])
    probs = []
    for k in range(c["requests"]):
        n = c["nmin"] + (k * (c["nmax"] - c["nmin"])) // max(c["requests"] - 1, 1)
        one = dict(c, nx=n, ny=n, nz=n, nside=4 if k % 2 else 2, optics="field")
        p = _problem(dict(one, mua=c["mua"] * (0.9 + 0.2 * u[k])), seed + 17 * k)
        for key in ("mua", "mus", "nidx"):
            p[key] = p[key].cpu().numpy()
        probs.append(p)
    return dict(case=c, server=T.Server(32 << 30, max_slots=4, steps_per_slice=32), probs=probs)


# ---- the calls

def _curves(fw):
    return torch.as_tensor(fw.detectors(), dtype=torch.float32)


def run(state):
    c = state["case"]
    if c["kind"] == "layer":
        s = state
        rc = s["fn"](c["na"], c["nvox"], s["P"].data_ptr(), s["Q"].data_ptr(), s["b1"].data_ptr(), s["eps"].data_ptr(),
                     s["Sp"].data_ptr(), s["S"].data_ptr(), s["I"].data_ptr(), 1e-6, 2000, None,
                     torch.cuda.current_stream().cuda_stream)
        if rc != 0:
            raise RuntimeError("source iteration failed: %d" % rc)
        return dict(S=s["S"], I=s["I"])
    if c["kind"] == "serve":
        srv = state["server"]
        ids = [srv.submit(p) for p in state["probs"]]
        out = []
        for rid in ids:
            st, rc, det, _ = srv.wait(rid)
            if st != T.REQ_DONE:
                raise RuntimeError("request failed: %d" % rc)
            out.append(torch.as_tensor(det, dtype=torch.float32))
        return out
    if c["kind"] == "grad":
        mua, mus = state["mua"], state["mus"]
        mua.grad = mus.grad = None
        E = detector_curves(mua, mus, state["prob"], c["steps"], c["every"])
        (E * state["weights"]).sum().backward()
        return dict(curves=E.detach().float(), mua=mua.grad, mus=mus.grad)
    fw = state["fw"]
    if c["kind"] == "solve":
        fw.reset()
    fw.run(c["steps"])
    return dict(curves=_curves(fw), I=fw.field(T.FIELD_I, out=state["I"]), S=fw.field(T.FIELD_S, out=state["S"]))


def work(case):
    c = case
    if c["kind"] == "layer":  # Q, b1, S_prev in, S, I out; one product per voxel
        return dict(bytes=20.0 * c["na"] * c["nvox"], flops=2.0 * c["na"] ** 2 * c["nvox"])
    if c["kind"] == "serve":
        tot = dict(bytes=0.0, flops=0.0)
        for k in range(c["requests"]):
            n = c["nmin"] + (k * (c["nmax"] - c["nmin"])) // max(c["requests"] - 1, 1)
            w = work(dict(c, kind="solve", nx=n, ny=n, nz=n, nside=4 if k % 2 else 2))
            tot = {key: tot[key] + w[key] for key in tot}
        return tot
    nv = c["nx"] * c["ny"] * c["nz"]
    na, ns = 12 * c["nside"] ** 2, 12 * (c.get("nside_scatter") or c["nside"]) ** 2
    # a step reads I and S at the two retarded levels and writes one level of each
    step = 12.0 * nv * (na + ns)
    times = c["steps"] * (3 if c["kind"] == "grad" else 1)  # a gradient: forward, forward again, reverse
    return dict(bytes=step * times, flops=2.0 * ns * ns * nv * times)


# ---- the same outputs in 64 bits, from the method's equations

def _f64(x):
    return torch.as_tensor(x, device="cuda", dtype=torch.float64)


def _directions(nside):
    """HEALPix RING pixel centres."""
    zs, ps = [], []
    for i in range(1, 4 * nside):
        ii = min(i, 4 * nside - i)
        if ii < nside:
            z, j, n = 1.0 - ii * ii / (3.0 * nside * nside), 0.5, 4 * ii
            z = z if i < nside else -z
        else:
            z, j, n = 4.0 / 3.0 - 2.0 * i / (3.0 * nside), 0.5 * ((i - nside + 1) % 2), 4 * nside
        zs.append(np.full(n, z))
        ps.append((np.arange(1, n + 1) - j) * 2.0 * np.pi / n)
    z, p = np.concatenate(zs), np.concatenate(ps)
    s = np.sqrt((1 - z) * (1 + z))
    return np.stack([s * np.cos(p), s * np.sin(p), z], axis=1)


def _parents(nside, coarse):
    """Coarse RING pixel that holds each fine pixel's centre (HEALPix pixel boundaries)."""
    d = _directions(nside)
    N, out = coarse, []
    for x, y, z in d:
        t = 2.0 * (math.atan2(y, x) % (2 * math.pi)) / math.pi  # [0, 4)
        if abs(z) <= 2.0 / 3.0:
            off = (N - 1) / 2.0
            a = math.floor(N * t + 0.75 * N * z - off + 0.5) + off
            b = math.floor(N * t - 0.75 * N * z - off + 0.5) + off
            i = int(round(2 * N - (a - b)))
            j = (int(round((a + b + (i - N + 1) % 2) / 2.0)) - 1) % (4 * N)
            out.append(2 * N * (N - 1) + 4 * N * (i - N) + j)
        else:
            q = min(int(t), 3)
            s = N * math.sqrt(3.0 * (1.0 - abs(z)))
            kx, ky = int((t - q) * s), int((1.0 - (t - q)) * s)
            i = kx + ky + 1
            j = q * i + kx
            out.append(2 * i * (i - 1) + j if z > 0 else 12 * N * N - 2 * i * (i + 1) + j)
    return np.array(out)


def _phase(nside, g):
    """P = D K D, K Henyey-Greenstein, unit row sums, mean cosine g."""
    d = _directions(nside)
    mu = np.clip(d @ d.T, -1.0, 1.0)

    def build(ge):
        K = (1 - ge * ge) / (1 + ge * ge - 2 * ge * mu) ** 1.5 / len(d)
        s = np.ones(len(d))
        for _ in range(5000):
            r = K @ s
            if np.max(np.abs(s * r - 1)) < 1e-14:
                break
            s = np.sqrt(s / r)
        return s[:, None] * K * s[None, :]

    lo, hi = 0.0, 1.0
    for _ in range(52):
        mid = 0.5 * (lo + hi)
        lo, hi = (mid, hi) if (build(mid) * mu).sum() / len(d) < g else (lo, mid)
    return _f64(build(0.5 * (lo + hi)))


def _cone(dirs, axis, inward_sign, eu, ev):
    """Share of a 15-degree cone around the face normal that is nearest to each direction."""
    ct = math.cos(math.radians(15.0))
    m, p = np.meshgrid(1 - (np.arange(64) + 0.5) * (1 - ct) / 64, 2 * np.pi * (np.arange(256) + 0.5) / 256, indexing="ij")
    m, p = m.ravel(), p.ravel()
    s = np.sqrt((1 - m) * (1 + m))
    pts = np.zeros((m.size, 3))
    pts[:, axis], pts[:, eu], pts[:, ev] = inward_sign * m, s * np.cos(p), s * np.sin(p)
    return np.bincount(np.argmax(pts @ dirs.T, axis=1), minlength=len(dirs)) / float(m.size)


class _Exact:
    """The method on one grid with vacuum faces and a uniform refractive index, 64 bits."""

    def __init__(self, c, prob):
        self.c = c
        nx, ny, nz = c["nx"], c["ny"], c["nz"]
        self.nv, n = nx * ny * nz, (nx, ny, nz)
        d = _directions(c["nside"])
        self.na, self.w = len(d), 4 * math.pi / len(d)
        self.dt = 0.5 * 1.4 / C0
        self.par = None
        if c.get("nside_scatter"):
            self.par = torch.as_tensor(_parents(c["nside"], c["nside_scatter"]), device="cuda")
        self.P = _phase(c.get("nside_scatter") or c["nside"], 0.9)
        self.mua, self.mus = (_f64(prob[k].detach()).reshape(-1) for k in ("mua", "mus"))
        dom = np.array([2 if abs(v[2]) >= max(abs(v[0]), abs(v[1])) - 1e-12 else (1 if abs(v[1]) >= abs(v[0]) - 1e-12 else 0)
                        for v in d])
        big = np.abs(d[np.arange(self.na), dom])
        self.ds = _f64(1.0 / big)
        nidx = float(prob["nidx"].reshape(-1)[0])
        delta = nidx / big / (C0 * self.dt)
        self.m, self.f = torch.as_tensor(np.floor(delta).astype(np.int64), device="cuda"), _f64(delta - np.floor(delta))
        # upwind voxel of every (direction, voxel): -1 outside the box
        snap = lambda y: np.where(np.abs(y - np.round(y)) < 1e-9, np.round(y), np.floor(y)).astype(np.int64)  # noqa: E731
        v = torch.arange(self.nv, device="cuda")
        pos = [v % nx, (v // nx) % ny, v // (nx * ny)]
        self.up = torch.empty(self.na, self.nv, dtype=torch.int64, device="cuda")
        for k in range(self.na):
            a, sg = int(dom[k]), 1 if d[k, dom[k]] > 0 else -1
            kp = pos[a] if sg > 0 else n[a] - 1 - pos[a]
            q = list(pos)
            q[a] = pos[a] - sg
            for b in range(3):
                if b != a:
                    s = np.arange(n[a], dtype=np.float64)
                    t = d[k, b] / big[k]
                    off = snap(0.5 + s * t) - snap(0.5 + (s - 1) * t)
                    off[0] = 0
                    q[b] = pos[b] - torch.as_tensor(off, device="cuda")[kp]
            inside = torch.ones_like(v, dtype=torch.bool)
            for b in range(3):
                inside &= (q[b] >= 0) & (q[b] < n[b])
            self.up[k] = torch.where(inside, (q[2] * ny + q[1]) * nx + q[0], torch.full_like(v, -1))
        # source inflow and detectors on the -z face
        src = prob["source"]
        amp = _cone(d, 2, 1.0, 0, 1)
        self.amp = _f64(np.where(amp > 0, amp / (self.w * np.where(amp > 0, d[:, 2], 1.0) * self.dt), 0.0))
        self.spot = int(src["v_mm"]) * nx + int(src["u_mm"])
        det = _cone(d, 2, -1.0, 0, 1) * 2 * math.pi * (1 - math.cos(math.radians(15.0)))
        self.det_w = _f64(np.where(det > 0, det * -d[:, 2], 0.0) * self.dt)
        self.det_v = []
        yy, xx = np.meshgrid(np.arange(ny) + 0.5, np.arange(nx) + 0.5, indexing="ij")
        for q in prob["detectors"]:
            hit = (xx - q["u_mm"]) ** 2 + (yy - q["v_mm"]) ** 2 <= q["radius_mm"] ** 2 * (1 + 1e-12)
            self.det_v.append(torch.as_tensor(np.nonzero(hit.ravel())[0], device="cuda"))
        self.nbins = prob["nbins"]
        self.weights()

    def weights(self):
        mut = self.mua + self.mus
        x = self.ds[:, None] * mut[None, :]
        self.Tr = torch.exp(-x)
        self.b0, self.b1 = (1 - (1 + x) * self.Tr) / x, (x - 1 + self.Tr) / x
        self.alb = self.mus / mut
        self.b1s = self.b1 if self.par is None else self.mean(self.b1)

    def mean(self, X):
        """Mean over the children of each coarse direction."""
        out = torch.zeros(self.P.shape[0], X.shape[1], device="cuda", dtype=X.dtype)
        return out.index_add_(0, self.par, X) / (self.na // self.P.shape[0])

    def solve(self, Q, S):
        """S = a P (Q + b1 S) in every voxel."""
        if self.c["optics"] == "uniform":
            if not hasattr(self, "M"):
                A = self.alb[0] * self.P
                self.M = torch.linalg.solve(torch.eye(len(A), device="cuda", dtype=A.dtype) - A * self.b1s[:, 0], A)
            return self.M @ Q
        den = len(self.P) - self.alb * self.b1s.sum(0)
        for k in range(2000):
            Sn = self.alb * (self.P @ (Q + self.b1s * S))
            D = Sn - S
            if k % 8 == 7 and float((D.abs().max(0).values / (Sn.abs().max(0).values + 1e-300)).max()) < 1e-11:
                return Sn
            S = Sn + self.alb * (self.b1s * D).sum(0) / den
        return S

    def steps(self, nsteps, hist=None):
        """(curves, I, S) after nsteps from hist = (I, S) held for ever before, or from nothing."""
        dev = dict(device="cuda", dtype=torch.float64)
        zero = (torch.zeros(self.na, self.nv, **dev), torch.zeros(len(self.P), self.nv, **dev))
        lev = {k: zero if hist is None else hist for k in range(-4, 0)}
        E = torch.zeros(len(self.det_v), self.nbins, **dev)
        dd = torch.arange(self.na, device="cuda")[:, None]
        for n in range(nsteps):
            Q = 0.0
            for back in (0, 1):
                wt = (1 - self.f if back == 0 else self.f)[:, None]
                for m in range(1, 4):
                    rows = torch.nonzero(self.m == m).reshape(-1)
                    if not len(rows):
                        continue
                    I, S = lev[n - m - back]
                    u = self.up[rows]
                    ok = u >= 0
                    u = u.clamp(min=0)
                    Iu = torch.where(ok, torch.gather(I[rows], 1, u), 0.0)
                    if n - m - back == 0:  # the pulse lasts one level
                        add = torch.zeros_like(Iu)
                        add[:, self.spot] = self.amp[rows] * (self.up[rows, self.spot] < 0)
                        Iu = Iu + add
                    Sr = S[rows] if self.par is None else S[self.par[rows]]
                    Su = torch.where(ok, torch.gather(Sr, 1, u), 0.0)
                    part = wt[rows] * (Iu * self.Tr[rows] + Su * self.b0[rows])
                    Q = Q + torch.zeros(self.na, self.nv, **dev).index_copy(0, rows, part)
            S = self.solve(Q if self.par is None else self.mean(Q), lev[n - 1][1])
            I = Q + self.b1 * (S if self.par is None else S[self.par])
            lev = {k: lev[k] for k in range(n - 3, n)}
            lev[n] = (I, S)
            b = math.floor((n + 0.5) * self.dt / 0.01 + 1e-9)
            if b < self.nbins:
                col = torch.stack([(self.det_w[:, None] * I[:, v]).sum() for v in self.det_v])
                E = E + torch.zeros_like(E).index_copy(1, torch.tensor([b], device="cuda"), col[:, None])
        return E, I, S


class _ExactGrad(_Exact):
    """The same with a direct, differentiable per-voxel solve."""

    def weights(self):
        self.mua.requires_grad_()
        self.mus.requires_grad_()
        super().weights()
        A = self.alb[:, None, None] * self.P
        self.M = torch.linalg.solve(torch.eye(len(self.P), device="cuda", dtype=A.dtype) - A * self.b1.T[:, None, :], A)

    def solve(self, Q, S):
        return torch.matmul(self.M, Q.T[:, :, None])[:, :, 0].T


def exact(case, seed):
    c = case
    if c["kind"] == "serve" or c.get("optics") == "phantom":
        return None  # too long in 64 bits; interface splits
    if c["kind"] == "layer":
        s = _prepare_layer(c, seed)
        P, Q, b1, a = s["P"].double(), s["Q"].double(), s["b1"].double(), 1 - s["eps"].double()
        P = P + torch.diag(1 - P.sum(1))
        S, den = s["Sp"].double(), len(P) - a * b1.sum(0)
        for k in range(300):
            Sn = a * (P @ (Q + b1 * S))
            S = Sn + a * (b1 * (Sn - S)).sum(0) / den
        return dict(S=S, I=Q + b1 * S)
    nv, na = c["nx"] * c["ny"] * c["nz"], 12 * c["nside"] ** 2
    if c["optics"] == "field" and c["kind"] != "grad" and 2.0 * nv * na * na * 150 * c["steps"] > 1.2e13:
        return None
    prob = _problem(c, seed)
    if c["kind"] == "grad":
        x = _ExactGrad(c, prob)
        w = _f64(0.5 + _uniform01(seed + 3, 8 * prob["nbins"]).reshape(8, -1))
        E = x.steps(c["steps"])[0]
        (E * w).sum().backward()
        shape = (c["nz"], c["ny"], c["nx"])
        return dict(curves=E.detach(), mua=x.mua.grad.reshape(shape), mus=x.mus.grad.reshape(shape))
    x = _Exact(c, prob)
    hist = tuple(t.double() for t in _glow(c, seed)) if c["kind"] == "window" else None
    E, I, S = x.steps(c["steps"], hist)
    return dict(curves=E, I=I, S=S)
