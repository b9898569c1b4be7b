"""Performance cases of the GKE evaluator: what its users have it do, through
the public entry points (the binding of include/gke.h and include/gke1h.h).

A case is a dict of plain values.  ``path`` is one of

  channel   the plane-channel GKE of nsnap snapshots on an nx x nz x ny grid.
            ``precision`` f64 / bf16x3 / f32; ``domain`` triangle / wedge
            (mirror sampling); ``under_x``, ``under_z`` the undersampling of
            the separations, "t1,t2,s1,s2"; ``call``: compute (one call),
            batches (Step-1 mean, snapshots in two or more batches, Step 3),
            graph (the pass replayed as a CUDA graph), noalloc (the
            allocation-free entry point); ``memory``: device, or pinned (host
            buffers for the snapshots and the terms);
  duct      the variant with one homogeneous direction, nx x ny x nz;
  step1     u, v, w, p of nsnap snapshots from velocity-vorticity data.

Inputs are synthetic: complex Gaussian half spectra with the amplitude
(1 + k^2)^(-5/6), shaped to vanish at the walls, plus a laminar mean profile.
"""
from __future__ import annotations

import math

import numpy as np
import torch

import paper_1910_06409_gb300._native as N

LX, LZ, NU = 4.0 * math.pi, 2.0 * math.pi, 1.0 / 200.0
PRECISION = {"f64": N.GKE_PREC_F64, "bf16x3": N.GKE_PREC_BF16X3, "f32": N.GKE_PREC_F32}
DOMAIN = {"triangle": N.GKE_DOMAIN_TRIANGLE, "wedge": N.GKE_DOMAIN_WEDGE}
FULL = "0,0,0,0"


def _channel(name, nx, nz, ny, nsnap, precision, domain="triangle", under_x=FULL, under_z=FULL, call="compute",
             batch=0, memory="device"):
    return {"name": name, "path": "channel", "nx": nx, "nz": nz, "ny": ny, "nsnap": nsnap, "precision": precision,
            "domain": domain, "under_x": under_x, "under_z": under_z, "call": call, "batch": batch or nsnap,
            "memory": memory}


def _duct(name, nx, ny, nz, nsnap, precision):
    return {"name": name, "path": "duct", "nx": nx, "ny": ny, "nz": nz, "nsnap": nsnap, "precision": precision}


def _step1(name, nx, nz, ny, nsnap):
    return {"name": name, "path": "step1", "nx": nx, "nz": nz, "ny": ny, "nsnap": nsnap}


def listed():
    return [
        # a toy grid inside a program that may not allocate on the device: a
        # handful of launches, nothing but latency
        _channel("noalloc_16x16x17_s2_f64", 16, 16, 17, 2, "f64", call="noalloc"),
        # a quick look at a coarse run: the plan's call at the size where
        # launches and synchronisations still count
        _channel("tiny_32x32x33_s4_f64", 32, 32, 33, 4, "f64"),
        # the same grid replayed as a graph, once per new set of snapshots, on
        # the tensor-core path
        _channel("graph_32x32x33_s4_bf16x3", 32, 32, 33, 4, "bf16x3", call="graph"),
        # a ragged grid (3 2^a points, ny off every tile), mirror sampling,
        # thresholded separations, the snapshots in two batches, FP32
        _channel("wedge_96x48x41_s6_f32", 96, 48, 41, 6, "f32", domain="wedge", under_x="6,20,2,4",
                 under_z="5,12,2,3", call="batches", batch=3),
        # an ordinary data set in full precision: many snapshots, ny = 64 + 1
        _channel("group_128x128x65_s32_f64", 128, 128, 65, 32, "f64"),
        # large planes in full precision (256-point transforms): the largest
        # full-precision grid whose plan leaves room for two more
        _channel("plane_256x256x65_s16_f64", 256, 256, 65, 16, "f64"),
        # the Re_tau = 200 data set of the benchmark on the tensor-core path
        _channel("retau200_256x256x129_s16_bf16x3", 256, 256, 129, 16, "bf16x3"),
        # an ordinary data set end to end: snapshots from pinned host memory,
        # terms to pinned host memory
        _channel("group_128x128x65_s32_bf16x3_pinned", 128, 128, 65, 32, "bf16x3", memory="pinned"),
        # the memory-bounded streaming mode: wedge, every fourth separation,
        # batches of four
        _channel("stream_256x256x129_s8_bf16x3", 256, 256, 129, 8, "bf16x3", domain="wedge", under_x="0,0,0,4",
                 under_z="0,0,0,4", call="batches", batch=4),
        # the benchmark's straight duct, both precisions
        _duct("duct_256x33x33_s16_f64", 256, 33, 33, 16, "f64"),
        _duct("duct_256x33x33_s16_f32", 256, 33, 33, 16, "f32"),
        # Step 1 for a velocity-vorticity database at the Re_tau = 200 grid,
        # a few snapshots at a time
        _step1("step1_256x256x129_s4", 256, 256, 129, 4),
    ]


# ---------------------------------------------------------------- drawn cases

LENGTHS = (8, 12, 16, 24, 32, 48, 64, 96, 128, 192, 256)     # transform lengths, 2^a and 3 2^a


def _log_int(rng, lo, hi):
    return min(hi, max(lo, round(math.exp(rng.uniform(math.log(lo), math.log(hi))))))


def _under(rng, n):
    kind = rng.randrange(3)
    if kind == 0:
        t1 = rng.randint(1, max(1, n // 8))
        t2 = rng.randint(t1, max(t1, n // 3))
        return "%d,%d,%d,%d" % (t1, t2, rng.randint(1, 3), rng.randint(2, 5))
    if kind == 1 and n >= 16:
        return "0,0,0,%d" % rng.choice((2, 4))
    return FULL


def _state_bytes(c):
    """Rough device bytes of one state (inputs, plan, terms)."""
    n8 = 8 if c.get("precision") == "f64" else 4
    nxh = c["nx"] // 2 + 1
    if c["path"] == "duct":
        P = c["ny"] * c["nz"]
        npair = P * (P + 1) // 2
        return 2 * n8 * (8 * npair + 11 * c["nsnap"] * P) * nxh + 8 * n8 * npair * c["nx"]
    nk, ny = c["nz"] * nxh, c["ny"]
    pad = 8 * ((ny + 7) // 8)
    npair = ny * (ny + 1) // 2
    return (2 * n8 * nk * (7 * pad * pad + 7 * npair + (11 * c["nsnap"] + 22) * ny) + 64 * nk * ny * c["nsnap"]
            + 11 * n8 * npair * c["nx"] * c["nz"])


def _budget(kind):
    """Largest contraction work of the listed cases of a kind."""
    return max(work(c)["flops"] for c in listed() if (c["path"], c.get("precision")) == kind)


def draw(rng):
    while True:
        path = rng.choices(("channel", "duct", "step1"), (7, 2, 1))[0]
        nx, nz = rng.choice(LENGTHS), rng.choice(LENGTHS)
        if path == "channel":
            precision = rng.choice(("f64", "f64", "bf16x3", "bf16x3", "f32"))
            ny, nsnap = _log_int(rng, 5, 129), _log_int(rng, 1, 32)
            c = _channel("", nx, nz, ny, nsnap, precision)
            if rng.random() < 0.3:
                c["domain"] = "wedge"
            if rng.random() < 0.3:
                c["under_x"], c["under_z"] = _under(rng, nx), _under(rng, nz)
            if rng.random() < 0.25 and nsnap > 1:
                c["call"], c["batch"] = "batches", rng.randint((nsnap + 3) // 4, (nsnap + 1) // 2)
            elif rng.random() < 0.15:
                c["call"] = "graph"
            limit = _budget(("channel", "f64" if precision == "f64" else "bf16x3"))
            if precision == "f32":
                limit /= 4
        elif path == "duct":
            precision = rng.choice(("f64", "f32"))
            ny, n2 = _log_int(rng, 5, 33), _log_int(rng, 5, 33)
            c = _duct("", nx, ny, n2, _log_int(rng, 1, 16), precision)
            limit = _budget(("duct", precision))
        else:
            c = _step1("", nx, nz, _log_int(rng, 5, 129), _log_int(rng, 1, 4))
            limit = _budget(("step1", None))
        del c["name"]
        if work(c)["flops"] <= limit and _state_bytes(c) <= 64e9 and work(c)["bytes"] > 2e4:
            return c


# --------------------------------------------------------------------- inputs

def _grid(n):
    """Chebyshev-Gauss-Lobatto points on [-1, 1], exactly antisymmetric."""
    y = -np.cos(np.pi * np.arange(n) / (n - 1))
    return 0.5 * (y - y[::-1])


def _device():
    return torch.device("cuda" if torch.cuda.is_available() else "cpu")


def _generator(seed, dev):
    g = torch.Generator(device=dev)
    g.manual_seed(int(seed) * 1000003 + 191006409)
    return g


def _amplitude2(nx, nz, dev):
    kx = 2 * math.pi / LX * torch.arange(nx // 2 + 1, device=dev, dtype=torch.float64)
    kz = 2 * math.pi / LZ * torch.fft.fftfreq(nz, d=1.0 / nz, device=dev, dtype=torch.float64)
    amp = (1.0 + kz[:, None] ** 2 + kx[None, :] ** 2) ** (-5.0 / 6.0)
    amp[0, 0] = 0.0
    amp[:, nx // 2] = 0.0
    amp[nz // 2, :] = 0.0
    return amp


def _planes(g, nf, ny, nz, nx, amp, env, dev):
    """rfft2 (forward) of nf random real fields on ny planes, times env(y)."""
    shape = (nf, ny, nz, nx // 2 + 1, 2)
    c = torch.view_as_complex(torch.randn(shape, generator=g, device=dev, dtype=torch.float64)) * amp
    a = torch.fft.irfft2(c, s=(nz, nx), norm="forward") * env[None, :, None, None]
    return torch.fft.rfft2(a, norm="forward")


def _channel_fields(c, seed):
    nx, nz, ny, ns, dev = c["nx"], c["nz"], c["ny"], c["nsnap"], _device()
    g, amp = _generator(seed, dev), _amplitude2(nx, nz, dev)
    y = torch.from_numpy(_grid(ny)).to(dev)
    f = torch.empty((ns, 4, ny, nz, nx // 2 + 1), dtype=torch.complex128, device=dev)
    for s in range(ns):
        f[s] = _planes(g, 4, ny, nz, nx, amp, 1.0 - y * y, dev)
        f[s, 0, :, 0, 0] += 1.0 - y * y
    return f


def _step1_inputs(c, seed):
    nx, nz, ny, ns, dev = c["nx"], c["nz"], c["ny"], c["nsnap"], _device()
    g, amp = _generator(seed, dev), _amplitude2(nx, nz, dev)
    y = torch.from_numpy(_grid(ny)).to(dev)
    env = 1.0 - y * y
    f = torch.empty((ns, 2, ny, nz, nx // 2 + 1), dtype=torch.complex128, device=dev)
    mean = torch.empty((ns, 2, ny), dtype=torch.float64, device=dev)
    for s in range(ns):
        f[s, 0:1] = _planes(g, 1, ny, nz, nx, amp, env * env, dev)
        f[s, 1:2] = _planes(g, 1, ny, nz, nx, amp, env, dev)
        r = torch.randn((2, ny), generator=g, device=dev, dtype=torch.float64)
        mean[s, 0] = env * (1.0 + 0.05 * r[0])
        mean[s, 1] = 0.02 * env * r[1]
    return f, mean


def _duct_fields(c, seed):
    nx, ny, nz, ns, dev = c["nx"], c["ny"], c["nz"], c["nsnap"], _device()
    g = _generator(seed, dev)
    kx = 2 * math.pi / LX * torch.arange(nx // 2 + 1, device=dev, dtype=torch.float64)
    amp = (1.0 + kx * kx) ** (-5.0 / 6.0)
    amp[0] = 0.0
    amp[nx // 2] = 0.0
    y, z = torch.from_numpy(_grid(ny)).to(dev)[:, None], torch.from_numpy(_grid(nz)).to(dev)[None, :]
    env = (1.0 - y * y) * (1.0 - z * z)
    r = torch.randn((ns, 4, ny, nz, nx // 2 + 1, 2), generator=g, device=dev, dtype=torch.float64)
    a = torch.fft.irfft(torch.view_as_complex(r) * amp, n=nx, norm="forward") * env[..., None]
    f = torch.fft.rfft(a, norm="forward")
    f[:, 0, :, :, 0] += env
    f[:, 1, :, :, 0] += 0.02 * z * env
    f[:, 2, :, :, 0] += 0.02 * y * env
    return f


# ------------------------------------------------------------- the calls

class _Plan:
    """A plan handle that goes with its last reference."""

    def __init__(self, handle, destroy):
        self.handle, self._destroy = handle, destroy

    def __del__(self):
        self._destroy(self.handle)


def _ints(text):
    return tuple(int(v) for v in text.split(","))


def _real(c):
    return torch.float64 if c["precision"] == "f64" else torch.float32


def prepare(case, seed):
    c = case
    s = {"case": c}
    if c["path"] == "duct":
        s["fields"] = _duct_fields(c, seed)
        s["y"], s["z"] = _grid(c["ny"]), _grid(c["nz"])
        P = c["ny"] * c["nz"]
        s["plan"] = _Plan(N.gke1h_plan(c["nx"], c["ny"], c["nz"], LX, NU, s["y"], s["z"], c["nsnap"],
                                       precision=PRECISION[c["precision"]]), N.gke1h_destroy)
        s["terms"] = torch.zeros((N.GKE1H_NTERM, P * (P + 1) // 2, c["nx"]), dtype=_real(c), device="cuda")
        s["profiles"] = torch.zeros((N.GKE1H_NPROF, P), dtype=torch.float64, device="cuda")
        return s
    s["y"] = _grid(c["ny"])
    if c["path"] == "step1":
        s["v_eta"], s["mean_uw"] = _step1_inputs(c, seed)
        s["plan"] = _Plan(N.gke_plan(c["nx"], c["nz"], c["ny"], LX, LZ, NU, s["y"], c["nsnap"], N.GKE_PREC_BF16X3),
                          N.gke_destroy)
        s["fields"] = torch.zeros((c["nsnap"], 4) + tuple(s["v_eta"].shape[2:]), dtype=torch.complex128, device="cuda")
        return s
    s["fields"] = _channel_fields(c, seed)
    ny, npair = c["ny"], c["ny"] * (c["ny"] + 1) // 2
    nrz, nrx = c["nz"], c["nx"]
    if c["call"] != "noalloc":
        stream = None
        if c["call"] == "graph":
            s["stream"] = torch.cuda.Stream()
            stream = s["stream"].cuda_stream
        s["plan"] = _Plan(N.gke_plan(c["nx"], c["nz"], ny, LX, LZ, NU, s["y"], c["batch"], PRECISION[c["precision"]],
                                     stream, DOMAIN[c["domain"]], _ints(c["under_x"]), _ints(c["under_z"])),
                          N.gke_destroy)
        mz, mx = N.gke_separation_labels(s["plan"].handle)
        npair, nrz, nrx = N.gke_npair(s["plan"].handle), len(mz), len(mx)
    s["terms"] = torch.zeros((N.GKE_NTERM, npair, nrz, nrx), dtype=_real(c), device="cuda")
    s["profiles"] = torch.zeros((N.GKE_NPROF, ny), dtype=torch.float64, device="cuda")
    if c["memory"] == "pinned":
        for k in ("fields", "terms", "profiles"):
            s[k] = torch.empty(s[k].shape, dtype=s[k].dtype, pin_memory=True).copy_(s[k])
    return s


def run(state):
    s, c = state, state["case"]
    if c["path"] == "duct":
        N.gke1h_compute(s["plan"].handle, s["fields"], c["nsnap"], s["terms"], s["profiles"])
        return {"terms": s["terms"], "profiles": s["profiles"]}
    if c["path"] == "step1":
        N.gke_velocity_vorticity(s["plan"].handle, s["v_eta"], s["mean_uw"], c["nsnap"], s["fields"])
        return {"fields": s["fields"]}
    if c["call"] == "noalloc":
        N.gke_compute_noalloc(c["nx"], c["nz"], c["ny"], LX, LZ, NU, s["y"], s["fields"], c["nsnap"], s["terms"],
                              s["profiles"])
    elif c["call"] == "graph":
        N.gke_compute_graph(s["plan"].handle, s["fields"], c["nsnap"], s["terms"], s["profiles"])
    elif c["call"] == "batches":
        plan, n, b = s["plan"].handle, c["nsnap"], c["batch"]
        N.gke_reset(plan)
        for i in range(0, n, b):
            N.gke_accumulate_mean(plan, s["fields"][i:i + b], min(b, n - i))
        for i in range(0, n, b):
            N.gke_accumulate_snapshot(plan, s["fields"][i:i + b], min(b, n - i))
        N.gke_finalize_terms(plan, s["terms"], s["profiles"])
    else:
        N.gke_compute(s["plan"].handle, s["fields"], c["nsnap"], s["terms"], s["profiles"])
    return {"terms": s["terms"], "profiles": s["profiles"]}


# ------------------------------------------------------------------ the work

def _kept(n, under):
    t1, t2, s1, s2 = under
    if not any(under):
        return list(range(n))
    d = [min(m, n - m) for m in range(n)]
    return [m for m in range(n) if d[m] < t1 or (d[m] % s1 == 0 if d[m] < t2 else d[m] % s2 == 0)]


def _fft_flops(n, batch):
    return 5.0 * n * math.log2(n) * batch


def work(case):
    """Bytes: the snapshots read once, the terms written once.  Operations:
    the contractions over snapshots (8 per complex multiply-add) and the
    Fourier transforms (5 n log2 n)."""
    c = case
    nx, nz, ny, ns = c["nx"], c["nz"], c["ny"], c["nsnap"]
    nxh = nx // 2 + 1
    if c["path"] == "duct":
        P = ny * nz
        npair = P * (P + 1) // 2
        real = 8 if c["precision"] == "f64" else 4
        return {"bytes": 64 * ns * P * nxh + 8 * npair * nx * real + 88 * P,
                "flops": 8.0 * 37 * ns * npair * nxh + _fft_flops(nx, 11 * ns * P / 2 + 4 * npair)}
    nk = nz * nxh
    plane = _fft_flops(nx, nz / 2) + _fft_flops(nz, nxh)
    if c["path"] == "step1":
        return {"bytes": 16 * nk * ny * ns * 6 + 16 * ny * ns, "flops": 9 * ns * ny * plane + 2 * 26.0 * nk * ny * ns}
    npair = ny * (ny + 1) // 2
    nout = sum(ny - 2 * i for i in range((ny + 1) // 2)) if c["domain"] == "wedge" else npair
    nr = len(_kept(nz, _ints(c["under_z"]))) * len(_kept(nx, _ints(c["under_x"])))
    real = 8 if c["precision"] == "f64" else 4
    cmac = nk * ns * (3 * npair + 14 * ny * ny)
    ratio = nr / (nx * nz) if "0,0,0," in c["under_x"] and "0,0,0," in c["under_z"] else 1.0
    return {"bytes": 64 * ns * ny * nk + 7 * nout * nr * real + 48 * ny,
            "flops": 8.0 * cmac + 11 * ns * ny * plane + 7 * nout * plane * ratio}


# ------------------------------------------------- the same in 64 bits, plainly

def _fd(x, order):
    """Dense matrix of the 5-point derivative on the nodes x (window shifted at
    the ends), by the derivatives of the Lagrange polynomials."""
    n = len(x)
    D = np.zeros((n, n))
    for j in range(n):
        l0 = min(max(j - 2, 0), n - 5)
        t = x[l0:l0 + 5] - x[j]
        for i in range(5):
            o = [k for k in range(5) if k != i]
            den = np.prod([t[i] - t[k] for k in o])
            if order == 1:
                num = sum(np.prod([-t[k] for k in o if k != a]) for a in o)
            else:
                num = 2 * sum(np.prod([-t[k] for k in o if k not in (a, b)]) for a in o for b in o if a < b)
            D[j, l0 + i] = num / den
    return D


def _signed(n, half, length, dev, true=False):
    m = torch.arange(n // 2 + 1 if half else n, device=dev, dtype=torch.float64)
    m = torch.where(m > n // 2, m - n, m)
    if not true:
        m[n // 2] = 0.0
    return 2 * math.pi / length * m


def _exact_channel(c, seed):
    dev = _device()
    nx, nz, ny = c["nx"], c["nz"], c["ny"]
    nxh = nx // 2 + 1
    nk = nz * nxh
    f = _channel_fields(c, seed)
    if c["domain"] == "wedge":                       # the mirror images are samples too
        g = f.flip(2).clone()
        g[:, 1] *= -1
        f = torch.cat([f, g])
    ns = f.shape[0]
    mean = f[:, :, :, 0, 0].real.mean(0)
    f[:, :, :, 0, 0] -= mean
    y = _grid(ny)
    D = torch.from_numpy(_fd(y, 1)).to(dev)
    kx, kz = _signed(nx, True, LX, dev), _signed(nz, False, LZ, dev)
    U, dU1 = mean[0], D @ mean[0]
    hat = {n: torch.empty((nk, ns, ny), dtype=torch.complex128, device=dev)
           for n in ("u", "v", "w", "p", "q", "uu", "vv", "ww", "uv", "uw", "vw")}
    one = {n: torch.zeros(ny, dtype=torch.float64, device=dev) for n in ("q", "uv", "pv", "qu", "qv", "qw", "eps")}

    def put(name, s, a):
        hat[name][:, s] = a.reshape(ny, nk).T

    for s in range(ns):
        ph = torch.fft.irfft2(f[s], s=(nz, nx), norm="forward")
        u, v, w, p = ph
        q = u * u + v * v + w * w
        for n, a in zip("uvwp", f[s]):
            put(n, s, a)
        for n, a in (("q", q), ("uu", u * u), ("vv", v * v), ("ww", w * w), ("uv", u * v), ("uw", u * w), ("vw", v * w)):
            put(n, s, torch.fft.rfft2(a, norm="forward"))
        for n, a in (("q", q), ("uv", u * v), ("pv", p * v), ("qu", q * u), ("qv", q * v), ("qw", q * w)):
            one[n] += a.mean((1, 2)) / ns
        for a, h in zip((u, v, w), f[s]):
            for d in (torch.fft.irfft2(1j * kx * h, s=(nz, nx), norm="forward"),
                      torch.fft.irfft2(1j * kz[:, None] * h, s=(nz, nx), norm="forward"),
                      (D @ a.reshape(ny, -1)).reshape(a.shape)):
                one["eps"] += NU * (d * d).mean((1, 2)) / ns
    del f

    def corr(*pairs):                                # mean over samples of conj(a(y1)) b(y2), [nk][y1][y2]
        out = 0
        for scale, a, b in pairs:
            out = out + scale / ns * torch.bmm(hat[a].conj().transpose(1, 2), hat[b])
        return out

    H = lambda S: S.transpose(1, 2).conj()  # noqa: E731
    KX = kx.repeat(nz)[:, None, None]
    KZ = kz.repeat_interleave(nxh)[:, None, None]
    dU = U[None, :] - U[:, None]

    def inverse(S):
        out = torch.empty((ny, ny, nz, nx), dtype=torch.float64, device=dev)
        for i in range(ny):
            out[i] = torch.fft.irfft2(S[:, i, :].T.reshape(ny, nz, nxh), s=(nz, nx), norm="forward")
        return out

    def d1(F):
        return (D @ F.reshape(ny, -1)).reshape(F.shape)

    def d2(F):
        return torch.stack([(D @ F[i].reshape(ny, -1)).reshape(F[i].shape) for i in range(ny)])

    def plus(F, a, b):                               # the one-point part a(y1) + b(y2)
        F += (a[:, None] + b[None, :])[:, :, None, None]
        return F

    i1, i2 = np.triu_indices(ny)
    if c["domain"] == "wedge":
        keep = i1 + i2 <= ny - 1
        i1, i2 = i1[keep], i2[keep]
    i1, i2 = torch.from_numpy(i1).to(dev), torch.from_numpy(i2).to(dev)
    mz = torch.tensor(_kept(nz, _ints(c["under_z"])), device=dev)
    mx = torch.tensor(_kept(nx, _ints(c["under_x"])), device=dev)
    terms = torch.empty((7, len(i1), len(mz), len(mx)), dtype=torch.float64, device=dev)

    def store(t, F):
        terms[t] = F[:, :, mz][:, :, :, mx][i1, i2] if len(mz) < nz or len(mx) < nx else F[i1, i2]

    S0 = corr((1, "u", "u"), (1, "v", "v"), (1, "w", "w"))
    res = 0
    for t, fa, k, base in ((1, ("uu", "uv", "uw"), KX, "u"), (3, ("uw", "vw", "ww"), KZ, "w")):
        S = corr((1, "q", base), (2, fa[0], "u"), (2, fa[1], "v"), (2, fa[2], "w"))
        S = S - H(S) + 4j * NU * k * S0
        if t == 1:
            S = S - 2 * dU * S0
        res = res + 1j * k * S
        F = plus(inverse(S), -one["q" + base], one["q" + base])
        if t == 1:
            F += (dU * (one["q"][:, None] + one["q"][None, :]))[:, :, None, None]
        store(t, F)
        del S, F
    S = corr((1, "u", "v"))
    S1, S2 = S + H(S), H(S) - S
    Um, dUp = dU1[:, None] + dU1[None, :], dU1[None, :] - dU1[:, None]
    S = Um * S1 - dUp * S2
    del S1, S2
    res = res - S
    uv, ep = one["uv"], one["eps"]
    xi0 = -Um * (uv[:, None] + uv[None, :]) - dUp * (uv[None, :] - uv[:, None]) - 2 * (ep[:, None] + ep[None, :])
    store(5, inverse(S) + xi0[:, :, None, None])
    res = inverse(res)
    res -= xi0[:, :, None, None]
    A = plus(inverse(-2 * S0), one["q"], one["q"])
    del S0, S
    store(0, A)
    A1, A2 = d1(A), d2(A)
    del A
    QV, X = corr((1, "q", "v")), corr((2, "uv", "u"), (2, "vv", "v"), (2, "vw", "w"))
    S = QV + X
    F = plus(inverse(S - H(S)), -one["qv"], one["qv"])
    F -= NU * (A2 - A1)
    store(2, F)
    res += 0.5 * (d2(F) - d1(F))
    del F
    P = corr((1, "p", "v"))
    S = QV - X
    S = 0.5 * (S + H(S)) - 2 * (P + H(P))
    del QV, X, P
    F = plus(inverse(S), 0.5 * one["qv"] + 2 * one["pv"], 0.5 * one["qv"] + 2 * one["pv"])
    F -= 0.5 * NU * (A1 + A2)
    store(4, F)
    res += d1(F) + d2(F)
    store(6, res)
    return {"terms": terms, "profiles": torch.stack([mean[0], mean[1], mean[2], mean[3], dU1, ep])}


def _exact_duct(c, seed):
    dev = _device()
    nx, ny, nz, ns = c["nx"], c["ny"], c["nz"], c["nsnap"]
    nxh, P = nx // 2 + 1, ny * nz
    f = _duct_fields(c, seed).reshape(ns, 4, P, nxh)
    mean = f[..., 0].real.mean(0)
    f[..., 0] -= mean
    D = {1: torch.kron(torch.from_numpy(_fd(_grid(ny), 1)), torch.eye(nz, dtype=torch.float64)).to(dev),
         2: torch.kron(torch.eye(ny, dtype=torch.float64), torch.from_numpy(_fd(_grid(nz), 1))).to(dev)}
    kx = _signed(nx, True, LX, dev)
    g = {(i, k): D[k] @ mean[i] for i in range(3) for k in (1, 2)}
    ph = torch.fft.irfft(f, n=nx, norm="forward")
    u, p = [ph[:, i] for i in range(3)], ph[:, 3]
    q = u[0] * u[0] + u[1] * u[1] + u[2] * u[2]
    cols = lambda a: torch.fft.rfft(a, norm="forward").permute(2, 0, 1).contiguous()  # noqa: E731
    hu, hq, hp = [cols(a) for a in u], cols(q), cols(p)
    hp2 = {(i, k): cols(u[i] * u[k]) for i in range(3) for k in range(i, 3)}
    for i in range(3):
        for k in range(i):
            hp2[(i, k)] = hp2[(k, i)]
    avg = lambda a: a.mean((0, 2))  # noqa: E731
    eps = 0
    for i in range(3):
        parts = [torch.fft.irfft(1j * kx * f[:, i], n=nx, norm="forward")] + [D[k] @ u[i] for k in (1, 2)]
        eps = eps + NU * sum(avg(d * d) for d in parts)

    def corr(a, b):                                  # [nxh][P][P]
        return torch.bmm(a.conj().transpose(1, 2), b) / ns

    def inverse(S):
        out = torch.empty((P, P, nx), dtype=torch.float64, device=dev)
        for i in range(0, P, 64):
            out[i:i + 64] = torch.fft.irfft(S[:, i:i + 64].permute(1, 2, 0).contiguous(), n=nx, norm="forward")
        return out

    def d1(F, k):
        return (D[k] @ F.reshape(P, -1)).reshape(F.shape)

    def d2(F, k):
        return torch.matmul(D[k], F)

    i1, i2 = (torch.from_numpy(a).to(dev) for a in np.triu_indices(P))
    terms = torch.empty((8, len(i1), nx), dtype=torch.float64, device=dev)
    K = avg(q)
    U = mean[:3]
    dU, Us = U[:, None, :] - U[:, :, None], 0.5 * (U[:, None, :] + U[:, :, None])
    S0 = corr(hu[0], hu[0]) + corr(hu[1], hu[1]) + corr(hu[2], hu[2])
    KK = K[:, None] + K[None, :]
    A = inverse(-2 * S0) + KK[..., None]
    terms[0] = A[i1, i2]
    res = 0
    for k in range(3):
        Sk, pk = avg(q * u[k]), avg(p * u[k])
        Q1, Q2 = corr(hq, hu[k]), corr(hu[k], hq)
        X1 = sum(corr(hp2[(i, k)], hu[i]) for i in range(3))
        X2 = sum(corr(hu[i], hp2[(i, k)]) for i in range(3))
        S = Q1 + 2 * X1 - Q2 - 2 * X2 - 2 * dU[k] * S0
        if k == 0:
            S = S + 4j * NU * kx[:, None, None] * S0
        F = inverse(S) + (Sk[None, :] - Sk[:, None] + dU[k] * KK)[..., None]
        if k:
            F -= NU * (d2(A, k) - d1(A, k))
            res += 0.5 * (d2(F, k) - d1(F, k))
        else:
            res = inverse(1j * kx[:, None, None] * S)
        terms[1 + k] = F[i1, i2]
        if k:
            S = 0.5 * (Q1 + Q2) - X1 - X2 - 2 * Us[k] * S0 - 2 * (corr(hp, hu[k]) + corr(hu[k], hp))
            o = 0.5 * (Sk[:, None] + Sk[None, :]) + 2 * (pk[:, None] + pk[None, :]) + Us[k] * KK
            F = inverse(S) + o[..., None]
            F -= 0.5 * NU * (d1(A, k) + d2(A, k))
            res += d1(F, k) + d2(F, k)
            terms[3 + k] = F[i1, i2]
    S = 0
    for a in range(3):
        for b in range(3):
            co = 0
            if b:
                co = co + 2 * g[(a, b)][None, :]
            if a:
                co = co + 2 * g[(b, a)][:, None]
            if a or b:
                S = S + co * corr(hu[a], hu[b])
    Pi = -sum(avg(u[i] * u[k]) * g[(i, k)] for i in range(3) for k in (1, 2))
    F = inverse(S) + (2 * (Pi - eps)[:, None] + 2 * (Pi - eps)[None, :])[..., None]
    terms[6] = F[i1, i2]
    res -= F
    terms[7] = res[i1, i2]
    prof = [mean[i] for i in range(4)] + [g[(i, k)] for i in range(3) for k in (1, 2)] + [eps]
    return {"terms": terms, "profiles": torch.stack(prof)}


def _exact_step1(c, seed):
    dev = _device()
    nx, nz, ny, ns = c["nx"], c["nz"], c["ny"], c["nsnap"]
    nxh = nx // 2 + 1
    f, mean = _step1_inputs(c, seed)
    y = _grid(ny)
    D1, D2 = torch.from_numpy(_fd(y, 1)).to(dev), torch.from_numpy(_fd(y, 2)).to(dev)
    dy = lambda M, a: (M.to(a.dtype) @ a.reshape(ny, -1)).reshape(a.shape)  # noqa: E731
    kx, kz = _signed(nx, True, LX, dev)[None, :], _signed(nz, False, LZ, dev)[:, None]
    k2 = kx * kx + kz * kz
    k2t = _signed(nx, True, LX, dev, True)[None, :] ** 2 + _signed(nz, False, LZ, dev, True)[:, None] ** 2
    inv = torch.where(k2 > 0, 1.0 / torch.where(k2 > 0, k2, 1.0), 0.0)
    out = torch.empty((ns, 4, ny, nz, nxh), dtype=torch.complex128, device=dev)
    rhs = torch.empty((ns, ny, nz, nxh), dtype=torch.complex128, device=dev)
    for s in range(ns):
        v, eta = f[s, 0], f[s, 1]
        Dv = dy(D1, v)
        u, w = 1j * inv * (kx * Dv - kz * eta), 1j * inv * (kz * Dv + kx * eta)
        u[:, 0, 0], w[:, 0, 0] = mean[s, 0].to(u.dtype), mean[s, 1].to(u.dtype)
        out[s, 0], out[s, 1], out[s, 2] = u, v, w
        P = [torch.fft.irfft2(a, s=(nz, nx), norm="forward") for a in (u, v, w)]
        pr = lambda a, b: torch.fft.rfft2(P[a] * P[b], norm="forward")  # noqa: E731
        kxt2 = _signed(nx, True, LX, dev, True)[None, :] ** 2
        kzt2 = _signed(nz, False, LZ, dev, True)[:, None] ** 2
        r = (kxt2 * pr(0, 0) + kzt2 * pr(2, 2) - dy(D2, pr(1, 1)) + 2 * kx * kz * pr(0, 2)
             - 2j * kx * dy(D1, pr(0, 1)) - 2j * kz * dy(D1, pr(1, 2)))
        d2v = dy(D2, v)
        r[0], r[-1] = NU * d2v[0], NU * d2v[-1]
        r[0, 0, 0] = 0.0
        rhs[s] = r
    # per wavenumber: D2 - k^2, Neumann rows at the walls, the (0, 0) mode pinned
    # (k^2 is the same at kz and -kz: solved together)
    for iz in range(nz // 2 + 1):
        rows = sorted({iz, (nz - iz) % nz})
        M = D2[None] - k2t[iz][:, None, None] * torch.eye(ny, dtype=torch.float64, device=dev)
        M[:, 0], M[:, -1] = D1[0], D1[-1]
        if iz == 0:
            M[0, 0] = 0.0
            M[0, 0, 0] = 1.0
        b = rhs[:, :, rows].permute(3, 1, 0, 2).reshape(nxh, ny, -1)
        x = torch.linalg.solve(M, torch.cat([b.real, b.imag], -1))
        n = b.shape[-1]
        x = torch.complex(x[..., :n].contiguous(), x[..., n:].contiguous()).reshape(nxh, ny, ns, len(rows))
        out[:, 3, :, rows] = x.permute(2, 1, 3, 0)
    return {"fields": out}


def exact(case, seed):
    with torch.no_grad():
        if case["path"] == "duct":
            return _exact_duct(case, seed)
        if case["path"] == "step1":
            return _exact_step1(case, seed)
        return _exact_channel(case, seed)
