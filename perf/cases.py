"""Performance cases: what a program that redatums seismic data has this library do.

Kernels are sums of hyperbolic events with a 15 Hz Ricker spectrum between points of a 20 m
grid (the structure of a reflection response), scaled so that the operator's norm is about 0.5.
Inputs are Ricker arrivals: focusing functions and windows of point targets for the Marchenko
solvers, recorded traces with noise for the operator itself.  Everything is made on the device
with torch from the seed alone; the operator handles (the library's copy of the kernel in the
storage format asked for) belong to the state, as a program keeps them over many calls.

``exact`` evaluates the same formulas in complex128 with torch, on the kernel as it is stored
(for 16-bit and E4M3 storage: rounded to nearest after the documented scaling of each row).
"""
import math

import numpy as np
import torch

import paper_2011_11120_gb300 as mdc

DT = 0.004            # s
AREA = 400.0          # m^2 per point of the 20 m grid
SPEED = 2000.0        # m/s above the target
FPEAK = 15.0          # Hz
QMAX = {"c16f": (32768.0, torch.float16), "cbf16": (1.0, torch.bfloat16), "ce4m3": (448.0, torch.float8_e4m3fn)}
STORED_BYTES = {"c64": 8, "c32s": 8, "c16f": 4, "cbf16": 4, "ce4m3": 2}


def listed():
    def case(name, kind, storage, nr, ns, nt, nf, nv, niter=0):
        return {"name": name, "kind": kind, "storage": storage, "nr": nr, "ns": ns, "nt": nt, "nf": nf, "nv": nv,
                "niter": niter}

    return [
        # one forward and one adjoint application on a small aperture, two points: call latency
        case("mdc_81_c64_nv2", "mdc", "c64", 81, 81, 128, 40, 2),
        # the 21 x 21 survey, one point: a kernel of 0.1 GB, launches and transforms count
        case("mdc_441_c64_nv1", "mdc", "c64", 441, 441, 256, 64, 1),
        # the 61 x 61 survey, one point: streaming the 22 GB kernel
        case("mdc_3721_c64_nv1", "mdc", "c64", 3721, 3721, 1024, 200, 1),
        # the same survey with 64 points at once, in the default storage
        case("mdc_3721_c64_nv64", "mdc", "c64", 3721, 3721, 1024, 200, 64),
        # an irregular survey (half the points missing), long traces, bfloat16 storage
        case("mdc_1861x997_cbf16_nv37", "mdc", "cbf16", 1861, 997, 2048, 300, 37),
        # the 91 x 91 survey, a quarter of its band: a few points on E4M3, many on float16
        case("mdc_8281_ce4m3_nv16", "mdc", "ce4m3", 8281, 8281, 1024, 40, 16),
        case("mdc_8281_c16f_nv128", "mdc", "c16f", 8281, 8281, 1024, 40, 128),
        # one target point on the small survey, ten iterations: a chain of short kernels
        case("marchenko_441_c64_nv1", "marchenko", "c64", 441, 441, 256, 64, 1, 10),
        # a 3 x 3 patch of target points on the 41 x 41 survey, float32 throughout
        case("marchenko_1681_c64_nv9", "marchenko", "c64", 1681, 1681, 512, 150, 9, 20),
        # a 16 x 16 patch of target points: float16 kernel in LSQR, one refinement step on split float16
        case("refined_1681_c16f_nv256", "refined", "c16f", 1681, 1681, 512, 150, 256, 20),
        # one batch of virtual sources of the deconvolution with a rectangular kernel
        case("mdd_3721x841_c64_nv20", "mdd", "c64", 3721, 841, 1024, 200, 20, 10),
        # five jobs of uneven size from host memory through the server
        case("serving_900_c16f_nv16", "serving", "c16f", 900, 900, 512, 150, 16, 12),
    ]


KINDS = ["mdc"] * 6 + ["marchenko"] * 2 + ["refined", "mdd", "neumann", "serving"]


def draw(rng):
    """A case of the same ranges: 25 .. 8281 traces, 64 .. 4096 samples, 1 .. 256 columns."""
    def log_int(lo, hi):
        return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))

    while True:
        kind = rng.choice(KINDS)
        nt = rng.choice([64, 128, 256, 256, 512, 512, 1024, 1024, 1024, 2048, 4096])
        c = {"kind": kind, "storage": rng.choice(["c64", "c64", "c64", "c16f", "c32s", "cbf16", "ce4m3"]),
             "nr": log_int(25, 8281), "ns": log_int(25, 8281), "nt": nt, "nf": rng.randint(min(nt // 8, 150), min(nt // 3, 300)),
             "nv": log_int(1, 256), "niter": 0}
        if kind != "mdc":
            c["niter"] = rng.randint(4, 20)
        if kind in ("marchenko", "neumann", "refined", "serving"):
            c["nr"] = c["ns"] = log_int(25, 2000)
        if kind in ("refined", "serving"):
            c["storage"] = rng.choice(["c16f", "c16f", "cbf16"])
        if kind == "serving":
            c["nv"] = log_int(1, 24)
        kernel = 8 * c["nf"] * c["nr"] * c["ns"]
        vectors = 4 * nt * max(c["nr"], c["ns"]) * c["nv"]
        w = work(c)
        if kernel > 12e9 or vectors > (0.9e9 if kind != "serving" else 0.1e9):
            continue
        if w["flops"] <= 2.8e12 and w["bytes"] + 10 * _passes(c) * vectors <= 100e9:
            return c


def _job_columns(case):
    """Columns and iterations of the jobs of a serving case."""
    return [(1 + (j * 37 + 11 + case["nv"]) % case["nv"], case["niter"] + (3 * j) % 8) for j in range(5)]


def _passes(case):
    """Applications of the kernel to nv columns in one run (an LSQR iteration of the Marchenko
    system applies R and R* forward and adjoint)."""
    k, n = case["kind"], case["niter"]
    if k == "mdc":
        return 2
    if k == "mdd":
        return 2 * n + 1
    if k == "neumann":
        return 1 + 2 * (n - 1) + 2
    if k == "refined":
        return (1 + 2 + 4 * n) + 2 + (2 + 4 * 5) + 2 + 2
    return 1 + 2 + 4 * n + 2


def _sweeps(case):
    """Times the whole kernel has to be read: once per dependent product."""
    k, n = case["kind"], case["niter"]
    if k == "mdc":
        return 2
    if k == "mdd":
        return 2 * n + 1
    if k == "neumann":
        return 1 + (n - 1) + 1
    if k == "refined":
        return (1 + 1 + 2 * n) + 1 + (1 + 2 * 5) + 1 + 1
    return 1 + 1 + 2 * n + 1


def work(case):
    """Kernel reads of every dependent product, inputs read and outputs written once; the complex
    products (8 flops per kernel entry and column) and nothing for the transforms."""
    entries = case["nf"] * case["nr"] * case["ns"]
    col_in, col_out = 4 * case["nt"] * case["ns"], 4 * case["nt"] * case["nr"]
    size = entries * STORED_BYTES[case["storage"]]
    k, nv = case["kind"], case["nv"]
    if k == "mdc":
        return {"bytes": 2 * size + 2 * nv * (col_in + col_out), "flops": 2 * 8 * entries * nv}
    if k == "mdd":
        return {"bytes": _sweeps(case) * size + nv * (col_in + col_out), "flops": _passes(case) * 8 * entries * nv}
    if k == "serving":
        jobs = _job_columns(case)
        nv = sum(v for v, _ in jobs)
        sweeps = max(_sweeps({**case, "kind": "marchenko", "niter": n}) for _, n in jobs)
        flops = sum(_passes({**case, "kind": "marchenko", "niter": n}) * 8 * entries * v for v, n in jobs)
        return {"bytes": sweeps * size + nv * 5 * col_in, "flops": flops}
    return {"bytes": _sweeps(case) * size + nv * 5 * col_in, "flops": _passes(case) * 8 * entries * nv}


def tolerance(case):
    """About four times the largest error against ``exact`` seen on the device: single products 3.8e-7
    (complex64), 2.6e-4 (float16 spectra, short columns), 2e-3 (bfloat16 spectra); solves 3e-6 in the
    Green's functions (complex64), 1.8e-3 (float16 throughout), 6e-6 (refined)."""
    if case["kind"] == "mdc":
        return {"rel": {"c64": 2e-6, "c32s": 8e-6, "c16f": 1e-3, "cbf16": 8e-3, "ce4m3": 1e-3}[case["storage"]]}
    if case["kind"] == "refined":
        return {"rel": 5e-5 if case["storage"] == "c16f" else 5e-4}
    return {"rel": {"c64": 1.5e-5, "c32s": 4e-5, "c16f": 6e-3, "cbf16": 2e-2, "ce4m3": 6e-3}[case["storage"]]}


# ------------------------------------------------------------------ inputs
def _generator(seed, part):
    return torch.Generator(device="cuda").manual_seed(1000003 * part + seed)


def _points(n, g):
    """n points of the smallest square 20 m grid that holds them, in a fixed scan order."""
    side = math.isqrt(n - 1) + 1
    keep = torch.sort(torch.randperm(side * side, generator=g, device="cuda")[:n]).values
    return torch.stack([20.0 * (keep % side), 20.0 * (keep // side)], 1).double()


def _ricker(t):
    a = (math.pi * FPEAK * t) ** 2
    return (1.0 - 2.0 * a) * torch.exp(-a)


def _distances(a, b):
    return torch.sqrt((a[:, None, 0] - b[None, :, 0]) ** 2 + (a[:, None, 1] - b[None, :, 1]) ** 2)


def _survey(case, seed):
    """Receiver and source points (the same ones for a square kernel) and the kernel
    complex64 [nf, nr, ns], its operator norm scaled to about 0.5."""
    g = _generator(seed, 1)
    src = _points(case["ns"], g)
    rec = src if case["nr"] == case["ns"] else _points(case["nr"], g)
    u = torch.rand(3, 5, generator=g, device="cuda", dtype=torch.float64).cpu()
    t0, vel = 0.2 + 0.6 * u[0], 1500.0 + 1500.0 * u[1]
    amp = torch.randn(5, generator=g, device="cuda", dtype=torch.float64).cpu()
    d2 = _distances(rec, src) ** 2
    tau = [torch.sqrt(d2 / float(v) ** 2 + float(t) ** 2) for t, v in zip(t0, vel)]
    del d2
    nf, df = case["nf"], 1.0 / (case["nt"] * DT)
    G = torch.empty((nf, case["nr"], case["ns"]), dtype=torch.complex64, device="cuda")
    for k in range(nf):
        f = max(k, 0.25) * df
        w = (f / FPEAK) ** 2 * math.exp(1.0 - (f / FPEAK) ** 2) + 1e-3
        acc = G[k]
        acc.zero_()
        for e in range(5):
            ph = (f * tau[e]).frac_().mul_(-2.0 * math.pi).float()
            acc.add_(torch.polar(torch.full_like(ph, w * float(amp[e])), ph))
    del tau
    # the largest singular value over the frequencies, by a few power iterations
    v = torch.randn((nf, case["ns"], 1), generator=g, device="cuda").to(torch.complex64)
    norm = None
    for _ in range(6):
        v = v / torch.linalg.vector_norm(v, dim=1, keepdim=True)
        z = torch.bmm(G, v)
        norm = torch.linalg.vector_norm(z, dim=1).max()
        v = torch.stack([torch.mv(G[k].T, z[k, :, 0].conj()).conj() for k in range(nf)])[:, :, None]
    G.mul_(0.5 / (DT * AREA * float(norm)))
    return rec, src, G


def _traces(nt, pts, nv, g):
    """Recorded traces [nt, n, nv]: the arrival from a random point per column, with a second,
    weaker one and one per cent of noise."""
    ext = float(pts.max()) + 20.0
    x = torch.randn((nt, len(pts), nv), generator=g, device="cuda")
    x.mul_(0.01)
    tgt = ext * torch.rand((nv, 2), generator=g, device="cuda", dtype=torch.float64)
    t1 = torch.sqrt(600.0 ** 2 + _distances(pts, tgt) ** 2) / SPEED
    tt = DT * torch.arange(nt, device="cuda", dtype=torch.float64)
    for a in range(0, nt, 64):
        t = tt[a:a + 64, None, None]
        x[a:a + 64] += (_ricker(t - t1) - 0.4 * _ricker(t - 1.3 * t1)).float()
    return x


def _focusing(nt, pts, nv, g):
    """Window cut-offs int32 [n, nv] and direct focusing function [nt, n, nv] of random target
    points; their depth keeps the direct arrival inside the causal half of the traces."""
    ext = float(pts.max()) + 20.0
    depth = min(800.0, 0.25 * nt * DT * SPEED)
    tgt = ext * torch.rand((nv, 2), generator=g, device="cuda", dtype=torch.float64)
    td = torch.sqrt(depth ** 2 + _distances(pts, tgt) ** 2) / SPEED
    cut = (torch.round(td / DT).long() - 4).int()
    tau = torch.arange(nt, device="cuda", dtype=torch.float64)
    tau = DT * torch.where(tau < nt // 2, tau, tau - nt)
    fd = torch.empty((nt, len(pts), nv), device="cuda")
    for a in range(0, nt, 64):
        fd[a:a + 64] = _ricker(tau[a:a + 64, None, None] + td).float()
    return cut.contiguous(), fd


class _Server:
    """A server over an operator, its jobs' pinned inputs and outputs."""

    def __init__(self, op, case, pts, g):
        self.op = op
        self.jobs = []
        for nv, niter in _job_columns(case):
            cut, fd = _focusing(case["nt"], pts, nv, g)
            outs = [torch.empty(fd.shape, pin_memory=True).numpy() for _ in range(4)]
            host = torch.empty(fd.shape, pin_memory=True)
            host.copy_(fd)
            self.jobs.append((cut.cpu().numpy(), host.numpy(), nv, niter, outs))
        self.srv = mdc.srv_create(op.h, None, 1 << 35, 512)

    def __del__(self):
        if getattr(self, "srv", None) is not None:
            mdc.srv_destroy(self.srv)


def prepare(case, seed):
    rec, src, G = _survey(case, seed)
    kind, nt, nv = case["kind"], case["nt"], case["nv"]
    g = _generator(seed, 2)
    s = {"case": case, "op": mdc.MDC(G, nt, DT, AREA, storage=case["storage"])}
    if kind == "refined":
        s["ref"] = mdc.MDC(G, nt, DT, AREA, storage="c32s")
    del G
    if kind == "mdc":
        s["x"] = _traces(nt, src, nv, g)
        s["y"] = _traces(nt, rec, nv, g)
    elif kind == "mdd":
        s["d"] = _traces(nt, rec, nv, g)
    elif kind == "serving":
        s["server"] = _Server(s["op"], case, src, g)
    else:
        s["cut"], s["fd"] = _focusing(nt, src, nv, g)
    torch.cuda.empty_cache()        # the library allocates outside torch's pool
    return s


# ------------------------------------------------------------------ one pass
FIELDS = ("f_minus", "f_mplus", "g_minus", "g_plus")


def run(s):
    c, op = s["case"], s["op"]
    kind = c["kind"]
    if kind == "mdc":
        return {"y": op.forward(s["x"]), "x": op.adjoint(s["y"])}
    if kind == "mdd":
        out = op.mdd(s["d"], c["niter"])
        return {"r": out["r"], "resid": np.array(out["resid"])}
    if kind == "serving":
        srv, jobs = s["server"].srv, s["server"].jobs
        ids = [mdc.srv_submit(srv, cut, fd, nv, niter, 0.0, outs) for cut, fd, nv, niter, outs in jobs]
        done = 0
        while done < len(ids):
            done += mdc.srv_step(srv)
        for i in ids:
            mdc.srv_release(srv, i)
        return [dict(zip(FIELDS, outs)) for _, _, _, _, outs in jobs]
    if kind == "neumann":
        out = op.neumann(s["cut"], s["fd"], c["niter"])
        return {k: out[k] for k in FIELDS}
    if kind == "refined":
        out = op.marchenko_refined(s["ref"], s["cut"], s["fd"], c["niter"], nrefine=1, niter_refine=5)
        return {**{k: out[k] for k in FIELDS}, "history": np.array(out["resid"] + [out["final_residual"]])}
    out = op.marchenko(s["cut"], s["fd"], c["niter"])
    return {**{k: out[k] for k in FIELDS}, "resid": np.array(out["resid"])}


# ------------------------------------------------------------------ the same in 64 bits
def _as_stored(Gk, storage):
    """One frequency [nr, ns] of the kernel as the storage format holds it, in complex128."""
    if storage not in QMAX:
        return Gk.to(torch.complex128)
    qmax, dtype = QMAX[storage]
    v = torch.view_as_real(Gk)
    top = v.abs().amax(dim=(1, 2), keepdim=True)
    inv = torch.where(top > 0, qmax / top, torch.zeros_like(top))
    q = (v * inv).to(dtype).double()
    return torch.view_as_complex(q * (top / qmax).double())


class _Exact:
    """C and C^H in complex128, one frequency after the other."""

    def __init__(self, G, storage, nt):
        self.nt, self.nf = nt, G.shape[0]
        # small kernels are converted once, large ones frequency by frequency
        self.G = [_as_stored(G[k], storage) for k in range(self.nf)] if G.numel() <= 6e8 else None
        self.raw, self.storage = G, storage

    def _apply(self, x, adjoint, conj):
        X = torch.fft.rfft(x.double(), dim=0)[:self.nf]
        X = X.conj() if conj else X
        out = None
        for k in range(self.nf):
            Gk = self.G[k] if self.G is not None else _as_stored(self.raw[k], self.storage)
            yk = (Gk.mH if adjoint else Gk) @ X[k]
            if out is None:
                out = torch.zeros((self.nt // 2 + 1,) + tuple(yk.shape), dtype=torch.complex128, device="cuda")
            out[k] = yk
        out = out.conj() if conj else out
        out[0].imag.zero_()
        return torch.fft.irfft(out * (DT * AREA), n=self.nt, dim=0)

    def fwd(self, x, conj=False):
        return self._apply(x, False, conj)

    def adj(self, y, conj=False):
        return self._apply(y, True, conj)


def _lsqr(matvec, rmatvec, b, niter):
    """Paige and Saunders (1982) on tuples of tensors, x0 = 0: (x, residual norms)."""
    def norm(v):
        return math.sqrt(sum(float(torch.sum(t * t)) for t in v))

    beta = norm(b)
    u = tuple(t / beta for t in b)
    v = rmatvec(u)
    alpha = norm(v)
    v = tuple(t / alpha for t in v)
    w, x = v, tuple(torch.zeros_like(t) for t in v)
    phibar, rhobar, resid = beta, alpha, [beta]
    for _ in range(niter):
        u = tuple(p - alpha * q for p, q in zip(matvec(v), u))
        beta = norm(u)
        u = tuple(t / beta for t in u)
        v = tuple(p - beta * q for p, q in zip(rmatvec(u), v))
        alpha = norm(v)
        v = tuple(t / alpha for t in v)
        rho = math.hypot(rhobar, beta)
        c, sn = rhobar / rho, beta / rho
        theta, rhobar, phi, phibar = sn * alpha, -c * alpha, c * phibar, sn * phibar
        x = tuple(p + (phi / rho) * q for p, q in zip(x, w))
        w = tuple(p - (theta / rho) * q for p, q in zip(v, w))
        resid.append(phibar)
    return x, resid


def _solve_exact(case, cut, fd, lo, ref):
    """The Marchenko system of one group of points, as the call of this kind solves it."""
    nt, niter = case["nt"], case["niter"]
    t = torch.arange(nt, device="cuda")
    win = (torch.where(t < nt // 2, t, nt - t)[:, None, None] < cut[None]).double()
    fd = fd.double()

    def m(op):
        return lambda f: (f[0] - win * op.fwd(f[1]), f[1] - win * op.fwd(f[0], True))

    def mh(op):
        return lambda h: (h[0] - op.adj(win * h[1], True), h[1] - op.adj(win * h[0]))

    d = (win * ref.fwd(fd), torch.zeros_like(fd))
    history = []
    if case["kind"] == "neumann":
        x = d
        for _ in range(niter - 1):
            x = (d[0] + win * ref.fwd(x[1]), win * ref.fwd(x[0], True))
    else:
        x, history = _lsqr(m(lo), mh(lo), d, niter)
        if case["kind"] == "refined":
            r = tuple(p - q for p, q in zip(d, m(ref)(x)))
            dx, more = _lsqr(m(lo), mh(lo), r, 5)
            x = tuple(p + q for p, q in zip(x, dx))
            r = tuple(p - q for p, q in zip(d, m(ref)(x)))
            size = [math.sqrt(sum(float(torch.sum(q * q)) for q in z)) for z in (r, d)]
            history = history + more + [size[0] / size[1]]
    fplus = fd + x[1]
    gps = fplus - ref.fwd(x[0], True)
    return {"f_minus": x[0], "f_mplus": x[1], "g_minus": ref.fwd(fplus) - x[0],
            "g_plus": torch.roll(torch.flip(gps, (0,)), 1, 0)}, history


def exact(case, seed):
    flops = work(case)["flops"]
    if flops > 8e12:                                   # over 20 seconds in 64 bits
        return None
    kind, nt, nv = case["kind"], case["nt"], case["nv"]
    rec, src, G = _survey(case, seed)
    g = _generator(seed, 2)
    op = _Exact(G, case["storage"], nt)
    if kind == "mdc":
        x, y = _traces(nt, src, nv, g), _traces(nt, rec, nv, g)
        return {"y": op.fwd(x), "x": op.adj(y)}
    if kind == "mdd":
        d = _traces(nt, rec, nv, g).double()
        (r,), resid = _lsqr(lambda v: (op.fwd(v[0]),), lambda u: (op.adj(u[0]),), (d,), case["niter"])
        return {"r": r, "resid": np.array(resid)}
    if kind == "serving":
        outs = []
        for cols, niter in _job_columns(case):
            cut, fd = _focusing(nt, src, cols, g)
            one = {**case, "kind": "marchenko", "niter": niter}
            outs.append({k: v.cpu().numpy() for k, v in _solve_exact(one, cut, fd, op, op)[0].items()})
        return outs
    cut, fd = _focusing(nt, src, nv, g)
    ref = _Exact(G, "c32s", nt) if kind == "refined" else op
    out, history = _solve_exact(case, cut, fd, op, ref)
    if kind == "neumann":
        return out
    return {**out, ("history" if kind == "refined" else "resid"): np.array(history)}
