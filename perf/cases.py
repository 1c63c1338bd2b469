"""What this framework's speed is measured on: the calls its users make, over the
sizes they make them at.

Every case is one call (or one pair of calls) of the Python binding of include/wf.h:

  flat      wf_solve on the periodic flat grid (FP64)
  synth     wf_alm2map: the basis change harmonic -> pixels
  adjoint   wf_map2alm_adjoint: the basis change pixels -> harmonic
  solve     wf_solve on the sphere, temperature (ncomp 1) or I, Q, U (ncomp 3)
  batch     wf_solve_batch: Wiener-filter and fluctuation solves of one geometry, paired

Solves run a fixed list of (lambda, L), the cooling levels of the heuristic schedule
(wf_set_schedule, the call that replays or resumes a recorded run), so a pass is the same
work whatever the last bits of chi^2 are.  In a real solve about half of the iterations
are at lambda = 1 on the full band and the others are spread over the levels; so are these.

Inputs are made on the device from the seed: CMB-like C_l, a hit pattern that rises to
the ecliptic poles, a galactic cut and point-source disks, plane waves with the power of
C_l as the signal, white noise of the pixel variance.

FP64 plans return FP64 arrays.  The mixed-precision plans compute their transforms in
FP32 (or in splits of FP32) and store them in FP64 arrays; a program that chose such a
plan keeps its maps and a_lm in single precision, as sky-map files do, and so does
run(): it hands back float32 maps and complex64 a_lm.
"""
import math

import numpy as np
import torch

import paper_1210_4931_gb300 as wf

DEV = torch.device("cuda" if torch.cuda.is_available() else "cpu")
F8, C16 = torch.float64, torch.complex128


def _c(name, kind, **kw):
    return {"name": name, "kind": kind, **kw}


def listed():
    return [
        # the 128 x 128 flat-sky problem (the repository's first configuration), a few cooling levels of it
        _c("flat_128", "flat", n=128, iters=300),
        # a small patch filtered on its own: the smallest solve, latency counts
        _c("flat_32", "flat", n=32, iters=25),
        # the smallest map of the request loop: one transform, launches count
        _c("synth_64", "synth", nside=64, lmax=128, precision="mixed", ncomp=1),
        # one transform of a large map: simulating a sky
        _c("synth_1024", "synth", nside=1024, lmax=2048, precision="mixed", ncomp=1),
        # its adjoint at a grid that is no power of two, ragged band limit
        _c("adjoint_768", "adjoint", nside=768, lmax=1499, precision="mixed", ncomp=1),
        # double precision, the accuracy reference of every other plan
        _c("synth_256_fp64", "synth", nside=256, lmax=512, precision="fp64", ncomp=1),
        # an FP64 solve of a small odd grid
        _c("solve_100_fp64", "solve", nside=100, lmax=187, precision="fp64", ncomp=1, iters=6, sweeps=0),
        # the request loop's commonest sizes: a whole short solve with host decisions in between
        _c("solve_128", "solve", nside=128, lmax=256, precision="mixed", ncomp=1, iters=24, sweeps=0),
        # the nside 512 temperature map, ending in double-float correction sweeps
        _c("solve_512_sweeps", "solve", nside=512, lmax=1024, precision="mixed", ncomp=1, iters=16, sweeps=1),
        # the benchmark's map: nside 2048, lmax 4096
        _c("solve_2048", "solve", nside=2048, lmax=4096, precision="mixed", ncomp=1, iters=5, sweeps=0),
        # polarised maps of the constrained-realisation workload
        _c("solve_pol_512", "solve", nside=512, lmax=1024, precision="mixed", ncomp=3, iters=4, sweeps=0),
        # four constrained realisations of one geometry (a Wiener filter and a fluctuation solve each),
        # their synthesis shared on the tensor cores
        _c("batch_256_tf32", "batch", nside=256, lmax=512, precision="tf32", maps=4, iters=4),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["flat", "synth", "adjoint", "solve", "solve", "batch"])
    if kind == "flat":
        return {"kind": kind, "n": rng.choice([16, 32, 64, 128]), "iters": _log(rng, 20, 300)}
    prec = rng.choice(["mixed", "mixed", "mixed", "fp64", "tf32", "bf16"])
    nc = rng.choice([1, 1, 3])
    hi = {"synth": 1100, "adjoint": 1100, "solve": 700, "batch": 200}[kind]
    if prec == "fp64":
        hi = min(hi, 256)
    if nc == 3:
        hi = min(hi, 420)
    nside = _log(rng, 24, hi)
    if rng.random() < 0.4:
        nside = 1 << int(round(math.log2(nside)))
    lmax = 2 * nside if rng.random() < 0.5 else rng.randint(nside, 2 * nside)
    case = {"kind": kind, "nside": nside, "lmax": lmax, "precision": prec}
    if kind == "batch":
        return {**case, "maps": rng.randint(2, 5), "iters": rng.randint(3, 8)}
    case["ncomp"] = nc
    if kind == "solve":
        case["iters"] = rng.randint(3, 12)
        case["sweeps"] = rng.choice([0, 0, 1]) if prec != "fp64" and nc == 1 else 0
    return case


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------
def _gen(seed, k=0):
    g = torch.Generator(device=DEV)
    g.manual_seed(int(seed) * 1000 + k)
    return g


def _randn(g, *shape):
    return torch.randn(*shape, dtype=F8, device=DEV, generator=g)


def _rings(nside):
    """z, first longitude and length of every ring of the HEALPix RING grid."""
    i = np.arange(1, 4 * nside)
    k = np.minimum(i, 4 * nside - i)
    cap = k < nside
    z = np.where(cap, 1.0 - k * k / (3.0 * nside * nside), 4.0 / 3.0 - 2.0 * np.minimum(i, 4 * nside - i) / (3.0 * nside))
    z = np.where(i > 2 * nside, -z, z)
    z[2 * nside - 1] = 0.0
    nr = np.where(cap, 4 * k, 4 * nside)
    q = np.where(cap, 1, np.where((i + nside) % 2 == 1, 0, 1))
    return z, q, nr


def _pixels(nside):
    """Unit vectors of every pixel, 3 x npix."""
    z, q, nr = (torch.as_tensor(np.ascontiguousarray(a), device=DEV) for a in _rings(nside))
    off = torch.cumsum(nr, 0) - nr
    n = torch.repeat_interleave(nr, nr)
    j = torch.arange(12 * nside * nside, device=DEV, dtype=F8) - torch.repeat_interleave(off, nr)
    phi = (2.0 * j + torch.repeat_interleave(q, nr)) * math.pi / n
    zz = torch.repeat_interleave(z.to(F8), nr)
    s = torch.sqrt((1.0 - zz) * (1.0 + zz))
    return torch.stack([s * torch.cos(phi), s * torch.sin(phi), zz])


def _cl(lmax):
    """CMB-like spectrum with a beam of 2.2 resolution elements, C_0 = C_1 = 0."""
    l = np.arange(lmax + 1, dtype=np.float64)
    sb = 2.2 * math.pi / lmax / math.sqrt(8.0 * math.log(2.0))
    l1 = np.maximum(l, 1.0)
    c = 2.0 * math.pi / (l1 * (l1 + 1.0)) * (1.0 + 0.3 * np.sin(l / 45.0)) * np.exp(-((l * sb) ** 2))
    c[:2] = 0.0
    return c


def _alm_index(lmax):
    m = torch.repeat_interleave(torch.arange(lmax + 1, device=DEV), torch.arange(lmax + 1, 0, -1, device=DEV))
    base = (m * (2 * lmax + 3 - m)) // 2
    l = torch.arange(m.numel(), device=DEV) - base + m
    return l, m


def _unit_alm(g, lmax):
    """Unit complex Gaussian a_lm of a real field, m-major (m = 0 real)."""
    n = (lmax + 1) * (lmax + 2) // 2
    a = torch.complex(_randn(g, n), _randn(g, n)) * math.sqrt(0.5)
    a[: lmax + 1] = (a[: lmax + 1].real * math.sqrt(2.0)).to(C16)
    return a


def _wave_map(g, vec, cl, waves=40):
    """Plane waves of random direction with the power of cl around l = |k|."""
    lmax = len(cl) - 1
    edges = np.unique(np.round(np.geomspace(2, lmax + 1, waves + 1)).astype(int))
    out = torch.zeros(vec.shape[1], dtype=F8, device=DEV)
    par = _randn(g, len(edges), 3)
    par = (par / par.norm(dim=1, keepdim=True)).cpu().numpy()
    ph = (torch.rand(len(edges), dtype=F8, device=DEV, generator=g) * 2 * math.pi).cpu().numpy()
    for b in range(len(edges) - 1):
        l = np.arange(edges[b], edges[b + 1])
        var = float(np.sum((2 * l + 1) * cl[l]) / (4 * math.pi))
        k = float(l.mean())
        arg = vec[0] * (k * par[b, 0]) + vec[1] * (k * par[b, 1]) + vec[2] * (k * par[b, 2]) + float(ph[b])
        out += math.sqrt(2.0 * var) * torch.cos(arg)
    return out


_POLE = (-0.0964, -0.8623, 0.4971)  # ecliptic pole in galactic coordinates


def _sky(case, seed):
    """Noise variance, mask and spectrum of one geometry (all maps of a case share them)."""
    nside, lmax = case["nside"], case["lmax"]
    g = _gen(seed)
    vec = _pixels(nside)
    npix = vec.shape[1]
    sb = (vec[0] * _POLE[0] + vec[1] * _POLE[1] + vec[2] * _POLE[2]).abs()
    hits = (1.0 + 4.0 * sb ** 3) * torch.exp(0.2 * _randn(g, npix))
    mask = vec[2].abs() >= math.sin(math.radians(15.0))
    cen = _randn(g, 48, 3)
    cen = (cen / cen.norm(dim=1, keepdim=True)).cpu().numpy()
    for c in cen:
        mask &= vec[0] * c[0] + vec[1] * c[1] + vec[2] * c[2] < math.cos(math.radians(1.2))
    cl = _cl(lmax)
    omega = 4.0 * math.pi / npix
    nv = cl[max(2, lmax // 2)] * float(hits.mean()) / omega / hits
    return g, vec, nv, mask.to(torch.uint8), cl


def _problem(case, seed):
    """Everything a solve of the sphere takes, on the device."""
    nc = case.get("ncomp", 1)
    g, vec, nv, mask, cl = _sky(case, seed)
    npix, lmax = vec.shape[1], case["lmax"]
    P = {"mask": mask, "maps": []}
    if nc == 1:
        P["noise"] = nv
        P["cl"] = torch.as_tensor(cl, device=DEV)
        eig = cl
    else:
        rho = (torch.rand(3, npix, dtype=F8, device=DEV, generator=g) - 0.5) * 0.2
        sI, sP = nv, 2.0 * nv
        P["noise"] = torch.stack([sI, sP, sP, rho[0] * (sI * sP).sqrt(), rho[1] * (sI * sP).sqrt(), rho[2] * sP])
        tt, ee = cl, 0.05 * cl
        te = 0.5 * np.sqrt(tt * ee)
        P["cl"] = torch.as_tensor(np.stack([tt, ee, np.zeros_like(tt), te]), device=DEV)
        eig = 0.5 * (tt + ee) + np.sqrt(0.25 * (tt - ee) ** 2 + te ** 2)
    for _ in range(case.get("maps", 1)):
        comp = []
        for c in range(nc):
            var = nv if c == 0 else 2.0 * nv
            comp.append(_wave_map(g, vec, cl * (1.0 if c == 0 else 0.05)) + var.sqrt() * _randn(g, npix))
        d = {"d": torch.stack(comp) if nc == 3 else comp[0]}
        if case["kind"] == "batch":
            d["g1"] = _randn(g, npix)
            d["g2"] = _unit_alm(g, lmax)
        P["maps"].append(d)
    # the heuristic schedule's levels (lambda, L); tau is about the smallest variance: any value of
    # that size cools the same way, and the list is plain numbers of the problem
    tau_h = float(nv[mask > 0].min()) * 4.0 * math.pi / npix
    levels, li = [], 20
    while True:
        li = min(li, lmax)
        lam = max(1.0, float(eig[li]) / tau_h) if li < lmax else 1.0
        levels.append((lam, min(lmax, li + 100) if li < lmax else lmax))
        if li >= lmax:
            break
        li += min(li, 500)
    k = case["iters"]
    nf = (k + 1) // 2
    cool = [levels[int(i * (len(levels) - 1) / max(1, k - nf))] for i in range(k - nf)]
    P["schedule"] = cool + [(1.0, lmax)] * nf
    return P


def _flat_problem(case, seed):
    n = case["n"]
    g = _gen(seed)
    ky = np.fft.fftfreq(n) * n
    k = np.sqrt(ky[:, None] ** 2 + np.arange(n // 2 + 1)[None, :] ** 2)
    p = (k + 2.0) ** -2.5
    w = np.full(p.shape, 2.0)
    w[:, 0] = w[:, -1] = 1.0
    S = torch.as_tensor(n * n / float((w * p).sum()) * p, device=DEV)
    nv = 10.0 ** (-2.0 * torch.rand(n, n, dtype=F8, device=DEV, generator=g))
    mask = torch.ones(n, n, dtype=torch.uint8, device=DEV)
    mask[n // 2 - n // 32: n // 2 + n // 32] = 0
    mask[torch.rand(n, n, dtype=F8, device=DEV, generator=g) < 0.05] = 0
    d = torch.fft.irfft2(torch.fft.rfft2(_randn(g, n, n), norm="ortho") * S.sqrt(), s=(n, n), norm="ortho")
    d = d + nv.sqrt() * _randn(g, n, n)
    k, lam = case["iters"], []
    for i in range(k):
        lam.append(max(1.0, 100.0 * 0.25 ** (8 * i // max(1, k))))
    return {"d": d.contiguous(), "noise": nv, "mask": mask, "S": S.contiguous(), "lam": lam}


def _transform_input(case, seed):
    lmax, nc = case["lmax"], case["ncomp"]
    g = _gen(seed)
    cl = _cl(lmax)
    amp = (1.0, 0.05, 0.01)
    if case["kind"] == "synth":
        l, _ = _alm_index(lmax)
        sc = torch.as_tensor(np.sqrt(cl), device=DEV)[l]
        return torch.stack([_unit_alm(g, lmax) * sc * math.sqrt(amp[c]) for c in range(nc)]).reshape(-1)
    vec = _pixels(case["nside"])
    npix = vec.shape[1]
    white = math.sqrt(cl[max(2, lmax // 2)] * npix / (4.0 * math.pi))
    return torch.stack([_wave_map(g, vec, cl * amp[c]) + white * math.sqrt(amp[c]) * _randn(g, npix)
                        for c in range(nc)]).reshape(-1)


# ---------------------------------------------------------------------------
# a pass
# ---------------------------------------------------------------------------
def _keep(case, t):
    """Results as the program keeps them: FP64 of an FP64 plan, single precision of a mixed one."""
    if case.get("precision", "fp64") == "fp64":
        return t
    return t.to(torch.complex64 if t.is_complex() else torch.float32)


def _plan(case):
    return wf.wf_plan_create("healpix", nside=case["nside"], lmax=case["lmax"], precision=case["precision"],
                             ncomp=case.get("ncomp", 1))


def prepare(case, seed):
    kind = case["kind"]
    st = {"case": case}
    if kind == "flat":
        n = case["n"]
        P = _flat_problem(case, seed)
        st["plan"] = wf.wf_plan_create("flat", n=n)
        wf.wf_set_schedule(st["plan"], P["lam"])
        st["P"] = P
        st["s"] = torch.empty(n, n, dtype=F8, device=DEV)
        st["alm"] = torch.empty(n, n // 2 + 1, dtype=C16, device=DEV)
        return st
    if kind in ("synth", "adjoint"):
        st["plan"] = p = _plan(case)
        st["in"] = _transform_input(case, seed)
        nc = case["ncomp"]
        st["out"] = torch.empty(nc * p.npix, dtype=F8, device=DEV) if kind == "synth" else \
            torch.empty(nc * p.nalm, dtype=C16, device=DEV)
        return st
    P = _problem(case, seed)
    lam, L = [x[0] for x in P["schedule"]], [x[1] for x in P["schedule"]]
    st["P"] = P
    if kind == "solve":
        st["plan"] = p = _plan(case)
        if case["sweeps"]:
            wf.wf_set_options(p, refine_sweeps=case["sweeps"])
        wf.wf_set_schedule(p, lam, L)
        st["s"] = torch.empty(p.ncomp * p.npix, dtype=F8, device=DEV)
        st["alm"] = torch.empty(p.ncomp * p.nalm, dtype=C16, device=DEV)
        return st
    st["plans"], st["items"] = [], []
    for q in P["maps"]:
        for k in ("wf", "fluct"):
            p = _plan(case)
            wf.wf_set_schedule(p, lam, L)
            it = {"kind": k, "noise_var": P["noise"], "mask": P["mask"], "C_ell": P["cl"], "tol": 1e-9,
                  "s_out": torch.empty(p.npix, dtype=F8, device=DEV),
                  "alm_out": torch.empty(p.nalm, dtype=C16, device=DEV)}
            it.update({"d": q["d"]} if k == "wf" else {"g1": q["g1"], "g2": q["g2"]})
            st["plans"].append(p)
            st["items"].append(it)
    return st


def run(st):
    case = st["case"]
    kind = case["kind"]
    if kind == "flat":
        P = st["P"]
        wf.wf_solve(st["plan"], P["d"], P["noise"], P["mask"], P["S"], 1e-9, st["s"], st["alm"])
        return {"map": st["s"], "alm": st["alm"]}
    if kind == "synth":
        wf.wf_alm2map(st["plan"], st["in"], case["lmax"], st["out"])
        return {"map": _keep(case, st["out"])}
    if kind == "adjoint":
        wf.wf_map2alm_adjoint(st["plan"], st["in"], case["lmax"], st["out"])
        return {"alm": _keep(case, st["out"])}
    P = st["P"]
    if kind == "solve":
        wf.wf_solve(st["plan"], P["maps"][0]["d"], P["noise"], P["mask"], P["cl"], 1e-9, st["s"], st["alm"])
        return {"map": _keep(case, st["s"]), "alm": _keep(case, st["alm"])}
    wf.wf_solve_batch(st["plans"], st["items"])
    return {"map": [_keep(case, it["s_out"]) for it in st["items"]],
            "alm": [_keep(case, it["alm_out"]) for it in st["items"]]}


def _transform_work(nside, lmax, L, spin2):
    """Operations of one transform to band limit L: per (l, m, ring pair) the recurrence (3) and
    the complex contraction with the even/odd symmetry (4), twice the recurrence and four times
    the contraction for the spin-2 pair; 5 n log2 n per ring DFT."""
    tri = 2.0 * nside * (L + 1) * (L + 2) / 2
    _, _, nr = _rings(nside)
    fft = float(np.sum(2.5 * nr * np.log2(np.maximum(nr, 2))))
    return tri * (7 + (22 if spin2 else 0)) + fft * (3 if spin2 else 1)


def work(case):
    kind = case["kind"]
    if kind == "flat":
        n = case["n"]
        it = case["iters"]
        per = 2 * 2.5 * n * n * 2 * math.log2(n) + 20.0 * n * n
        return {"bytes": n * n * (8 + 8 + 1 + 8) + n * (n // 2 + 1) * 24, "flops": it * per}
    nside, lmax = case["nside"], case["lmax"]
    nc = case.get("ncomp", 1)
    npix, nalm = 12 * nside * nside, (lmax + 1) * (lmax + 2) // 2
    pol = nc == 3
    if kind in ("synth", "adjoint"):
        return {"bytes": nc * (8 * npix + 16 * nalm), "flops": _transform_work(nside, lmax, lmax, pol)}
    # a solve: its inputs and outputs once; two transforms an iteration, the output map
    k = case["iters"]
    nf = (k + 1) // 2
    levels = max(1, k - nf)
    band = [lmax] * nf + [min(lmax, 120 + int((lmax - 120) * i / levels)) if lmax > 120 else lmax for i in range(k - nf)]
    sw = case.get("sweeps", 0)
    f = sum(2 * _transform_work(nside, lmax, L, pol) for L in band) + (2 * sw + 1) * _transform_work(nside, lmax, lmax, pol)
    n_solves = 2 * case["maps"] if kind == "batch" else 1
    b = nc * (16 * npix + 16 * nalm) + (6 if pol else 1) * 8 * npix + npix
    return {"bytes": b * n_solves, "flops": f * n_solves}


# ---------------------------------------------------------------------------
# the same results in 64 bits from plain torch: the textbook three-term recurrences
# with a carried exponent, FFTs of the rings, Eqs. (3)-(4) as they stand
# ---------------------------------------------------------------------------
class _Sht:
    def __init__(self, nside, lmax):
        self.nside, self.lmax, self.np = nside, lmax, 2 * nside
        z, q, nr = _rings(nside)
        k = np.arange(1, 2 * nside + 1)
        # sin^2 theta without cancellation near the pole
        u = np.where(k < nside, k * k / (3.0 * nside * nside), 1.0 - z[: 2 * nside])
        self.x = torch.as_tensor(z[: 2 * nside].copy(), device=DEV)
        self.s2 = torch.as_tensor(u * (2.0 - u), device=DEV)
        self.q, self.nr = q[: 2 * nside], nr[: 2 * nside]
        self.off = (np.cumsum(nr) - nr)
        m = np.arange(lmax + 1)
        lg = np.array([0.5 * (math.log(2 * i + 1.0) - math.log(4 * math.pi) + math.lgamma(2 * i + 1.0)
                              - 2 * math.lgamma(i + 1.0) - 2 * i * math.log(2.0)) / math.log(2.0) for i in m])
        self.lgm = torch.as_tensor(lg, device=DEV)
        self.lgs = 0.5 * torch.log2(self.s2)
        self.m = torch.arange(lmax + 1, device=DEV, dtype=F8)

    def columns(self, L):
        """Yields (l, lambda_l of m = 0..l, lambda_{l-1}), each (l + 1) x ring pairs."""
        M, Pn = L + 1, self.np
        cur = torch.zeros(M, Pn, dtype=F8, device=DEV)
        prev = torch.zeros(M, Pn, dtype=F8, device=DEV)
        E = torch.zeros(M, Pn, dtype=torch.int32, device=DEV)
        m = self.m[:M]
        for l in range(L + 1):
            if l > 0:
                ml = m[:l]
                c1 = torch.sqrt((4.0 * l * l - 1.0) / (l * l - ml * ml))
                c0 = torch.sqrt(((l - 1.0) ** 2 - ml * ml).clamp(min=0.0) / (4.0 * (l - 1.0) ** 2 - 1.0)) if l > 1 else torch.zeros_like(ml)
                new = (cur[:l] * self.x - prev[:l] * c0[:, None]) * c1[:, None]
                prev[:l], cur[:l] = cur[:l], new
            lg = self.lgm[l] + l * self.lgs
            e = torch.ceil(lg / 512.0).clamp(max=0.0)
            cur[l] = torch.exp2(lg - 512.0 * e) * (-1.0 if l & 1 else 1.0)
            E[l] = e.to(torch.int32)
            if l % 8 == 0:
                up = (E[: l + 1] < 0) & (cur[: l + 1].abs() > 1.0)
                f = torch.where(up, torch.full_like(self.x[:1], 2.0 ** -512), torch.ones_like(self.x[:1]))
                cur[: l + 1] *= f
                prev[: l + 1] *= f
                E[: l + 1] += up.to(torch.int32)
            live = (E[: l + 1] == 0).to(F8)
            yield l, cur[: l + 1] * live, prev[: l + 1] * live

    def _spin(self, l, lam, lam1):
        """W = (2lambda + -2lambda) / 2 and X = (2lambda - -2lambda) / 2 at l >= 2."""
        m = self.m[: l + 1][:, None]
        N = 2.0 / math.sqrt((l + 2.0) * (l + 1.0) * l * (l - 1.0))
        R = torch.sqrt((2 * l + 1.0) / (2 * l - 1.0) * (l * l - m * m))
        W = N * (-((l - m * m) / self.s2 + 0.5 * l * (l - 1.0)) * lam + R * (self.x / self.s2) * lam1)
        X = N * (m / self.s2) * (-(l - 1.0) * self.x * lam + R * lam1)
        return W, X

    def grid(self, alm, L):
        """a_lm, m-major -> (L + 1) x (L + 1), [l, m]."""
        out = torch.zeros(L + 1, L + 1, dtype=C16, device=DEV)
        for m in range(L + 1):
            b = m * (2 * self.lmax + 3 - m) // 2
            out[m:, m] = alm[b: b + L + 1 - m]
        return out

    def pack(self, g, L):
        out = torch.zeros((self.lmax + 1) * (self.lmax + 2) // 2, dtype=C16, device=DEV)
        for m in range(L + 1):
            b = m * (2 * self.lmax + 3 - m) // 2
            out[b: b + L + 1 - m] = g[m:, m]
        return out

    def _caps(self):
        """Bluestein tables of all polar-cap ring lengths n = 4, 8, ... at once (one FFT length)."""
        n = torch.as_tensor(self.nr[: self.nside - 1].astype(np.int64), device=DEV)[:, None]
        N = 4 * (self.nside - 1)
        M = 1 << (2 * N - 1).bit_length()
        j = torch.arange(N, device=DEV)
        ang = ((j * j) % (2 * n)).to(F8) * (-math.pi) / n
        c = torch.polar((j < n).to(F8), ang)
        b = torch.zeros(len(n), M, dtype=C16, device=DEV)
        b[:, :N] = c.conj()
        b[:, M - N + 1:] += c[:, 1:].conj().flip(1)
        return n, N, M, c, torch.fft.fft(b)

    def _cap_dft(self, v, tab):
        """Forward DFT of every cap ring of its own length (v: pair, hemisphere, N; zero beyond n)."""
        n, N, M, c, B = tab
        return torch.stack([c * torch.fft.ifft(torch.fft.fft(v[:, h] * c, n=M) * B)[:, :N] for h in range(2)], 1)

    def _phase(self, ps, n, M, sign):
        md = torch.arange(M, device=DEV, dtype=F8)
        q = torch.as_tensor(self.q[ps].astype(np.float64), device=DEV)[:, None]
        return torch.exp(1j * (sign * math.pi / n * q * md))[:, None, :]  # pair, 1, m

    def _pieces(self):
        """(ring pairs, ring length) of the caps (None: each its own) and of the belt."""
        ns = self.nside
        return ([(np.arange(ns - 1), None)] if ns > 1 else []) + [(np.arange(ns - 1, 2 * ns), 4 * ns)]

    def _pixel_index(self, ps, N):
        """Pixel of (pair, hemisphere, j), and whether it exists."""
        R = 4 * self.nside - 1
        off = torch.as_tensor(np.stack([self.off[ps], self.off[R - 1 - ps]], 1), device=DEV)
        n = torch.as_tensor(self.nr[ps].astype(np.int64), device=DEV)[:, None, None]
        j = torch.arange(N, device=DEV)
        ok = (j < n).expand(len(ps), 2, N).clone()
        eq = torch.as_tensor(ps == 2 * self.nside - 1, device=DEV)
        ok[:, 1] &= ~eq[:, None]
        return (off[:, :, None] + j), ok

    def rings_out(self, G):
        """G: (m, pair, hemisphere) -> map."""
        M = G.shape[0]
        out = torch.empty(12 * self.nside ** 2, dtype=F8, device=DEV)
        mm = torch.arange(M, device=DEV)
        for ps, n in self._pieces():
            tab = self._caps() if n is None else None
            N = tab[1] if tab else n
            g = G[:, ps[0]: ps[-1] + 1].permute(1, 2, 0)
            ph = self._phase(ps, tab[0].to(F8) if tab else n, M, 1.0)
            g = g * ph
            nl = tab[0] if tab else torch.full((len(ps), 1), n, device=DEV)
            row = torch.arange(len(ps) * 2, device=DEV).reshape(len(ps), 2, 1) * N
            H = torch.zeros(len(ps) * 2 * N, 2, dtype=F8, device=DEV)
            H.index_add_(0, (row + (mm % nl)[:, None]).reshape(-1), torch.view_as_real(g.contiguous()).reshape(-1, 2))
            gc = g[..., 1:].conj().resolve_conj()
            H.index_add_(0, (row + ((-mm[1:]) % nl)[:, None]).reshape(-1),
                         torch.view_as_real(gc.contiguous()).reshape(-1, 2))
            H = torch.view_as_complex(H).reshape(len(ps), 2, N)
            f = self._cap_dft(H.conj().resolve_conj(), tab).real if tab else torch.fft.ifft(H).real * n
            idx, ok = self._pixel_index(ps, N)
            out[idx[ok]] = f[ok]
        return out

    def rings_in(self, f, M):
        """map -> F: (m, pair, hemisphere)."""
        F = torch.zeros(M, self.np, 2, dtype=C16, device=DEV)
        mm = torch.arange(M, device=DEV)
        for ps, n in self._pieces():
            tab = self._caps() if n is None else None
            N = tab[1] if tab else n
            idx, ok = self._pixel_index(ps, N)
            v = torch.where(ok, f[torch.where(ok, idx, torch.zeros_like(idx))], torch.zeros(1, dtype=F8, device=DEV)).to(C16)
            V = self._cap_dft(v, tab) if tab else torch.fft.fft(v)
            nl = tab[0] if tab else torch.full((len(ps), 1), n, device=DEV)
            V = torch.gather(V, 2, (mm % nl)[:, None].expand(len(ps), 2, M))
            F[:, ps[0]: ps[-1] + 1] = (V * self._phase(ps, tab[0].to(F8) if tab else n, M, -1.0)).permute(2, 0, 1)
        return F

    def synth(self, alms, L):
        """[T] or [T, E, B] (m-major) -> maps."""
        gs = [self.grid(a, L) for a in alms]
        G = [torch.zeros(2, 2, L + 1, self.np, dtype=F8, device=DEV) for _ in alms]  # hemisphere, re/im
        for l, lam, lam1 in self.columns(L):
            k = l + 1
            sg = (1.0 - 2.0 * ((l + self.m[:k]) % 2))
            a = gs[0][l, :k]
            for h in range(2):
                s = sg if h else torch.ones_like(sg)
                G[0][h, 0, :k].addcmul_(lam, (s * a.real)[:, None].expand_as(lam))
                G[0][h, 1, :k].addcmul_(lam, (s * a.imag)[:, None].expand_as(lam))
            if len(alms) == 3 and l >= 2:
                W, X = self._spin(l, lam, lam1)
                e, b = gs[1][l, :k], gs[2][l, :k]
                for h in range(2):
                    w = W * sg[:, None] if h else W
                    x = -X * sg[:, None] if h else X
                    # Q_m = -sum (E W + i B X),  U_m = -sum (B W - i E X)
                    G[1][h, 0, :k] -= e.real[:, None] * w - b.imag[:, None] * x
                    G[1][h, 1, :k] -= e.imag[:, None] * w + b.real[:, None] * x
                    G[2][h, 0, :k] -= b.real[:, None] * w + e.imag[:, None] * x
                    G[2][h, 1, :k] -= b.imag[:, None] * w - e.real[:, None] * x
        return [self.rings_out(torch.complex(g[:, 0], g[:, 1]).permute(1, 2, 0)) for g in G]

    def adjoint(self, maps, L):
        """maps -> Y^T map, [T] or [T, E, B], m-major."""
        Fs = [self.rings_in(f, L + 1) for f in maps]
        out = [torch.zeros(L + 1, L + 1, dtype=C16, device=DEV) for _ in maps]
        N = [(F[..., 0].real.contiguous(), F[..., 0].imag.contiguous()) for F in Fs]
        S = [(F[..., 1].real.contiguous(), F[..., 1].imag.contiguous()) for F in Fs]
        for l, lam, lam1 in self.columns(L):
            k = l + 1
            sg = (1.0 - 2.0 * ((l + self.m[:k]) % 2))[:, None]
            f = [(n[0][:k] + sg * s[0][:k], n[1][:k] + sg * s[1][:k]) for n, s in zip(N, S)]
            out[0][l, :k] = torch.complex((lam * f[0][0]).sum(1), (lam * f[0][1]).sum(1))
            if len(maps) == 3 and l >= 2:
                W, X = self._spin(l, lam, lam1)
                d = [(n[0][:k] - sg * s[0][:k], n[1][:k] - sg * s[1][:k]) for n, s in zip(N, S)]
                # E = -sum (W Q_m + i X U_m),  B = -sum (W U_m - i X Q_m) over both hemispheres
                out[1][l, :k] = -torch.complex((W * f[1][0] - X * d[2][1]).sum(1), (W * f[1][1] + X * d[2][0]).sum(1))
                out[2][l, :k] = -torch.complex((W * f[2][0] + X * d[1][1]).sum(1), (W * f[2][1] - X * d[1][0]).sum(1))
        return [self.pack(o, L) for o in out]


def _cost(case):
    """Seconds that exact() takes, about."""
    nside, lmax = case["nside"], case["lmax"]
    pol = case.get("ncomp", 1) == 3
    one = (lmax * (60e-6 if not pol else 300e-6) + nside * 400e-6 * (3 if pol else 1)
           + nside * float(lmax) ** 2 * (2.5e-11 if not pol else 1.5e-10))
    if case["kind"] in ("synth", "adjoint"):
        return one
    return one * (1.6 * case["iters"] + 2 + 2 * case.get("sweeps", 0)) * 2 * case.get("maps", 0.5)


def _inv3(a, b, c, d, e, f):
    """Inverse of the symmetric [[a, d, e], [d, b, f], [e, f, c]], n x 3 x 3."""
    A, B, C = b * c - f * f, a * c - e * e, a * b - d * d
    D, E, F = e * f - d * c, d * f - e * b, d * e - a * f
    det = a * A + d * D + e * E
    rows = [torch.stack(r, -1) for r in ((A, D, E), (D, B, F), (E, F, C))]
    return torch.stack(rows, -2) / det[:, None, None]


def _eig_min(N6, mask):
    a, b, c, d, e, f = (N6[:, mask > 0]).cpu().numpy()
    N = np.stack([np.stack([a, d, e], -1), np.stack([d, b, f], -1), np.stack([e, f, c], -1)], -2)
    return float(np.linalg.eigvalsh(N).min())


def _exact_solve(case, P, q, fluct=False):
    nside, lmax, nc = case["nside"], case["lmax"], case.get("ncomp", 1)
    sht = _Sht(nside, lmax)
    npix = 12 * nside * nside
    om = 4.0 * math.pi / npix
    l, _ = _alm_index(lmax)
    obs = (P["mask"] > 0).to(F8)
    sched = P["schedule"] + [(1.0, lmax)] * case.get("sweeps", 0)
    if nc == 1:
        S = P["cl"][l]
        nu = obs / P["noise"]
        tau = float(P["noise"][P["mask"] > 0].min())
        if fluct:
            h = torch.where(S > 0, q["g2"] / torch.where(S > 0, S, 1.0).sqrt(), torch.zeros_like(q["g2"]))
            r = nu.sqrt() * q["g1"] + om * sht.synth([h], lmax)[0]
        else:
            r = nu * q["d"]
        a = torch.zeros(l.numel(), dtype=C16, device=DEV)
        for lam, L in sched:
            s = sht.synth([a], L)[0]
            t = s + lam * tau * (r - nu * s) / (1.0 + (lam - 1.0) * tau * nu)
            a = S / (S + lam * tau * om) * om * sht.adjoint([t], L)[0]
        return sht.synth([a], lmax)[0], a
    nu = _inv3(*P["noise"]) * obs[:, None, None]
    tau = _eig_min(P["noise"], P["mask"])
    r = torch.einsum("nij,jn->in", nu, q["d"])
    tt, ee, te = P["cl"][0][l], P["cl"][1][l], P["cl"][3][l]
    a = [torch.zeros(l.numel(), dtype=C16, device=DEV) for _ in range(3)]
    eye = torch.eye(3, dtype=F8, device=DEV)
    for lam, L in sched:
        s = torch.stack(sht.synth(a, L))
        A = eye + (lam - 1.0) * tau * nu
        Ai = _inv3(A[:, 0, 0], A[:, 1, 1], A[:, 2, 2], A[:, 0, 1], A[:, 0, 2], A[:, 1, 2])
        rhs = r - torch.einsum("nij,jn->in", nu, s)
        t = s + lam * tau * torch.einsum("nij,jn->in", Ai, rhs)
        b = [om * v for v in sht.adjoint(list(t), L)]
        th = lam * tau * om
        det = (tt + th) * (ee + th) - te * te  # S (S + th)^-1 of the TE block
        a = [((tt * (ee + th) - te * te) * b[0] + te * th * b[1]) / det,
             (te * th * b[0] + (ee * (tt + th) - te * te) * b[1]) / det, torch.zeros_like(b[2])]
    return torch.cat(sht.synth(a, lmax)), torch.cat(a)


def exact(case, seed):
    kind = case["kind"]
    if kind == "flat":
        P = _flat_problem(case, seed)
        nu = (P["mask"] > 0).to(F8) / P["noise"]
        tau = float(P["noise"][P["mask"] > 0].min())
        r, S = nu * P["d"], P["S"]
        n = case["n"]
        a = torch.zeros(n, n // 2 + 1, dtype=C16, device=DEV)
        for lam in P["lam"]:
            s = torch.fft.irfft2(a, s=(n, n), norm="ortho")
            t = s + lam * tau * (r - nu * s) / (1.0 + (lam - 1.0) * tau * nu)
            a = S / (S + lam * tau) * torch.fft.rfft2(t, norm="ortho")
        return {"map": torch.fft.irfft2(a, s=(n, n), norm="ortho"), "alm": a}
    if _cost(case) > 20.0:
        return None
    if kind in ("synth", "adjoint"):
        v = _transform_input(case, seed).reshape(case["ncomp"], -1)
        sht = _Sht(case["nside"], case["lmax"])
        if kind == "synth":
            return {"map": torch.cat(sht.synth(list(v), case["lmax"]))}
        return {"alm": torch.cat(sht.adjoint(list(v), case["lmax"]))}
    P = _problem(case, seed)
    if kind == "solve":
        s, a = _exact_solve(case, P, P["maps"][0])
        return {"map": s, "alm": a}
    res = [_exact_solve(case, P, q, fluct=f) for q in P["maps"] for f in (False, True)]
    return {"map": [x[0] for x in res], "alm": [x[1] for x in res]}
