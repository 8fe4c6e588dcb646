"""What a user of this package has it do, as timed passes through its public entry points.

The listed cases follow the repository's own workloads (Nside 64 / lmax 128 / order 3 / T, Nside 512 /
lmax 1024 / order 4 / TQU, Nside 1024 / lmax 2048 for gradients, uneven batches of up to Nside 2048 /
lmax 3000); `draw` spreads over the same ranges. `exact` is a double-precision restatement of each
operation in plain torch: the three-term recurrence in l with its theta-derivatives by Leibniz's
rule, one FFT per ring length, the geodesic displacement, ang2pix and the Taylor sum.
"""
from __future__ import annotations

import math

import torch

from paper_1307_0719_gb300 import api

ARCMIN = math.pi / (180.0 * 60.0)
PRECISIONS = {"fp64": api.FP64, "fp32": api.MIXED_FP32, "tf32x3": api.MIXED_TF32x3, "bf16x3": api.MIXED_BF16x3}


# --------------------------------------------------------------------------- the cases

def _case(name, op, nside, lmax, order, pol, precision, nreal=1, lmax_phi=0, geoms=""):
    return {"name": name, "op": op, "nside": nside, "lmax": lmax, "order": order, "pol": pol, "precision": precision,
            "nreal": nreal, "lmax_phi": lmax_phi, "geoms": geoms}


def listed():
    return [
        # a quick look at one small temperature sky in double precision: launches and latency
        _case("lens_nside64_T_fp64", "lens", 64, 128, 3, False, "fp64"),
        # three small skies with an odd band limit in one call (patches, unit tests of a user's pipeline)
        _case("batch3_nside32_odd", "batch", 32, 75, 3, True, "bf16x3", nreal=3),
        # one polarised sky, interactively: one realisation in the default precision form
        _case("lens_nside512", "lens", 512, 1024, 4, True, "bf16x3"),
        # the same sky in double precision, the form that others are checked against
        _case("lens_nside512_fp64", "lens", 512, 1024, 4, True, "fp64"),
        # the potential taken to the paper's band limit of 8 Nside, above the fields' own
        _case("lens_nside512_phi8", "lens", 512, 1024, 4, True, "fp32", lmax_phi=4096),
        # Monte Carlo production at moderate resolution: sixteen skies a call
        _case("batch16_nside512", "batch", 512, 1024, 4, True, "bf16x3", nreal=16),
        # Monte Carlo production at full resolution, where most GPU hours go
        _case("batch16_nside2048", "batch", 2048, 3000, 4, True, "bf16x3", nreal=16),
        # skies in pinned host memory, maps back to it
        _case("host8_nside512", "host", 512, 1024, 4, True, "bf16x3", nreal=8),
        # an uneven set of skies as one replayed graph
        _case("uneven12_graph", "uneven", 1024, 2048, 4, True, "bf16x3", nreal=12,
              geoms="256x512,512x1024,512x1024,1024x2048,256x512,512x1024,1024x2048,256x512,512x1024,256x512,"
                    "512x1024,1024x2048"),
        # one step of a map-level fit: the lensed maps and the gradients of a misfit
        _case("fit_nside1024", "fit", 1024, 2048, 4, True, "fp32"),
        # derivative maps of the polarisation, for a user's own expansion
        _case("derivs_nside1024_spin2", "derivs", 1024, 2048, 4, True, "fp32"),
        # harmonic coefficients of lensed maps, for their spectra
        _case("map2alm_nside1024", "map2alm", 1024, 2048, 4, True, "fp32"),
    ]


def _log_uniform(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _cost(c):
    """Legendre work of a case in units of (ring, l, m) steps, weighted by precision and fields."""
    if c["op"] == "uneven":
        g = [tuple(map(int, s.split("x"))) for s in c["geoms"].split(",")]
        return sum(n * l * l for n, l in set(g)) * 16.0 + sum(n * l * l for n, l in g) * 6.0
    w = c["nside"] * c["lmax"] ** 2 * (c["order"] + 2.0) * (3.0 if c["pol"] else 1.0)
    w += c["nside"] * c["lmax_phi"] ** 2 * 3.0
    w *= {"fp64": 40.0, "fp32": 1.0, "tf32x3": 1.5, "bf16x3": 1.0}[c["precision"]]
    return w * {"batch": 0.7 + 0.1 * c["nreal"], "host": 0.7 + 0.3 * c["nreal"], "fit": 4.0}.get(c["op"], 1.0)


def draw(rng):
    """One more case of the listed ranges: any operation, Nside 16 to 2048, band limits of 0.5 to 3 Nside,
    orders 3 to 6 where maps are lensed in single precision (below that the series itself jumps by more
    than rounding from cell to cell) and 1 to 6 otherwise."""
    most = 0.9 * max(_cost(c) for c in listed() if c["op"] == "batch")
    while True:
        op = rng.choice(["lens", "lens", "batch", "batch", "host", "uneven", "fit", "derivs", "map2alm"])
        top = {"lens": 11, "batch": 11, "host": 10, "uneven": 10, "fit": 10, "derivs": 11, "map2alm": 11}[op]
        nside = 2 ** rng.randint(4, top)
        lmax = _log_uniform(rng, max(6, nside // 2), 3 * nside)
        pol = rng.random() < 0.75
        precision = "bf16x3" if op in ("batch", "host", "uneven") else rng.choice(["fp32", "bf16x3", "fp64"])
        if op in ("derivs", "map2alm", "fit") and precision == "bf16x3":
            precision = "fp32"
        if op in ("batch", "lens") and precision == "bf16x3" and rng.random() < 0.2:
            precision = "tf32x3"
        if precision == "fp64" and nside > 512:
            continue
        order = rng.randint(1 if op in ("derivs",) else 3, 6)
        if op == "fit":
            order = rng.randint(3, 5)
        nreal = {"batch": rng.randint(1, 20), "host": rng.randint(2, 10), "uneven": rng.randint(4, 12)}.get(op, 1)
        lmax_phi = 0
        if op == "lens" and precision != "tf32x3" and nside <= 512 and rng.random() < 0.3:
            lmax_phi = _log_uniform(rng, lmax, 8 * nside)
            lmax_phi = 0 if lmax_phi == lmax else lmax_phi
        geoms = ""
        if op == "uneven":
            sizes = [(n, _log_uniform(rng, n, 3 * n)) for n in sorted({2 ** rng.randint(4, 10) for _ in range(3)})]
            geoms = ",".join("%dx%d" % rng.choice(sizes) for _ in range(nreal))
            g = [tuple(map(int, s.split("x"))) for s in geoms.split(",")]
            nside, lmax = max(g)
        c = _case("", op, nside, lmax, order, pol, precision, nreal, lmax_phi, geoms)
        del c["name"]
        # a state (plan and maps) fits the card three times over
        planes = (3 if pol else 1) * (order + 1) + 2
        state = 4.0 * nside * lmax * 8 * planes * (16 if precision in ("bf16x3", "tf32x3") else 1)
        state += 12.0 * nside * nside * 4 * ((3 if pol else 1) * ((order + 1) * (order + 2) / 2 + nreal) + 3)
        if op == "fit":
            state += 12.0 * nside * nside * 4 * 3 * (order + 1) * (order + 2) / 2
        if _cost(c) <= most and state < 6.5e10:
            return c


# --------------------------------------------------------------------------- inputs

def _nalm(lmax):
    return (lmax + 1) * (lmax + 2) // 2


def _lm(lmax):
    """(l, m) of every coefficient in storage order, idx = m (2 lmax + 1 - m) / 2 + l."""
    m = torch.repeat_interleave(torch.arange(lmax + 1, device="cuda"), torch.arange(lmax + 1, 0, -1, device="cuda"))
    idx = torch.arange(_nalm(lmax), device="cuda")
    return idx - m * (2 * lmax + 1 - m) // 2, m


def _alm(cl, lm, gen):
    """Gaussian coefficients of a real field with spectrum cl."""
    l, m = lm
    x = torch.randn((l.numel(), 2), dtype=torch.float64, device="cuda", generator=gen)
    x *= torch.sqrt(0.5 * cl[l])[:, None]
    x[:, 0] *= 1.0 + (math.sqrt(2.0) - 1.0) * (m == 0).to(torch.float64)
    x[:, 1] *= (m > 0)
    return torch.view_as_complex(x)


def _spectra(nside, lmax, lmax_phi):
    """T, E, B and potential spectra: the repository's analytic ones, damped at 100 (Nside / 512)."""
    l = torch.arange(max(lmax, lmax_phi) + 1, dtype=torch.float64, device="cuda")
    damp = max(8.0, 100.0 * nside / 512)
    tt = 2e3 * math.pi / (l * (l + 1)).clamp(min=1.0) * torch.exp(-(l / damp) ** 2)
    tt[:2] = 0.0
    ee = 0.05 * tt * torch.exp(-(l / (8.0 * damp)) ** 2)
    pp = torch.where(l >= 1, (l + 1) ** -4.0, 0.0)
    p = pp[: lmax_phi + 1]
    lp = l[: lmax_phi + 1]
    pp = p * (2.5 * ARCMIN) ** 2 / ((2 * lp + 1) / (4 * math.pi) * lp * (lp + 1) * p).sum()
    return tt[: lmax + 1], ee[: lmax + 1], 0.3 * ee[: lmax + 1], pp


def _skies(case, seed):
    """The unlensed skies and potentials of a case: dicts T (E, B) and phi of complex128 CUDA tensors."""
    gen = torch.Generator(device="cuda")
    gen.manual_seed(int(seed))
    geoms = [tuple(map(int, s.split("x"))) for s in case["geoms"].split(",")] if case["geoms"] else \
        [(case["nside"], case["lmax"])] * case["nreal"]
    out, known = [], {}
    for nside, lmax in geoms:
        lp = case["lmax_phi"] or lmax
        if (nside, lmax) not in known:
            known[nside, lmax] = (_spectra(nside, lmax, lp), _lm(lmax), _lm(lp) if lp != lmax else None)
        (tt, ee, bb, pp), lm, lmp = known[nside, lmax]
        sky = {"T": _alm(tt, lm, gen)}
        if case["pol"]:
            sky["E"], sky["B"] = _alm(ee, lm, gen), _alm(bb, lm, gen)
        sky["phi"] = _alm(pp, lmp or lm, gen)
        out.append(sky)
    return geoms, out


def _maps(case, seed):
    """T, Q, U maps for the analysis and the fit: white noise over a few large-scale waves."""
    gen = torch.Generator(device="cuda")
    gen.manual_seed(int(seed) + 977)
    npix = 12 * case["nside"] ** 2
    n = 3 if case["pol"] else 1
    x = torch.randn((n, npix), dtype=torch.float64, device="cuda", generator=gen)
    t = torch.linspace(0.0, 1.0, npix, dtype=torch.float64, device="cuda")
    x += torch.sin(2 * math.pi * t * torch.arange(2, 2 + n, dtype=torch.float64, device="cuda")[:, None])
    return x.to(torch.float64 if case["precision"] == "fp64" else torch.float32)


def prepare(case, seed):
    op, pol, precision = case["op"], case["pol"], PRECISIONS[case["precision"]]
    s = {"op": op, "pol": pol}
    if op == "uneven":
        geoms, s["skies"] = _skies(case, seed)
        s["batch"] = api.Batch([g[0] for g in geoms], [g[1] for g in geoms], case["order"], pol=pol, precision=precision)
        s["outs"] = s["batch"].outputs()
        return s
    s["plan"] = plan = api.Plan(case["nside"], case["lmax"], case["order"], pol=pol, precision=precision,
                                lmax_phi=case["lmax_phi"] or None)
    if op == "map2alm":
        s["maps"] = list(_maps(case, seed).unbind(0))
        return s
    _, skies = _skies(case, seed)
    if op == "fit":
        # a fit keeps its parameters and its data in the plan's map precision
        single = case["precision"] != "fp64"
        s["params"] = [skies[0][k].to(torch.complex64 if single else torch.complex128).requires_grad_()
                       for k in (("T", "E", "B", "phi") if pol else ("T", "phi"))]
        s["data"] = _maps(case, seed)
    elif op == "derivs":
        a = torch.cat([skies[0]["E"], skies[0]["B"]]) if pol else skies[0]["T"]
        s["alm"], s["spin"] = a, 2 if pol else 0
    elif op == "host":
        s["skies"] = [{k: v.cpu().pin_memory() for k, v in sky.items()} for sky in skies]
        s["outs"] = [torch.empty((3 if pol else 1, plan.npix), dtype=plan.dtype, pin_memory=True) for _ in skies]
    else:
        s["skies"] = skies
        s["outs"] = [torch.empty((3 if pol else 1, plan.npix), dtype=plan.dtype, device="cuda") for _ in skies]
    return s


# --------------------------------------------------------------------------- the passes

def run(state):
    op = state["op"]
    if op == "lens":
        sky = state["skies"][0]
        return state["plan"].lens(sky["T"], sky.get("E"), sky.get("B"), sky["phi"], out=state["outs"][0])
    if op == "batch":
        return state["plan"].lens_batch(state["skies"], outs=state["outs"])
    if op == "host":
        return state["plan"].lens_batch_host(state["skies"], outs=state["outs"])
    if op == "uneven":
        return state["batch"].lens(state["skies"], state["outs"], mode="graph")
    if op == "derivs":
        return state["plan"].synth_derivs(state["alm"], state["spin"])
    if op == "map2alm":
        m = state["maps"]
        out = state["plan"].map2alm(m[0], *m[1:])
        # coefficients are kept in the maps' precision
        return {k: v.to(torch.complex64) if m[0].dtype == torch.float32 else v for k, v in out.items()}
    # fit: the lensed maps of the current parameters and the misfit's gradients
    params = state["params"]
    full = [p.to(torch.complex128) for p in params]
    if not state["pol"]:
        full = [full[0], None, None, full[1]]
    maps = api.LensFunction.apply(state["plan"], *full)
    loss = 0.5 * (maps - state["data"]).square().sum()
    return [maps.detach(), list(torch.autograd.grad(loss, params))]


def work(case):
    """Coefficients read and maps written once; flops of the recurrence (once per geometry), of the contraction,
    the ring FFTs and the Taylor sums. A third of the (ring, l, m) steps are evanescent and count nothing."""
    geoms = [tuple(map(int, s.split("x"))) for s in case["geoms"].split(",")] if case["geoms"] else \
        [(case["nside"], case["lmax"])] * case["nreal"]
    n, nf, op = case["order"], 3 if case["pol"] else 1, case["op"]
    el = 8 if case["precision"] == "fp64" else 4
    if op == "map2alm":
        n = 0
    K = (n + 1) * (n + 2) // 2
    fields = nf - 1 if op == "derivs" and case["pol"] else nf
    nbytes = flops = 0.0
    rec = sum(2 * j + 3 for j in range(n + 1))
    for i, (nside, lmax) in enumerate(geoms):
        npix, na, lp = 12 * nside * nside, _nalm(lmax), case["lmax_phi"] or lmax
        steps = 2 * nside * na * 2.0 / 3.0
        if geoms.index((nside, lmax)) == i:
            flops += steps * rec * (3 if case["pol"] else 1)
        flops += steps * 4 * (n + 1) * (1 + (4 if case["pol"] else 0)) + npix * fields * K * 2.5 * math.log2(4 * nside)
        if op == "derivs":
            nbytes += na * 16 * fields + npix * el * fields * K
        elif op == "map2alm":
            nbytes += na * (8 if el == 4 else 16) * nf + npix * el * nf
        else:
            flops += 2 * nside * _nalm(lp) * 2.0 / 3.0 * 16 + npix * nf * K * 2
            nbytes += (na * nf + _nalm(lp)) * 16 + npix * el * nf
            if op == "fit":
                nbytes += (na * nf + _nalm(lp)) * 8 + npix * el * nf
                flops += steps * 4 * (n + 1) * (1 + (4 if case["pol"] else 0)) + npix * nf * K * (2.5 * math.log2(4 * nside) + 6)
    return {"bytes": nbytes, "flops": flops}


# --------------------------------------------------------------------------- double-precision values

class _Rings:
    """The HEALPix RING grid, rings 0 .. 4 Nside - 2 from the north."""

    def __init__(self, nside):
        self.nside, self.npix, self.n = nside, 12 * nside * nside, 4 * nside - 1
        i = torch.arange(1, 4 * nside, dtype=torch.float64, device="cuda")
        inorth = torch.minimum(i, 4 * nside - i)
        cap = inorth < nside
        om = inorth ** 2 / (3.0 * nside ** 2)  # 1 - |z| in the caps
        z = torch.where(cap, 1 - om, (4.0 * nside - 2 * inorth) / (3.0 * nside))
        s = torch.where(cap, torch.sqrt(om * (2 - om)), torch.sqrt((1 - z) * (1 + z)))
        south = i > 2 * nside
        self.z, self.s = torch.where(south, -z, z), s
        self.theta = torch.atan2(self.s, self.z)
        self.ni = torch.minimum(inorth, torch.full_like(inorth, nside)).long()
        self.nphi = 4 * self.ni
        shifted = cap | (inorth.long() == nside) | (((inorth.long() - nside) & 1) == 0)
        self.phi0 = torch.where(shifted, math.pi / self.nphi.double(), 0.0)
        self.first = torch.cumsum(self.nphi, 0) - self.nphi
        # tan(theta/2), log2 sin(theta/2) and log2 cos(theta/2); the southern rings mirror the northern ones,
        # where 1 + cos(theta) does not cancel
        t = self.s / (1 + self.z.abs())
        self.t = torch.where(south, 1 / t, t)
        lc = 0.5 * torch.log2(0.5 * (1 + self.z.abs()))
        ls = torch.log2(t) + lc
        self.lsh, self.lch = torch.where(south, lc, ls), torch.where(south, ls, lc)

    def log_derivs(self, K):
        """d^k/dtheta^k of ln sin(theta/2) and ln cos(theta/2), k = 1 .. K."""
        def poly(p, x):
            r = torch.zeros_like(x)
            for c in reversed(p):
                r = r * x + c
            return r

        def step(p, sign):  # d/dtheta of p(x) with x' = sign (1 + x^2) / 2
            d = [k * c for k, c in enumerate(p)][1:] or [0.0]
            out = [0.0] * (len(d) + 2)
            for k, c in enumerate(d):
                out[k] += 0.5 * sign * c
                out[k + 2] += 0.5 * sign * c
            return out
        ps, pc, ls, lc = [0.0, 0.5], [0.0, -0.5], [], []
        for _ in range(K):
            ls.append(poly(ps, 1 / self.t))
            lc.append(poly(pc, self.t))
            ps, pc = step(ps, -1.0), step(pc, 1.0)
        return ls, lc


def _steps(g, lmax, nder, spin):
    """Yields (l, W) for l = spin .. lmax: W[ring, j, m] = d^j/dtheta^j of spin-weighted lambda_lm / L^j for
    m <= l, L = lmax + 1. Values carry a power of 2^400 until they are representable."""
    R, M, NJ, L = g.n, lmax + 1, nder + 1, lmax + 1.0
    f8 = dict(dtype=torch.float64, device="cuda")
    mm = torch.arange(M, **f8)
    E = torch.zeros((R, NJ, NJ), **f8)
    cyc = [g.z, -g.s, -g.z, g.s]  # cos^(i)(theta)
    for j in range(NJ):
        for i in range(j + 1):
            E[:, j, j - i] = math.comb(j, i) * cyc[i % 4] / L ** i
    ls, lc = g.log_derivs(nder)
    V, Vo, N = (torch.zeros((R, NJ, M), **f8) for _ in range(3))
    sc = torch.zeros((R, M), dtype=torch.int16, device="cuda")

    def seed(m):
        if m >= spin:
            lg = 0.5 * (math.log2((2 * m + 1) / (4 * math.pi)) +
                        (math.lgamma(2 * m + 1) - 2 * math.lgamma(m + 1)) / math.log(2.0))
            if spin:
                lg += 0.5 * math.log2(m * (m - 1) / ((m + 1) * (m + 2)))
            a, b = m + spin, m - spin
        else:
            lg = 0.5 * math.log2(5 / (4 * math.pi) * (6 if m == 0 else 4))
            a, b = 2 + m, 2 - m
        e = lg + a * g.lsh + b * g.lch
        s0 = torch.clamp(torch.ceil((e - 200.0) / 400.0), max=0.0)
        v = (-1.0) ** m * torch.exp2(e - 400.0 * s0)
        gk = [a * x + b * y for x, y in zip(ls, lc)]
        B = [torch.ones_like(v)]
        for j in range(nder):
            B.append(sum(math.comb(j, i) * gk[i] * B[j - i] for i in range(j + 1)))
        for j in range(NJ):
            V[:, j, m] = v * B[j] / L ** j
        Vo[:, :, m] = 0
        sc[:, m] = s0.to(torch.int16)

    def alpha(l, n):
        d = (l * l - mm[:n] ** 2).clamp(min=1e-300)
        return torch.where(mm[:n] < l, torch.sqrt((4.0 * l * l - 1) * l * l / (d * max(l * l - spin * spin, 1))), 0.0)

    for l in range(spin, lmax + 1):
        for m in (range(0, spin + 1) if l == spin else (l,)):
            seed(m)
        n = l + 1
        yield l, V[:, :, :n] * (sc[:, None, :n] == 0)
        if l == lmax:
            return
        a1, a0 = alpha(l + 1, n), alpha(l, n)
        if l == spin:
            a0 = torch.zeros_like(a0)
        beta = torch.where(a0 > 0, a1 / a0.clamp(min=1e-300), 0.0)
        new = torch.bmm(E, V[:, :, :n])
        if spin:
            new.addcmul_(V[:, :, :n], mm[:n] * spin / (l * (l + 1.0)))
        new *= a1
        new.addcmul_(Vo[:, :, :n], beta, value=-1.0)
        N[:, :, :n] = new
        V, Vo, N = N, V, Vo
        if l % 8 == 0:
            up = (sc[:, :n] < 0) & (V[:, 0, :n].abs() > 2.0 ** 200)
            f = torch.exp2(-400.0 * up.to(torch.float64))[:, None]
            V[:, :, :n] *= f
            Vo[:, :, :n] *= f
            sc[:, :n] += up.to(torch.int16)


def _dense(alm, lmax):
    """[l, m] real and imaginary parts of a coefficient vector; Im = 0 at m = 0."""
    l, m = _lm(lmax)
    out = torch.zeros((lmax + 1, lmax + 1), dtype=torch.complex128, device="cuda")
    out[l, m] = alm.to(torch.complex128)
    re, im = out.real.contiguous(), out.imag.contiguous()
    im[:, 0] = 0
    return re, im


def _analyse0(g, alms, lmax, nder):
    """Per field, the planes F[ring, j, m] of spin-0 coefficients."""
    M = lmax + 1
    co = [_dense(a, lmax) for a in alms]
    F = [[torch.zeros((g.n, nder + 1, M), dtype=torch.float64, device="cuda") for _ in range(2)] for _ in alms]
    for l, W in _steps(g, lmax, nder, 0):
        for (re, im), (fr, fi) in zip(co, F):
            fr[:, :, :l + 1].addcmul_(W, re[l, :l + 1])
            fi[:, :, :l + 1].addcmul_(W, im[l, :l + 1])
    return [torch.complex(fr, fi) for fr, fi in F]


def _analyse2(g, pairs, lmax, nder):
    """Per (E, B) pair, S1 = sum (E + iB) lambda and S2' = sum (-1)^(l+m) (E - iB) lambda (mirror rings)."""
    M = lmax + 1
    sg = 1.0 - 2.0 * (torch.arange(M, device="cuda") % 2).to(torch.float64)
    co = []
    for e, b in pairs:
        (er, ei), (br, bi) = _dense(e, lmax), _dense(b, lmax)
        co.append((er - bi, ei + br, er + bi, ei - br))
    S = [[torch.zeros((g.n, nder + 1, M), dtype=torch.float64, device="cuda") for _ in range(4)] for _ in pairs]
    for l, W in _steps(g, lmax, nder, 2):
        n = l + 1
        p = sg[:n] * (1.0 - 2.0 * (l % 2))
        for c, s in zip(co, S):
            s[0][:, :, :n].addcmul_(W, c[0][l, :n])
            s[1][:, :, :n].addcmul_(W, c[1][l, :n])
            s[2][:, :, :n].addcmul_(W, c[2][l, :n] * p)
            s[3][:, :, :n].addcmul_(W, c[3][l, :n] * p)
    return [(torch.complex(s[0], s[1]), torch.complex(s[2], s[3])) for s in S]


def _qu(S1, S2):
    """F^Q and F^U planes from S1 and the mirror rings' S2'."""
    j = torch.arange(S1.shape[1], device="cuda")
    S2 = torch.flip(S2, [0]) * (1.0 - 2.0 * (j % 2).to(torch.float64))[:, None]
    return -0.5 * (S1 + S2), 0.5j * (S1 - S2)


def _ring_maps(g, F, jks):
    """Maps d_theta^j d_phi^k / L^(j+k), [len(jks), npix], from the planes F[ring, j, m]."""
    M = F.shape[2]
    L = float(M)
    m = torch.arange(M, dtype=torch.float64, device="cuda")
    w = torch.where(m > 0, 2.0, 1.0).to(torch.float64)
    powers = [((1j * m) / L) ** k * w for k in range(max(k for _, k in jks) + 1)]
    parts, where = [], []
    for ni in range(1, g.nside + 1):
        rings = torch.nonzero(g.ni == ni).flatten()
        N = 4 * ni
        X = F[rings] * torch.exp(1j * g.phi0[rings, None] * m)[:, None, :]
        X = torch.stack([X[:, j] * powers[k] for j, k in jks])  # [maps, rings, m]
        pad = (-M) % N
        X = torch.nn.functional.pad(X, (0, pad)).reshape(len(jks), len(rings), -1, N).sum(2)
        parts.append((torch.fft.ifft(X, dim=-1).real * N).reshape(len(jks), -1))
        where.append((g.first[rings, None] + torch.arange(N, device="cuda")).flatten())
    out = torch.cat(parts, 1)
    inv = torch.empty(g.npix, dtype=torch.int64, device="cuda")
    inv[torch.cat(where)] = torch.arange(g.npix, device="cuda")
    return out[:, inv]


def _jks(order):
    return [(j, n - j) for n in range(order + 1) for j in range(n + 1)]


def _ang2pix(g, z, omz, phi):
    """(ring, index in ring) of the pixels holding the points; omz = 1 - |z|."""
    N = g.nside
    tt = torch.remainder(phi / (0.5 * math.pi), 4.0)
    belt = z.abs() <= 2.0 / 3.0
    t1, t2 = N * (0.5 + tt), 0.75 * N * z
    jp, jm = torch.floor(t1 - t2).long(), torch.floor(t1 + t2).long()
    ir = N + 1 + jp - jm
    kshift = 1 - (ir & 1)
    ip = torch.remainder(torch.div(jp + jm - N + kshift + 1, 2, rounding_mode="floor"), 4 * N)
    tp = tt - torch.floor(tt)
    tmp = N * torch.sqrt(3.0 * omz)
    jp, jm = torch.floor(tp * tmp).long(), torch.floor((1.0 - tp) * tmp).long()
    irc = jp + jm + 1
    ipc = torch.remainder(torch.floor(tt * irc).long(), 4 * irc)
    ring = torch.where(belt, ir + N - 2, torch.where(z > 0, irc - 1, g.n - irc))
    return ring, torch.where(belt, ip, ipc)


def _lensed(g, order, lmax, D, alpha, pol, keep=None):
    """The lensed maps from the derivative planes D (per field [K, npix], / (j! k! L^(j+k))) and alpha; `keep`
    holds the expansion pixels fixed where gradients are taken."""
    L = lmax + 1.0
    pix = torch.repeat_interleave(torch.arange(g.n, device="cuda"), g.nphi)
    idx = torch.arange(g.npix, device="cuda") - g.first[pix]
    phi = g.phi0[pix] + 2 * math.pi * idx.double() / g.nphi[pix]
    z, s = g.z[pix], g.s[pix]
    at, ap = alpha[0], alpha[1]
    d2 = (at * at + ap * ap).clamp(min=1e-60)
    d = torch.sqrt(d2)
    sinc, h = torch.sin(d) / d, 2 * torch.sin(0.5 * d) ** 2 / d2
    cosd = 1 - d2 * h
    X, Y, Z = s * cosd + z * at * sinc, ap * sinc, z * cosd - s * at * sinc
    rho = torch.sqrt(X * X + Y * Y)
    th, dphi = torch.atan2(rho, Z), torch.atan2(Y, X)
    with torch.no_grad():
        ring, iq = _ang2pix(g, Z, rho * rho / (1 + Z.abs()), phi + dphi)
        q = g.first[ring] + iq
        phq = g.phi0[ring] + 2 * math.pi * iq.double() / g.nphi[ring]
        wrap = torch.round((phi + dphi - phq) / (2 * math.pi)) * 2 * math.pi
    x, y = L * (th - g.theta[ring]), L * (phi + dphi - phq - wrap)
    vals = []
    for M in D:
        v = 0.0
        for k, (j, n) in enumerate(_jks(order)):
            v = v + x ** j * y ** n * M[k][q]
        vals.append(v)
    if pol:
        ct = 1 - at * at * h
        tx, ty, tz = ct * z - at * sinc * s, -ap * at * h, -ct * s - at * sinc * z
        cb, sb = Z * (tx * X + ty * Y) / rho - tz * rho, (ty * X - tx * Y) / rho
        n2 = cb * cb + sb * sb
        c2, s2 = (cb * cb - sb * sb) / n2, 2 * cb * sb / n2
        vals = [vals[0], c2 * vals[1] + s2 * vals[2], -s2 * vals[1] + c2 * vals[2]]
    return torch.stack(vals)


def _scaled(g, F, order):
    D = _ring_maps(g, F, _jks(order))
    f = torch.tensor([1.0 / (math.factorial(j) * math.factorial(k)) for j, k in _jks(order)], dtype=torch.float64,
                     device="cuda")
    return D * f[:, None]


def _alpha(g, FP):
    """The deflection from the potential's planes (j <= 1)."""
    L = float(FP.shape[2])
    a = _ring_maps(g, FP, [(1, 0), (0, 1)]) * L
    return torch.stack([a[0], a[1] / torch.repeat_interleave(g.s, g.nphi)])


def _exact_lens(nside, lmax, order, pol, skies, lmax_phi):
    g = _Rings(nside)
    FT = _analyse0(g, [s["T"] for s in skies], lmax, order)
    FP = _analyse0(g, [s["phi"] for s in skies], lmax_phi, 1)
    S = _analyse2(g, [(s["E"], s["B"]) for s in skies], lmax, order) if pol else [None] * len(skies)
    out = []
    for t, p, s in zip(FT, FP, S):
        D = [_scaled(g, f, order) for f in ([t, *_qu(*s)] if pol else [t])]
        out.append(_lensed(g, order, lmax, D, _alpha(g, p), pol))
    return out


def _exact_fit(case, seed):
    g, lmax, order, pol = _Rings(case["nside"]), case["lmax"], case["order"], case["pol"]
    _, skies = _skies(case, seed)
    single = case["precision"] != "fp64"
    sky = {k: v.to(torch.complex64).to(torch.complex128) if single else v for k, v in skies[0].items()}
    leaves = [_analyse0(g, [sky["T"]], lmax, order)[0]]
    if pol:
        leaves += list(_analyse2(g, [(sky["E"], sky["B"])], lmax, order)[0])
    leaves.append(_analyse0(g, [sky["phi"]], lmax, 1)[0])
    for f in leaves:
        f.requires_grad_()
    fields = [leaves[0], *(_qu(leaves[1], leaves[2]) if pol else ())]
    maps = _lensed(g, order, lmax, [_scaled(g, f, order) for f in fields], _alpha(g, leaves[-1]), pol)
    loss = 0.5 * (maps - _maps(case, seed).double()).square().sum()
    G = torch.autograd.grad(loss, leaves)
    maps = maps.detach()
    del loss, leaves, fields
    l, m = _lm(lmax)

    def flat(re, im):
        im = im.clone()
        im[:, 0] = 0
        return torch.complex(re[l, m], im[l, m])

    def back0(F, nder):
        out = torch.zeros((2, lmax + 1, lmax + 1), dtype=torch.float64, device="cuda")
        fr, fi = F.real.contiguous(), F.imag.contiguous()
        for ll, W in _steps(g, lmax, nder, 0):
            out[0, ll, :ll + 1] = torch.einsum("rjm,rjm->m", W, fr[:, :, :ll + 1])
            out[1, ll, :ll + 1] = torch.einsum("rjm,rjm->m", W, fi[:, :, :ll + 1])
        return flat(out[0], out[1])
    grads = [back0(G[0], order)]
    if pol:
        E, B = (torch.zeros((lmax + 1, lmax + 1), dtype=torch.complex128, device="cuda") for _ in range(2))
        parts = [G[1].real.contiguous(), G[1].imag.contiguous(), G[2].real.contiguous(), G[2].imag.contiguous()]
        sg = 1.0 - 2.0 * (torch.arange(lmax + 1, device="cuda") % 2).to(torch.float64)
        for ll, W in _steps(g, lmax, order, 2):
            v = [torch.einsum("rjm,rjm->m", W, x[:, :, :ll + 1]) for x in parts]
            s1 = torch.complex(v[0], v[1])
            s2 = torch.complex(v[2], v[3]) * sg[:ll + 1] * (1.0 - 2.0 * (ll % 2))
            E[ll, :ll + 1] = s1 + s2
            B[ll, :ll + 1] = -1j * (s1 - s2)
        grads += [flat(E.real.contiguous(), E.imag.contiguous()), flat(B.real.contiguous(), B.imag.contiguous())]
    grads.append(back0(G[-1], 1))
    return [maps, grads]


def _exact_map2alm(case, seed):
    g, lmax, pol = _Rings(case["nside"]), case["lmax"], case["pol"]
    maps = _maps(case, seed).double()
    M = lmax + 1
    m = torch.arange(M, device="cuda")
    X = torch.zeros((len(maps), g.n, M), dtype=torch.complex128, device="cuda")
    for ni in range(1, g.nside + 1):
        rings = torch.nonzero(g.ni == ni).flatten()
        N = 4 * ni
        p = g.first[rings, None] + torch.arange(N, device="cuda")
        f = torch.fft.fft(maps[:, p].to(torch.complex128), dim=-1)[:, :, m % N]
        X[:, rings] = f * torch.exp(-1j * g.phi0[rings, None] * m.double())
    w = 4 * math.pi / g.npix
    l, mi = _lm(lmax)

    def back(spin, field):
        out = torch.zeros((2, M, M), dtype=torch.float64, device="cuda")
        fr, fi = field.real.contiguous(), field.imag.contiguous()
        for ll, W in _steps(g, lmax, 0, spin):
            out[0, ll, :ll + 1] = (W[:, 0] * fr[:, :ll + 1]).sum(0)
            out[1, ll, :ll + 1] = (W[:, 0] * fi[:, :ll + 1]).sum(0)
        return torch.complex(out[0], out[1]) * w

    def flat(a):
        a = a.clone()
        a[:, 0] = a[:, 0].real.to(torch.complex128)
        return a[l, mi]
    out = {"T": flat(back(0, X[0]))}
    if pol:
        sg = (1.0 - 2.0 * ((l + mi) % 2).to(torch.float64))
        a2 = back(2, X[1] + 1j * X[2])
        am = back(2, torch.flip(X[1] - 1j * X[2], [0]))
        am[l, mi] *= sg
        out["E"], out["B"] = flat(-0.5 * (a2 + am)), flat(0.5j * (a2 - am))
    return out


def exact(case, seed):
    """What run() returns, in double precision. Of a batch, the first and the last sky; None above Nside 1024 and
    for band limits where the recurrence over every ring takes too long."""
    op, nside, lmax, order, pol = case["op"], case["nside"], case["lmax"], case["order"], case["pol"]
    lp = case["lmax_phi"] or lmax
    if nside > 1024 or 4.0 * nside * (lmax ** 2 * (order + 1) * (3 if pol else 1) + 2 * lp ** 2) > 6e11:
        return None
    with torch.no_grad():
        if op in ("lens", "batch", "host"):
            _, skies = _skies(case, seed)
            n = len(skies)
            pick = sorted({0, n - 1})
            got = dict(zip(pick, _exact_lens(nside, lmax, order, pol, [skies[i] for i in pick], lp)))
            return got[0] if op == "lens" else [got.get(i) for i in range(n)]
        if op == "uneven":
            geoms, skies = _skies(case, seed)
            out = [None] * len(skies)
            for i in {geoms.index(x): None for x in geoms}:
                out[i] = _exact_lens(*geoms[i], order, pol, [skies[i]], geoms[i][1])[0]
            return out
        if op == "derivs":
            _, skies = _skies(case, seed)
            g = _Rings(nside)
            L = torch.tensor([(lmax + 1.0) ** (j + k) for j, k in _jks(order)], dtype=torch.float64, device="cuda")
            if pol:
                F = _qu(*_analyse2(g, [(skies[0]["E"], skies[0]["B"])], lmax, order)[0])
            else:
                F = _analyse0(g, [skies[0]["T"]], lmax, order)
            return torch.cat([_ring_maps(g, f, _jks(order)) * L[:, None] for f in F])
        if op == "map2alm":
            return _exact_map2alm(case, seed)
    return _exact_fit(case, seed)
