"""Performance cases of the measurement operator: what a user of this package
has it do, through `Plan`, the differentiable operator and the kernel
evaluation, over image sizes, visibility counts, supports, precisions, kernel
modes and options.

    listed()            the fixed cases
    draw(rng)           one more case of the same ranges
    prepare(case, seed) what a user's program holds before the call
    run(state)          one pass and its outputs
    work(case)          bytes and operations a pass cannot do without
    exact(case, seed)   the outputs in 64 bits, from plain torch

Observations are synthetic: Earth-rotation tracks of a random 128-antenna
array (the MWA-like snapshot's recipe, the array scaled so that its baselines
fill the grid of the image size as they do there) or, for the smallest
images, baselines uniform in a disk.
"""
import math

import numpy as np
import torch

import paper_1903_06555_gb300 as phi
from paper_1903_06555_gb300 import autograd

SUPPORT = 4          # J, the default taper
OVERSAMPLE = 2.0


def _case(name, op, **kw):
    c = dict(name=name, op=op, mode="quadrature", precision="f32", image_n=2048, fov_deg=25.0,
             n_vis=1950720, n_stacks=8, conj_fold=1, wmax=500.0, tracks=1, rule="stack",
             weighted=0, deterministic=0, staging=0, tol=1e-6, dde_taps=0)
    c.update(kw)
    return c


def listed():
    return [
        # the smallest observation: 128^2, 5,000 baselines in a 60-wavelength disk, one stack
        # (J_w 26); what a unit check or a calibration loop calls again and again
        _case("tiny-degrid", "degrid", image_n=128, fov_deg=20.0, n_vis=5000, n_stacks=1,
              conj_fold=0, wmax=40.0, tracks=0),
        # the same observation in the FP64 path at its parity tolerance, the adjoint direction
        _case("tiny-f64-grid", "grid", precision="f64", tol=1e-12, image_n=128, fov_deg=20.0,
              n_vis=5000, n_stacks=1, conj_fold=0, wmax=40.0, tracks=0),
        # the headline: prediction for the MWA-like snapshot (2048^2, 1.95M visibilities,
        # 8 stacks, fold on, J_w 26-36), every tap by quadrature
        _case("snapshot-degrid", "degrid"),
        # its dirty image
        _case("snapshot-grid", "grid"),
        # one gradient of a least-squares fit through the differentiable operator: forward,
        # residual, backward, on a 1024^2 image with an odd number of visibilities
        _case("gradient-1024", "gradient", image_n=1024, n_vis=300007, n_stacks=4, wmax=200.0),
        # the same in the radial interpolation mode, at the snapshot's image size
        _case("gradient-radial", "gradient", mode="radial", n_vis=700001, weighted=1),
        # pre-sampled w-planes with w-row staging, forward and backward
        _case("gradient-table", "gradient", mode="table", staging=2, n_vis=1200000),
        # a small served request: 512^2, support per visibility, weights, reproducible gridding
        _case("served-512-grid", "grid", image_n=512, n_vis=50021, n_stacks=6, wmax=300.0,
              rule="vis", weighted=1, deterministic=1),
        # the same request's precision study, FP64 prediction at 1e-12
        _case("served-512-f64-degrid", "degrid", precision="f64", tol=1e-12, image_n=512,
              n_vis=8009, n_stacks=6, wmax=150.0),
        # direction-dependent effects, 5 x 5 separable kernels, fold off, 16 stacks
        _case("dde-degrid", "dde_degrid", n_vis=200003, n_stacks=16, conj_fold=0, dde_taps=5),
        # kernel values at given radii and w offsets (kernel plots, fits and checks)
        _case("kernel-values", "kernel", image_n=512, n_vis=40009, n_stacks=1, wmax=60.0),
        # an observation from its baselines to its dirty image, plan and all, at the paper's
        # many-stack setting (50 stacks, small supports)
        _case("observation-50-stacks", "observation", n_vis=1000003, n_stacks=50, wmax=600.0),
    ]


def draw(rng):
    def odd_log(lo, hi):
        return int(math.exp(rng.uniform(math.log(lo), math.log(hi))))

    op = rng.choice(["degrid", "grid", "degrid", "grid", "gradient", "dde_degrid", "dde_grid",
                     "kernel", "observation"])
    mode = rng.choice(["quadrature", "quadrature", "quadrature", "radial", "table"])
    f64 = rng.random() < 0.25
    image_n = 2 * odd_log(64, 1024)
    fov = rng.choice([15.0, 20.0, 25.0])
    fold = 0 if op.startswith("dde") else rng.choice([0, 1])
    stacks = rng.randint(1, 24)
    half = rng.uniform(2.0, 24.0)          # half the mean width of a stack in w
    n_vis = odd_log(1000, 8000 if f64 else 1000000)
    if mode == "table" and op == "observation":
        mode = "quadrature"
    if op.startswith("dde"):
        mode = "quadrature" if mode == "table" else mode
        n_vis = min(n_vis, 200000)
    if f64 and op == "gradient":
        n_vis = min(n_vis, 4000)
    if op == "kernel":
        n_vis = min(n_vis, 40000)
    return _case(None, op, mode=mode, precision="f64" if f64 else "f32",
                 tol=1e-12 if f64 and mode != "table" else 1e-6, image_n=image_n, fov_deg=fov,
                 n_vis=n_vis, n_stacks=stacks, conj_fold=fold,
                 wmax=half * stacks * (2.0 if fold else 1.0),
                 tracks=1 if rng.random() < 0.7 else 0,
                 rule=rng.choice(["stack", "stack", "vis"]),
                 weighted=rng.choice([0, 1]),
                 deterministic=1 if rng.random() < 0.2 else 0,
                 staging=rng.choice([0, 2]) if mode == "table" else 0,
                 dde_taps=rng.choice([3, 5, 7]) if op.startswith("dde") else 0)


# ----------------------------------------------------------------------------
# Inputs
# ----------------------------------------------------------------------------

def _generator(seed, salt):
    return torch.Generator(device="cuda").manual_seed(1000003 * int(seed) + salt)


def _rand(g, *shape):
    return torch.rand(*shape, generator=g, device="cuda", dtype=torch.float64)


def _randn(g, *shape):
    return torch.randn(*shape, generator=g, device="cuda", dtype=torch.float64)


def _uvw(case, seed):
    """Baselines (n_vis, 3) in wavelengths, max |w| = wmax."""
    g = _generator(seed, 1)
    M, N, fov = case["n_vis"], case["image_n"], math.radians(case["fov_deg"])
    extent = N / (2.0 * fov)               # half side of the uv grid, wavelengths
    if not case["tracks"]:
        r = min(60.0, 0.8 * extent) * torch.sqrt(_rand(g, M))
        t = 2.0 * math.pi * _rand(g, M)
        w = case["wmax"] * (2.0 * _rand(g, M) - 1.0)
        return torch.stack([r * torch.cos(t), r * torch.sin(t), w], 1).contiguous()
    # 128 antennas in a disk whose longest baselines just leave the grid
    n_ant = 128
    r = 0.64 * extent * torch.sqrt(_rand(g, n_ant))
    t = 2.0 * math.pi * _rand(g, n_ant)
    east, north = r * torch.cos(t), r * torch.sin(t)
    i, j = torch.triu_indices(n_ant, n_ant, 1, device="cuda")
    e, n = east[j] - east[i], north[j] - north[i]
    lat, dec = math.radians(-26.7), math.radians(-37.2)
    X, Y, Z = -math.sin(lat) * n, e, math.cos(lat) * n
    n_times = -(-M // e.numel())
    ha = torch.linspace(-n_times / 240.0, n_times / 240.0, n_times, device="cuda",
                        dtype=torch.float64) * (2.0 * math.pi / 1440.0)
    sh, ch = torch.sin(ha)[:, None], torch.cos(ha)[:, None]
    u = sh * X + ch * Y
    v = -math.sin(dec) * ch * X + math.sin(dec) * sh * Y + math.cos(dec) * Z
    w = math.cos(dec) * ch * X - math.cos(dec) * sh * Y + math.sin(dec) * Z
    uvw = torch.stack([u.ravel(), v.ravel(), w.ravel()], 1)
    if M < e.numel():                      # part of a snapshot: baselines of every length
        uvw = uvw[torch.randperm(e.numel(), generator=g, device="cuda")]
    uvw = uvw[:M].contiguous()
    uvw[:, 2] *= case["wmax"] / uvw[:, 2].abs().max()
    return uvw


def _inputs(case, seed):
    real = torch.float64 if case["precision"] == "f64" else torch.float32
    cplx = torch.complex128 if case["precision"] == "f64" else torch.complex64
    N, M = case["image_n"], case["n_vis"]
    s = dict(uvw=_uvw(case, seed))
    g = _generator(seed, 2)
    # a sky of point sources over faint diffuse emission
    x = 1e-3 * _rand(g, N, N)
    at = torch.randint(0, N * N, (200,), generator=g, device="cuda")
    x.view(-1)[at] += 0.1 + 0.9 * _rand(g, 200)
    s["x"] = x.to(real)
    s["y"] = torch.complex(_randn(g, M), _randn(g, M)).to(cplx)
    s["weights"] = 0.5 + _rand(g, M) if case["weighted"] else None
    if case["dde_taps"]:
        t = case["dde_taps"]
        off = torch.arange(t, device="cuda", dtype=torch.float64) - t // 2
        for key in ("a", "b"):             # blur, sub-pixel shift and phase ramp
            sig, mid = 0.4 + 0.8 * _rand(g, M, 1), _rand(g, M, 1) - 0.5
            ramp = _rand(g, M, 1) - 0.5
            k = torch.exp(-0.5 * ((off - mid) / sig) ** 2)
            k = torch.polar(k / k.sum(1, keepdim=True), ramp * off)
            s[key] = k.to(cplx)
    if case["op"] == "kernel":
        s["rho"] = 24.0 * _rand(g, M)
        s["dw"] = case["wmax"] * (2.0 * _rand(g, M) - 1.0)
    return s


def _plan(case, uvw, weights):
    return phi.Plan(uvw, weights, image_n=case["image_n"], fov_rad=math.radians(case["fov_deg"]),
                    oversample=OVERSAMPLE, support=SUPPORT, n_stacks=case["n_stacks"],
                    conj_fold=case["conj_fold"], precision=case["precision"],
                    support_rule=case["rule"], kernel_mode=case["mode"],
                    grid_staging=case["staging"], grid_deterministic=case["deterministic"],
                    quad_rel_tol=case["tol"], quad_abs_tol=case["tol"], max_support=128)


def prepare(case, seed):
    s = _inputs(case, seed)
    s["op"] = case["op"]
    if case["op"] == "observation":
        s["case"] = dict(case)
    elif case["op"] == "kernel":
        s["plan"] = _plan(case, s["uvw"][:1000], None)
    else:
        s["plan"] = _plan(case, s["uvw"], s["weights"])
        del s["uvw"]
    return s


def run(s):
    op = s["op"]
    if op == "degrid":
        return {"vis": s["plan"].degrid(s["x"])}
    if op == "grid":
        return {"image": s["plan"].grid(s["y"])}
    if op == "gradient":                   # of 1/2 ||Phi x - y||^2
        x = s["x"].detach().requires_grad_(True)
        model = autograd.degrid(x, s["plan"])
        r = model - s["y"]
        (0.5 * torch.sum(r.real ** 2 + r.imag ** 2)).backward()
        return {"vis": model.detach(), "gradient": x.grad}
    if op == "dde_degrid":
        return {"vis": s["plan"].degrid_dde(s["x"], s["a"], s["b"])}
    if op == "dde_grid":
        return {"image": s["plan"].grid_dde(s["y"], s["a"], s["b"])}
    if op == "kernel":
        k, missed = s["plan"].wkernel(s["rho"], s["dw"])
        return {"kernel": k, "missed": missed}
    if op == "observation":
        with _plan(s["case"], s["uvw"], s["weights"]) as plan:
            image = plan.grid(s["y"])
            info = plan.info()
        return {"image": image, "kept": info["n_kept"], "support": info["max_jw"],
                "sweeps": info["kmeans_sweeps"]}
    raise ValueError(op)


def work(case):
    """Bytes: baselines, visibilities, DDE kernels and the image once each.
    Operations: 8 per tap to apply it, counted at the support of a stack of
    the mean width, the FFTs of the stacks with 5 n log2 n each, and for kernel
    values one 31-point rule per point."""
    N, M, K = case["image_n"], case["n_vis"], case["n_stacks"]
    size = 8 if case["precision"] == "f64" else 4
    if case["op"] == "kernel":
        return {"bytes": M * (16 + 2 * size), "flops": M * 31 * 4.0}
    fov = math.radians(case["fov_deg"])
    c = 2.0 * fov * fov / math.sqrt(1.0 - fov * fov)
    half = case["wmax"] / K / (2.0 if case["conj_fold"] else 1.0)
    jw = SUPPORT + 2 * math.ceil(half * c) + max(0, case["dde_taps"] - 1)
    passes = 2 if case["op"] == "gradient" else 1
    n = (OVERSAMPLE * N) ** 2
    flops = passes * (8.0 * M * jw * jw + K * 5.0 * n * math.log2(n))
    data = passes * (M * (24 + 2 * size * (1 + 2 * case["dde_taps"])) + size * N * N)
    return {"bytes": data, "flops": flops}


# ----------------------------------------------------------------------------
# The operator in 64 bits, from its definition
# ----------------------------------------------------------------------------

_PIECE = 2.0      # grid pixels of rho per interpolation piece
_TERMS = 26       # Chebyshev terms per piece: below 1e-16 of the kernel's scale


def _bessel_j(n, x):
    """J_n(x) by the trapezoidal rule on its integral over one period, exact to
    rounding once the points outnumber |x| (torch.special's is off by 4e-7 near 5)."""
    m = int(float(x.abs().max())) + 40
    tot = torch.zeros_like(x)
    for k in range(m):
        t = math.pi * (k + 0.5) / m
        tot += torch.cos(n * t - x * math.sin(t))
    return tot / m


class _Exact:
    """y = Phi x and x = Re(Phi^H y) with every kernel value from one
    Gauss-Legendre rule over the whole window (interpolated in rho to rounding
    by a Chebyshev series), all in float64."""

    def __init__(self, case, uvw, weights):
        self.case = case
        N = self.N = case["image_n"]
        self.npad = int(round(OVERSAMPLE * N))
        fov = math.radians(case["fov_deg"])
        self.dl, self.R = fov / N, 0.5
        self.du = 1.0 / (self.npad * self.dl)
        l_win = self.R / self.du
        self.c = l_win / (math.sqrt(1.0 - l_win * l_win) * self.du)
        self.beta = math.pi * math.sqrt((SUPPORT / OVERSAMPLE) ** 2 * (OVERSAMPLE - 0.5) ** 2 - 0.8)
        if uvw is None:
            return
        K = case["n_stacks"]
        self.flag = (uvw[:, 2] < 0) if case["conj_fold"] else torch.zeros_like(uvw[:, 2], dtype=torch.bool)
        sgn = torch.where(self.flag, -1.0, 1.0).double()
        uvw = uvw * sgn[:, None]
        w = uvw[:, 2].contiguous()
        self.stack, self.centres, self.sweeps = self._kmeans(w, K)
        self.dw = w - self.centres[self.stack]
        up, vp = uvw[:, 0] / self.du, uvw[:, 1] / self.du
        h = self.npad // 2
        self.keep = (up >= -h) & (up < h) & (vp >= -h) & (vp < h)
        jw = SUPPORT + 2 * torch.ceil(self.dw.abs() * self.c).long()
        top = torch.zeros(K, dtype=torch.long, device="cuda")
        top.scatter_reduce_(0, self.stack[self.keep], jw[self.keep], "amax")
        self.jw = jw if case["rule"] == "vis" else top[self.stack]
        self.max_jw = int(top.max())
        self.bu, self.bv = torch.floor(up), torch.floor(vp)
        self.fu, self.fv = up - self.bu, vp - self.bv
        self.bu, self.bv = self.bu.long(), self.bv.long()
        self.weight = torch.ones_like(w) if weights is None else weights

    @staticmethod
    def _kmeans(w, K):
        lo, hi = float(w.min()), float(w.max())
        c = torch.linspace(lo, hi, K, device="cuda", dtype=torch.float64) if K > 1 else \
            torch.full((1,), 0.5 * (lo + hi), device="cuda", dtype=torch.float64)
        if K > 1:
            c = lo + torch.arange(K, device="cuda", dtype=torch.float64) * (hi - lo) / (K - 1)
        eps = (hi - lo) / K
        eps = eps if eps > 0 else 1.0
        sweeps = 0
        while True:
            s = torch.cat([torch.argmin((c[None, :] - p[:, None]) ** 2, 1) for p in w.split(1 << 20)])
            n = torch.bincount(s, minlength=K)
            tot = torch.zeros(K, device="cuda", dtype=torch.float64).index_add_(0, s, w)
            new = torch.where(n > 0, tot / n.clamp(min=1), torch.zeros_like(tot))
            d = float(((new - c).abs() / c.abs().clamp(min=eps)).mean())
            c, sweeps = new, sweeps + 1
            if d < 1e-3 or sweeps >= 100:
                return s, c, sweeps

    def taper(self, r):
        """g(r): the 2-D transform of the radial Kaiser-Bessel kernel."""
        a = 0.5 * SUPPORT
        z2 = self.beta ** 2 - (2.0 * math.pi * a * r) ** 2
        z = torch.sqrt(z2.abs()).clamp(min=1e-9)
        f = torch.where(z2 > 0, torch.special.i1(z) / z, _bessel_j(1, z) / z)
        i0 = torch.special.i0(torch.tensor(self.beta, dtype=torch.float64, device=r.device))
        return 2.0 * math.pi * a * a * f / i0

    def rule(self, rho_max, dw_max):
        """Nodes 1 - n(r_j) and weighted 2 pi g r, and r_j itself."""
        cycles = self.R * (rho_max + dw_max * self.c)
        x, wt = np.polynomial.legendre.leggauss(64 + int(4 * cycles))
        r = torch.from_numpy(0.5 * self.R * (x + 1.0)).cuda()
        wt = torch.from_numpy(0.5 * self.R * wt).cuda()
        l2 = (r / self.du) ** 2
        return l2 / (1.0 + torch.sqrt(1.0 - l2)), 2.0 * math.pi * wt * self.taper(r) * r, r

    def series(self, rho_max, r):
        """(pieces * _TERMS, nodes): Chebyshev coefficients in rho of J0(2 pi rho r_j)."""
        pieces = int(rho_max / _PIECE) + 1
        t = math.pi * (torch.arange(_TERMS, device="cuda", dtype=torch.float64) + 0.5) / _TERMS
        rho = _PIECE * (torch.arange(pieces, device="cuda", dtype=torch.float64)[:, None]
                        + 0.5 * (1.0 + torch.cos(t)))
        J = _bessel_j(0, 2.0 * math.pi * rho.reshape(-1, 1) * r)
        m = torch.arange(_TERMS, device="cuda", dtype=torch.float64)[:, None]
        dct = torch.cos(m * t) * (2.0 / _TERMS)
        dct[0] *= 0.5
        return torch.matmul(dct, J.view(pieces, _TERMS, -1)).reshape(pieces * _TERMS, -1), pieces

    def kernels(self, J, sel):
        """Kernel box (len(sel), J, J), rows v, of visibilities `sel`."""
        off = torch.arange(J, device="cuda", dtype=torch.float64) - J // 2 + 1
        omn, hk, r = self.rule(J * 0.75 + 2, float(self.dw.abs().max()))
        A, pieces = self.series(J / math.sqrt(2.0) + 1e-9, r)
        ph = 2.0 * math.pi * torch.remainder(self.dw[sel][:, None] * omn, 1.0)
        re, im = (hk * torch.cos(ph)) @ A.T, (hk * torch.sin(ph)) @ A.T
        rho = torch.sqrt((self.fu[sel][:, None] - off)[:, None, :] ** 2
                         + (self.fv[sel][:, None] - off)[:, :, None] ** 2).reshape(len(sel), -1)
        return torch.complex(self.clenshaw(re, rho, pieces), self.clenshaw(im, rho, pieces)
                             ).view(len(sel), J, J)

    @staticmethod
    def clenshaw(coef, rho, pieces):
        p = (rho / _PIECE).long().clamp(max=pieces - 1)
        x2 = 2.0 * (2.0 * (rho / _PIECE - p) - 1.0)
        p *= _TERMS
        b1 = torch.zeros_like(rho)
        b2 = torch.zeros_like(rho)
        for m in range(_TERMS - 1, 0, -1):
            b1, b2 = torch.gather(coef, 1, p + m).sub_(b2).addcmul_(x2, b1), b1
        return torch.gather(coef, 1, p).sub_(b2).addcmul_(x2, b1, value=0.5)

    def boxes(self, a=None, b=None):
        """Chunks (sel, J, K box, cells) of the kept visibilities, DDE applied."""
        taps = 1 if a is None else a.shape[1]
        for J in sorted(set(self.jw[self.keep].tolist())):
            rows = torch.nonzero(self.keep & (self.jw == J)).ravel()
            for sel in rows.split(max(1, 6000000 // (J + taps - 1) ** 2)):
                k = self.kernels(J, sel)
                if taps > 1:               # C[cv, cu] = sum b a K[cv - 2h + sv, cu - 2h + su]
                    pad = torch.nn.functional.pad(k, (taps - 1,) * 4)
                    L = J + taps - 1
                    row = sum(a[sel, s].view(-1, 1, 1) * pad[:, :, s:s + L] for s in range(taps))
                    k = sum(b[sel, s].view(-1, 1, 1) * row[:, s:s + L, :] for s in range(taps))
                L = J + taps - 1
                off = torch.arange(L, device="cuda") - taps // 2 - J // 2 + 1
                qu = torch.remainder(self.bu[sel][:, None] + off, self.npad)
                qv = torch.remainder(self.bv[sel][:, None] + off, self.npad)
                yield sel, k, qv[:, :, None] * self.npad + qu[:, None, :] \
                    + (self.stack[sel] * self.npad ** 2)[:, None, None]

    def screen(self):
        """Per pixel 1 - n and 1 / (g n)."""
        l = (torch.arange(self.N, device="cuda", dtype=torch.float64) - self.N // 2) * self.dl
        s = l[:, None] ** 2 + l[None, :] ** 2
        n = torch.sqrt(1.0 - s)
        return s / (1.0 + n), 1.0 / (self.taper(self.du * torch.sqrt(s)) * n)

    def degrid(self, x, a=None, b=None):
        omn, corr = self.screen()
        o = (self.npad - self.N) // 2
        grids = torch.zeros(self.centres.numel(), self.npad, self.npad, device="cuda",
                            dtype=torch.complex128)
        for k, wb in enumerate(self.centres.tolist()):
            ph = 2.0 * math.pi * torch.remainder(wb * omn, 1.0)
            grids[k, o:o + self.N, o:o + self.N] = torch.polar(x * corr, torch.zeros_like(ph)) \
                * torch.polar(torch.ones_like(ph), ph)
            grids[k] = torch.fft.fft2(torch.fft.ifftshift(grids[k]))
        flat = grids.view(-1)
        y = torch.zeros(self.dw.numel(), device="cuda", dtype=torch.complex128)
        for sel, k, cell in self.boxes(a, b):
            y[sel] = (k * flat[cell]).sum((1, 2)) * self.weight[sel]
        return torch.where(self.flag, y.conj(), y)

    def grid(self, y, a=None, b=None):
        omn, corr = self.screen()
        o = (self.npad - self.N) // 2
        K = self.centres.numel()
        flat = torch.zeros(K * self.npad ** 2, 2, device="cuda", dtype=torch.float64)
        y = torch.where(self.flag, y.conj(), y).resolve_conj() * self.weight
        for sel, k, cell in self.boxes(a, b):
            v = (k.conj() * y[sel].view(-1, 1, 1)).resolve_conj().reshape(-1)
            flat.index_add_(0, cell.reshape(-1), torch.view_as_real(v))
        grids = torch.view_as_complex(flat).view(K, self.npad, self.npad)
        x = torch.zeros(self.N, self.N, device="cuda", dtype=torch.float64)
        for k, wb in enumerate(self.centres.tolist()):
            f = torch.fft.fftshift(torch.fft.ifft2(grids[k], norm="forward"))[o:o + self.N, o:o + self.N]
            ph = 2.0 * math.pi * torch.remainder(wb * omn, 1.0)
            x += corr * (f.real * torch.cos(ph) + f.imag * torch.sin(ph))
        return x


def exact(case, seed):
    s = _inputs(case, seed)
    op = case["op"]
    if op == "kernel":
        E = _Exact(case, None, None)
        omn, hk, r = E.rule(float(s["rho"].max()), case["wmax"])
        out = []
        for rho, dw in zip(s["rho"].split(8192), s["dw"].split(8192)):
            ph = 2.0 * math.pi * torch.remainder(dw[:, None] * omn, 1.0)
            J = hk * _bessel_j(0, 2.0 * math.pi * rho[:, None] * r)
            out.append(torch.complex((J * torch.cos(ph)).sum(1), (J * torch.sin(ph)).sum(1)))
        return {"kernel": torch.cat(out), "missed": None}
    E = _Exact(case, s["uvw"], s["weights"])
    x, y = s["x"].double(), s["y"].to(torch.complex128)
    a = s["a"].to(torch.complex128) if "a" in s else None
    b = s["b"].to(torch.complex128) if "b" in s else None
    if op in ("degrid", "dde_degrid"):
        return {"vis": E.degrid(x, a, b)}
    if op in ("grid", "dde_grid"):
        return {"image": E.grid(y, a, b)}
    if op == "observation":
        return {"image": E.grid(y), "kept": None, "support": None, "sweeps": None}
    model = E.degrid(x)
    return {"vis": model, "gradient": E.grid(model - y)}
