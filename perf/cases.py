"""The work that users of the ray tracer have it do, as timed cases over its public entry points.

``listed()`` gives the standard cases, ``draw(rng)`` one more of the same ranges. ``prepare`` makes
what a user's program holds before the call (a context with its model and camera, image buffers,
network weights), ``run`` is one pass through the binding, ``work`` what a pass cannot do without,
and ``exact`` the same outputs from a plain torch FP64 restatement of the method (sizes permitting).

Models: the semi-analytic ADAF with seeded normalisations, and the Fishbone-Moncrief torus on the
288 x 128 x 128 FMKS grid with seeded log-normal density and field factors.
"""
import functools
import math

import numpy as np
import torch

from paper_2302_02733_gb300 import polrt, synth

DEV = "cuda"
FORMS = {"fp64": polrt.RT_FP64, "mixed": polrt.RT_MIXED, "unpol": polrt.RT_UNPOL, "surrogate": polrt.RT_SURROGATE}
STEPS_PER_RAY = 351.0   # mean RK4 steps of a ray at the default step size
# the surrogate's input box (ln nu/nu_c, theta_B, ln Theta_e, kappa) around the torus images' features
BOX_LO, BOX_HI = (1.2, 0.001, -3.75, 3.2), (27.5, math.pi / 2, 2.1, 8.0)


def listed():
    return [
        # the first thing a user renders, and the smallest call: the plain FP64 ADAF image
        dict(name="adaf64_fp64", call="render", model="adaf", form="fp64", nx=64, ny=64, incl=60.0, kappa=0.0, depths=False),
        # an ADAF image of odd, ragged size with its optical and Faraday depth maps
        dict(name="adaf_ragged_depths", call="render", model="adaf", form="mixed", nx=333, ny=257, incl=60.0, kappa=0.0, depths=True),
        # the headline: a GRMHD-shaped snapshot at 1024^2, FP64 geodesics and FP32 transfer
        dict(name="torus1024_mixed", call="render", model="torus", form="mixed", nx=1024, ny=1024, incl=20.0, kappa=0.0, depths=False),
        # the same snapshot in plain FP64, the form that errors are stated against
        dict(name="torus300_fp64", call="render", model="torus", form="fp64", nx=300, ny=300, incl=20.0, kappa=0.0, depths=False),
        # one likelihood evaluation of a fit: a 128^2 unpolarized image, its flux and its visibilities
        dict(name="fit128_unpol", call="fit", model="torus", form="unpol", nx=128, ny=128, incl=50.0),
        # an image library: images of several sizes, inclinations and model parameters in one call
        dict(name="library6_mixed", call="batch", form="mixed", images=6, table=7, sizes="128,256,512", mode=1),
        # an ADAF image traced adaptively, on a size that the lattice does not divide
        dict(name="adaptive250_mixed", call="adaptive", model="adaf", form="mixed", nx=250, ny=250, incl=60.0, base=8, tol=1e-3),
        # nonthermal electrons by quadrature along every ray, FP32 transfer
        dict(name="kappa64_mixed", call="render", model="torus", form="mixed", nx=64, ny=64, incl=20.0, kappa=4.5, depths=False),
        # a small FP64 image of the snapshot, as an oracle check or a preview takes it
        dict(name="torus126_fp64", call="render", model="torus", form="fp64", nx=126, ny=130, incl=70.0, kappa=0.0, depths=True),
        # nonthermal electrons through the network that stands in for the quadrature
        dict(name="surrogate384", call="surrogate", model="torus", form="surrogate", nx=384, ny=384, incl=20.0, kappa=4.78),
        # coefficients of a list of plasma points by quadrature (training sets, checks of the network)
        dict(name="coeffs60k", call="coeffs", n=60000, thermal_every=0),
        # training the network: forward, backward and Adam on the tensor cores
        dict(name="train300", call="train", n=131072, steps=300, batch=8192),
    ]


def _log(rng, lo, hi):
    return lo * (hi / lo) ** rng.random()


def draw(rng):
    k = rng.random()
    if k < 0.45:
        form = rng.choice(["fp64", "mixed", "mixed"])
        nx = int(_log(rng, 40, 340 if form == "fp64" else 1000))
        ny = min(int(nx * rng.uniform(0.7, 1.3)), 340 if form == "fp64" else 1000)
        return dict(call="render", model=rng.choice(["adaf", "torus"]), form=form, nx=nx, ny=ny,
                    incl=round(rng.uniform(10.0, 170.0), 2), kappa=0.0, depths=rng.random() < 0.3)
    if k < 0.58:
        n = int(_log(rng, 60, 500))
        return dict(call="fit", model=rng.choice(["adaf", "torus"]), form="unpol", nx=n, ny=n, incl=round(rng.uniform(10.0, 170.0), 2))
    if k < 0.70:
        return dict(call="batch", form=rng.choice(["mixed", "unpol"]), images=rng.randint(2, 8), table=rng.randint(1, 10**6),
                    sizes=rng.choice(["128", "128,256", "128,256,512"]), mode=1)
    if k < 0.80:
        n = int(_log(rng, 100, 400))
        return dict(call="adaptive", model="adaf", form=rng.choice(["mixed", "fp64"]), nx=n, ny=n, incl=round(rng.uniform(10.0, 170.0), 2),
                    base=rng.choice([4, 8]), tol=1e-3)
    if k < 0.86:
        n = int(_log(rng, 24, 64))
        return dict(call="render", model="torus", form="mixed", nx=n, ny=n, incl=round(rng.uniform(10.0, 170.0), 2),
                    kappa=round(rng.uniform(4.3, 7.9), 3), depths=False)
    if k < 0.94:
        n = int(_log(rng, 96, 420))
        return dict(call="surrogate", model="torus", form="surrogate", nx=n, ny=n, incl=round(rng.uniform(10.0, 170.0), 2),
                    kappa=round(rng.uniform(3.3, 7.9), 3))
    return dict(call="coeffs", n=int(_log(rng, 500, 60000)), thermal_every=rng.choice([0, 16]))


# ----------------------------------------------------------------------------------------------
# inputs

@functools.lru_cache(maxsize=1)
def _torus_base():
    """The unperturbed torus, axisymmetric: [n1][n2][1][8] on the device, and the grid it lies on."""
    prims, g = synth.fm_torus_grid(1, synth.GridParams(n3=1), synth.TorusParams(sigma_pert=0.0))
    g.n3 = 128
    return torch.from_numpy(prims).to(DEV), g


def _torus(seed):
    """The snapshot: log-normal factors (sigma 0.5) on density and field, cell by cell, from the seed."""
    base, g = _torus_base()
    gen = torch.Generator(device=DEV).manual_seed(seed)
    prims = base.expand(g.n1, g.n2, g.n3, 8).contiguous()
    f = torch.exp(0.5 * torch.randn((2, g.n1, g.n2, g.n3), generator=gen, device=DEV) - 0.125)
    prims[..., 0] *= f[0]
    prims[..., 5:8] *= f[1].unsqueeze(-1)
    return prims, g


def _camera(case):
    return synth.Camera(incl_deg=case["incl"], nx=case["nx"], ny=case["ny"])


def _model(case, seed):
    """(the C ABI's model, what it points to) of a case's plasma."""
    kappa = case.get("kappa", 0.0)
    if case.get("model") == "adaf":
        return polrt.adaf_model(synth.adaf_params(seed), kappa), None
    prims, g = _torus(seed)
    return polrt.grid_model(prims, g, kappa), prims


class State:
    """A context with its model, its camera and its buffers; the context goes with the object."""

    def __init__(self, case):
        self.case = case
        self.form = FORMS.get(case.get("form"))
        self.ctx = polrt.rt_create(0, torch.cuda.current_stream().cuda_stream)

    def __del__(self):
        if getattr(self, "ctx", None):
            polrt.rt_destroy(self.ctx)
            self.ctx = None


def _image(ny, nx, form):
    if form == polrt.RT_UNPOL:
        return torch.zeros((ny, nx), dtype=torch.float32, device=DEV)
    return torch.zeros((ny, nx, 4), dtype=torch.float64 if form == polrt.RT_FP64 else torch.float32, device=DEV)


def _library(case):
    """The image table of a batch: (camera, M_unit, R_high) for each image."""
    sizes = [int(s) for s in case["sizes"].split(",")]
    jobs = []
    for j in range(case["images"]):
        u = synth.uniform(case["table"], [4 * j + k for k in range(4)])
        n = sizes[j % len(sizes)]
        jobs.append((synth.Camera(incl_deg=10.0 + 160.0 * float(u[0]), nx=n, ny=n), 10.0 ** (17.0 + 3.0 * float(u[1])),
                     160.0 ** float(u[2])))
    return jobs


def _points(case, seed):
    """Plasma points (n_e, Theta_e, B, nu, theta_B, kappa) as images meet them."""
    gen = torch.Generator(device=DEV).manual_seed(seed)
    u = torch.rand((6, case["n"]), generator=gen, device=DEV, dtype=torch.float64)
    p = torch.stack([10.0 ** (3 + 5 * u[0]), 10.0 ** (-1 + 2.5 * u[1]), 10.0 ** (2 * u[2]), 86e9 * 10.0 ** (0.9 * u[3]),
                     0.02 + (math.pi - 0.04) * u[4], 3.2 + 4.8 * u[5]], dim=1)
    if case["thermal_every"]:
        p[:: case["thermal_every"], 5] = 0.0
    return p.contiguous()


@functools.lru_cache(maxsize=2)
def _network(seed):
    """Weights of a trained surrogate's kind: the cubic baseline fitted to coefficients of the
    distribution in the box, and a network whose residual is of the size that training leaves."""
    gen = torch.Generator(device=DEV).manual_seed(seed)
    n = 3072
    x = 2.0 * torch.rand((n, 4), generator=gen, device=DEV, dtype=torch.float64) - 1.0
    lo, hi = (torch.tensor(v, dtype=torch.float64, device=DEV) for v in (BOX_LO, BOX_HI))
    f = lo + 0.5 * (x + 1.0) * (hi - lo)
    th, te = f[:, 1].clamp(min=1e-3), torch.exp(f[:, 2])
    nu = torch.full_like(te, 230e9)
    B = nu / torch.exp(f[:, 0]) / (1.5 * CB * torch.sin(th) * te * te)
    c = _kappa_coeffs(torch.ones_like(te), te, B, nu, th.sin(), th.cos(), f[:, 3], h=0.2)
    y = torch.stack(_targets(te, B, nu, th.sin(), th.cos(), c), dim=1)
    ok = torch.isfinite(y).all(dim=1)
    phi = _monomials(x)
    base = torch.linalg.lstsq(phi[ok], y[ok]).solution.T        # [8][35]
    res = y[ok] - phi[ok] @ base.T
    norm = polrt.mlp_norm(BOX_LO, BOX_HI, y_mean=res.mean(0).tolist(), y_std=(0.05 * res.std(0)).tolist())
    b = base.tolist()
    for k in range(8):
        for q in range(35):
            norm.base[k][q] = b[k][q]
    w = []
    for o, i in ((64, 4), (64, 64), (64, 64), (8, 64)):
        w.append(torch.cat([(2.0 * torch.rand((o, i), generator=gen, device=DEV) - 1.0) * math.sqrt(3.0 / i),
                            torch.zeros((o, 1), device=DEV)], dim=1).flatten())
    return torch.cat(w).float().contiguous(), norm


def _monomials(x):
    cols = [torch.ones_like(x[:, 0])] + [x[:, i] for i in range(4)]
    cols += [x[:, i] * x[:, j] for i in range(4) for j in range(i, 4)]
    cols += [x[:, i] * x[:, j] * x[:, k] for i in range(4) for j in range(i, 4) for k in range(j, 4)]
    return torch.stack(cols, dim=1)


def prepare(case, seed):
    s = State(case)
    call = case["call"]
    if call == "coeffs":
        s.inp = _points(case, seed)
        s.out = torch.zeros((case["n"], 8), dtype=torch.float64, device=DEV)
        return s
    if call == "train":
        gen = torch.Generator(device=DEV).manual_seed(seed)
        s.x = (2.0 * torch.rand((case["n"], 4), generator=gen, device=DEV) - 1.0).contiguous()
        a = torch.randn((4, 8), generator=gen, device=DEV)
        t = torch.sin(2.0 * s.x @ a) + 0.3 * (s.x @ a) ** 2
        s.t = ((t - t.mean(0)) / t.std(0)).contiguous()
        s.theta, s.norm = _network(1)
        s.new = torch.zeros_like(s.theta)
        s.curve = np.zeros(case["steps"], dtype=np.float32)
        return s
    if call == "batch":
        prims, g = _torus(seed)
        polrt.rt_load_model(s.ctx, polrt.grid_model(prims, g))
        polrt.rt_set_batch_config(s.ctx, polrt.RT_MIXED, 3, 1, 2, case["mode"], 4)
        table = _library(case)
        s.imgs = [_image(c.ny, c.nx, s.form) for c, _, _ in table]
        s.jobs = polrt.make_jobs([(c, mu, rh, o, None, None) for (c, mu, rh), o in zip(table, s.imgs)])
        return s
    model, keep = _model(case, seed)
    polrt.rt_load_model(s.ctx, model)  # copies the grid
    polrt.rt_set_camera(s.ctx, _camera(case))
    s.img = _image(case["ny"], case["nx"], s.form)
    if call == "surrogate":
        theta, norm = _network(1)
        polrt.rt_mlp_set_params(s.ctx, theta, norm)
    if call == "render":
        s.status = torch.zeros((case["ny"], case["nx"]), dtype=torch.uint8, device=DEV)
        s.depth = torch.zeros((case["ny"], case["nx"], 2), dtype=s.img.dtype, device=DEV) if case["depths"] else None
    if call == "fit":
        s.vis = torch.zeros((case["ny"], case["nx"]), dtype=torch.complex64, device=DEV)
    return s


def run(s):
    call = s.case["call"]
    if call == "render":
        if s.depth is not None:
            polrt.rt_render_depths(s.ctx, s.form, s.img, s.depth, s.status)
            return {"img": s.img, "status": s.status, "depth": s.depth}
        polrt.rt_render(s.ctx, s.form, s.img, s.status)
        return {"img": s.img, "status": s.status}
    if call == "fit":
        polrt.rt_render(s.ctx, s.form, s.img)
        flux, _, _ = polrt.rt_image_stats(s.ctx, s.img, s.form)
        polrt.rt_image_visibilities(s.ctx, s.img, s.form, 0, s.vis)
        return {"img": s.img, "flux": flux, "vis": s.vis}
    if call == "batch":
        polrt.rt_render_batch(s.ctx, s.form, s.jobs)
        return s.imgs
    if call == "adaptive":
        polrt.rt_render_adaptive(s.ctx, s.form, s.img, None, s.case["base"], s.case["tol"])
        return s.img
    if call == "surrogate":
        polrt.rt_render(s.ctx, s.form, s.img)
        return s.img
    if call == "coeffs":
        polrt.rt_kappa_coeffs(s.ctx, s.inp, s.out)
        return s.out
    polrt.rt_mlp_set_params(s.ctx, s.theta, s.norm)  # training starts from the same weights each pass
    polrt.rt_mlp_train(s.ctx, s.x, s.t, s.case["steps"], s.case["batch"], 2e-3, 2302, s.curve)
    polrt.rt_mlp_get_params(s.ctx, s.new)
    return {"theta": s.new, "loss": s.curve}


def work(case):
    """Bytes: the grid and the other inputs read once, the outputs written once. Flops: 612 for an
    RK4 step of the geodesic, 900 for a point of the polarized transfer (300 unpolarized), 400
    quadrature nodes of 60 operations for a kappa point, 25,088 for a row of the network."""
    call, grid = case["call"], 288 * 128 * 128 * 32
    if call == "coeffs":
        return {"bytes": case["n"] * 14 * 8, "flops": case["n"] * 400 * 60}
    if call == "train":
        return {"bytes": case["steps"] * case["batch"] * 48, "flops": case["steps"] * case["batch"] * 3 * 25088}
    if call == "batch":
        rays = sum(c.nx * c.ny for c, _, _ in _library(case))
    else:
        rays = case["nx"] * case["ny"]
    if call == "adaptive":
        rays = rays // 8
    size = {"fp64": 32, "mixed": 16, "unpol": 4, "surrogate": 16}[case["form"]]
    point = 300 if case["form"] == "unpol" else 900
    if case.get("kappa") and case["form"] != "surrogate":
        point += 400 * 60
    if case["form"] == "surrogate":
        point += 25088
    return {"bytes": (0 if case.get("model") == "adaf" else grid) + rays * size, "flops": rays * STEPS_PER_RAY * (612 + point)}


# ----------------------------------------------------------------------------------------------
# the method in plain torch FP64, all rays (or all points) at once

G, C, ME, MP, QE, KB, H = 6.67430e-8, 2.99792458e10, 9.1093837015e-28, 1.67262192369e-24, 4.80320471257e-10, 1.380649e-16, 6.62607015e-27
CB = QE / (2 * math.pi * ME * C)  # nu_B / B
S3 = math.sqrt(3.0)


class _Kerr:
    """Kerr-Schild metric at (r, theta): components by index pair, its derivatives and inverse."""

    def __init__(self, a, r, th):
        s, c = torch.sin(th), torch.cos(th)
        s2, sc, a2 = s * s, s * c, a * a
        sig = r * r + a2 * c * c
        q = 2 * r / sig
        qr, qt = 2 / sig - q * q, 2 * a2 * sc * q / sig
        self.s, self.sig, self.q, self.r, self.s2 = s, sig, q, r, s2
        z = torch.zeros_like(q)
        self.g = {(0, 0): q - 1, (0, 1): q, (0, 3): -a * s2 * q, (1, 1): 1 + q, (1, 3): -a * s2 * (1 + q), (2, 2): sig,
                  (3, 3): s2 * (sig + a2 * s2 * (1 + q))}
        self.gr = {(0, 0): qr, (0, 1): qr, (0, 3): -a * s2 * qr, (1, 1): qr, (1, 3): -a * s2 * qr, (2, 2): 2 * r,
                   (3, 3): s2 * (2 * r + a2 * s2 * qr)}
        self.gt = {(0, 0): qt, (0, 1): qt, (0, 3): -a * (2 * sc * q + s2 * qt), (1, 1): qt,
                   (1, 3): -a * (2 * sc * (1 + q) + s2 * qt), (2, 2): -2 * a2 * sc,
                   (3, 3): 2 * sc * (sig + 2 * a2 * s2 * (1 + q)) - 2 * a2 * sc * s2 + a2 * s2 * s2 * qt}
        self.inv = {(0, 0): -(1 + q), (0, 1): q, (1, 1): (r * r - 2 * r + a2) / sig, (1, 3): a / sig, (2, 2): 1 / sig,
                    (3, 3): 1 / (sig * s2)}
        self.z = z

    def mul(self, m, v):
        o = [self.z] * 4
        for (i, j), x in m.items():
            o[i] = o[i] + x * v[j]
            if i != j:
                o[j] = o[j] + x * v[i]
        return o

    def lower(self, v):
        return self.mul(self.g, v)

    def dot(self, u, v):
        return sum(x * y for x, y in zip(self.lower(u), v))

    def accel(self, k):
        pr, pt = self.mul(self.gr, k), self.mul(self.gt, k)
        f = [k[1] * x + k[2] * y for x, y in zip(pr, pt)]
        f[1] = f[1] - 0.5 * sum(x * y for x, y in zip(pr, k))
        f[2] = f[2] - 0.5 * sum(x * y for x, y in zip(pt, k))
        return [-x for x in self.mul(self.inv, f)]

    def connection(self, k):
        """T^m_b = Gamma^m_ab k^a as a [..., 4, 4] tensor."""
        full = lambda m: [[m.get((min(i, j), max(i, j)), self.z) for j in range(4)] for i in range(4)]  # noqa: E731
        gr, gt, inv = full(self.gr), full(self.gt), full(self.inv)
        pr, pt = self.mul(self.gr, k), self.mul(self.gt, k)
        low = [[k[1] * gr[n][b] + k[2] * gt[n][b] for b in range(4)] for n in range(4)]
        for n in range(4):
            low[n][1] = low[n][1] + pr[n]
            low[n][2] = low[n][2] + pt[n]
        for b in range(4):
            low[1][b] = low[1][b] - pr[b]
            low[2][b] = low[2][b] - pt[b]
        low = torch.stack([torch.stack(x, -1) for x in low], -2)
        inv = torch.stack([torch.stack(x, -1) for x in inv], -2)
        return 0.5 * inv @ low


def _legs(m, zero):
    """Static observer's frame by Gram-Schmidt (d_t; then d_phi, d_theta, d_r), as lists of components."""
    one = zero + 1.0
    e = [None] * 4
    e[0] = [1 / torch.sqrt(-m.g[0, 0]), zero, zero, zero]
    for i in (3, 2, 1):
        v = [zero] * 4
        v[i] = one
        w = [x + m.dot(v, e[0]) * y for x, y in zip(v, e[0])]
        for j in range(3, i, -1):
            d = m.dot(v, e[j])
            w = [x - d * y for x, y in zip(w, e[j])]
        n = torch.sqrt(m.dot(w, w))
        e[i] = [x / n for x in w]
    return e


def _trace(cam, eps=0.05, nmax=20000):
    """Every ray's saved states [steps][8][rays] (r, th, ph, K^t..K^ph, signed h), the mask of states
    that a step left from, the status codes and each ray's sky direction and camera frame."""
    n = cam.nx * cam.ny
    idx = torch.arange(n, device=DEV)
    x = ((idx % cam.nx) + 0.5 - 0.5 * cam.nx).double() * cam.fov_M / cam.nx / cam.r_cam
    y = (torch.div(idx, cam.nx, rounding_mode="floor") + 0.5 - 0.5 * cam.ny).double() * cam.fov_M / cam.nx / cam.r_cam
    nn = torch.rsqrt(1 + x * x + y * y)
    sky = [-nn, -y * nn, x * nn]
    zero = torch.zeros_like(x)
    r, th, ph = zero + cam.r_cam, zero + math.radians(cam.incl_deg), zero
    frame = _legs(_Kerr(cam.a, r, th), zero)
    k = [-frame[0][c] + sum(sky[i] * frame[i + 1][c] for i in range(3)) for c in range(4)]
    st = torch.stack([r, th, ph] + k)
    rh = 1 + math.sqrt(1 - cam.a ** 2)
    live, status = torch.ones_like(idx, dtype=torch.bool), torch.zeros_like(idx, dtype=torch.uint8)
    states, masks = [], []

    def rate(v):
        return torch.cat([v[4:7], torch.stack(_Kerr(cam.a, v[0], v[1]).accel(v[3:7]))])

    for step in range(nmax):
        tt = torch.minimum(st[1], math.pi - st[1]).clamp(min=0.01)
        h = eps / (st[4].abs() / st[0] + st[5].abs() / tt + st[6].abs())
        k1 = rate(st)
        k2 = rate(st + 0.5 * h * k1)
        k3 = rate(st + 0.5 * h * k2)
        k4 = rate(st + h * k3)
        nw = st + h / 6 * (k1 + 2 * (k2 + k3) + k4)
        under, over = nw[1] < 0, nw[1] > math.pi
        flip = under | over
        nw[1] = torch.where(under, -nw[1], torch.where(over, 2 * math.pi - nw[1], nw[1]))
        nw[2] = torch.where(flip, nw[2] + math.pi, nw[2])
        nw[5] = torch.where(flip, -nw[5], nw[5])
        states.append(torch.cat([st, torch.where(flip, -h, h)[None]]))
        masks.append(live)
        st = torch.where(live, nw, st)
        hor, esc = live & (st[0] < 1.05 * rh), live & (st[0] > cam.r_cam) & (st[4] > 0)
        status = torch.where(hor, torch.full_like(status, 1), torch.where(esc & ~hor, torch.full_like(status, 2), status))
        live = live & ~hor & ~esc
        if step % 16 == 15 and not bool(live.any()):
            break
    return torch.stack(states), torch.stack(masks), status, sky, frame


def _isco(a):
    z1 = 1 + (1 - a * a) ** (1 / 3) * ((1 + a) ** (1 / 3) + (1 - a) ** (1 / 3))
    z2 = math.sqrt(3 * a * a + z1 * z1)
    return 3 + z2 - math.sqrt((3 - z1) * (3 + z1 + 2 * z2))


def _adaf(p, a, m, r):
    ne, te = p.n0 * r ** -1.5, p.T0 * KB / (ME * C * C) / r
    B = torch.sqrt(8 * math.pi * ne * KB * p.T0 / r * (1 + p.Ti_over_Te) / p.beta)
    s2, de, rr = m.s2, r * r - 2 * r + a * a, r * r + a * a
    big = rr * rr - a * a * de * s2
    gtt, gtp, gpp, grr = -big / (m.sig * de), -2 * a * r / (m.sig * de), (de - a * a * s2) / (m.sig * de * s2), de / m.sig
    rk = r.clamp(min=_isco(a))
    lk = (rk * rk - 2 * a * rk.sqrt() + a * a) / (rk ** 1.5 - 2 * rk.sqrt() + a)
    l = p.f_kep * lk * s2
    ur = -torch.sqrt((2 * r * rr / (m.sig * de) + 2 * gtp * l - gpp * l * l).clamp(min=0) / grr)
    u = [-gtt + gtp * l + 2 * r / de * grr * ur, grr * ur, torch.zeros_like(r), -gtp + gpp * l + a / de * grr * ur]
    nrm = torch.rsqrt(-m.dot(u, u))
    u = [x * nrm for x in u]
    ul = m.lower(u)
    bt = ul[1] + ul[3] / r
    b = [bt, (1 + bt * u[1]) / u[0], bt * u[2] / u[0], (1 / r + bt * u[3]) / u[0]]
    return r <= p.r_out, ne, te, B, u, b


def _fmks(g, w, x2):
    y = 2 * x2 - 1
    n = 0.5 * math.pi / (1 + 1 / ((g.poly_alpha + 1) * g.poly_xt ** g.poly_alpha))
    ya = (y.abs() / g.poly_xt) ** g.poly_alpha
    tg = math.pi * x2 + 0.5 * (1 - g.hslope) * torch.sin(2 * math.pi * x2)
    tj = n * y * (1 + ya / (g.poly_alpha + 1)) + 0.5 * math.pi
    dg = math.pi * (1 + (1 - g.hslope) * torch.cos(2 * math.pi * x2))
    return tg + w * (tj - tg), dg + w * (2 * n * (1 + ya) - dg), tj - tg


def _grid(prims, g, L, m, r, th, ph):
    x1 = torch.log(r)
    x1in = math.log(g.r_in)
    dx1 = (math.log(g.r_out) - x1in) / g.n1
    w = torch.exp(g.mks_smooth * (x1in - x1))
    lo, hi = torch.zeros_like(r), torch.ones_like(r)
    for _ in range(12):
        mid = 0.5 * (lo + hi)
        low = _fmks(g, w, mid)[0] < th
        lo, hi = torch.where(low, mid, lo), torch.where(low, hi, mid)
    x2 = 0.5 * (lo + hi)
    for _ in range(4):
        f, d, _ = _fmks(g, w, x2)
        x2 = (x2 - (f - th) / d).clamp(0.0, 1.0)
    _, d2, dd = _fmks(g, w, x2)
    fi, fj, fk = (x1 - x1in) / dx1 - 0.5, x2 * g.n2 - 0.5, ph * (g.n3 / (2 * math.pi)) - 0.5
    i0, j0, kf = fi.floor().clamp(0, g.n1 - 2), fj.floor().clamp(0, g.n2 - 2), fk.floor()
    wi, wj, wk = (fi - i0).clamp(0, 1), (fj - j0).clamp(0, 1), fk - kf
    i0, j0, k0 = i0.long(), j0.long(), kf.long() % g.n3
    P = 0
    for di in (0, 1):
        for dj in (0, 1):
            for dk in (0, 1):
                wt = (wi if di else 1 - wi) * (wj if dj else 1 - wj) * (wk if dk else 1 - wk)
                P = P + wt.unsqueeze(-1) * prims[i0 + di, j0 + dj, (k0 + dk) % g.n3].double()
    rho, uu = P[..., 0], P[..., 1]
    d1 = -g.mks_smooth * w * dd
    z = torch.zeros_like(r)
    U = [z, r * P[..., 2], d1 * P[..., 2] + d2 * P[..., 3], P[..., 4]]
    Bv = [z, r * P[..., 5], d1 * P[..., 5] + d2 * P[..., 6], P[..., 7]]
    gam = torch.sqrt(1 + m.dot(U, U))
    sop = torch.sqrt(1 + m.q)
    u = [gam * sop, U[1] - gam * m.q / sop, U[2], U[3]]
    bt = sum(x * y for x, y in zip(m.lower(u), Bv))
    b = [bt] + [(Bv[i] + bt * u[i]) / u[0] for i in (1, 2, 3)]
    bsq = m.dot(b, b)
    ok = (r >= g.r_in) & (r <= g.r_out) & (rho > 0) & (uu > 0) & ~(bsq > g.sigma_cut * rho)
    ib = (bsq / (2 * (g.gamma_ad - 1) * uu)) ** 2
    ratio = torch.where(ib < 1e30, (g.R_high + g.R_low * ib) / (1 + ib), z + g.R_low)
    unit = g.M_unit / L ** 3
    te = MP / ME * (g.gamma_ad - 1) * uu / (rho * (1 + ratio))
    return ok, rho * unit / (MP + ME), te, torch.sqrt(bsq.clamp(min=0)) * C * math.sqrt(4 * math.pi * unit), u, b


def _shcherbakov(X):
    f = 2.011 * torch.exp(-X ** 1.035 / 4.7) - torch.cos(0.5 * X) * torch.exp(-X ** 1.2 / 2.73) - 0.011 * torch.exp(-X / 47.2)
    tail = 0.011 * torch.exp(-X / 47.2) - 2 ** (-1 / 3) * 3 ** (-23 / 6) * 1e4 * math.pi * X ** (-8 / 3)
    f = torch.where(X > 1, f + tail * 0.5 * (1 + torch.tanh(10 * torch.log(X / 120))), f)
    return f, 1 - 0.11 * torch.log1p(0.035 * X)


def _cone(a, q, v):
    """(Q, V) scaled back where sqrt(Q^2 + V^2) exceeds |a|."""
    p = torch.sqrt((q / a) ** 2 + (v / a) ** 2)
    k = torch.where((a > 0) & (p > 1), 1 / p, torch.ones_like(p))
    return q * k, v * k


def _thermal(ne, te, B, nu, s, c):
    """j_I, j_Q, j_V, a_I, a_Q, a_V, r_Q, r_V of Maxwell-Juttner electrons."""
    rb = CB * B / nu
    X = te * torch.sqrt(math.sqrt(2.0) * s * 1e3 * rb)
    k0, k1 = torch.special.scaled_modified_bessel_k0(1 / te), torch.special.scaled_modified_bessel_k1(1 / te)
    k2 = k0 + 2 * te * k1
    f, gx = _shcherbakov(X)
    e2 = QE * QE / (ME * C)
    rq = e2 * ne * rb * rb / nu * s * s * f * (k1 / k2 + 6 * te)
    rv = 2 * e2 * ne * rb / nu * c * (k0 / k2) * gx
    x = nu / (1.5 * CB * B * s * te * te)
    x13 = x ** (1 / 3)
    ex = torch.exp(-1.8899 * x13)
    pre = QE * QE / (2 * S3 * C) * ne * nu / te ** 2 * 2.5651
    jI = pre * (1 + 1.92 / x13 + 0.9977 / x13 ** 2) * ex
    jQ = pre * (1 + 0.93193 / x13 + 0.499873 / x13 ** 2) * ex
    jV = 2 * QE * QE / (3 * S3 * C) * ne * nu * (c / s) / te ** 3 * (1.81348 / x + 3.42319 / x13 ** 2 + 0.0292545 / x.sqrt() + 2.03773 / x13) * ex
    jQ, jV = _cone(jI, jQ, jV)
    bb = 2 * H * nu ** 3 / (C * C) / torch.expm1(H * nu / (ME * C * C * te))
    on = (s >= 1e-12) & (jI > 1e-250)
    cf = [jI, jQ, jV, jI / bb, jQ / bb, jV / bb]
    return [torch.where(on, v, torch.zeros_like(v)) for v in cf] + [rq, rv]


def _kernels(x):
    """Synchrotron kernels F, G, H by the trapezoid rule on their cosh integrals."""
    ok = (x > 0) & (x < 740.0)
    x = torch.where(ok, x, torch.ones_like(x))
    h = 0.25 * torch.rsqrt(x).clamp(max=1.0)
    sums = [0.5 * torch.exp(-x) for _ in range(4)]
    for i in range(1, 400):
        t = i * h
        ch = torch.cosh(t)
        e = torch.exp(-x * ch)
        c13 = torch.cosh(t / 3)
        for j, v in enumerate((e * torch.cosh(5 * t / 3) / ch, e * torch.cosh(2 * t / 3), e * c13, e * c13 / ch)):
            sums[j] = sums[j] + torch.where(e > 0, v, torch.zeros_like(v))
        if i % 16 == 0 and float((e * torch.cosh(5 * t / 3)).max()) < 1e-19:
            break
    a, b, c, d = sums
    zero = torch.zeros_like(x)
    return [torch.where(ok, v, zero) for v in (x * h * a, x * h * b, x * h * c + h * d)]


@functools.lru_cache(maxsize=1)
def _kernel_table():
    """d^m ln K / d (ln x)^m is smooth: ln F, ln G, ln H + x at nodes fine enough for a degree-7 rule."""
    n, lo, hi = 6000, math.log(1e-13), math.log(740.0)
    u = torch.linspace(lo, hi, n, dtype=torch.float64, device=DEV)
    x = torch.exp(u)
    return lo, (hi - lo) / (n - 1), n, torch.stack([torch.log(k) + x for k in _kernels(x.clamp(max=739.999999))])


def _kernels_at(x):
    lo, h, n, tab = _kernel_table()
    ok = (x > 1e-13) & (x < 739.0)
    xs = torch.where(ok, x, torch.ones_like(x))
    u = (torch.log(xs) - lo) / h
    i = u.floor().long().clamp(3, n - 6)
    t = u - i
    out = [0, 0, 0]
    for a in range(-3, 5):  # Lagrange through 8 nodes
        wt = torch.ones_like(t)
        for b in range(-3, 5):
            if b != a:
                wt = wt * (t - b) / (a - b)
        for j in range(3):
            out[j] = out[j] + wt * tab[j][i + a]
    zero = torch.zeros_like(x)
    return [torch.where(ok, torch.exp(v - xs), zero) for v in out]


def _kappa_coeffs(ne, te, B, nu, s, c, kappa, h=0.05):
    """The coefficients of kappa electrons (kappa > 3; 0 selects Maxwell-Juttner) by the trapezoid
    rule in ln p, which converges geometrically for these integrands."""
    out = []
    kappa = kappa if torch.is_tensor(kappa) else torch.full_like(te, kappa)
    for lo in range(0, te.numel(), 1 << 16):
        sl = slice(lo, lo + (1 << 16))
        out.append(_kappa_some(*(v[sl] for v in (ne, te, B, nu, s, c, kappa)), h))
    return [torch.cat(v) for v in zip(*out)]


def _kappa_some(ne, te, B, nu, s, c, kappa, h):
    thermal = kappa <= 0
    kw = torch.where(thermal, torch.ones_like(te), (kappa - 3) * te)
    top = torch.where(thermal, torch.log(1 + 800 * te), torch.log(10 * (1 + kw)) + (45 / (kappa - 2.34)).clamp(max=600))
    hi = float(top.max())
    X = nu / (1.5 * CB * B * s.abs())
    nacc = rv = rq = 0
    e = [0] * 6
    zero = torch.zeros_like(te)
    # thermal electrons far above nu_c have a peak about 0.1 wide in ln p
    h = min(h, 0.02) if bool(thermal.any()) else h
    for i in range(int((hi - math.log(1e-7)) / h) + 2):
        sv = math.log(1e-7) + i * h
        if sv > 350.0:
            break
        p = math.exp(sv)
        g = math.sqrt(1 + p * p)
        gm1 = p * p / (g + 1)
        dg = h * p * p / g
        tq = torch.exp(-gm1 / te)
        kq = torch.exp(-(kappa + 1) * torch.log1p(gm1 / kw))
        q = torch.where(thermal, tq, kq)
        slope = torch.where(thermal, g * p / te, g * p * (kappa + 1) / (kw + gm1))
        N, D = g * p * q, q * (1 / p - slope)
        nacc = nacc + dg * N
        rv = rv + dg * N * math.asinh(p) / (g * p)
        rq = rq + dg * N * (2 * g - 1 / g)
        if p < 1e-4:
            continue
        k = _kernels_at(X / (g * g))
        for j in range(3):
            kj = k[j] if j < 2 else k[j] / g
            e[j] = e[j] + dg * N * kj
            e[3 + j] = e[3 + j] + dg * D * kj
    f, gx = _shcherbakov(te * torch.sqrt(math.sqrt(2.0) * s.abs() * 1e3 * CB * B / nu))
    nb = CB * B
    r6 = ne * QE * QE * nb * nb * s * s / (ME * C * nu ** 3) * f * rq / nacc
    r7 = 2 * ne * QE * QE * nb * c / (ME * C * nu * nu) * gx * rv / nacc
    A = S3 * QE ** 3 * B * s.abs() / (4 * math.pi * ME * C * C) * ne / nacc
    cot = c / s
    j = [A * e[0], A * e[1], A * (4 / 3) * cot * e[2]]
    al = [-A / (2 * nu * nu * ME) * v for v in (e[3], e[4], (4 / 3) * cot * e[5])]
    j[1], j[2] = _cone(j[0], j[1], j[2])
    al[1], al[2] = _cone(al[0], al[1], al[2])
    on = (s.abs() >= 1e-12) & (j[0] > 1e-250)
    return [torch.where(on, v, zero) for v in j + al] + [r6, r7]


def _targets(te, B, nu, s, c, cf):
    """Logarithms of the coefficients (n_e = 1) over the surrogate's prefactors."""
    e2, cot = QE * QE, c.abs() / s
    pj = e2 * nu / (2 * S3 * C * te * te)
    pa = e2 / (4 * S3 * ME * C * nu * te ** 3)
    f, gx = _shcherbakov(te * torch.sqrt(math.sqrt(2.0) * s * 1e3 * CB * B / nu))
    nb = CB * B
    pre = [pj, pj, pj * 4 / (3 * te) * cot, pa, pa, pa * cot, e2 * nb * nb * s * s / (ME * C * nu ** 3) * f,
           2 * e2 * nb * c.abs() / (ME * C * nu * nu) * gx]
    return [torch.log(x / y) for x, y in zip(cf, pre)]


def _tetrad(m, K, u, b):
    """The fluid frame's screen legs e1, e2, w = nu / nu_obs, sin and cos of the field angle."""
    w = m.dot(K, u)
    e3 = [-x - w * y for x, y in zip(K, u)]
    n = torch.rsqrt(m.dot(e3, e3))
    e3 = [x * n for x in e3]
    top = torch.stack([x.abs() for x in b]).amax(0)
    bn = [x / torch.where(top > 0, top, torch.ones_like(top)) for x in b]
    bb, b3 = m.dot(bn, bn), m.dot(bn, e3)
    e2 = [x - b3 * y for x, y in zip(bn, e3)]
    n2 = torch.sqrt(m.dot(e2, e2).clamp(min=0))
    has = bb > 0
    sth, cth = torch.where(has, n2 / bb.sqrt(), m.z), torch.where(has, b3 / bb.sqrt(), m.z + 1)
    alt = [m.z, m.z, m.z + 1, m.z]
    vu, ve = m.dot(alt, u), m.dot(alt, e3)
    bad = ~(n2 > 1e-10 * bb.clamp(min=0).sqrt())
    e2 = [torch.where(bad, x + vu * y - ve * z, v) for x, y, z, v in zip(alt, u, e3, e2)]
    n2 = torch.sqrt(m.dot(e2, e2))
    e2 = [x / n2 for x in e2]
    a, bv, cv = u, e2, e3

    def det(i, j, k):
        return (a[i] * (bv[j] * cv[k] - bv[k] * cv[j]) - a[j] * (bv[i] * cv[k] - bv[k] * cv[i])
                + a[k] * (bv[i] * cv[j] - bv[j] * cv[i]))

    sg = m.sig * m.s
    e1 = m.mul(m.inv, [-sg * det(1, 2, 3), sg * det(0, 2, 3), -sg * det(0, 1, 3), sg * det(0, 1, 2)])
    n1 = torch.rsqrt(m.dot(e1, e1))
    return [x * n1 for x in e1], e2, w, sth, cth


def _render(case, seed):
    """img [ny][nx][4] (or [ny][nx] unpolarized), status, depth, all FP64."""
    cam = _camera(case)
    states, masks, status, sky, frame = _trace(cam)
    L = G * cam.M_bh_g / (C * C)
    n = cam.nx * cam.ny
    f8 = dict(dtype=torch.float64, device=DEV)
    unpol, kappa = case["form"] == "unpol", case.get("kappa", 0.0)
    par = synth.adaf_params(seed) if case["model"] == "adaf" else None
    prims, g = (None, None) if par else _torus(seed)
    S = torch.zeros((n,) if unpol else (n, 4), **f8)
    tau, phi = torch.zeros(n, **f8), torch.zeros(n, **f8)
    basis = torch.zeros(n, dtype=torch.bool, device=DEV)
    E, TE = torch.zeros((n, 4, 2), **f8), torch.zeros((n, 4, 2), **f8)
    turn = torch.ones(4, 1, **f8)
    turn[2] = -1
    width = max(1, (1 << 19) // n)
    for top in range(states.shape[0], 0, -width):
        lo = max(0, top - width)
        q = states[lo:top]
        r, th, ph, hs = q[:, 0], q[:, 1], q[:, 2], q[:, 7]
        K = [q[:, 3 + i] for i in range(4)]
        m = _Kerr(cam.a, r, th)
        ok, ne, te, B, u, b = _adaf(par, cam.a, m, r) if par else _grid(prims, g, L, m, r, th, ph)
        ok = ok & masks[lo:top]
        e1, e2, w, sth, cth = _tetrad(m, K, u, b)
        nu = w * cam.freq_hz
        if kappa:
            cf = [torch.zeros_like(r) for _ in range(8)]
            got = _kappa_coeffs(*(v[ok] for v in (ne, te, B, nu, sth, cth)), kappa, h=0.125)
            for v, x in zip(cf, got):
                v[ok] = x
        else:
            cf = _thermal(ne, te, B, nu, sth, cth)
        cf = [torch.where(ok, v, torch.zeros_like(v)) for v in cf]
        ds = w * hs.abs() * L
        if unpol:
            t = cf[3] * ds
            p1 = torch.where(t == 0, torch.ones_like(t), -torch.expm1(-t) / torch.where(t == 0, torch.ones_like(t), t))
            J = cf[0] * ds / w ** 3
            for k in range(top - lo - 1, -1, -1):
                S = torch.where(ok[k], S + (J[k] - t[k] * S) * p1[k], S)
            continue
        T = m.connection(K)
        M = torch.zeros(r.shape + (5, 5), **f8)
        aI, aQ, aV, rQ, rV = cf[3:]
        for i in range(4):
            M[..., i, i] = -aI * ds
        for i, j, v in ((0, 1, aQ), (0, 3, aV), (1, 0, aQ), (1, 2, rV), (2, 1, -rV), (2, 3, rQ), (3, 0, aV), (3, 2, -rQ)):
            M[..., i, j] = -v * ds
        scale = cf[0].max() * 1e20 + 1e-200
        for i, v in ((0, cf[0]), (1, cf[1]), (3, cf[2])):
            M[..., i, 4] = v * ds / w ** 3 / scale
        X = torch.zeros_like(M)
        X[ok] = torch.linalg.matrix_exp(M[ok])
        e = torch.stack([torch.stack(e1, -1), torch.stack(e2, -1)], -1)   # [k][ray][4][2]
        gl = torch.stack([torch.stack(m.lower(e1), -1), torch.stack(m.lower(e2), -1)], -1)
        for k in range(top - lo - 1, -1, -1):
            on = masks[lo + k]
            cross = (on & basis & (hs[k] < 0))[:, None, None]
            E, TE = torch.where(cross, E * turn, E), torch.where(cross, TE * turn, TE)
            h = hs[k].abs()[:, None, None]
            moved = E + 0.5 * h * (TE + T[k] @ (E + h * TE))
            E = torch.where((on & basis)[:, None, None], moved, E)
            old = ok[k] & basis
            cm = gl[k].transpose(-1, -2) @ E
            nn = 0.5 * torch.stack([torch.stack([S[:, 0] + S[:, 1], S[:, 2]], -1), torch.stack([S[:, 2], S[:, 0] - S[:, 1]], -1)], -2)
            nn = cm @ nn @ cm.transpose(-1, -2)
            det = cm[:, 0, 0] * cm[:, 1, 1] - cm[:, 0, 1] * cm[:, 1, 0]
            S2 = torch.stack([nn[:, 0, 0] + nn[:, 1, 1], nn[:, 0, 0] - nn[:, 1, 1], 2 * nn[:, 0, 1], det * S[:, 3]], -1)
            S = torch.where(old[:, None], S2, S)
            S = torch.where(ok[k][:, None], (X[k][:, :4, :4] @ S[..., None])[..., 0] + X[k][:, :4, 4] * scale, S)
            E = torch.where(ok[k][:, None, None], e[k], E)
            basis = basis | ok[k]
            TE = torch.where((on & basis)[:, None, None], T[k] @ E, TE)
            tau, phi = tau + torch.where(ok[k], aI[k] * ds[k], 0.0), phi + torch.where(ok[k], rV[k] * ds[k], 0.0)
    shape = (cam.ny, cam.nx)
    if unpol:
        return S.reshape(shape), status.reshape(shape), None
    # the camera's screen: x along e_phi, y along -e_theta, each normal to the ray
    sk = torch.stack(sky, -1)
    legs = torch.stack([torch.stack([x.expand(n) for x in v], -1) for v in frame[1:]], -2)  # [ray][3][4]
    xh = torch.zeros_like(sk)
    xh[:, 2] = 1
    yh = torch.zeros_like(sk)
    yh[:, 1] = -1
    xh = xh - (xh * sk).sum(-1, keepdim=True) * sk
    xh = xh / xh.norm(dim=-1, keepdim=True)
    yh = yh - (yh * sk).sum(-1, keepdim=True) * sk
    yh = yh - (yh * xh).sum(-1, keepdim=True) * xh
    yh = yh / yh.norm(dim=-1, keepdim=True)
    mc = _Kerr(cam.a, torch.full((n,), cam.r_cam, **f8), torch.full((n,), math.radians(cam.incl_deg), **f8))
    low = [torch.stack(mc.lower([(v[:, None, :] @ legs)[:, 0, i] for i in range(4)]), -1) for v in (xh, yh)]
    cm = torch.stack(low, -2) @ E
    nn = 0.5 * torch.stack([torch.stack([S[:, 0] + S[:, 1], S[:, 2]], -1), torch.stack([S[:, 2], S[:, 0] - S[:, 1]], -1)], -2)
    nn = cm @ nn @ cm.transpose(-1, -2)
    det = cm[:, 0, 0] * cm[:, 1, 1] - cm[:, 0, 1] * cm[:, 1, 0]
    S2 = torch.stack([nn[:, 0, 0] + nn[:, 1, 1], nn[:, 0, 0] - nn[:, 1, 1], 2 * nn[:, 0, 1], det * S[:, 3]], -1)
    S = torch.where(basis[:, None], S2, S)
    return S.reshape(shape + (4,)), status.reshape(shape), torch.stack([tau, phi], -1).reshape(shape + (2,))


def exact(case, seed):
    call = case["call"]
    if call == "coeffs":
        p = _points(case, seed)
        th = p[:, 4]
        return torch.stack(_kappa_coeffs(p[:, 0], p[:, 1], p[:, 2], p[:, 3], torch.sin(th), torch.cos(th), p[:, 5]), dim=1)
    # batches, adaptive and surrogate images and large ones take too long; training differs from 64
    # bits by design (BF16 operands, magnified by Adam's first steps)
    if call not in ("render", "fit") or case["nx"] * case["ny"] > (1024 if case.get("kappa") else 17000):
        return None
    img, status, depth = _render(case, seed)
    if call == "render":
        return {"img": img, "status": None, "depth": depth} if case["depths"] else {"img": img, "status": None}
    cam = _camera(case)
    pix = cam.fov_M * G * cam.M_bh_g / (C * C) / (cam.nx * cam.dist_cm)
    # V(u, v) by the direct sum over pixel centres
    half = lambda n: torch.arange(n, device=DEV, dtype=torch.float64)  # noqa: E731
    nx, ny = cam.nx, cam.ny
    wx = torch.exp(-2j * math.pi / nx * torch.outer(half(nx) - nx // 2, half(nx) + 0.5 - 0.5 * nx))
    wy = torch.exp(-2j * math.pi / nx * torch.outer(half(ny) - ny // 2, half(ny) + 0.5 - 0.5 * ny))
    vis = wy @ (img * pix * pix * 1e23).to(torch.complex128) @ wx.T
    return {"img": img, "flux": float(img.sum()) * pix * pix * 1e23, "vis": vis}
