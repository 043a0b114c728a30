"""Performance cases of the hybrid lattice Boltzmann library: what a user's
program has it do, through the public binding (paper_0902_3921_gb300.lbm).

Kinds of case:
  lattice   `steps` LB steps of one lattice that works in the caller's own
            device buffers (as a PyTorch program lends them); the results are
            the population lattice and the phi plane of the new time.  With
            diagnostics=1 the pass ends with the FP64 observables, as the
            Sec. III studies sample them;
  batch     `steps` LB steps of `count` independent drops of uneven size, then
            n, phi and u* of every one of them, as a parameter study reads them;
  forward   one prediction of the learned surrogate;
  train     one training step of the surrogate (loss and gradients).

Initial fields are a late state of phase separation (domains of phi = +-phi0
with interfaces of the scheme's own width, a little noise) or a drop, both in
a flow of a few hundredths of c_s.
"""
import math

import numpy as np
import torch

from paper_0902_3921_gb300 import inputs, lbm

# the benchmark's fluid (automatic m = 4 in 2D, 8 in 3D) and the paper's own
# (Sec. III, m = 1)
BENCH = dict(a=-0.1, b=0.1, kappa=0.14, tau=1.0, Gamma=0.5, N=0.3, Q=2.5)
BENCH3 = dict(BENCH, N=1.0 / 6.0, Q=1.0 / 3.0)
PAPER = dict(a=-1e-3, b=1e-3, kappa=3e-3, tau=0.8, Gamma=5.0, N=0.3, Q=2.5)
PRECISION = {"f64": lbm.LBM_F64, "f32": lbm.LBM_F32DEV, "f16": lbm.LBM_F16DEV}
_STREAM = []  # one stream for a program's lattices, made at the first use
DTYPE = {"f64": torch.float64, "f32": torch.float32, "f16": torch.float16}
F16_SCALE = 1024.0  # the default storage scale of FP16 deviations


def _lattice(Lx, Ly, Lz=1, precision="f32", fluid="bench", init="domains", steps=10, flux=0, stencil=0,
             force=0.0, diagnostics=0):
    return dict(kind="lattice", Lx=Lx, Ly=Ly, Lz=Lz, precision=precision, fluid=fluid, init=init, steps=steps,
                flux=flux, stencil=stencil, force=force, diagnostics=diagnostics)


def listed():
    return [
        # the smallest run of the validation set (64^2 drop): launches and latency count
        dict(_lattice(64, 64, init="drop", steps=64), name="drop_64_f32"),
        # the headline: spinodal decomposition at 1024^2, FP32 deviations
        dict(_lattice(1024, 1024, steps=20), name="spinodal_1024_f32"),
        # its large point, beyond L2
        dict(_lattice(4096, 4096, steps=4), name="spinodal_4096_f32"),
        # FP16 deviation storage, chosen for memory
        dict(_lattice(2048, 2048, precision="f16", steps=10), name="spinodal_2048_f16"),
        # the Sec. III studies (Table I, Fig. 4): an FP64 drop on 128^2, sampled as it relaxes
        dict(_lattice(128, 128, precision="f64", fluid="paper", init="drop", steps=50, diagnostics=1),
             name="table1_128_f64"),
        # an odd-sized box: a drop pushed by a body force, conservative advection
        dict(_lattice(509, 251, init="drop", steps=24, flux=1, force=1e-5), name="pushed_drop_509x251_f32"),
        # the 3D benchmark: D3Q19 at 256^3
        dict(_lattice(256, 256, 256, steps=2), name="drop3d_256_f32"),
        # a 3D box that is no power of two, FP16 deviations
        dict(_lattice(200, 144, 112, precision="f16", steps=4), name="spinodal3d_200x144x112_f16"),
        # the 3D accuracy runs: 64^3 in FP64
        dict(_lattice(64, 64, 64, precision="f64", init="drop", steps=4), name="drop3d_64_f64"),
        # the parameter study of 512 drops
        dict(kind="batch", count=512, steps=300, name="batch_512_drops"),
        # surrogate inference at 2048^2 and training on 512^2 crops
        dict(kind="forward", count=1, H=2048, W=2048, channels=32, layers=6, name="surrogate_forward_2048"),
        dict(kind="train", count=8, H=512, W=512, channels=32, layers=6, name="surrogate_train_8x512"),
    ]


def draw(rng):
    """One more case of these ranges: sides over their logarithm, multiples of
    16 and of 4 as programs choose them, and any size at all."""
    def side(lo, hi):
        v = math.exp(rng.uniform(math.log(lo), math.log(hi)))
        m = rng.choice([1, 1, 4, 16])
        return int(max(lo, min(hi, round(v / m) * m)))

    what = rng.choice(["2d", "2d", "2d", "study", "3d", "3d", "3d64", "batch", "forward", "train"])
    if what == "2d":
        Lx, Ly = side(48, 4096), side(48, 4096)
        return _lattice(Lx, Ly, precision=rng.choice(["f32", "f32", "f16"]),
                        init=rng.choice(["domains", "drop"]), flux=rng.choice([0, 0, 1]),
                        force=rng.choice([0.0, 1e-5]),
                        steps=max(2, min(64, int(6e7 / (Lx * Ly)))))
    if what == "study":
        Lx, Ly = side(64, 512), side(64, 512)
        return _lattice(Lx, Ly, precision="f64", fluid=rng.choice(["paper", "bench"]), init="drop",
                        stencil=rng.choice([0, 0, 1]), force=rng.choice([0.0, 3e-5]), diagnostics=1,
                        steps=max(4, min(50, int(8e5 / (Lx * Ly)))))
    if what == "3d":
        Lx, Ly, Lz = side(24, 256), side(24, 256), side(24, 256)
        return _lattice(Lx, Ly, Lz, precision=rng.choice(["f32", "f32", "f16"]),
                        init=rng.choice(["domains", "drop"]), flux=rng.choice([0, 0, 1]),
                        steps=max(1, min(16, int(1.5e7 / (Lx * Ly * Lz)))))
    if what == "3d64":
        Lx, Ly, Lz = side(24, 96), side(24, 96), side(24, 96)
        return _lattice(Lx, Ly, Lz, precision="f64", init="drop",
                        steps=max(1, min(8, int(1e6 / (Lx * Ly * Lz)))))
    if what == "batch":
        count = side(16, 512)
        return dict(kind="batch", count=count, steps=rng.choice([100, 200, 300]))
    if what == "forward":
        return dict(kind="forward", count=rng.randint(1, 4), H=8 * rng.randint(16, 128),
                    W=16 * rng.randint(8, 64), channels=rng.choice([32, 32, 16]), layers=rng.randint(4, 6))
    return dict(kind="train", count=rng.randint(1, 8), H=8 * rng.randint(16, 64), W=16 * rng.randint(8, 32),
                channels=rng.choice([32, 32, 16]), layers=rng.randint(4, 6))


# ---- inputs ------------------------------------------------------------------------


def _fluid(case):
    if case["fluid"] == "paper":
        return PAPER
    return BENCH3 if case["Lz"] > 1 else BENCH


def _generator(seed):
    return torch.Generator(device="cuda").manual_seed(int(seed) & 0x7FFFFFFF)


def _waves(shape, gen, wavelength, count=8):
    """Sum of `count` periodic plane waves of about this wavelength with random
    directions and phases, variance 1 (FP64, device)."""
    d = len(shape)
    out = torch.zeros(shape, dtype=torch.float64, device="cuda")
    r = torch.rand(count, d + 2, generator=gen, device="cuda", dtype=torch.float64).cpu().tolist()
    for row in r:
        v = [2.0 * x - 1.0 for x in row[:d]]
        norm = math.sqrt(sum(x * x for x in v)) or 1.0
        term = None
        for axis, L in enumerate(shape):
            k = round(v[axis] / norm * L / (wavelength * (0.7 + 0.6 * row[d])))
            ph = 2.0 * math.pi * k / L * torch.arange(L, dtype=torch.float64, device="cuda")
            e = torch.polar(torch.ones_like(ph), ph + (2.0 * math.pi * row[d + 1] if axis == 0 else 0.0))
            e = e.reshape([-1 if a == axis else 1 for a in range(d)])
            term = e if term is None else term * e
        out += term.real
    return out * math.sqrt(2.0 / count)


def _fields(shape, init, fluid, seed):
    """n, phi, u (FP64, device) of one lattice."""
    gen = _generator(seed)
    d = len(shape)
    phi0 = math.sqrt(-fluid["a"] / fluid["b"])
    xi = math.sqrt(-2.0 * fluid["kappa"] / fluid["a"])
    if init == "drop":
        R = 0.25 * min(shape) * (0.9 + 0.2 * torch.rand(1, generator=gen, device="cuda").item())
        r2 = 0.0
        for axis, L in enumerate(shape):
            x = torch.arange(L, dtype=torch.float64, device="cuda") - L / 2.0
            r2 = r2 + (x * x).reshape([-1 if a == axis else 1 for a in range(d)])
        phi = phi0 * torch.tanh((R - torch.sqrt(r2)) / xi)
    else:
        wavelength = min(24.0 * xi / 1.67, min(shape) / 1.5)
        w = _waves(shape, gen, wavelength)
        phi = 0.95 * phi0 * torch.tanh(w * wavelength / (2.0 * math.pi * xi))
    phi = phi + 0.01 * phi0 * (2.0 * torch.rand(shape, generator=gen, device="cuda", dtype=torch.float64) - 1.0)
    u = torch.stack([0.02 * _waves(shape, gen, max(32.0, min(shape) / 2.0), count=3) for _ in range(d)])
    n = 1.0 + 0.002 * _waves(shape, gen, max(32.0, min(shape) / 2.0), count=3)
    return n, phi, u


def _drops(case):
    """Sides, radii and body forces of the batch, as the benchmark draws them."""
    return inputs.batch_instances(case["count"], seed=case["count"])


def _weights(case, seed):
    """He-normal weights, the last layer scaled by 0.1, small biases (FP32, host):
    a list of (W [co][3][3][ci], b [co])."""
    gen = torch.Generator().manual_seed(int(seed) & 0x7FFFFFFF)
    C, layers = case["channels"], case["layers"]
    out = []
    for k in range(layers):
        ci, co = (4 if k == 0 else C), (4 if k == layers - 1 else C)
        W = torch.randn(co, 3, 3, ci, generator=gen) * math.sqrt(2.0 / (9 * ci))
        out.append(((0.1 if k == layers - 1 else 1.0) * W, 0.05 * torch.randn(co, generator=gen)))
    return out


IN_MEAN = [0.0, 0.0, 0.0, 0.0]
IN_STD = [0.6, 0.02, 0.02, 2e-3]
OUT_STD = [0.05, 2e-3, 2e-3, 5e-4]


def _states(case, seed):
    """Network states [count][H][W][4] (phi, u*_x, u*_y, n - 1), FP32, device."""
    xs = []
    for k in range(case["count"]):
        n, phi, u = _fields((case["H"], case["W"]), "domains", BENCH, seed * 64 + k)
        xs.append(torch.stack([phi, u[0], u[1], n - 1.0], dim=-1))
    return torch.stack(xs).float().contiguous()


def _targets(case, x0, seed):
    """The states a window later: the change of the normalised state is of the
    order of out_std."""
    gen = _generator(seed + 77)
    step = torch.randn(x0.shape, generator=gen, device="cuda") * torch.tensor(OUT_STD, device="cuda")
    return (x0 + 0.5 * step + 0.5 * torch.roll(step, 1, dims=2)).contiguous()


# ---- the passes --------------------------------------------------------------------


def prepare(case, seed):
    kind = case["kind"]
    if kind == "lattice":
        d3 = case["Lz"] > 1
        shape = (case["Lz"], case["Ly"], case["Lx"]) if d3 else (case["Ly"], case["Lx"])
        params = lbm.LbmParams(dims=3 if d3 else 2, Lx=case["Lx"], Ly=case["Ly"], Lz=case["Lz"],
                               precision=PRECISION[case["precision"]],
                               adv_variant=lbm.LBM_ADV_FLUX if case["flux"] else lbm.LBM_ADV_PAPER,
                               stencil_fd=case["stencil"], g=(case["force"], 0.0, 0.0),
                               force_steps=1000000 if case["force"] else 0, **_fluid(case))
        field = torch.float64 if case["precision"] == "f64" else torch.float32
        new = lambda k, dt: torch.empty((k,) + shape, dtype=dt, device="cuda")  # noqa: E731
        buffers = {"populations": [new(19 if d3 else 9, DTYPE[case["precision"]]) for _ in range(2)],
                   "phi": [torch.empty(shape, dtype=field, device="cuda") for _ in range(3)],
                   "u": new(len(shape), field)}
        if not _STREAM:
            _STREAM.append(torch.cuda.Stream())
        lattice = lbm.Lattice(params, stream=_STREAM[0].cuda_stream, buffers=buffers)
        n, phi, u = _fields(shape, case["init"], _fluid(case), seed)
        lattice.init_fields(n.cpu().numpy(), phi.cpu().numpy(), u.cpu().numpy())
        return dict(case=case, lattice=lattice)
    if kind == "batch":
        drops = _drops(case)
        batch = lbm.Batch(lbm.LbmParams(precision=lbm.LBM_F32DEV, **BENCH),
                          [(d["side"], d["side"], (1e-5 if d["forced"] else 0.0, 0.0),
                            1000000 if d["forced"] else 0) for d in drops])
        rng = np.random.RandomState(seed & 0x7FFFFFFF)
        for k, d in enumerate(drops):
            L = d["side"]
            phi = inputs.drop(2, L, L, R=d["R"], phi0=1.0, xi=math.sqrt(2.8))
            phi += 0.01 * (2.0 * rng.random_sample(phi.shape) - 1.0)
            y = 2.0 * np.pi * np.arange(L) / L
            u = np.empty((2, L, L))
            u[0] = 0.02 * np.sin(y + rng.uniform(0.0, 6.28))[:, None]
            u[1] = 0.02 * np.sin(y + rng.uniform(0.0, 6.28))[None, :]
            batch.init_fields(k, np.ones((L, L)), phi, u)
        return dict(case=case, batch=batch, sides=[d["side"] for d in drops])
    net = lbm.Net(case["channels"], case["layers"], seed=1)
    net.set_params(torch.cat([t.reshape(-1) for W, b in _weights(case, seed) for t in (W, b)]).numpy())
    net.set_normalisation(IN_MEAN, IN_STD, OUT_STD)
    x0 = _states(case, seed)
    x1 = torch.empty_like(x0) if kind == "forward" else _targets(case, x0, seed)
    torch.cuda.synchronize()
    return dict(case=case, net=net, x0=x0, x1=x1)


def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "lattice":
        lattice = state["lattice"]
        lattice.step(case["steps"])
        now = lattice.t % 2  # the two lattices alternate from step to step
        out = {"populations": lattice.buffers["populations"][now], "phi": lattice.buffers["phi"][now]}
        if case["diagnostics"]:
            d = lattice.diagnostics()
            out["observables"] = np.array([d["sum_n"], d["sum_phi"], d["u_max"], d["area"], d["R_eff"]]
                                          + d["r_cm"], dtype=np.float32)
        return out
    if kind == "batch":
        batch, sides = state["batch"], state["sides"]
        batch.step(case["steps"])
        total = sum(L * L for L in sides)
        n, phi, u = (np.empty(k * total, dtype=np.float32) for k in (1, 1, 2))  # as the lattices store them
        at = 0
        for k, L in enumerate(sides):
            nk, pk, uk = batch.moments(k)
            S = L * L
            n[at:at + S], phi[at:at + S], u[2 * at:2 * (at + S)] = nk.ravel(), pk.ravel(), uk.ravel()
            at += S
        return {"n": n, "phi": phi, "u": u}
    net, x0, x1 = state["net"], state["x0"], state["x1"]
    if kind == "forward":
        net.forward(x0.data_ptr(), case["count"], case["H"], case["W"], x1.data_ptr())
        return x1
    loss = net.train_step(x0.data_ptr(), x1.data_ptr(), case["count"], case["H"], case["W"], 1e-4)
    return {"loss": np.float32(loss), "gradients": net.get_grads()}


# ---- algorithmic work --------------------------------------------------------------


def work(case):
    """Bytes: per LB step and site the populations and phi read and written once
    (the method's own count); for the network each layer's input and output
    once.  Flops: collision and force, and m substeps of the phi equation."""
    kind = case["kind"]
    if kind == "lattice":
        d3 = case["Lz"] > 1
        updates = float(case["Lx"]) * case["Ly"] * case["Lz"] * case["steps"]
        pop = {"f64": 8, "f32": 4, "f16": 2}[case["precision"]]
        field = 8 if case["precision"] == "f64" else 4
        m = _substeps(case)
        return {"bytes": updates * 2 * ((19 if d3 else 9) * pop + field),
                "flops": updates * (480 + 55 * m if d3 else 210 + 41 * m)}
    if kind == "batch":
        sites = sum(d["side"] ** 2 for d in _drops(case))
        return {"bytes": sites * (80.0 * case["steps"] + 32.0), "flops": sites * 374.0 * case["steps"]}
    P, C, layers = float(case["count"]) * case["H"] * case["W"], case["channels"], case["layers"]
    macs = 9.0 * (2 * 4 * C + (layers - 2) * C * C)
    hidden = 2.0 * C * (layers - 1)  # BF16 activations between the layers, bytes per pixel
    if kind == "forward":
        return {"bytes": P * (32.0 + 2.0 * hidden), "flops": 2.0 * P * macs}
    return {"bytes": P * (32.0 + 6.0 * hidden), "flops": 6.0 * P * macs}


def _substeps(case):
    """The smallest m whose diffusive stiffness times 1/m is at most 1.5 (what
    fd_substeps = 0 asks for)."""
    f = _fluid(case)
    lam = 4.0 * (3 if case["Lz"] > 1 else 2)
    if case["stencil"]:
        lam = max(8.0 * f["Q"], 4.0)
    return max(1, math.ceil(f["Gamma"] * (-2.0 * f["a"] * lam + f["kappa"] * lam * lam) / 1.5 - 1e-12))


# ---- the same results in 64 bits, plain torch --------------------------------------

D2Q9 = [(0, 0), (1, 0), (0, 1), (-1, 0), (0, -1), (1, 1), (-1, 1), (-1, -1), (1, -1)]
D3Q19 = [(0, 0, 0), (1, 0, 0), (-1, 0, 0), (0, 1, 0), (0, -1, 0), (0, 0, 1), (0, 0, -1), (1, 1, 0), (-1, -1, 0),
         (1, -1, 0), (-1, 1, 0), (1, 0, 1), (-1, 0, -1), (1, 0, -1), (-1, 0, 1), (0, 1, 1), (0, -1, -1),
         (0, 1, -1), (0, -1, 1)]


def _at(f, e):
    """f(r + e) on the periodic lattice, e in (x, y, z) order."""
    d = len(e)
    dims = [a for a in range(d) if e[a]]
    return torch.roll(f, [-e[a] for a in dims], [d - 1 - a for a in dims]) if dims else f


def _weight(e):
    speed = sum(abs(c) for c in e)
    return ({0: 4.0 / 9.0, 1: 1.0 / 9.0, 2: 1.0 / 36.0} if len(e) == 2
            else {0: 1.0 / 3.0, 1: 1.0 / 18.0, 2: 1.0 / 36.0})[speed]


def _operators(d, N, Q):
    """The stencil derivative and Laplacian (Eqs. 30-31) over the lattice vectors."""
    vectors = (D2Q9 if d == 2 else D3Q19)[1:]
    M, R = ((1.0 - 2.0 * N) / 4.0, (1.0 - Q) / 2.0) if d == 2 else ((1.0 - 2.0 * N) / 8.0, (1.0 - Q) / 4.0)

    def diff(f, axis):
        return sum((N if sum(map(abs, e)) == 1 else M) * e[axis] * _at(f, e) for e in vectors if e[axis])

    def lap(f):
        return sum((Q if sum(map(abs, e)) == 1 else R) * (_at(f, e) - f) for e in vectors)

    return diff, lap


class _Exact:
    """The scheme of include/hybrid_lbm.h in FP64: step 1-5 at every site."""

    def __init__(self, case, n, phi, u):
        self.case, f = case, _fluid(case)
        self.d = d = 3 if case["Lz"] > 1 else 2
        self.e = D2Q9 if d == 2 else D3Q19
        self.w = [_weight(e) for e in self.e]
        self.p, self.m = f, _substeps(case)
        self.diff, self.lap = _operators(d, f["N"], f["Q"])
        self.unit = [tuple(int(a == b) for b in range(d)) for a in range(d)]
        self.phi = phi
        F = self.force(n)
        v = [u[a] - F[a] / (2.0 * n) for a in range(d)]
        self.f = [self.feq(i, n, v) for i in range(len(self.e))]

    def lap1(self, f):
        if self.case["stencil"]:
            return self.lap(f)
        return sum(_at(f, e) + _at(f, tuple(-c for c in e)) - 2.0 * f for e in self.unit)

    def force(self, n):
        p, phi = self.p, self.phi
        mu = p["a"] * phi + p["b"] * phi ** 3 - p["kappa"] * self.lap(phi)
        F = [-phi * self.diff(mu, a) for a in range(self.d)]
        F[0] = F[0] + n * self.case["force"]
        return F

    def feq(self, i, n, u):
        e, w = self.e[i], self.w[i]
        eu = sum(c * x for c, x in zip(e, u) if c)
        return w * n * (1.0 + 3.0 * eu + 4.5 * eu * eu - 1.5 * sum(x * x for x in u))

    def step(self, last):
        tau, d = self.p["tau"], self.d
        n = sum(self.f)
        F = self.force(n)
        u = [(sum(e[a] * f for e, f in zip(self.e, self.f) if e[a]) + 0.5 * F[a]) / n for a in range(d)]
        uF = sum(x * y for x, y in zip(u, F))
        for i, e in enumerate(self.e):
            eu = sum(c * x for c, x in zip(e, u) if c)
            eF = sum(c * x for c, x in zip(e, F) if c)
            S = (1.0 - 0.5 / tau) * self.w[i] * (3.0 * (eF - uF) + 9.0 * eu * eF)
            post = self.f[i] - (self.f[i] - self.feq(i, n, u)) / tau + S
            # the lattice's buffer holds the post-collision values at their source
            self.f[i] = post if last else _at(post, tuple(-c for c in e))
        for _ in range(self.m):
            self.substep(u)

    def substep(self, u):
        p, phi, dt = self.p, self.phi, 1.0 / self.m
        tend = 0.0
        for a, e in enumerate(self.unit):
            b = tuple(-c for c in e)
            if self.case["flux"]:
                face = 0.5 * (u[a] + _at(u[a], e))  # between r and r + e
                J = torch.where(face > 0, face * phi, face * _at(phi, e))
                tend = tend + J - _at(J, b)
            else:
                du = self.diff(u[a], a) if self.case["stencil"] else 0.5 * (_at(u[a], e) - _at(u[a], b))
                up = torch.where(u[a] < 0, _at(phi, e) - phi, phi - _at(phi, b))
                tend = tend + phi * du + u[a] * up
        half = phi - dt * tend
        psi = p["a"] * half + p["b"] * phi ** 3 - p["kappa"] * self.lap1(half)
        self.phi = half + dt * p["Gamma"] * self.lap1(psi)

    def populations(self):
        s = F16_SCALE if self.case["precision"] == "f16" else 1.0
        return torch.stack([(f - w) * s for f, w in zip(self.f, self.w)])


def _network(case, params, x):
    for k, (W, b) in enumerate(params):
        y = b
        for dy in (-1, 0, 1):
            for dx in (-1, 0, 1):
                y = y + torch.roll(x, (-dy, -dx), (1, 2)) @ W[:, dy + 1, dx + 1, :].T
        x = torch.relu(y) if k < len(params) - 1 else y
    return x


def exact(case, seed):
    kind = case["kind"]
    if kind == "batch":
        return None  # hundreds of lattices over hundreds of steps
    if kind == "lattice":
        shape = (case["Lz"], case["Ly"], case["Lx"]) if case["Lz"] > 1 else (case["Ly"], case["Lx"])
        ref = _Exact(case, *_fields(shape, case["init"], _fluid(case), seed))
        for k in range(case["steps"]):
            ref.step(last=k == case["steps"] - 1)
        out = {"populations": ref.populations(), "phi": ref.phi}
        if case["diagnostics"]:
            out["observables"] = None
        return out
    scale = torch.tensor(OUT_STD, device="cuda", dtype=torch.float64)
    x0 = _states(case, seed)
    x = (x0.double() - torch.tensor(IN_MEAN, device="cuda")) / torch.tensor(IN_STD, device="cuda", dtype=torch.float64)
    params = [(W.double().cuda(), b.double().cuda()) for W, b in _weights(case, seed)]
    if kind == "forward":
        return x0.double() + scale * _network(case, params, x)
    target = (_targets(case, x0, seed).double() - x0.double()) / scale
    leaves = [t.requires_grad_(True) for W, b in params for t in (W, b)]
    loss = ((_network(case, params, x) - target) ** 2).mean()
    grads = torch.autograd.grad(loss, leaves)
    return {"loss": loss.item(), "gradients": torch.cat([g.reshape(-1) for g in grads])}
