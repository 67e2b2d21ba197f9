"""The work whose speed is measured: what a user of the library has it do, through its public entry points.

A pass of a device case is one bias point of a sweep as a user's program runs it from a checkpoint: the saved
polarization is put back, the electrodes are set, the initial Poisson solve runs (from a zero potential, as the paper
starts) and a few coupled TDGL + Poisson time steps follow.  The batched case does the same for 64 devices at once.
The network cases are the learned warm start's inference and one training step of it, and the TDGL case is the update
entry that allocates nothing.  Sizes, materials, biases and tolerances are those of the device workloads in
`paper_2210_15668_gb300.inputs`, of the tests and of the benchmark.

`exact` solves the same problems with plain torch in 64 bits: an FFT / tridiagonal direct solve where no carriers are
present, damped Newton with preconditioned conjugate gradients where they are, and the network without its 16-bit
rounding.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2210_15668_gb300 import ferrox, inputs

GPU = "cuda:0"
DT = inputs.DT_DEFAULT
FP64, MIXED = "fp64", "mixed"


# ---- the listed cases -------------------------------------------------------------------

def _device(name, stack, nx, ny, nz, precision, steps, v, guess=0, inner=1, tol=1e-10, order=1, points=0):
    return dict(name=name, kind="device", stack=stack, nx=nx, ny=ny, nz=nz, precision=precision, steps=steps, v=v,
                guess=guess, inner=inner, tol=tol, order=order, points=points)


def listed():
    return [
        # the smallest device of the workloads: a short Q-V sweep with its charges read back per point (launches and
        # latency count)
        _device("qv_64x64x16_fp64", "mfim", 64, 64, 16, FP64, 4, 0.5, points=3),
        # the benchmark's device in its headline form: FP64, the paper's guess, one V-cycle per residual check
        _device("mfim_256x256x32_fp64", "mfim", 256, 256, 32, FP64, 3, -2.0),
        # the same device with FP32 V-cycles inside the FP64 defect correction, the paper's order
        _device("mfim_256x256x32_mixed", "mfim", 256, 256, 32, MIXED, 4, -2.0),
        # the form a sweep over many bias points uses: extrapolated guess, V-cycles per residual chosen on the device
        _device("mfim_256x256x32_fast", "mfim", 256, 256, 32, MIXED, 6, -2.0, guess=1, inner=-8),
        # MFISM stacks (p-Si with Boltzmann carriers, damped Newton), four V-cycles per Newton residual
        _device("mfism_256x256x64_fast", "mfism", 256, 256, 64, MIXED, 4, 0.0, guess=1, inner=4),
        # the largest workload: 33.5 M cells
        _device("mfism_512x512x128_fast", "mfism", 512, 512, 128, MIXED, 2, 0.0, guess=1, inner=4),
        # a ragged MFISM device: lateral sizes that are no powers of two and an odd number of planes
        _device("mfism_96x80x37_mixed", "mfism", 96, 80, 37, MIXED, 4, -0.7),
        # the convergence study of the paper: undoped Si with Fermi-Dirac carriers, the second-order integrator, FP64
        _device("cube_64_order2_fp64", "cube", 64, 64, 64, FP64, 2, 0.0, tol=1e-11, order=2),
        # 64 independent devices of 32 to 128 cells a side at their own biases, advanced together
        dict(name="batch_64_mixed", kind="batch", count=64, layout=3, nz=16, precision=MIXED, steps=3, tol=1e-10),
        # the warm-start network on the coarse level of the 256 x 256 x 32 device, as every learned step runs it
        dict(name="nn_forward_8x64x64", kind="nn_forward", d=8, h=64, w=64),
        # loss, gradients and the Adam step of one snapshot of the 256 x 256 x 64 device
        dict(name="nn_train_16x64x64", kind="nn_train", d=16, h=64, w=64),
        # the polarization update alone, through the entry that allocates nothing, at the most cells it takes
        dict(name="tdgl_128x128x16", kind="tdgl", nx=128, ny=128, nz=16, ncomp=1, v=0.5),
    ]


# ---- drawn cases ------------------------------------------------------------------------

def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _coarsest(nx, ny, nz):
    """Cells left where no direction halves any more: what the coarsest grid of a multigrid has to solve."""
    can = lambda n: n % 2 == 0 and (n == 2 or n % 4 == 0)  # noqa: E731
    while can(nx) or can(ny) or nz % 2 == 0:
        nx, ny, nz = nx // 2 if can(nx) else nx, ny // 2 if can(ny) else ny, nz // 2 if nz % 2 == 0 else nz
    return nx * ny * nz


def _draw_size(rng, most_side, most_cells, nz_lo, nz_hi):
    while True:
        # devices are mostly about as wide as deep; half of them have sides that are multiples of 16
        side, ratio = _log_int(rng, 16, most_side), math.exp(rng.uniform(-0.7, 0.7))
        nx, ny = (max(16, min(most_side, 2 * round(side * r / 2))) for r in (math.sqrt(ratio), 1 / math.sqrt(ratio)))
        if rng.random() < 0.5:
            nx, ny = nx // 16 * 16, ny // 16 * 16
        nz = _log_int(rng, nz_lo, nz_hi)
        if nx * ny * nz <= most_cells and _coarsest(nx, ny, nz) <= 1000:
            return nx, ny, nz


def draw(rng):
    kind = rng.choice(["fp64", "mixed", "mixed", "fast", "fast", "mfism", "mfism", "cube", "batch", "batch", "nn_forward",
                       "nn_train", "tdgl"])
    if kind == "fp64":
        nx, ny, nz = _draw_size(rng, 256, 1 << 21, 13, 64)
        return _drawn("mfim", nx, ny, nz, FP64, rng.randint(2, 4), rng.uniform(-2, 2), points=rng.choice([0, 0, 2]))
    if kind == "mixed":
        nx, ny, nz = _draw_size(rng, 384, 1 << 22, 13, 64)
        return _drawn("mfim", nx, ny, nz, MIXED, rng.randint(2, 5), rng.uniform(-2, 2))
    if kind == "fast":
        nx, ny, nz = _draw_size(rng, 384, 1 << 22, 13, 64)
        return _drawn("mfim", nx, ny, nz, MIXED, rng.randint(3, 6), rng.uniform(-2, 2), guess=1, inner=rng.choice([-8, 4]))
    if kind == "mfism":
        nx, ny, nz = _draw_size(rng, 512, 1 << 24, 24, 128)
        return _drawn("mfism", nx, ny, nz, MIXED, rng.randint(2, 4), rng.uniform(-1, 1), guess=rng.choice([0, 1]),
                      inner=rng.choice([1, 4]))
    if kind == "cube":
        n = rng.choice([32, 48, 64, 80, 96])
        return _drawn("cube", n, n, n, FP64, rng.randint(1, 3), 0.0, tol=1e-11, order=rng.choice([1, 2]))
    if kind == "batch":
        return dict(kind="batch", count=_log_int(rng, 4, 64), layout=rng.randrange(100), nz=rng.choice([14, 16, 20, 24]),
                    precision=rng.choice([MIXED, MIXED, FP64]), steps=rng.randint(2, 4), tol=1e-10)
    if kind in ("nn_forward", "nn_train"):
        # mostly the coarse levels of devices of 64 to 512 cells a side; some whose sides the 8 x 16 tiles do not divide
        side = lambda: 16 * rng.choice([1, 2, 3, 4, 6, 8]) if rng.random() < 0.75 else 2 * rng.randint(4, 40)  # noqa: E731
        return dict(kind=kind, d=2 * rng.randint(2, 12), h=side(), w=side())
    while True:
        nx, ny, nz = 2 * _log_int(rng, 8, 128), 2 * _log_int(rng, 8, 128), _log_int(rng, 12, 64)
        if nx * ny * nz <= 262144:
            return dict(kind="tdgl", nx=nx, ny=ny, nz=nz, ncomp=rng.choice([1, 1, 3]), v=round(rng.uniform(-2, 2), 3))


def _drawn(stack, nx, ny, nz, precision, steps, v, **more):
    c = _device("", stack, nx, ny, nz, precision, steps, round(v, 3), **more)
    del c["name"]
    return c


# ---- preparing and running --------------------------------------------------------------

def _geometry(case):
    nx, ny, nz = case["nx"], case["ny"], case["nz"]
    if case.get("stack") == "cube":
        return inputs.convergence_cube(nx)
    if case.get("stack") == "mfism":
        return inputs.make_geometry(nx, ny, inputs.mfism_stack(nz))
    return inputs.make_geometry(nx, ny, inputs.mfim_stack(nz), ncomp=case.get("ncomp", 1))


def _random_p(geom, seed, amp=1e-3):
    """P[c][z][y][x], uniform in [-amp, amp] on ferroelectric planes, as the paper starts; made on the GPU."""
    g = torch.Generator(GPU)
    g.manual_seed(int(seed))
    fe = torch.from_numpy(inputs.fe_plane_mask(geom)).to(GPU)
    shape = (geom["ncomp"], inputs.nz_of(geom), geom["ny"], geom["nx"])
    p = torch.rand(shape, dtype=torch.float64, device=GPU, generator=g)
    p.mul_(2.0).sub_(1.0).mul_(amp)
    p[:, ~fe] = 0.0
    return p


def _layout(case):
    """Lateral sizes and biases of a batch's devices (part of the case: a program keeps them and changes the states)."""
    return inputs.batch_sweep(n=case["count"], seed=case["layout"], nz=case["nz"])


def _precision(case):
    return ferrox.MIXED if case["precision"] == MIXED else ferrox.FP64


def _net_inputs(case, seed):
    """Features as the solver makes them: the scaled residual, the planes' materials and height, the bias; a smooth target."""
    g = torch.Generator(GPU)
    g.manual_seed(int(seed))
    d, h, w = case["d"], case["h"], case["w"]
    x = torch.zeros((d, h, w, 16), dtype=torch.float32, device=GPU)
    x[..., 0] = torch.randn((d, h, w), generator=g, device=GPU)
    z = ((torch.arange(d, device=GPU) + 0.5) / d)[:, None, None]
    fe = (z > 0.68).float()
    x[..., 1] = fe + (1 - fe) * 0.1625
    x[..., 2] = fe
    x[..., 4] = z
    x[..., 5] = 2.0 * torch.rand((), generator=g, device=GPU) - 1.0
    t = torch.randn((d, h, w), generator=g, device=GPU)
    t = sum(torch.roll(t, s, a) for s in (-1, 0, 1) for a in (1, 2)) / 6.0
    return x.reshape(-1, 16).contiguous(), t.reshape(-1).contiguous()


def prepare(case, seed):
    kind = case["kind"]
    if kind == "device":
        geom = _geometry(case)
        num = ferrox.make_numerics(DT, order=case["order"], tol=case["tol"], precision=_precision(case), guess=case["guess"],
                                   inner=case["inner"])
        p0 = _random_p(geom, seed)
        return dict(case=case, p0=p0, dev=ferrox.Device(geom, np.zeros(p0.shape), num))
    if kind == "batch":
        inst = _layout(case)
        p0 = torch.cat([_random_p(q["geom"], 1000 * int(seed) + i).reshape(-1) for i, q in enumerate(inst)])
        num = ferrox.make_numerics(DT, tol=case["tol"], precision=_precision(case))
        shapes = [(1, inputs.nz_of(q["geom"]), q["geom"]["ny"], q["geom"]["nx"]) for q in inst]
        dev = ferrox.Batch([q["geom"] for q in inst], [np.zeros(s) for s in shapes], num)
        return dict(case=case, p0=p0, dev=dev, v=[q["v_top"] for q in inst])
    if kind == "tdgl":
        geom = _geometry(case)
        p0 = _random_p(geom, seed)
        g = torch.Generator(GPU)
        g.manual_seed(int(seed) + 1)
        phi = 1e-2 * torch.randn(p0.shape[1:], dtype=torch.float64, device=GPU, generator=g)
        return dict(case=case, geom=geom, p0=p0, p=p0.clone(), phi=phi)
    x, t = _net_inputs(case, seed)
    return dict(case=case, x=x, t=t, net=ferrox.NN(case["d"], case["h"], case["w"], params=_weights(seed)))


def _weights(seed):
    """He-normal weights and small biases of the network's six layers ([27][Cin][Cout] each)."""
    rng = np.random.default_rng(int(seed))
    ws, bs = [], []
    for ci, co in ferrox.NN_LAYERS:
        ws.append((rng.standard_normal((27, ci, co)) * math.sqrt(2.0 / (27 * ci))).astype(np.float32))
        bs.append((0.05 * rng.standard_normal(co)).astype(np.float32))
    return ws, bs


def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "device":
        dev = state["dev"]
        dev.P.copy_(state["p0"])
        dev.phi.zero_()
        dev.set_bias(0.0, case["v"])
        dev.solve_poisson()
        if not case["points"]:
            dev.step(case["steps"])
            return dict(P=dev.P, phi=dev.phi)
        q = dev.qv_sweep(_sweep(case), case["steps"])
        return dict(P=dev.P, phi=dev.phi, Q=[r["Q_int"] for r in q], V_fe=[r["V_fe"] for r in q])
    if kind == "batch":
        dev = state["dev"]
        dev.P.copy_(state["p0"])
        dev.phi.zero_()
        dev.set_bias(0.0, state["v"])
        dev.solve_poisson()
        dev.step(case["steps"])
        return dict(P=dev.P, phi=dev.phi)
    if kind == "tdgl":
        state["p"].copy_(state["p0"])
        ferrox.tdgl_update_static(state["geom"], DT, 0.0, case["v"], state["p"], state["phi"])
        return dict(P=state["p"])
    net = state["net"]
    if kind == "nn_forward":
        return dict(y=net.forward(state["x"]))
    loss = net.loss_grad(state["x"], state["t"])
    _, _, gw, gb = net.params()
    net.adam_step(1e-12)   # clears the gradients; the rate leaves the next pass the same weights
    return dict(loss=loss, gw=gw, gb=gb)


def _sweep(case):
    return [case["v"] * (i + 1) / case["points"] for i in range(case["points"])]


def work(case):
    """State read and written once; the operations of a multigrid solve: about 60 a cell and V-cycle, one V-cycle a decimal."""
    kind = case["kind"]
    if kind in ("nn_forward", "nn_train"):
        m = case["d"] * case["h"] * case["w"]
        macs = 27 * m * (16 * 16 + 16 * 16 + (16 * 32 + 32 * 32) / 8 + 48 * 16 + 16 * 16)
        weights = 27 * sum(ci * co for ci, co in ferrox.NN_LAYERS) * 4
        if kind == "nn_forward":
            return dict(bytes=m * 68 + weights, flops=2 * macs)
        return dict(bytes=m * 68 + 2 * weights, flops=6 * macs)
    if kind == "tdgl":
        fe = 10 * case["nx"] * case["ny"]
        return dict(bytes=fe * (16 * case["ncomp"] + 8), flops=fe * 40 * case["ncomp"])
    if kind == "batch":
        geoms = [q["geom"] for q in _layout(case)]
    else:
        geoms = [_geometry(case)]
    cells = sum(inputs.nz_of(g) * g["nx"] * g["ny"] for g in geoms)
    fe = sum(int(inputs.fe_plane_mask(g).sum()) * g["nx"] * g["ny"] for g in geoms)
    steps = case["steps"] * max(1, case.get("points", 0)) * case.get("order", 1)
    return dict(bytes=16 * fe + 8 * cells,
                flops=(steps + 1) * cells * 60.0 * -math.log10(case["tol"]) + steps * fe * 40.0)


# ---- the same in 64 bits, without the library -------------------------------------------

EPS0, QE, KB = 8.8541878128e-12, 1.602176634e-19, 1.380649e-23
H_PLANCK, M_E = 6.62607015e-34, 9.1093837015e-31


def _at():
    return "cuda:0" if torch.cuda.is_available() else "cpu"


class _Stack:
    """Per-plane data of a layered stack and the coupled model's discrete equations, in float64."""

    def __init__(self, geom):
        self.g, self.h = geom, geom["h"]
        self.of = [l for l in geom["layers"] for _ in range(l["ncells"])]
        self.nz = len(self.of)
        col = lambda k: torch.tensor([float(l[k]) for l in self.of], dtype=torch.float64, device=_at())[:, None, None]  # noqa: E731
        self.eps = EPS0 * col("eps_r")
        self.fe = torch.tensor([l["kind"] == inputs.FE for l in self.of], device=_at())
        self.sc = torch.tensor([l["kind"] == inputs.SC for l in self.of], device=_at())
        self.al, self.be, self.ga, self.g11, self.g44, self.kin = (col(k) for k in ("alpha", "beta", "gamma", "g11", "g44", "Gamma"))
        e, h = self.eps, self.h
        cz = torch.empty((self.nz + 1, 1, 1), dtype=torch.float64, device=_at())
        cz[0], cz[-1] = 2 * e[0] / h ** 2, 2 * e[-1] / h ** 2
        cz[1:-1] = 2 * e[:-1] * e[1:] / (e[:-1] + e[1:]) / h ** 2
        self.cz = cz
        lam = lambda n: (2 - 2 * torch.cos(2 * math.pi * torch.arange(n, dtype=torch.float64, device=_at()) / n)) / h ** 2  # noqa: E731
        nx, ny = geom["nx"], geom["ny"]
        self.mu = lam(ny)[:, None] + lam(nx)[None, : nx // 2 + 1]
        self.carriers = bool(self.sc.any())
        if self.carriers:
            self._carriers()

    def _carriers(self):
        l = next(q for q in self.of if q["kind"] == inputs.SC)
        self.net = l["N_D"] - l["N_A"]
        self.vt = KB * l["T"] / QE
        self.fd = l["stats"] == inputs.STATS_FERMI_DIRAC
        if not self.fd:
            root = math.sqrt(0.25 * self.net ** 2 + l["n_i"] ** 2)
            if self.net <= 0:
                self.p0 = -0.5 * self.net + root
                self.n0 = l["n_i"] ** 2 / self.p0
            else:
                self.n0 = 0.5 * self.net + root
                self.p0 = l["n_i"] ** 2 / self.n0
            return
        dos = lambda m: 2.0 * (2.0 * math.pi * m * M_E * KB * l["T"] / H_PLANCK ** 2) ** 1.5  # noqa: E731
        self.nc, self.nv = dos(l["m_e"]), dos(l["m_p"])
        gap = l["E_g"] * QE / (KB * l["T"])
        half = lambda e: float(self._half(torch.tensor(e, dtype=torch.float64))[0])  # noqa: E731
        lo, hi = -gap - 60.0, 60.0
        for _ in range(200):
            mid = 0.5 * (lo + hi)
            if self.nv * half(-gap - mid) - self.nc * half(mid) + self.net > 0:
                lo = mid
            else:
                hi = mid
        self.ee = 0.5 * (lo + hi)
        self.ep = -gap - self.ee

    @staticmethod
    def _half(eta):
        """The paper's approximation of the Fermi-Dirac integral of order 1/2, and its derivative."""
        g = torch.exp(-0.17 * (eta + 1) ** 2)
        w = 1 - 0.68 * g
        v = eta ** 4 + 50 + 33.6 * eta * w
        dv = 4 * eta ** 3 + 33.6 * w + 33.6 * eta * 0.68 * 0.34 * (eta + 1) * g
        xi = 0.75 * math.sqrt(math.pi) * v ** -0.375
        em = torch.exp(-eta)
        f = 1 / (em + xi)
        return f, (em + 0.375 * xi * dv / v) * f * f

    def charge(self, phi):
        """Carrier charge and minus its derivative on the semiconductor planes."""
        u = phi[self.sc] / self.vt
        if self.fd:
            n, dn = self._half(self.ee + u)
            p, dp = self._half(self.ep - u)
            n, dn, p, dp = self.nc * n, self.nc * dn, self.nv * p, self.nv * dp
        else:
            n, p = self.n0 * torch.exp(u), self.p0 * torch.exp(-u)
            dn, dp = n, p
        return QE * (p - n + self.net), QE * (dn + dp) / self.vt

    def rhs(self, p, v):
        """-div P and the electrodes' part; p: the components, the last one P_z."""
        e, pz = self.eps, p[-1]
        f = torch.empty((self.nz + 1,) + pz.shape[1:], dtype=torch.float64, device=pz.device)
        f[0], f[-1] = pz[0], pz[-1]
        f[1:-1] = (e[1:] * pz[:-1] + e[:-1] * pz[1:]) / (e[:-1] + e[1:])
        b = -(f[1:] - f[:-1]) / self.h
        b[-1] += 2 * e[-1] * v / self.h ** 2
        return b

    def apply(self, x):
        lat = 4 * x - torch.roll(x, 1, 1) - torch.roll(x, -1, 1) - torch.roll(x, 1, 2) - torch.roll(x, -1, 2)
        y = self.eps / self.h ** 2 * lat + (self.cz[:-1] + self.cz[1:]) * x
        y[1:] -= self.cz[1:-1] * x[:-1]
        y[:-1] -= self.cz[1:-1] * x[1:]
        return y

    def direct(self, f, shift=None):
        """(A + diag(shift of the plane))^-1 f: Fourier modes in x and y, one tridiagonal system in z per mode."""
        t = torch.fft.rfft2(f, dim=(1, 2))
        cz, c = self.cz.reshape(-1).tolist(), []
        eps = self.eps.reshape(-1).tolist()
        sh = [0.0] * self.nz if shift is None else shift.tolist()
        for k in range(self.nz):
            d = eps[k] * self.mu + (cz[k] + cz[k + 1] + sh[k])
            if k:
                d = d + cz[k] * c[-1]
                t[k] = (t[k] + cz[k] * t[k - 1]) / d
            else:
                t[k] = t[k] / d
            c.append(-cz[k + 1] / d)
        for k in range(self.nz - 2, -1, -1):
            t[k] -= c[k] * t[k + 1]
        return torch.fft.irfft2(t, s=f.shape[1:], dim=(1, 2))

    def solve(self, p, v, phi):
        b = self.rhs(p, v)
        if not self.carriers:
            x = self.direct(b)
            return x + self.direct(b - self.apply(x))
        best, last = phi.clone(), math.inf
        for _ in range(40):
            rho, s = self.charge(best)
            f = b - self.apply(best)
            f[self.sc] += rho
            norm = float(f.norm() / max(float(b.norm()), float(rho.norm())))
            if norm < 1e-15 or (norm < 1e-12 and norm > 0.5 * last):
                break
            last = norm
            best = best + self._newton(f, s).clamp_(-10 * self.vt, 10 * self.vt)
        return best

    def _newton(self, f, s):
        """(A + diag s) d = f by conjugate gradients, preconditioned with the planes' mean of s."""
        full = torch.zeros(self.nz, dtype=torch.float64, device=f.device)
        full[self.sc] = s.mean(dim=(1, 2))
        d, r = torch.zeros_like(f), f.clone()
        z = self.direct(r, full)
        q, rz, start = z.clone(), float((r * z).sum()), float(f.norm())
        for _ in range(60):
            aq = self.apply(q)
            aq[self.sc] += s * q[self.sc]
            a = rz / float((q * aq).sum())
            d += a * q
            r -= a * aq
            if float(r.norm()) < 1e-6 * start:
                break
            z = self.direct(r, full)
            rz, old = float((r * z).sum()), rz
            q = z + rz / old * q
        return d

    def force(self, p, phi, v):
        """dP/dt of the Landau-Ginzburg-Devonshire equation on ferroelectric cells, every component."""
        g, h, e = self.g, self.h, self.eps
        out = []
        for c in range(p.shape[0]):
            q = p[c]
            lat = (torch.roll(q, 1, 1) + torch.roll(q, -1, 1) + torch.roll(q, 1, 2) + torch.roll(q, -1, 2) - 4 * q) / h ** 2
            dz = torch.zeros_like(q)
            for k in range(self.nz):
                if not self.of[k]["kind"] == inputs.FE:
                    continue
                dn = k > 0 and self.of[k - 1]["kind"] == inputs.FE
                up = k + 1 < self.nz and self.of[k + 1]["kind"] == inputs.FE
                if dn and up:
                    dz[k] = (q[k + 1] - 2 * q[k] + q[k - 1]) / h ** 2
                else:
                    o = q[k + 1] if up else q[k - 1]
                    face = g["lam"] * (9 * q[k] - o) / (3 * h + 8 * g["lam"])
                    dz[k] = 4 * (o - 3 * q[k] + 2 * face) / (3 * h ** 2)
            if c == p.shape[0] - 1:
                f = torch.empty((self.nz + 1,) + phi.shape[1:], dtype=torch.float64, device=phi.device)
                f[0], f[-1] = 0.0, v
                f[1:-1] = ((e[:-1] * phi[:-1] + e[1:] * phi[1:]) - 0.5 * h * (q[1:] - q[:-1])) / (e[:-1] + e[1:])
                grad = (f[1:] - f[:-1]) / h
            else:
                a = 2 if c == 0 else 1
                up = 0.5 * (phi + torch.roll(phi, -1, a)) - 0.25 * h * (torch.roll(q, -1, a) - q) / e
                grad = (up - torch.roll(up, 1, a)) / h
            r = -self.kin * (self.al * q + self.be * q ** 3 + self.ga * q ** 5 - self.g44 * lat - self.g11 * dz + grad)
            r[~self.fe] = 0.0
            out.append(r)
        return torch.stack(out)

    def advance(self, p, phi, v, steps, order):
        for _ in range(steps):
            f0 = self.force(p, phi, v)
            q = p + DT * f0
            phi = self.solve(q, v, phi)
            if order == 2:
                q = p + 0.5 * DT * (f0 + self.force(q, phi, v))
                phi = self.solve(q, v, phi)
            p = q
        return p, phi

    def q_int(self, p, phi, v):
        """-<D_z> on the lowest ferroelectric plane's bottom face, and V minus the mean potential there."""
        k = int(torch.nonzero(self.fe)[0])
        el, er, h = float(self.eps[k - 1]), float(self.eps[k]), self.h
        pl, pr = p[-1][k - 1], p[-1][k]
        dz = -2 * el * er / (el + er) * (phi[k] - phi[k - 1]) / h + (er * pl + el * pr) / (el + er)
        face = ((el * phi[k - 1] + er * phi[k]) - 0.5 * h * (pr - pl)) / (el + er)
        return -float(dz.mean()), v - float(face.mean())


def _net(params, x, shape):
    """The U-Net in float64: 3x3x3 convolutions periodic in x and y and zero beyond z, mean pooling, repeated upsampling."""
    def conv(q, a, relu):
        w, b = params[q]
        ci, co = ferrox.NN_LAYERS[q]
        a = torch.nn.functional.pad(a, (1, 1, 1, 1, 0, 0), mode="circular")
        a = torch.nn.functional.pad(a, (0, 0, 0, 0, 1, 1))
        w = w.reshape(3, 3, 3, ci, co)
        d, h, v = a.shape[2] - 2, a.shape[3] - 2, a.shape[4] - 2
        y = b[None, :, None, None, None].expand(1, co, d, h, v)
        for i in range(27):
            dz, dy, dx = i // 9, i // 3 % 3, i % 3
            y = y + torch.einsum("nczyx,cd->ndzyx", a[:, :, dz:dz + d, dy:dy + h, dx:dx + v], w[dz, dy, dx])
        return torch.relu(y) if relu else y

    a = x.reshape(*shape, 16).permute(3, 0, 1, 2)[None]
    s = conv(1, conv(0, a, True), True)
    c = conv(3, conv(2, torch.nn.functional.avg_pool3d(s, 2), True), True)
    for axis in (2, 3, 4):
        c = c.repeat_interleave(2, axis)
    return conv(5, conv(4, torch.cat([c, s], 1), True), False)[0, 0].reshape(-1)


def exact(case, seed):
    kind = case["kind"]
    if kind in ("nn_forward", "nn_train"):
        x, t = (q.to(_at(), torch.float64) for q in _net_inputs(case, seed))
        ws, bs = _weights(seed)
        params = [tuple(torch.tensor(q, dtype=torch.float64, device=_at()).requires_grad_(kind == "nn_train") for q in wb)
                  for wb in zip(ws, bs)]
        y = _net(params, x, (case["d"], case["h"], case["w"]))
        if kind == "nn_forward":
            return dict(y=y)
        loss = ((y - t) ** 2).mean()
        loss.backward()
        return dict(loss=float(loss.detach()), gw=[w.grad.reshape(-1) for w, _ in params], gb=[b.grad for _, b in params])
    if kind == "tdgl":
        geom = _geometry(case)
        st = prepare(case, seed)
        return dict(P=st["p0"] + DT * _Stack(geom).force(st["p0"], st["phi"], case["v"]))
    if kind == "batch":
        outs = []
        for i, q in enumerate(_layout(case)):
            st = _Stack(q["geom"])
            p = _random_p(q["geom"], 1000 * int(seed) + i)
            phi = st.solve(p, q["v_top"], torch.zeros_like(p[0]))
            outs.append(st.advance(p, phi, q["v_top"], case["steps"], 1))
        return dict(P=torch.cat([o[0].reshape(-1) for o in outs]), phi=torch.cat([o[1].reshape(-1) for o in outs]))
    geom = _geometry(case)
    st = _Stack(geom)
    p = _random_p(geom, seed)
    phi = st.solve(p, case["v"], torch.zeros_like(p[0]))
    if not case["points"]:
        p, phi = st.advance(p, phi, case["v"], case["steps"], case["order"])
        return dict(P=p, phi=phi)
    charge = []
    for v in _sweep(case):
        p, phi = st.advance(p, phi, v, case["steps"], case["order"])
        charge.append(st.q_int(p, phi, v))
    return dict(P=p, phi=phi, Q=[q for q, _ in charge], V_fe=[v for _, v in charge])
