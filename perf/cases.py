"""The work that users of the library have it do, as cases that can be timed.

Every case goes through the calls of ``paper_2103_14588_gb300.binding``:

* ``apply``   one application of the operator A = D_w22 (FP64 or FP32) on a 1+1, 2+1 or 3+1 mesh;
* ``step``    one FP64 Arnoldi step that a caller composes from the library's calls: w = A v_last,
              h = V^H w, w -= V h and ||w||^2;
* ``solve``   a whole solve to a tight tolerance (FP64 GMRES, or FP32 inner cycles with FP64 refinement);
* ``sweep``   one application of the Crank-Nicolson sweep preconditioner;
* ``unet``    the learned correction's network, forward (inference) or loss and gradients (training).

``prepare`` makes the inputs on the GPU from a seed, ``run`` is one pass, ``work`` the bytes and
operations that a pass cannot do without, ``exact`` the result in 64 bits from torch alone.
"""

import math

import numpy as np
import torch
import torch.nn.functional as F

from paper_2103_14588_gb300 import binding as B

BC = {"periodic": B.DST_BC_PERIODIC, "open": B.DST_BC_OPEN, "dirichlet": B.DST_BC_DIRICHLET}
CHANNELS = (16, 32, 64)
# (input level, output level, kernel) of the network's convolutions in order; -1: the field's channels
CONVS = ((-1, 0, 3), (0, 0, 3), (0, 1, 3), (1, 1, 3), (1, 2, 3), (2, 2, 3), (2, 1, 1), (1, 1, 3), (1, 0, 1), (0, 0, 3), (0, -1, 1))


def listed():
    return [
        # The smallest call: the operator of the 64 x 64 plane-wave mesh in FP64, where the launch and the
        # host path count.
        dict(name="apply_1p1_f64_64", kind="apply", precision="f64", d=1, nx=64, ny=1, nz=1, nt=64, bcx="periodic",
             bcy="periodic", bcz="periodic", potential="none", tuned=False),
        # The FP32 operator of the 2+1 Zitterbewegung benchmark, applied once per inner Krylov step.
        dict(name="apply_2p1_f32_96", kind="apply", precision="f32", d=2, nx=96, ny=96, nz=1, nt=96, bcx="periodic",
             bcy="periodic", bcz="periodic", potential="none", tuned=True),
        # The FP32 operator of the 3+1 Klein-step benchmark (x walls, potential step along x).
        dict(name="apply_3p1_f32_48", kind="apply", precision="f32", d=3, nx=48, ny=48, nz=48, nt=48,
             bcx="dirichlet", bcy="periodic", bcz="periodic", potential="x", tuned=True),
        # The same operator in FP64: the refinement's residual and every step of the plain FP64 solve.
        dict(name="apply_3p1_f64_48", kind="apply", precision="f64", d=3, nx=48, ny=48, nz=48, nt=48,
             bcx="dirichlet", bcy="periodic", bcz="periodic", potential="x", tuned=True),
        # A mesh of odd sizes with an open axis, a wall axis and a potential that varies along both axes.
        dict(name="apply_2p1_f64_general", kind="apply", precision="f64", d=2, nx=61, ny=45, nz=1, nt=33, bcx="open",
             bcy="dirichlet", bcz="periodic", potential="general", tuned=False),
        # A caller's own FP64 Arnoldi iteration on the 2+1 benchmark mesh in the middle of a 30-vector cycle.
        dict(name="step_2p1_f64_96", kind="step", d=2, nx=96, ny=96, nz=1, nt=96, bcx="periodic", bcy="periodic",
             bcz="periodic", potential="none", nvec=15),
        # The plain solve with the library's default options (FP64 GMRES(30)): many short kernels.
        dict(name="solve_1p1_f64_64", kind="solve", problem="plane_wave", precision="f64", nx=64, nt=64, rtol=1e-10,
             inner_cycles=1, ortho=0),
        # The 2+1 Zitterbewegung benchmark, mixed precision with the benchmark's options.
        dict(name="solve_2p1_mixed_96", kind="solve", problem="packet", precision="mixed", nx=96, nt=96, rtol=1e-10,
             inner_cycles=4, ortho=2),
        # The headline's problem: the 3+1 Klein step, 10M complex unknowns, mixed precision with the benchmark's options.
        dict(name="solve_3p1_mixed_40", kind="solve", problem="klein", precision="mixed", nx=40, nt=40, rtol=1e-10,
             inner_cycles=4, ortho=2),
        # One preconditioner application inside flexible GMRES on the 3+1 Klein mesh.
        dict(name="sweep_3p1_48", kind="sweep", d=3, nx=48, ny=48, nz=48, nt=48, bcx="dirichlet", potential="x"),
        # One application of the learned correction's network on the 48^3 mesh on which the benchmark takes it.
        dict(name="unet_forward_2p1_48", kind="unet", backward=False, d=2, nx=48, ny=48, nt=48),
        # One training step's loss and gradients there.
        dict(name="unet_grad_2p1_48", kind="unet", backward=True, d=2, nx=48, ny=48, nt=48),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _around(rng, n, least):
    return max(least, int(round(n * rng.uniform(0.75, 1.25))))


def draw(rng):
    kind = rng.choice(["apply", "apply", "apply", "step", "solve", "solve", "sweep", "unet"])
    if kind in ("apply", "step"):
        d = rng.choice([1, 2, 3])
        n = _log_int(rng, *({1: (32, 2048), 2: (16, 160), 3: (8, 38)} if kind == "apply" else
                            {1: (32, 640), 2: (16, 64), 3: (8, 19)})[d])
        c = dict(kind=kind, d=d, nx=_around(rng, n, 4), ny=_around(rng, n, 4) if d > 1 else 1,
                 nz=_around(rng, n, 4) if d > 2 else 1, nt=_around(rng, n, 3))
        for k, axis in enumerate(("bcx", "bcy", "bcz")):
            c[axis] = rng.choice(["periodic", "periodic", "dirichlet", "open"]) if k < d else "periodic"
        c["potential"] = rng.choice(["none", "x", "x", "general"])
        if kind == "apply":
            c.update(precision=rng.choice(["f32", "f64"]), tuned=rng.random() < 0.5)
        else:
            c.update(nvec=rng.randint(1, 30))
        return c
    if kind == "solve":
        problem = rng.choice(["plane_wave", "packet", "klein"])
        n = _log_int(rng, *{"plane_wave": (24, 128), "packet": (20, 80), "klein": (8, 28)}[problem])
        precision = "mixed" if problem != "plane_wave" and n > 24 else rng.choice(["f64", "mixed"])
        return dict(kind=kind, problem=problem, precision=precision, nx=n, nt=_around(rng, n, 4), rtol=1e-10,
                    inner_cycles=rng.choice([1, 4]), ortho=rng.choice([0, 2]))
    if kind == "sweep":
        d = rng.choice([1, 2, 2, 3])
        n = _log_int(rng, *{1: (32, 256), 2: (16, 96), 3: (8, 38)}[d])
        bcx = "dirichlet" if d == 3 else rng.choice(["periodic", "dirichlet"])
        return dict(kind=kind, d=d, nx=_around(rng, n, 4), ny=_around(rng, n, 4) if d > 1 else 1,
                    nz=_around(rng, n, 4) if d > 2 else 1, nt=_around(rng, n, 3), bcx=bcx,
                    potential="x" if bcx == "dirichlet" else "none")
    d = rng.choice([1, 2])
    n = _log_int(rng, *{1: (32, 256), 2: (12, 40)}[d])
    return dict(kind="unet", backward=rng.random() < 0.5, d=d, nx=_around(rng, n, 8),
                ny=_around(rng, n, 8) if d > 1 else 1, nt=_around(rng, n, 8))


# ---- meshes and physical inputs ---------------------------------------------


class Box:
    """A mesh description and its physical inputs, all from the case and the seed."""

    def __init__(self, case, seed):
        rng = np.random.default_rng(seed)
        kind = case["kind"]
        if kind == "solve":
            self._problem(case, rng)
        else:
            self.d = case["d"]
            self.n_el = [case["nx"], case["ny"], case.get("nz", 1), case["nt"]]
            self.lo, self.hi = [-6.0, -6.0, -6.0, 0.0], [6.0, 6.0, 6.0, 3.0]
            self.bc = [case.get("bcx", "periodic"), case.get("bcy", "periodic"), case.get("bcz", "periodic")]
            self.m = 1.0 + 0.2 * rng.random()
            self.psi0 = None
            shape = tuple(self.n_el[k] if k < self.d else 1 for k in (2, 1, 0))
            pot = case.get("potential", "none")
            if pot == "x":        # the Klein step
                cx = self.lo[0] + (np.arange(self.n_el[0]) + 0.5) * (self.hi[0] - self.lo[0]) / self.n_el[0]
                self.V = np.broadcast_to(np.where(cx >= 0, 2.5 + rng.random(), 0.0), shape).ravel().copy()
            elif pot == "general":
                self.V = rng.uniform(-1.0, 2.0, shape).ravel()
            else:
                self.V = None
        self.nc = 4 if self.d == 3 else 2
        self.h = [(self.hi[k] - self.lo[k]) / self.n_el[k] for k in range(4)]
        self.nodes = []
        for k in range(3):
            extra = {"periodic": 0, "open": 1, "dirichlet": -1}[self.bc[k]]
            self.nodes.append(self.n_el[k] + extra if k < self.d else 1)
        self.nt = self.n_el[3]
        self.shape = (self.nt, self.nodes[2], self.nodes[1], self.nodes[0], self.nc)
        self.n = int(np.prod(self.shape))

    def _problem(self, case, rng):
        n, nt, problem = case["nx"], case["nt"], case["problem"]
        per = "periodic"
        if problem == "plane_wave":      # a momentum eigenstate on a periodic axis
            self.d, self.n_el, self.bc = 1, [n, 1, 1, nt], [per] * 3
            self.lo, self.hi, self.m, self.V = [0.0] * 4, [2 * math.pi, 1.0, 1.0, 1.0], 1.0 + 0.2 * rng.random(), None
            k, x = 1.0, 2 * math.pi * np.arange(n) / n
            e = math.sqrt(k * k + self.m ** 2)
            up = np.array([e + self.m, k]) / math.sqrt(2 * e * (e + self.m))
            self.psi0 = (np.exp(1j * k * x + 2j * math.pi * rng.random())[:, None] * up).reshape(1, 1, n, 2)
            return
        if problem == "packet":          # a Zitterbewegung packet of positive- and negative-energy spinors
            self.d, self.n_el, self.bc = 2, [n, n, 1, nt], [per] * 3
            self.lo, self.hi, self.m, self.V = [-8.0, -8.0, 0.0, 0.0], [8.0, 8.0, 1.0, 4.0], 1.0, None
            x = -8.0 + 16.0 * np.arange(n) / n
            px = 2.0
            e = math.sqrt(px * px + 1)
            up = np.array([e + 1, px]) / math.sqrt(2 * e * (e + 1))
            um = np.array([-px, e + 1]) / math.sqrt(2 * e * (e + 1))
            env = np.exp(-(x[None, :] ** 2 + x[:, None] ** 2) + 1j * px * x[None, :])
            psi = env[..., None] * (up + np.exp(2j * math.pi * rng.random()) * um)
            self.psi0 = (psi / np.sqrt(np.sum(np.abs(psi) ** 2) * (16.0 / n) ** 2))[None]
            return
        # the Klein step: a packet in x, uniform in y and z, that meets a step between x walls
        self.d, self.n_el, self.bc = 3, [n, n, n, nt], ["dirichlet", per, per]
        self.lo, self.hi, self.m = [-6.0, -6.0, -6.0, 0.0], [6.0, 6.0, 6.0, 3.0], 1.0
        p0 = 1.0 + 2.0 * rng.random()
        x = -6.0 + 12.0 * np.arange(1, n) / n
        e = math.sqrt(p0 * p0 + 1)
        up = np.array([e + 1, 0.0, 0.0, p0]) / math.sqrt(2 * e * (e + 1))
        env = np.exp(-(x + 2.0) ** 2 + 1j * p0 * x)
        psi = np.broadcast_to(env[None, None, :, None] * up, (n, n, n - 1, 4))
        self.psi0 = psi / np.sqrt(np.sum(np.abs(psi) ** 2) * (12.0 / n) ** 3)
        cx = -6.0 + 12.0 * (np.arange(n) + 0.5) / n
        self.V = np.broadcast_to(np.where(cx >= 0, 2.5, 0.0), (n, n, n)).ravel().copy()

    def mesh(self):
        return B.Mesh(self.d, self.n_el, self.lo, self.hi, [BC[b] for b in self.bc], m=self.m, V=self.V, psi0=self.psi0)

    def field(self, seed, dtype, count=1):
        """Vectors such as a Krylov basis holds: noise under a packet's envelope, whose far tails are small."""
        g = torch.Generator(device="cuda").manual_seed(seed)
        env = torch.ones((), dtype=torch.float64, device="cuda")
        for axis, n in ((1, self.shape[1]), (2, self.shape[2]), (3, self.shape[3])):
            u = torch.linspace(-1.0, 1.0, n, dtype=torch.float64, device="cuda") if n > 1 else torch.zeros(1, dtype=torch.float64, device="cuda")
            sz = [1] * 5
            sz[axis] = n
            env = env * torch.exp(-4.0 * (u - 0.2) ** 2).view(sz)
        real = torch.float64 if dtype == torch.complex128 else torch.float32
        out = torch.empty((count,) + self.shape, dtype=dtype, device="cuda")
        for j in range(count):
            v = torch.randn(self.shape + (2,), generator=g, dtype=real, device="cuda")
            out[j] = torch.view_as_complex(v) * env.to(real)
            out[j] /= torch.linalg.vector_norm(out[j])
        return out.view(count, self.n)


def prepare(case, seed):
    if case["kind"] == "unet":
        box = Box(dict(case, potential="none"), seed)
        mesh = box.mesh()
        net = B.UNet(mesh.handle)
        net.set_params(_parameters(case, seed))
        s = dict(case=case, mesh=mesh, net=net, x=box.field(seed + 1, torch.complex64)[0])
        if case["backward"]:
            s["target"] = box.field(seed + 2, torch.complex64)[0]
        else:
            s["y"] = torch.empty_like(s["x"])
        return s
    box = Box(case, seed)
    mesh = box.mesh()
    s = dict(case=case, mesh=mesh)
    if case["kind"] == "apply":
        if case["tuned"]:
            B.dst_tune_apply(mesh.handle)
        s["x"] = box.field(seed + 1, torch.complex128 if case["precision"] == "f64" else torch.complex64)[0]
        s["y"] = torch.empty_like(s["x"])
    elif case["kind"] == "step":
        s["V"] = _orthonormal(box.field(seed + 1, torch.complex128, case["nvec"]))
        s["w"] = torch.empty(box.n, dtype=torch.complex128, device="cuda")
        s["h"] = torch.empty(case["nvec"], dtype=torch.complex128, device="cuda")
        s["nrm2"] = torch.empty(1, dtype=torch.float64, device="cuda")
    elif case["kind"] == "solve":
        s["psi"] = torch.zeros(box.n, dtype=torch.complex128, device="cuda")
        s["opts"] = {"restart": 30, "rtol": case["rtol"], "max_iters": 20000, "ortho": case["ortho"]}
        if case["precision"] == "mixed":
            s["opts"].update(mixed_precision=1, inner_rtol=1e-4, inner_cycles=case["inner_cycles"])
    else:
        s["v"] = box.field(seed + 1, torch.complex64)[0]
        s["z"] = torch.empty_like(s["v"])
    return s


def run(s):
    case, mesh = s["case"], s["mesh"].handle
    kind = case["kind"]
    if kind == "apply":
        B.dst_apply_operator(mesh, B.DST_FP64 if case["precision"] == "f64" else B.DST_FP32, s["x"], s["y"])
        return s["y"]
    if kind == "step":
        n, k = s["w"].numel(), case["nvec"]
        B.dst_apply_operator(mesh, B.DST_FP64, s["V"][k - 1], s["w"])
        B.dst_arnoldi_project(n, k, s["V"], s["w"], s["h"])
        B.dst_arnoldi_update(n, k, s["V"], s["h"], s["w"], s["nrm2"])
        return {"h": s["h"], "w": s["w"], "nrm2": s["nrm2"]}
    if kind == "solve":
        B.dst_solve(mesh, s["opts"], s["psi"])
        return s["psi"]
    if kind == "sweep":
        B.dst_precond_apply(mesh, B.DST_PRECOND_CN_SWEEP, s["v"], s["z"])
        return s["z"]
    if case["backward"]:
        loss, grad = s["net"].loss_grad(s["x"], s["target"])
        return {"loss": loss, "grad": grad}
    s["net"].forward(s["x"], s["y"])
    return s["y"]


def work(case):
    box = Box(dict(case, potential=case.get("potential", "none")), 0)
    n, d = box.n, box.d
    # sum-factorised operator: x stencils, y and z passes, spin combination, time stencils, potential
    apply_flops = n * ({1: 26, 2: 44, 3: 68}[d] + (0 if box.V is None else {1: 10, 2: 16, 3: 22}[d]))
    kind = case["kind"]
    if kind == "apply":
        return {"bytes": n * (32 if case["precision"] == "f64" else 16), "flops": apply_flops}
    if kind == "step":
        return {"bytes": 16 * n * (case["nvec"] + 1), "flops": apply_flops + 16 * n * case["nvec"] + 4 * n}
    if kind == "solve":
        return {"bytes": 16 * (n + n // box.nt), "flops": apply_flops}
    if kind == "sweep":
        # layer solves (2 x 2 or 4 x 4 blocks), the time recurrences and two FFTs of each plane
        return {"bytes": 16 * n, "flops": n * (16 * box.nc + 20 + 10 * math.log2(max(2, case["ny"] * case["nz"])))}
    flops = 0
    for cin, cout, k in CONVS:
        ci, co = (2 * box.nc if c < 0 else CHANNELS[c] for c in (cin, cout))
        level = 2 if (cin, cout) in ((1, 2), (2, 2)) else 1 if cout == 1 else 0
        cells = box.nt * box.nodes[0] * box.nodes[1] / 2 ** ((d + 1) * level)
        flops += 2 * cells * ci * co * k ** (d + 1)
    p = _parameters(case, 0).size
    if case["backward"]:
        return {"bytes": 16 * n + 8 * p, "flops": 3 * flops}
    return {"bytes": 16 * n + 4 * p, "flops": flops}


# ---- exact results in 64 bits -------------------------------------------------


def exact(case, seed):
    if case["kind"] == "unet":
        return _exact_unet(case, seed)
    box = Box(case, seed)
    if case["kind"] == "apply":
        x = box.field(seed + 1, torch.complex128 if case["precision"] == "f64" else torch.complex64)[0]
        return _operator(box, x.to(torch.complex128))
    if case["kind"] == "step":
        V = _orthonormal(box.field(seed + 1, torch.complex128, case["nvec"]))
        w = _operator(box, V[-1])
        h = V.conj() @ w
        w = w - h @ V
        return {"h": h, "w": w, "nrm2": torch.linalg.vector_norm(w).square().view(1)}
    if case["kind"] == "solve":
        return _exact_packet(box) if case["problem"] == "packet" else _exact_line(box)
    return _exact_sweep(box, box.field(seed + 1, torch.complex64)[0].to(torch.complex128))


def _orthonormal(V):
    """Rows made orthonormal by a Cholesky factor of their Gram matrix."""
    L = torch.linalg.cholesky(V.conj() @ V.T)
    return torch.linalg.solve_triangular(L.conj(), V, upper=False).contiguous()


def _axis(n_el, h, bc, weight=None):
    """1D Q1 mass matrix (of a weight per element) and convection matrix on the unknown nodes."""
    e = np.arange(n_el)
    a, b = e, (e + 1) % n_el if bc == "periodic" else e + 1
    size = n_el if bc == "periodic" else n_el + 1
    w = np.ones(n_el) if weight is None else weight
    M, C = np.zeros((size, size)), np.zeros((size, size))
    for i, j, mass, conv in ((a, a, 2, -0.5), (a, b, 1, 0.5), (b, a, 1, -0.5), (b, b, 2, 0.5)):
        np.add.at(M, (i, j), w * h * mass / 6)
        np.add.at(C, (i, j), conv)
    cut = slice(1, n_el) if bc == "dirichlet" else slice(None)
    return M[cut, cut], C[cut, cut]


def _times(h, nt):
    """Time stencils over the layers 0..N_t: (mass, convection), rows of the unknown layers 1..N_t."""
    M, C = _axis(nt, h, "open")
    return M[1:], C[1:]


def _spin(d):
    s = [np.array([[0, 1], [1, 0]], complex), np.array([[0, -1j], [1j, 0]]), np.array([[1, 0], [0, -1]], complex)]
    if d < 3:
        return s[:d], s[2]
    z = np.zeros((2, 2))
    return [np.block([[z, a], [a, z]]) for a in s], np.diag([1, 1, -1, -1]).astype(complex)


def _on(A, x, axis):
    """A (dense, or None for the identity) applied along one axis of x."""
    if A is None:
        return x
    A = torch.as_tensor(A, dtype=x.dtype, device=x.device)
    return torch.movedim(torch.tensordot(A, x, dims=([1], [axis])), 0, axis)


def _operator(box, v):
    """A v: i D^t + i sum_k alpha_k D^k - (m beta + V) D^0."""
    x = v.view(box.shape)
    ax = [_axis(box.n_el[k], box.h[k], box.bc[k]) if k < box.d else (None, None) for k in range(3)]
    Mt, Ct = (A[:, 1:] for A in _times(box.h[3], box.nt))
    alpha, beta = _spin(box.d)

    def space(conv):
        y = x
        for k in range(box.d):
            y = _on(ax[k][1 if k == conv else 0], y, 3 - k)
        return y

    mass = space(-1)
    y = 1j * _on(Ct, mass, 0)
    in_time = -box.m * _on(beta, mass, 4)
    for k in range(box.d):
        in_time = in_time + 1j * _on(alpha[k], space(k), 4)
    if box.V is not None:
        in_time = in_time - _weighted(box, x)
    return (y + _on(Mt, in_time, 0)).reshape(-1)


def _weighted(box, x):
    """The mass of a potential that is constant on each spatial element, corner pair by corner pair."""
    full = [box.n_el[k] + (box.bc[k] != "periodic") if k < box.d else 1 for k in range(3)]
    cut = [slice(1, box.n_el[k]) if box.bc[k] == "dirichlet" else slice(None) for k in range(3)]
    u = torch.zeros((box.nt, full[2], full[1], full[0], box.nc), dtype=x.dtype, device=x.device)
    u[:, cut[2], cut[1], cut[0]] = x
    out = torch.zeros_like(u)
    V = torch.as_tensor(box.V, device=x.device).view([box.n_el[k] if k < box.d else 1 for k in (2, 1, 0)])

    def corner(bits):
        return [(torch.arange(box.n_el[k], device=x.device) + (bits >> k & 1)) % full[k] if k < box.d
                else torch.zeros(1, dtype=torch.long, device=x.device) for k in (2, 1, 0)]

    for a in range(1 << box.d):
        acc = 0
        for b in range(1 << box.d):
            w = 1.0
            for k in range(box.d):
                w *= box.h[k] / 6 * (2 if (a ^ b) >> k & 1 == 0 else 1)
            z, y, c = corner(b)
            acc = acc + w * V[None, :, :, :, None] * u[:, z[:, None, None], y[None, :, None], c[None, None, :]]
        z, y, c = corner(a)
        _scatter(out, z, y, c, acc)
    return out[:, cut[2], cut[1], cut[0]]


def _scatter(out, z, y, c, acc):
    """out[:, z, y, c] += acc."""
    plane = (z[:, None, None] * out.shape[2] + y[None, :, None]) * out.shape[3] + c[None, None, :]
    out.view(out.shape[0], -1, out.shape[4]).index_add_(1, plane.reshape(-1), acc.reshape(acc.shape[0], -1, acc.shape[4]))


def _solve_line(Mx, Cx, Wp, Wm, Mt, Ct, first):
    """Two components over x and t: rows (t, x, c); Wp, Wm: the masses of m + V and V - m."""
    nt, nx = Mt.shape[0], Mx.shape[0]
    Z = np.zeros_like(Mx)
    K = np.block([[-Wp + 0j, 1j * Cx], [1j * Cx, -Wm + 0j]])     # rows (c, x)
    Ms = np.block([[Mx, Z], [Z, Mx]])
    dev = "cuda"
    t = lambda a: torch.as_tensor(a, dtype=torch.complex128, device=dev)
    A = torch.kron(t(1j * Ct[:, 1:]), t(Ms)) + torch.kron(t(Mt[:, 1:]), t(K))
    b = -(torch.kron(t(1j * Ct[:, :1]), t(Ms)) + torch.kron(t(Mt[:, :1]), t(K))) @ t(first.T.reshape(-1, 1))
    return torch.linalg.solve(A, b).view(nt, 2, nx).permute(0, 2, 1)


def _exact_line(box):
    """The solution of data uniform in y and z: the two-component problem over x and t."""
    n = box.n_el[0]
    if box.n // box.nt // max(1, box.nodes[1] * box.nodes[2]) * box.nt > 13000:
        return None
    V = np.zeros(n) if box.V is None else box.V.reshape(-1, n)[0]
    Mx, Cx = _axis(n, box.h[0], box.bc[0])
    Wp, Wm = (_axis(n, box.h[0], box.bc[0], V + s * box.m)[0] for s in (1, -1))
    Mt, Ct = _times(box.h[3], box.nt)
    comps = [0, 3] if box.d == 3 else [0, 1]
    x = _solve_line(Mx, Cx, Wp, Wm, Mt, Ct, np.ascontiguousarray(box.psi0[0, 0][:, comps]))
    if box.d == 1:
        return x.reshape(-1)
    out = torch.zeros(box.shape, dtype=torch.complex128, device=x.device)
    out[..., comps] = x[:, None, None]
    return out.view(-1)


def _exact_packet(box):
    """Periodic mesh without potential: a small dense system over t for each frequency."""
    n, nt = box.n_el[0], box.nt
    th = 2 * math.pi * torch.arange(n, dtype=torch.float64, device="cuda") / n
    m1, s1 = box.h[0] * (2 + torch.cos(th)) / 3, torch.sin(th)
    mass = (m1[:, None] * m1[None, :]).reshape(-1)
    sx, sy = (m1[:, None] * s1[None, :]).reshape(-1), (s1[:, None] * m1[None, :]).reshape(-1)
    (ax, ay), beta = _spin(2)
    t = lambda a: torch.as_tensor(a, dtype=torch.complex128, device="cuda")
    # i alpha_k (i sin) - m beta mass
    K = -sx[:, None, None] * t(ax) - sy[:, None, None] * t(ay) - box.m * mass[:, None, None] * t(beta)
    Ms = mass[:, None, None] * t(np.eye(2))
    Mt, Ct = (t(a) for a in _times(box.h[3], nt))
    f = torch.fft.fft2(t(box.psi0[0]), dim=(0, 1)).reshape(-1, 2, 1)
    out = torch.empty((n * n, nt, 2), dtype=torch.complex128, device="cuda")
    step = max(1, int(2e9 / (16 * (2 * nt) ** 2)))
    for at in range(0, n * n, step):
        k, ms = K[at:at + step], Ms[at:at + step]
        A = torch.einsum("ts,fcd->ftcsd", 1j * Ct[:, 1:], ms) + torch.einsum("ts,fcd->ftcsd", Mt[:, 1:], k)
        b = -(torch.einsum("t,fcd->ftcd", 1j * Ct[:, 0], ms) + torch.einsum("t,fcd->ftcd", Mt[:, 0], k))
        b = (b.reshape(len(k), 2 * nt, 2) @ f[at:at + step])
        out[at:at + step] = torch.linalg.solve(A.reshape(len(k), 2 * nt, 2 * nt), b).view(-1, nt, 2)
    out = torch.fft.ifft2(out.view(n, n, nt, 2), dim=(0, 1))
    return out.permute(2, 0, 1, 3).reshape(-1)


def _exact_sweep(box, v):
    """B^-1 S^-1 v: layers averaged backwards in time, then the Crank-Nicolson march, frequency by frequency."""
    s = v.view(box.shape).clone()
    s[-1] *= 2
    for t in range(box.nt - 2, -1, -1):
        s[t] = 2 * s[t] - s[t + 1]
    s = torch.fft.fftn(s, dim=(1, 2))
    n, nc = box.n_el[0], box.nc
    V = np.zeros(n) if box.V is None else box.V.reshape(-1, n)[0]
    Mx, Cx = _axis(n, box.h[0], box.bc[0])
    Vx = _axis(n, box.h[0], box.bc[0], V)[0]
    alpha, beta = _spin(box.d)
    dev = v.device
    t_ = lambda a: torch.as_tensor(a, dtype=torch.complex128, device=dev)
    sym = []
    for k in (1, 2):
        th = 2 * math.pi * torch.arange(box.nodes[k], dtype=torch.float64, device=dev) / box.nodes[k]
        sym.append((box.h[k] * (2 + torch.cos(th)) / 3, torch.sin(th)) if k < box.d else (torch.ones_like(th), torch.zeros_like(th)))
    my, sy = (a[None, :].expand(box.nodes[2], -1).reshape(-1, 1, 1) for a in sym[0])
    mz, sz = (a[:, None].expand(-1, box.nodes[1]).reshape(-1, 1, 1) for a in sym[1])
    kron = lambda a, b: torch.kron(t_(a), t_(b))[None]
    eye = np.eye(nc)
    K = my * mz * (kron(1j * Cx, alpha[0]) - kron(box.m * Mx, beta) - kron(Vx, eye))
    if box.d > 1:
        K = K - sy * mz * kron(Mx, alpha[1])
    if box.d > 2:
        K = K - my * sz * kron(Mx, alpha[2])
    M = 1j * my * mz * kron(Mx, eye)
    LU = torch.linalg.lu_factor(M + 0.5 * box.h[3] * K)
    low = -M + 0.5 * box.h[3] * K
    f = s.reshape(box.nt, box.nodes[2] * box.nodes[1], box.nodes[0] * nc, 1)
    x = torch.zeros_like(f[0])
    for t in range(box.nt):
        x = torch.linalg.lu_solve(*LU, f[t] - low @ x)
        f[t] = x
    return torch.fft.ifftn(f.view(box.shape), dim=(1, 2)).reshape(-1)


# ---- the network ----------------------------------------------------------------


def _shapes(d):
    C = 4 if d < 3 else 8
    for cin, cout, k in CONVS:
        ci, co = (C if c < 0 else CHANNELS[c] for c in (cin, cout))
        yield (co, ci) + (k,) * (d + 1)


def _parameters(case, seed):
    """The flat parameter vector a training starts from: He-normal weights, small biases."""
    rng, out = np.random.default_rng(seed + 3), []
    for shape in _shapes(case["d"]):
        fan_in = int(np.prod(shape[1:]))
        out += [rng.standard_normal(shape).ravel() * math.sqrt(2.0 / fan_in), 0.1 * rng.standard_normal(shape[0])]
    return np.concatenate(out).astype(np.float32)


def _exact_unet(case, seed):
    box = Box(dict(case, potential="none"), seed)
    d, dev = case["d"], "cuda"
    flat = torch.as_tensor(_parameters(case, seed), device=dev).double().requires_grad_(case["backward"])
    grid = (box.nt,) + ((box.nodes[1],) if d == 2 else ()) + (box.nodes[0],)
    conv = F.conv2d if d == 1 else F.conv3d

    def to_grid(v):
        return torch.movedim(torch.view_as_real(v.to(torch.complex128)).reshape(grid + (2 * box.nc,)), -1, 0)[None]

    layers, at = [], 0
    for shape in _shapes(d):
        size = int(np.prod(shape))
        layers.append((flat[at:at + size].view(shape), flat[at + size:at + size + shape[0]]))
        at += size + shape[0]

    def c(i, x):
        w, b = layers[i]
        return conv(x, w, b, padding=w.shape[2] // 2)

    def pool(x):
        pad = []
        for n in reversed(x.shape[2:]):
            pad += [0, n % 2]
        return (F.avg_pool2d if d == 1 else F.avg_pool3d)(F.pad(x, pad), 2)

    def up(x, like):
        for k, n in enumerate(like.shape[2:]):
            x = x.repeat_interleave(2, dim=2 + k).narrow(2 + k, 0, n)
        return x

    v = box.field(seed + 1, torch.complex64)[0]
    norm = torch.linalg.vector_norm(v.to(torch.complex128))
    with torch.backends.cudnn.flags(enabled=False):
        s1 = F.relu(c(1, F.relu(c(0, to_grid(v) / norm))))
        s2 = F.relu(c(3, F.relu(c(2, pool(s1)))))
        h = F.relu(c(5, F.relu(c(4, pool(s2)))))
        h = F.relu(c(7, c(6, up(h, s2)) + s2))
        y = c(10, F.relu(c(9, c(8, up(h, s1)) + s1)))
        if not case["backward"]:
            y = torch.movedim(y[0], 0, -1).reshape(-1, 2).contiguous() * norm
            return torch.view_as_complex(y).reshape(-1)
        t = to_grid(box.field(seed + 2, torch.complex64)[0]) / norm
        loss = (y - t).square().sum() / t.square().sum()
        (grad,) = torch.autograd.grad(loss, flat)
    return {"loss": loss.detach(), "grad": grad}
