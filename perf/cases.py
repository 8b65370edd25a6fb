"""The work that users of this framework have it do, as cases to be measured.

A simulation pass is what a user's program repeats until its run is over:
some time steps through the public binding, then the observables of the new
state.  The state goes on from pass to pass, as in a run.  The other cases
are a checkpoint restart (populations in, steps, populations out) and the
gradient of the learned closure's training loss.

Fields are built on the GPU from the seed alone; species constants and
transport inputs come from the repository's recipes (workloads.py).  `exact`
restates the method in 64-bit torch: equilibria as full populations,
propagation by rolls, gradients by the 26-point sum, no stored deviations.
FP32 and 16-bit handles compute in FP32, so their observables, which cross
the interface as float64, are returned as the float32 values they carry.
"""

from __future__ import annotations

import math
import types

import numpy as np
import torch

from paper_2004_11286_gb300 import binding, workloads as W

F64 = torch.float64


def _case(name, kind, shape, precision, steps, **kw):
    nz, ny, nx = shape
    c = dict(kind=kind, nz=nz, ny=ny, nx=nx, precision=precision, steps=steps)
    c.update(kw)
    if name:
        c["name"] = name
    return c


def listed():
    return [
        # The ternary uphill-diffusion tube in the parity mode: a thousand nodes, latency and launches.
        _case("tube_fp64", "tube", (4, 4, 64), "fp64", 20),
        # The closed Loschmidt tube (Sec. 4.2), tens of thousands of steps on a line of nodes.
        _case("loschmidt_fp32", "loschmidt", (1, 1, 96), "fp32", 20),
        # The planar opposed jets (Sec. 4.3) at the paper's size, four species, with their boundary set.
        _case("jets_fp32", "jets", (1, 400, 200), "fp32", 20),
        # The sound-speed box (Sec. 4.4).
        _case("pulse_fp32", "pulse", (128, 128, 128), "fp32", 20),
        # The Kelvin-Helmholtz flow (Sec. 4.5) at the benchmark's grid, plain FP32.
        _case("layers_fp32", "layers", (256, 256, 256), "fp32", 10),
        # The same flow with 16-bit storage.
        _case("layers_bf16", "layers", (256, 256, 256), "bf16", 10),
        # A ternary mixture on a ragged grid (rows of no multiple of anything).
        _case("ternary_ragged_fp32", "mixture", (45, 75, 101), "fp32", 20, M=3),
        # The eight-species mixture, plain FP32, and at the configured size with 16-bit storage.
        _case("mixture8_fp32", "mixture", (128, 128, 128), "fp32", 8, M=8),
        _case("mixture8_bf16", "mixture", (192, 192, 192), "bf16", 4, M=8),
        # The batched ensemble of uneven ternary domains, edges 32..96.
        _case("ensemble_bf16", "ensemble", (32, 64, 96), "bf16", 8, domains=16),
        # A restart: populations loaded, a short run, populations saved (FP16 storage).
        _case("restart_fp16", "restart", (96, 96, 96), "fp16", 20),
        # One mini-batch of the closure's training: loss and gradient for eight species.
        dict(name="closure_grad", kind="closure", M=8, rows=4096),
    ]


def draw(rng):
    def edge(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    kind = rng.choice(["tube", "loschmidt", "jets", "pulse", "layers", "layers", "mixture", "mixture", "mixture",
                       "ensemble", "restart", "closure"])
    if kind == "closure":
        return dict(kind=kind, M=rng.randint(2, 8), rows=edge(256, 16384))
    precision = rng.choice(["fp32", "fp32", "bf16", "fp16"])
    kw = {}
    if kind == "tube":
        shape, precision = (edge(1, 12), edge(1, 12), edge(32, 256)), rng.choice(["fp64", "fp64", "fp32"])
    elif kind == "loschmidt":
        shape, precision = (1, 1, edge(48, 864)), rng.choice(["fp64", "fp32", "fp32"])
    elif kind == "jets":
        nx = edge(40, 300)
        shape, precision = (rng.choice([1, 1, 3]), 2 * nx + rng.randint(-9, 9), nx), "fp32"
    elif kind == "ensemble":
        shape, kw["domains"] = (edge(16, 32), edge(33, 64), edge(65, 96)), rng.randint(2, 24)
    else:
        # whole warps and rows that are multiples of nothing
        shape = [edge(24, 200) for _ in range(3)]
        if rng.random() < 0.5:
            shape = [max(24, s // 4 * 4) for s in shape]
        cap = 4_000_000
        if kind == "mixture":
            kw["M"] = rng.randint(1, 8)
            cap = 8_000_000 // (kw["M"] + 2)
            if rng.random() < 0.2:
                precision, kw["heats"] = "fp32", True
            elif rng.random() < 0.3:
                kw["weak"] = True
        while shape[0] * shape[1] * shape[2] > cap:
            shape[shape.index(max(shape))] = max(24, max(shape) * 3 // 4)
    return _case(None, kind, shape, precision, rng.choice([4, 8, 9, 20]), **kw)


# ---------------------------------------------------------------------------
# Inputs
# ---------------------------------------------------------------------------
def _grid(case):
    """Cell indices along z, y, x, broadcastable, on the GPU."""
    nz, ny, nx = case["nz"], case["ny"], case["nx"]
    z = torch.arange(nz, dtype=F64, device="cuda").view(nz, 1, 1)
    y = torch.arange(ny, dtype=F64, device="cuda").view(1, ny, 1)
    x = torch.arange(nx, dtype=F64, device="cuda").view(1, 1, nx)
    return z, y, x


def _ripple(case, rng, amplitude, modes=4):
    """1 + amplitude times a smooth periodic field of a few Fourier modes."""
    z, y, x = _grid(case)
    out = torch.ones(case["nz"], case["ny"], case["nx"], dtype=F64, device="cuda")
    for _ in range(modes):
        kz, ky, kx = rng.integers(-3, 4, size=3)
        ph = rng.uniform(0.0, 2.0 * math.pi)
        arg = (2.0 * math.pi * float(kx) / case["nx"]) * x + (2.0 * math.pi * float(ky) / case["ny"]) * y \
            + (2.0 * math.pi * float(kz) / case["nz"]) * z + ph
        out += (amplitude / modes * rng.uniform(0.2, 1.0)) * torch.cos(arg)
    return out


def _recipe(case):
    """The repository's recipe of this kind on a grid of a few nodes: species
    constants, transport inputs, ambient T and P."""
    kind, ny, nx = case["kind"], case["ny"], case["nx"]
    if kind == "tube":
        return W.ternary_tube(nx=nx, ny=1, nz=1)
    if kind == "loschmidt":
        return W.loschmidt_tube("1T", L=nx)
    if kind == "pulse":
        return W.acoustic_pulse(shape=(2, 2, 2), x1=0.5)
    if kind == "layers":
        # the lattice viscosity of the full 800-cell-high box at its Reynolds number
        return W.khi_n2_h2o(shape=(1, ny, 1), reynolds=11963.46 * ny / 800.0, width=4.0)
    if kind == "restart":
        return W.shear_layer(shape=(1, ny, 1))
    if kind == "jets":
        return W.opposed_jets(nx=nx, ny=ny, nz=1)[0]
    return W.random_mixture(M=case["M"], shape=(4, 4, 4), seed=7)


def _fields(case, wl, seed):
    """X (M, nz, ny, nx), u, T, P in float64 on the GPU."""
    rng = np.random.Generator(np.random.PCG64(seed))
    nz, ny, nx, M = case["nz"], case["ny"], case["nx"], wl.M
    kind = case["kind"]
    z, y, x = _grid(case)
    full = (nz, ny, nx)
    T = torch.full(full, float(wl.T.flat[0]), dtype=F64, device="cuda")
    P = torch.full(full, float(wl.P.flat[0]), dtype=F64, device="cuda")
    u = torch.zeros((3,) + full, dtype=F64, device="cuda")
    if kind in ("tube", "loschmidt", "jets"):          # profiles along x
        X = torch.as_tensor(wl.X, device="cuda").reshape(M, -1, nx)[:, :1].view(M, 1, 1, nx).expand((M,) + full)
    elif kind in ("layers", "restart"):                # bands along y, velocity with the bands
        X = torch.as_tensor(wl.X, device="cuda").reshape(M, 1, ny, 1).expand((M,) + full)
        ux = torch.as_tensor(wl.u[0], device="cuda").reshape(1, ny, 1)
        u[0] = ux
        top = float(np.abs(wl.u[0]).max())
        u[1] = 0.02 * top * torch.sin(2.0 * math.pi * x / nx + rng.uniform(0.0, 6.0))
        u[2] = 0.02 * top * torch.sin(2.0 * math.pi * z / nz + rng.uniform(0.0, 6.0))
    elif kind == "pulse":
        x1 = rng.uniform(0.2, 0.8)
        X = torch.tensor([x1, 1.0 - x1], dtype=F64, device="cuda").view(2, 1, 1, 1).expand((2,) + full)
        r2 = (x - nx / 2.0) ** 2 + (y - ny / 2.0) ** 2 + (z - nz / 2.0) ** 2
        P = P * (1.0 + 1e-3 * torch.exp(-r2 / 72.0))
    else:                                              # smooth mixture
        X = torch.ones((M,) + full, dtype=F64, device="cuda")
    amplitude = {"mixture": 0.5, "pulse": 0.0}.get(kind, 0.02)
    if amplitude and M > 1:
        X = torch.stack([X[a] * _ripple(case, rng, amplitude) for a in range(M)])
        X = X / X.sum(dim=0, keepdim=True)
    else:
        X = X.contiguous()
        P = P * _ripple(case, rng, 1e-3)
    return X, u, T, P


def _slaved(X, wl):
    """The species whose smallest mass fraction is largest (strong coupling)."""
    Y = X * torch.as_tensor(wl.molar_mass, device=X.device).view(-1, 1, 1, 1)
    return int(torch.argmax((Y / Y.sum(dim=0, keepdim=True)).flatten(1).amin(dim=1)))


def _jets(case):
    """The nozzles in grid rows (one frame node beyond every x and y face)."""
    inl = W.opposed_jets(nx=case["nx"], ny=case["ny"], nz=1)[1]
    return types.SimpleNamespace(y0=inl.y0 + 1, y1=inl.y1 + 1, X=inl.X, u=inl.u, T=inl.T, P=inl.P)


def _pad_frame(a):
    return torch.nn.functional.pad(a.flatten(0, -3)[None], (1, 1, 1, 1), mode="replicate")[0] \
        .reshape(a.shape[:-2] + (a.shape[-2] + 2, a.shape[-1] + 2)).contiguous()


def _heats(case, wl):
    return W.variable_heats(wl.molar_mass, seed=3) if case.get("heats") else None


def _setup(case, seed):
    """(recipe, fields, slaved species) of a single-domain case."""
    wl = _recipe(case)
    fields = _fields(case, wl, seed)
    return wl, fields, _slaved(fields[0], wl)


def _domains(case, seed):
    """The ensemble's grids and recipes: edges drawn from the seed's own numbers within [nz, nx]."""
    shapes = W.ensemble_shapes(case["domains"], seed=4, lo=case["nz"], hi=case["nx"])
    return [W.ensemble_domain(s, 100 * (seed % 100_000) + k) for k, s in enumerate(shapes)]


def _checkpoint(case, seed):
    """Populations of a run under way: equilibria of the initial fields moved off equilibrium by 0.1 %."""
    wl, fields, slaved = _setup(case, seed)
    m = Method(wl, slaved)
    pops = m.initial(*fields)
    g = torch.Generator(device="cuda").manual_seed(seed)
    pops *= 1.0 + 1e-3 * (2.0 * torch.rand(pops.shape, dtype=F64, device="cuda", generator=g) - 1.0)
    return wl, slaved, pops


def _closure_dims(M):
    def pad16(n):
        return (n + 15) // 16 * 16
    return pad16(4 * M + M * (M - 1) // 2 + 1), pad16(3 * M)


def _closure_inputs(case, seed):
    """Mini-batch (features, exact corrections) of random mixture states, and packed He-initialised weights."""
    M, rows = case["M"], case["rows"]
    F, O = _closure_dims(M)
    wl = W.random_mixture(M=M, shape=(2, 2, 2), seed=7)
    g = torch.Generator(device="cuda").manual_seed(seed)
    rand = lambda *s: torch.rand(*s, dtype=F64, device="cuda", generator=g)  # noqa: E731
    mass = torch.as_tensor(wl.molar_mass, device="cuda")
    D = torch.as_tensor(wl.D, device="cuda").clone()
    D.fill_diagonal_(1.0)
    X = 0.3 + rand(rows, M)
    X = X / X.sum(dim=1, keepdim=True)
    m = X @ mass
    Y = X * mass / m[:, None]
    itab = 0.2 * m[:, None, None] / (D * mass[:, None] * mass[None, :])
    r = rand(rows, M, 3) - 0.5
    r -= Y[:, :, None] * r.sum(dim=1, keepdim=True)
    r = r / r.abs().flatten(1).amax(dim=1)[:, None, None]
    off = itab * (1.0 - torch.eye(M, dtype=F64, device="cuda"))
    A = -0.5 * off * Y[:, :, None] + torch.diag_embed(1.0 + 0.5 * (off * Y[:, None, :]).sum(dim=2))
    J = torch.linalg.solve(A, r) - r / torch.diagonal(A, dim1=1, dim2=2)[:, :, None]
    feat, tgt = torch.zeros(rows, F, dtype=F64, device="cuda"), torch.zeros(rows, O, dtype=F64, device="cuda")
    feat[:, :M], feat[:, M:4 * M] = X, r.flatten(1)
    k = 4 * M
    for a in range(M):
        for b in range(a + 1, M):
            h = 0.5 * itab[:, a, b] * (Y[:, a] + Y[:, b])
            feat[:, k] = h / (1.0 + h)
            k += 1
    feat[:, k] = 1.0
    tgt[:, :3 * M] = J.flatten(1)
    parts = []
    for rows_w, cols, s in ((128, F, 1.0), (128, 128, 1.0), (O, 128, 0.1)):
        w = (2.0 * rand(rows_w, cols) - 1.0) * (s * math.sqrt(6.0 / cols))
        if rows_w == O:
            w[3 * M:] = 0.0
        parts += [w.flatten(), torch.zeros(rows_w, dtype=F64, device="cuda")]
    return feat.float(), tgt.float(), torch.cat(parts).float()


# ---------------------------------------------------------------------------
# The framework's side
# ---------------------------------------------------------------------------
def _handle(case, wl, slaved):
    kw = {}
    shape = (case["nz"], case["ny"], case["nx"])
    if case["kind"] == "jets":
        shape, kw["jets"] = (shape[0], shape[1] + 2, shape[2] + 2), _jets(case)
    return binding.LbmMix(wl.molar_mass, wl.cv_molar, wl.D, mu=wl.mu, lam=wl.lam, shape=shape,
                          precision=case["precision"], slaved=slaved,
                          coupling="weak" if case.get("weak") else "strong",
                          walls_x=case["kind"] == "loschmidt", cv_poly=_heats(case, wl), device="cuda", **kw)


def prepare(case, seed):
    kind = case["kind"]
    if kind == "closure":
        feat, tgt, w = _closure_inputs(case, seed)
        wl = W.random_mixture(M=case["M"], shape=(2, 2, 2), seed=7)
        h = binding.LbmMix(wl.molar_mass, wl.cv_molar, wl.D, mu=wl.mu, lam=wl.lam, shape=(2, 2, 2), device="cuda")
        h.set_closure_weights(w)
        return dict(case=case, h=h, feat=feat, tgt=tgt)
    if kind == "ensemble":
        wls = _domains(case, seed)
        b = binding.LbmBatch([binding.workload_params(v, precision=case["precision"], slaved=W.slaved_species(v))
                              for v in wls], device="cuda")
        outs = []
        for d, v in enumerate(wls):
            b.domain(d).init_fields(*(torch.as_tensor(f, device="cuda") for f in (v.X, v.u, v.T, v.P)))
            outs.append(torch.empty(b.domain(d).n_outputs * v.nodes, dtype=F64, device="cuda"))
        b.set_mode(1, 8)          # what the autotuner settles on for such ensembles
        return dict(case=case, batch=b, outs=outs)
    if kind == "restart":
        wl, slaved, pops = _checkpoint(case, seed)
        return dict(case=case, h=_handle(case, wl, slaved), pops=pops, out=torch.empty_like(pops))
    wl, fields, slaved = _setup(case, seed)
    h = _handle(case, wl, slaved)
    h.init_fields(*(_pad_frame(f) if kind == "jets" else f for f in fields))
    return dict(case=case, h=h, out=torch.empty(h.n_outputs * h.N, dtype=F64, device="cuda"))


def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "closure":
        loss, grad = state["h"].closure_loss_grad(state["feat"], state["tgt"])
        return dict(loss=np.float32(loss), grad=grad)
    if kind == "ensemble":
        b = state["batch"]
        b.step(case["steps"])
        return [b.domain(d).moments(o).float() for d, o in enumerate(state["outs"])]
    h = state["h"]
    if kind == "restart":
        h.set_populations(state["pops"])
        h.step(case["steps"])
        return h.populations(state["out"]).float()
    h.step(case["steps"])
    out = h.moments(state["out"])
    if kind == "jets":            # the frame's nodes hold boundary values
        return out.view((h.n_outputs,) + h.shape)[..., 1:-1, 1:-1].float()
    return out if case["precision"] == "fp64" else out.float()


def work(case):
    """Every stored population read and written once per step and the
    outputs written once; arithmetic of the moments, the equilibria, the
    relaxation and the species coupling."""
    M = case.get("M", {"tube": 3, "loschmidt": 3, "jets": 4, "ensemble": 3}.get(case["kind"], 2))
    if case["kind"] == "closure":
        F, O = _closure_dims(M)
        weights = 128 * (F + 128 + O)
        return dict(bytes=4.0 * (case["rows"] * (F + O) + 2 * weights),
                    flops=2.0 * case["rows"] * (3 * weights - 128 * F))
    b = {"fp64": 8, "fp32": 4}.get(case["precision"], 2)
    if case["kind"] == "ensemble":
        nodes = sum(nz * ny * nx for nz, ny, nx in W.ensemble_shapes(case["domains"], seed=4, lo=case["nz"], hi=case["nx"]))
    else:
        nodes = case["nz"] * case["ny"] * case["nx"]
    lattices = M + 2
    out = 27 * lattices * 8 * 2 if case["kind"] == "restart" else (6 + 5 * M) * 8
    per_step = 27 * (lattices * 16 + 2 * M * M) + 12 * M * M + 4 * M ** 3 // 3
    return dict(bytes=float(nodes) * (case["steps"] * 54 * lattices * b + out),
                flops=float(nodes) * case["steps"] * per_step)


# ---------------------------------------------------------------------------
# The method in 64-bit torch
# ---------------------------------------------------------------------------
_C = [(i % 3 - 1, (i // 3) % 3 - 1, i // 9 - 1) for i in range(27)]      # (cx, cy, cz)
_XREF = [i - 2 * _C[i][0] for i in range(27)]


class Method:
    """The step on full populations [M + 2, 27, nz, ny, nx]: collide, then move every population one link."""

    def __init__(self, wl, slaved, weak=False, walls=False, frame=None, cv_poly=None):
        t = lambda a: torch.as_tensor(np.asarray(a, dtype=np.float64), device="cuda")  # noqa: E731
        self.M, self.slaved, self.weak, self.walls, self.frame = wl.M, slaved, weak, walls, frame
        self.m_a, self.mu, self.lam = t(wl.molar_mass), t(wl.mu), t(wl.lam)
        self.R_a = wl.R_U / self.m_a
        D = np.array(wl.D, dtype=np.float64)
        for a in range(wl.M):
            if D[a, a] <= 0.0:      # self-diffusivity: geometric mean of the row
                D[a, a] = math.exp(np.mean([math.log(D[a, b]) for b in range(wl.M) if b != a]))
        self.D = t(D)
        # molar heats C_v / R_U = sum_k c_k T^k
        self.cv = t(cv_poly if cv_poly is not None else wl.cv_molar[:, None]) * self.R_a[:, None]
        mr, ur = self.m_a[None, :] / self.m_a[:, None], self.mu[:, None] / self.mu[None, :]
        self.wilke = (1.0 + torch.sqrt(ur * torch.sqrt(mr))) ** 2 / (math.sqrt(8.0) * torch.sqrt(1.0 + 1.0 / mr))

    def _sum(self, per_species, T, down):
        """sum over species of Y_a-like weights times int^T of the heats (down = 1) or the heats (0)."""
        s = torch.zeros_like(T)
        for k in range(self.cv.shape[1]):
            s += torch.einsum("a,a...->...", self.cv[:, k], per_species) * T ** (k + down) / (k + 1 if down else 1)
        return s

    def enthalpy_a(self, a, T):
        return sum(self.cv[a, k] * T ** (k + 1) / (k + 1) for k in range(self.cv.shape[1])) + self.R_a[a] * T

    @staticmethod
    def product(xi, zeta):
        """prod over axes of (1 - xi^2 - zeta | (+-xi + xi^2 + zeta) / 2)."""
        out = torch.empty((27,) + zeta.shape, dtype=F64, device="cuda")
        f = []
        for d in range(3):
            s = xi[d] * xi[d] + zeta
            f.append(((s - xi[d]) / 2.0, 1.0 - s, (s + xi[d]) / 2.0))
        for i, (cx, cy, cz) in enumerate(_C):
            torch.mul(f[0][cx + 1] * f[1][cy + 1], f[2][cz + 1], out=out[i])
        return out

    @staticmethod
    def energy(theta, M0, m, Mt):
        """The energy lattice's expansion of moments M0, m, Mt (dict of the six components)."""
        out = torch.empty((27,) + theta.shape, dtype=F64, device="cuda")
        w = ((theta / 2.0), 1.0 - theta, (theta / 2.0))
        N = {(a, b): Mt[a, b] - (theta * M0 if a == b else 0.0) for a, b in Mt}
        Z = [(1.0 - 3.0 * theta) / (2.0 * theta) * N[a, a] for a in range(3)]
        for i, c in enumerate(_C):
            second = sum(N[a, a] * (c[a] * c[a] - theta) for a in range(3))
            for a, b in ((0, 1), (0, 2), (1, 2)):
                if c[a] * c[b]:
                    second = second + 2.0 * c[a] * c[b] * N[a, b]
            h = M0 + second / (2.0 * theta * theta)
            for a in range(3):
                if c[a]:
                    h = h + c[a] * m[a] / theta
            h = h * w[c[0] + 1] * w[c[1] + 1] * w[c[2] + 1]
            n = sum(abs(v) for v in c)
            if n == 0:
                h = h + (Z[0] + Z[1] + Z[2])
            elif n == 1:
                h = h - 0.5 * sum(Z[a] for a in range(3) if c[a])
            out[i] = h
        return out

    def _pad(self, phi, odd):
        """One node beyond every face of a field (nz, ny, nx)."""
        p = torch.cat([phi[-1:], phi, phi[:1]], dim=0)
        if self.frame is None:
            p = torch.cat([p[:, -1:], p, p[:, :1]], dim=1)
            if self.walls:
                s = -1.0 if odd else 1.0
                return torch.cat([s * p[..., :1], p, s * p[..., -1:]], dim=2)
            return torch.cat([p[..., -1:], p, p[..., :1]], dim=2)
        p = torch.cat([p[:, :1], p, p[:, -1:]], dim=1)
        s = torch.ones(p.shape[1], dtype=F64, device="cuda").view(1, -1, 1)
        if odd:
            s = torch.where(self._nozzle(phi.shape[1]).view(1, -1, 1), s, -s)
        return torch.cat([s * p[..., :1], p, s * p[..., -1:]], dim=2)

    def _nozzle(self, ny):
        row = torch.clamp(torch.arange(ny + 2, device="cuda") - 1, 0, ny - 1) + 1      # nearest interior row, grid rows
        return (row >= self.frame.y0) & (row < self.frame.y1)

    def derivative(self, phi, axis, odd=False):
        p = self._pad(phi, odd)
        nz, ny, nx = phi.shape
        out = torch.zeros_like(phi)
        for c in _C:
            if c[axis]:
                w = {1: 2.0 / 27.0, 2: 1.0 / 54.0, 3: 1.0 / 216.0}[sum(abs(v) for v in c)]
                out += (3.0 * w * c[axis]) * p[1 + c[2]:1 + c[2] + nz, 1 + c[1]:1 + c[1] + ny, 1 + c[0]:1 + c[0] + nx]
        return out

    @staticmethod
    def _first(k):
        """Zeroth and first moments of one lattice."""
        j = [torch.zeros_like(k[0]) for _ in range(3)]
        for i, c in enumerate(_C):
            for d in range(3):
                if c[d]:
                    j[d] += c[d] * k[i]
        return k.sum(dim=0), torch.stack(j)

    def state(self, pops):
        M = self.M
        rho_a, j_a = (torch.stack(v) for v in zip(*(self._first(pops[a]) for a in range(M))))
        rho, j = self._first(pops[M])
        rhoE, q = self._first(pops[M + 1])
        if self.weak:
            rho_sp = rho_a.sum(dim=0)
            u_sp = j_a.sum(dim=0) / rho_sp
        else:
            s = self.slaved
            rho_a[s] += rho - rho_a.sum(dim=0)
            j_a[s] += j - j_a.sum(dim=0)
            rho_sp, u_sp = rho, j / rho
        u = j / rho
        usq = (u * u).sum(dim=0)
        Y = rho_a / rho_sp
        m = 1.0 / torch.einsum("a...,a->...", Y, 1.0 / self.m_a)
        X = torch.einsum("a...,a->a...", Y * m, 1.0 / self.m_a)
        R = 1.0 / m
        e = rhoE / rho - 0.5 * usq
        T = e / torch.einsum("a,a...->...", self.cv[:, 0], Y)
        if self.cv.shape[1] > 1:
            for _ in range(12):
                T = T - (self._sum(Y, T, 1) - e) / self._sum(Y, T, 0)
        Cp = self._sum(Y, T, 0) + R
        P = rho * R * T
        mu = sum(self.mu[a] * X[a] / torch.einsum("b,b...->...", self.wilke[a], X) for a in range(M))
        lam = 0.5 * (torch.einsum("a,a...->...", self.lam, X) + 1.0 / torch.einsum("a,a...->...", 1.0 / self.lam, X))
        om, om1 = 2.0 * P / (P + 2.0 * mu), 2.0 * P * Cp / (P * Cp + 2.0 * lam)
        # fluxes J_a = rho_a V_a: J_a + sum_b (Y_b J_a - Y_a J_b) / (2 tau_ab) = j_a - rho_a u
        tm = T * m
        Cab = 1.0 / (self.D * self.m_a[:, None] * self.m_a[None, :])
        off = Cab * (1.0 - torch.eye(M, dtype=F64, device="cuda"))
        r = j_a - rho_a[:, None] * u_sp[None]
        A = [[-0.5 * off[a, b] * tm * Y[a] if a != b else 1.0 + 0.5 * tm * torch.einsum("b,b...->...", off[a], Y)
              for b in range(M)] for a in range(M)]
        r = [r[a] for a in range(M)]
        for k in range(M):                              # elimination (columns are diagonally dominant)
            for i in range(k + 1, M):
                l = A[i][k] / A[k][k]
                for b in range(k + 1, M):
                    A[i][b] = A[i][b] - l * A[k][b]
                r[i] = r[i] - l[None] * r[k]
        J = [None] * M
        for k in range(M - 1, -1, -1):
            s = r[k]
            for b in range(k + 1, M):
                s = s - A[k][b][None] * J[b]
            J[k] = s / A[k][k][None]
        V = torch.stack([torch.where(rho_a[a] > 1e-14 * rho_sp, J[a] / rho_a[a], torch.zeros_like(J[a])) for a in range(M)])
        return types.SimpleNamespace(rho_a=rho_a, rho=rho, rho_sp=rho_sp, j=j, rhoE=rhoE, q=q, u=u, u_sp=u_sp, usq=usq, Y=Y,
                                     X=X, m=m, R=R, T=T, Cp=Cp, P=P, om=om, om1=om1, V=V, Cab=Cab, tm=tm)

    def observables(self, pops):
        s = self.state(pops)
        rows = [s.rho, *s.u, s.T, s.P, *s.X, *s.Y, *s.V.flatten(0, 1)]
        return torch.stack(rows)

    def _energy_moments(self, rho, u, P, h):
        Mt = {}
        for a, b in ((0, 0), (1, 1), (2, 2), (0, 1), (0, 2), (1, 2)):
            Mt[a, b] = h * (rho * u[a] * u[b] + (P if a == b else 0.0)) + P * u[a] * u[b]
        return Mt

    def initial(self, X, u, T, P):
        M = self.M
        m = torch.einsum("a...,a->...", X, self.m_a)
        Y = torch.einsum("a...,a->a...", X, self.m_a) / m
        rho = P * m / T
        usq = (u * u).sum(dim=0)
        U = self._sum(Y, T, 1)
        h = U + T / m + 0.5 * usq
        pops = torch.empty((M + 2, 27) + T.shape, dtype=F64, device="cuda")
        for a in range(M):
            pops[a] = Y[a] * rho * self.product(u, self.R_a[a] * T)
        pops[M] = rho * self.product(u, T / m)
        pops[M + 1] = self.energy(T / m, rho * (U + 0.5 * usq), h * rho * u, self._energy_moments(rho, u, P, h))
        return pops

    def collide(self, pops):
        """In place."""
        M, s = self.M, self.state(pops)
        u, rho, T, P, theta = s.u, s.rho, s.T, s.P, s.R * s.T
        # non-local terms
        Xc = []
        for a in range(3):
            G = (1.0 / s.om - 0.5) * self.derivative(s.j[a] * (1.0 - 3.0 * theta) - rho * u[a] ** 3, a, odd=a == 0)
            Xc.append(-self.derivative(G, a))
        flux = torch.zeros_like(u)                      # sum_a H_a grad Y_a
        for a in range(M):
            H = self.enthalpy_a(a, T)
            for d in range(3):
                flux[d] += H * self.derivative(s.Y[a], d)
        flux *= 0.5 * (2.0 - s.om1) * P
        for a in range(M):
            flux += (s.om1 * rho * self.enthalpy_a(a, T) * s.Y[a])[None] * s.V[a]
        # energy lattice: om1 (g_eq - g) + (om - om1) (g* - g), g* carrying q* (affine in it)
        H = self._sum(s.Y, T, 1) + s.R * T
        h = H + 0.5 * s.usq
        Mt = self._energy_moments(rho, u, P, h)
        qeq = h * s.j
        f = pops[M]
        qb = s.q.clone()
        for a in range(3):
            for b in range(3):
                Pi = torch.zeros_like(rho)
                for i, c in enumerate(_C):
                    if c[a] * c[b]:
                        Pi += c[a] * c[b] * f[i]
                qb[a] -= u[b] * (Pi - rho * u[a] * u[b] - (P if a == b else 0.0))
        drive = s.om * qeq + (s.om - s.om1) * (qb - qeq) + flux     # om times the first moment relaxed to
        geq = self.energy(theta, s.rhoE, drive / s.om, Mt)
        pops[M + 1] += s.om * (geq - pops[M + 1])
        del geq
        # momentum lattice
        f += s.om * (rho * self.product(u, theta) - f)
        for i, c in enumerate(_C):
            if sum(abs(v) for v in c) == 1:
                d = [abs(v) for v in c].index(1)
                f[i] += 0.5 * c[d] * Xc[d]
        # species
        eq = [s.rho_a[a] * self.product(s.u_sp, self.R_a[a] * T) for a in range(M)]
        dif = torch.stack([eq[b] - s.rho_a[b] * self.product(s.u_sp + s.V[b], self.R_a[b] * T) for b in range(M)])
        for a in range(M):
            it = s.tm * torch.einsum("b,b...->...", s.Cab[a], s.Y)
            beta = it / (2.0 + it)
            F = torch.einsum("b,b...->...", s.Cab[a], dif) * (s.tm * s.Y[a])
            pops[a] += 2.0 * beta * (eq[a] - pops[a]) + (beta - 1.0) * F
        return pops

    def stream(self, post):
        out = torch.empty_like(post)
        if self.frame is not None:
            nz, ny, nx = post.shape[-3:]
            pad = torch.empty(post.shape[:-2] + (ny + 2, nx + 2), dtype=F64, device="cuda")
            pad[..., 1:-1, 1:-1] = post
            pad[..., 0, 1:-1], pad[..., -1, 1:-1] = post[..., 0, :], post[..., -1, :]
            row = torch.clamp(torch.arange(ny + 2, device="cuda") - 1, 0, ny - 1)
            noz = self._nozzle(ny).view(1, 1, 1, -1)
            for k, (xo, xb) in enumerate(((0, 0), (-1, -1))):
                wall = post[:, _XREF][..., row, xb]
                pad[..., xo] = torch.where(noz, self.inlets[k].view(self.M + 2, 27, 1, 1), wall)
            for i, (cx, cy, cz) in enumerate(_C):
                out[:, i] = torch.roll(pad[:, i], (cz, cy, cx), (-3, -2, -1))[..., 1:-1, 1:-1]
            return out
        for i, c in enumerate(_C):
            out[:, i] = torch.roll(post[:, i], (c[2], c[1], c[0]), (-3, -2, -1))
            if self.walls and c[0]:
                x = 0 if c[0] > 0 else -1
                out[:, i, ..., x] = post[:, 26 - i, ..., x]
        return out

    def run(self, pops, steps):
        for _ in range(steps):
            pops = self.stream(self.collide(pops))
        return pops


def _exact_domain(case, wl, fields, slaved):
    frame = _jets(case) if case["kind"] == "jets" else None
    m = Method(wl, slaved, weak=bool(case.get("weak")), walls=case["kind"] == "loschmidt", frame=frame,
               cv_poly=_heats(case, wl))
    if frame is not None:
        m.inlets = []
        for k in range(2):
            X = torch.as_tensor(frame.X[k], device="cuda").view(-1, 1, 1, 1)
            u = torch.tensor([frame.u[k], 0.0, 0.0], dtype=F64, device="cuda").view(3, 1, 1, 1)
            T, P = (torch.full((1, 1, 1), float(v[k]), dtype=F64, device="cuda") for v in (frame.T, frame.P))
            m.inlets.append(m.initial(X, u, T, P)[..., 0, 0, 0])
    return m.observables(m.run(m.initial(*fields), case["steps"]))


def exact(case, seed):
    kind = case["kind"]
    if kind == "closure":
        M = case["M"]
        F, O = _closure_dims(M)
        feat, tgt, w = (t.double() for t in _closure_inputs(case, seed))
        w.requires_grad_(True)
        parts, k = [], 0
        for rows, cols in ((128, F), (128, 128), (O, 128)):
            parts.append((w[k:k + rows * cols].view(rows, cols), w[k + rows * cols:k + rows * cols + rows]))
            k += rows * cols + rows
        gelu = torch.nn.functional.gelu
        a = gelu(torch.nn.functional.linear(feat, *parts[0]))
        a = gelu(torch.nn.functional.linear(a, *parts[1]))
        out = torch.nn.functional.linear(a, *parts[2])
        loss = ((out - tgt)[:, :3 * M] ** 2).mean()
        loss.backward()
        return dict(loss=loss.detach(), grad=w.grad)
    if kind == "ensemble":
        outs = []
        for v in _domains(case, seed):
            fields = tuple(torch.as_tensor(f, device="cuda") for f in (v.X, v.u, v.T, v.P))
            outs.append(_exact_domain(case, v, fields, W.slaved_species(v)).flatten())
        return outs
    if kind == "restart":
        wl, slaved, pops = _checkpoint(case, seed)
        return Method(wl, slaved).run(pops, case["steps"])
    wl, fields, slaved = _setup(case, seed)
    out = _exact_domain(case, wl, fields, slaved)
    return out if kind == "jets" else out.flatten()
