"""Performance cases of the APFC library: what a program that uses it asks of it.

Every case goes through the package's public entry points (``Context``, ``Batch``,
``Rollout``) with amplitudes in device memory, as a simulation that lives on the GPU
drives them:

* ``step``    amplitudes in, ``n`` time steps, amplitudes out, on one 2D hexagonal or 3D
              bcc grid, in either precision (and with Picard iterations and the Jacobian);
* ``batch``   independent hexagonal runs of several sizes advanced together;
* ``rollout`` a checkpointed rollout and the gradient of its loss with respect to the
              initial amplitudes and to dB;
* ``analyse`` the free energy, its gradient, and the rotation field with the adaptivity
              map of one state (what a run writes out between steps).

``exact`` evaluates the same quantities in complex128 with torch: Fourier
diagonalisation of the constant-coefficient Schur complement (conjugate gradients
preconditioned by it where the Jacobian makes the coefficient vary), autograd for the
gradient.
"""
import math

import numpy as np
import torch

from paper_1902_09761_gb300 import apfc as A
from paper_1902_09761_gb300 import inputs
from paper_1902_09761_gb300.autograd import Rollout

DB, BX, T, V = 0.02, 0.98, 0.5, 1.0 / 3.0  # the library's standard parameter set
H = math.pi / 2  # the grid spacing of every recorded configuration
ADAPT = {"n": 10.0, "h_int": 0.5, "h_max": 20.0, "eps": 1e-3, "A_min": 0.05}


# ---------------------------------------------------------------------------
# Cases
# ---------------------------------------------------------------------------
def _step(name, lattice, shape, n=1, precision="fp32", dt=1.0, picard=1, jacobian=False):
    c = {"name": name, "kind": "step", "lattice": lattice, "precision": precision, "dt": dt, "n": n,
         "picard": picard, "jacobian": jacobian}
    for key, size in zip(("nz", "ny", "nx")[3 - len(shape):], shape):
        c[key] = size
    return c


def listed():
    return [
        # the smallest configuration (one grain, 128^2): a few steps between two looks at the
        # state, where launches and latency are all there is
        _step("grain-128", "hex", (128, 128), n=4),
        # an ordinary polycrystal on the grid of the gradient workload
        _step("voronoi-1024", "hex", (1024, 1024), n=2),
        # a box cut to fit a measured sample: odd row length, odd number of rows
        _step("voronoi-ragged", "hex", (1531, 997), n=2, dt=0.5),
        # the benchmark's polycrystal: 50 M amplitude values
        _step("voronoi-4096", "hex", (4096, 4096), n=2),
        # plain FP64, the library's default precision, on an ordinary grid
        _step("fp64-512", "hex", (512, 512), n=2, precision="fp64"),
        # Picard iterations with the Jacobian, for larger time steps
        _step("picard-512", "hex", (512, 512), dt=2.0, picard=3, jacobian=True),
        # the 3D benchmark: a rotated sphere in a bcc matrix
        _step("bcc-256", "bcc", (256, 256, 256)),
        # a small 3D box with odd sides
        _step("bcc-ragged", "bcc", (70, 90, 101), n=2),
        # plain FP64 in 3D
        _step("bcc-fp64", "bcc", (64, 64, 64), precision="fp64"),
        # a parameter study: independent runs of mixed sizes advanced together
        {"name": "batch-24", "kind": "batch", "runs": 24, "smallest": 128, "largest": 512, "dt": 1.0, "n": 2},
        # fitting to data: forward rollout and gradient with checkpoints
        {"name": "rollout-256", "kind": "rollout", "ny": 256, "nx": 256, "dt": 1.0, "n": 12, "every": 4,
         "precision": "fp32"},
        # what is written out between steps
        {"name": "analyse-1024", "kind": "analyse", "lattice": "hex", "ny": 1024, "nx": 1024},
    ]


def _size(rng, lo, hi):
    """A grid size over the logarithm of [lo, hi]; a third each a multiple of 64, even, odd."""
    v = int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))
    how = rng.randrange(3)
    if how == 0:
        v = max(64, (v + 32) // 64 * 64)
    elif how == 1:
        v += v & 1
    else:
        v |= 1
    return max(lo, min(hi, v))


def draw(rng):
    kind = rng.choice(["hex", "hex", "hex", "hex64", "picard", "bcc", "bcc", "bcc64", "batch", "rollout", "analyse"])
    dt = rng.choice([0.5, 1.0, 2.0])
    if kind == "hex":
        c = _step("", "hex", (_size(rng, 96, 3000), _size(rng, 96, 3000)), n=rng.choice([1, 2, 3]), dt=dt)
    elif kind == "hex64":
        c = _step("", "hex", (_size(rng, 96, 700), _size(rng, 96, 700)), n=rng.choice([1, 2]), precision="fp64", dt=dt)
    elif kind == "picard":
        c = _step("", "hex", (_size(rng, 96, 700), _size(rng, 96, 700)), dt=dt, picard=rng.choice([2, 3]),
                  jacobian=rng.choice([True, False]), precision=rng.choice(["fp32", "fp32", "fp64"]))
    elif kind == "bcc":
        c = _step("", "bcc", tuple(_size(rng, 32, 180) for _ in range(3)), n=rng.choice([1, 2]), dt=dt)
    elif kind == "bcc64":
        c = _step("", "bcc", tuple(_size(rng, 24, 72) for _ in range(3)), precision="fp64", dt=dt)
    elif kind == "batch":
        c = {"kind": "batch", "runs": rng.randrange(4, 33), "smallest": rng.choice([64, 128]),
             "largest": rng.choice([256, 384, 512]), "dt": dt, "n": rng.choice([1, 2])}
    elif kind == "rollout":
        precision = rng.choice(["fp32", "fp32", "fp64"])
        most = 500 if precision == "fp32" else 250
        c = {"kind": "rollout", "ny": _size(rng, 64, most), "nx": _size(rng, 64, most), "dt": dt,
             "n": rng.randrange(4, 13), "every": rng.randrange(2, 6), "precision": precision}
    else:
        c = {"kind": "analyse", "lattice": "hex", "ny": _size(rng, 96, 2500), "nx": _size(rng, 96, 2500)}
    c.pop("name", None)
    return c


def _shape(case):
    return tuple(case[k] for k in ("nz", "ny", "nx") if k in case)


def _lattice(name):
    return (inputs.hex_vectors(), A.APFC_LATTICE_HEX2D) if name == "hex" else (inputs.bcc_vectors(), A.APFC_LATTICE_BCC3D)


def _batch_shapes(case):
    """The grids of a batch: sides over the logarithm of [smallest, largest], some odd."""
    lo, hi = math.log(case["smallest"]), math.log(case["largest"])
    r = np.random.default_rng(12345)  # the study's grids belong to the case, not to the seed
    sides = np.exp(r.uniform(lo, hi, size=(case["runs"], 2))).astype(int)
    sides[::2, 1] = sides[::2, 0]  # half of the boxes are square
    sides[0], sides[-1] = case["smallest"], case["largest"]
    return [(int(a), int(b)) for a, b in sides]


# ---------------------------------------------------------------------------
# Inputs
# ---------------------------------------------------------------------------
def _amplitude(k, kind):
    return A.apfc_uniform_amplitude(A.make_lattice(k, kind), A.make_params(DB, BX, T, V))


def _grid(shape, device):
    """Node coordinates, in (x, y[, z]) order, broadcastable to the grid."""
    dim = len(shape)
    out = []
    for d in range(dim):
        view = [1] * dim
        view[dim - 1 - d] = shape[dim - 1 - d]
        out.append((torch.arange(shape[dim - 1 - d], dtype=torch.float64, device=device) * H).reshape(view))
    return out


def _grains(k, phi, shape, seed, ngrains, device, matrix=None, radius=None):
    """Rotated grains with noise: Voronoi grains that fill the periodic box or, with a
    radius, one round grain at its centre (in liquid, or in a solid of amplitude matrix)."""
    rng = np.random.default_rng(seed)
    dim = len(shape)
    box = np.array([shape[dim - 1 - d] * H for d in range(dim)])
    coords = _grid(shape, device)
    if radius is None:
        centres = rng.uniform(0.0, 1.0, size=(ngrains, dim)) * box
    else:
        centres = 0.5 * box[None, :]
    angles = np.deg2rad(rng.uniform(2.0, 10.0, size=len(centres)) * rng.choice([-1.0, 1.0], size=len(centres)))
    owner = torch.full(shape, -1, dtype=torch.int64, device=device)
    best = torch.full(shape, math.inf if radius is None else radius * radius, dtype=torch.float64, device=device)
    for g, c in enumerate(centres):
        d2 = torch.zeros(shape, dtype=torch.float64, device=device)
        for d in range(dim):
            u = coords[d] - c[d]
            d2 = d2 + (u - box[d] * torch.round(u / box[d])) ** 2
        owner = torch.where(d2 < best, g, owner)
        best = torch.minimum(best, d2)
    inside, at = owner >= 0, owner.clamp(min=0)
    dk = torch.from_numpy(np.stack([inputs.delta_k(k, a) for a in angles])).to(device)
    cen = torch.from_numpy(centres).to(device)
    gen = torch.Generator(device=device)
    gen.manual_seed(seed)
    eta = torch.empty((len(k),) + tuple(shape), dtype=torch.complex128, device=device)
    for j in range(len(k)):
        phase = torch.zeros(shape, dtype=torch.float64, device=device)
        for d in range(dim):
            phase += dk[at, j, d] * (coords[d] - cen[at, d])
        wave = torch.polar(torch.full_like(phase, phi), phase)
        wave = torch.where(inside, wave, torch.full_like(wave, 0.0 if matrix is None else matrix))
        noise = torch.randn((2,) + tuple(shape), dtype=torch.float64, device=device, generator=gen)
        eta[j] = wave + 1e-3 * torch.complex(noise[0], noise[1])
    return eta


def _initial(case, seed, device="cuda"):
    """Initial amplitudes of a case ([J] + grid; a list of them for a batch)."""
    k, kind = _lattice(case.get("lattice", "hex"))
    phi = _amplitude(k, kind)
    if case["kind"] == "batch":
        return [_grains(k, phi, s, seed * 1009 + r, 1, device, radius=0.25 * min(s) * H)
                for r, s in enumerate(_batch_shapes(case))]
    shape = _shape(case)
    if len(shape) == 3:
        return _grains(k, phi, shape, seed, 1, device, matrix=phi, radius=0.3 * min(shape) * H)
    if max(shape) <= 160:
        return _grains(k, phi, shape, seed, 1, device, radius=0.3 * min(shape) * H)
    return _grains(k, phi, shape, seed, 16, device)


def _opts(case):
    return A.apfc_default_opts(precision=A.APFC_FP64 if case["precision"] == "fp64" else A.APFC_FP32_REFINED)


def prepare(case, seed):
    k, kind = _lattice(case.get("lattice", "hex"))
    params = (DB, BX, T, V)
    s = {"case": case, "eta0": _initial(case, seed)}
    if case["kind"] == "step":
        o = _opts(case)
        o.picard_iters, o.jacobian = case["picard"], int(case["jacobian"])
        shape = _shape(case)
        s["ctx"] = A.Context(k, kind, params, shape, (H,) * len(shape), o)
        s["out"] = torch.empty_like(s["eta0"])
    elif case["kind"] == "batch":
        s["batch"] = A.Batch(k, kind, params, _batch_shapes(case), (H, H))
        s["out"] = [torch.empty_like(e) for e in s["eta0"]]
    elif case["kind"] == "rollout":
        s["ro"] = Rollout(k, kind, params, _shape(case), (H, H), case["dt"], case["n"], case["every"], _opts(case),
                          device="cuda")
        s["target"] = _target(case, seed)
        s["eta0"].requires_grad_(True)
        s["dB"] = torch.tensor(DB, dtype=torch.float64, requires_grad=True)
    else:
        s["ctx"] = A.Context(k, kind, params, _shape(case), (H, H))
        s["grad"] = torch.empty_like(s["eta0"])
    return s


def _target(case, seed, device="cuda"):
    gen = torch.Generator(device=device)
    gen.manual_seed(seed + 77)
    u = torch.randn((2, 3) + _shape(case), dtype=torch.float64, device=device, generator=gen)
    return 0.1 * torch.complex(u[0], u[1])


# ---------------------------------------------------------------------------
# One pass
# ---------------------------------------------------------------------------
def _loss(etaN, F, target):
    return 0.5 * H * H * (etaN - target).abs().pow(2).sum() + F


def run(s):
    case = s["case"]
    if case["kind"] == "step":
        ctx = s["ctx"]
        ctx.set_amplitudes(s["eta0"])
        ctx.step(case["dt"], case["n"])
        return ctx.get_amplitudes(s["out"])
    if case["kind"] == "batch":
        b = s["batch"]
        for r, e in enumerate(s["eta0"]):
            b.set_amplitudes(r, e)
        b.step(case["dt"], case["n"])
        return [b.get_amplitudes(r, out) for r, out in enumerate(s["out"])]
    if case["kind"] == "rollout":
        s["eta0"].grad = s["dB"].grad = None
        etaN, F = s["ro"](s["eta0"], s["dB"])
        loss = _loss(etaN, F, s["target"])
        loss.backward()
        return {"eta": etaN.detach(), "loss": loss.detach(), "grad": s["eta0"].grad, "grad_dB": s["dB"].grad}
    ctx = s["ctx"]
    ctx.set_amplitudes(s["eta0"])
    F = ctx.energy()
    grad, dF = ctx.energy_gradient(s["eta0"], s["grad"])
    omega, amp, h = ctx.rotation_field(ADAPT, device="cuda")
    return {"F": F, "grad": grad, "dF": dF, "omega": omega, "A": amp, "h": h}


def work(case):
    """Amplitudes are read once and written once (16 bytes a value); the operations are those of
    the nonlinear term and one residual per step (or iteration), not of any solver."""
    if case["kind"] == "batch":
        dof = sum(3 * a * b for a, b in _batch_shapes(case))
        return {"bytes": 32.0 * dof, "flops": 130.0 * dof * case["n"]}
    shape = _shape(case)
    J = 6 if len(shape) == 3 else 3
    dof = float(J * math.prod(shape))
    if case["kind"] == "analyse":
        return {"bytes": 32.0 * dof + 24.0 * dof / J, "flops": 200.0 * dof}
    if case["kind"] == "rollout":
        return {"bytes": 64.0 * dof, "flops": 3.0 * 130.0 * dof * case["n"]}
    return {"bytes": 32.0 * dof, "flops": (400.0 if J == 6 else 130.0) * dof * case["n"] * case["picard"]}


# ---------------------------------------------------------------------------
# The same in 64 bits
# ---------------------------------------------------------------------------
def _symbol(k, shape, device):
    """Fourier symbol of G_h = L_h + 2i k.D_h on the periodic grid (real)."""
    dim = len(shape)
    g = torch.zeros(shape, dtype=torch.float64, device=device)
    for d in range(dim):
        n = shape[dim - 1 - d]
        view = [1] * dim
        view[dim - 1 - d] = n
        q = (2 * math.pi / n * torch.arange(n, dtype=torch.float64, device=device)).reshape(view)
        g = g + (2.0 * torch.cos(q) - 2.0) / (H * H) - 2.0 * float(k[d]) * torch.sin(q) / H
    return g


def _G(u, k):
    """G_h u on the grid."""
    dim = u.dim()
    out = torch.zeros_like(u)
    for d in range(dim):
        p, m = torch.roll(u, -1, dim - 1 - d), torch.roll(u, 1, dim - 1 - d)
        out = out + (p + m - 2.0 * u) / (H * H) + 1j * float(k[d]) / H * (p - m)
    return out


def _terms(k, p):
    """Sets of p signed modes (j, s) whose wavevectors sum to zero, with their multiplicities."""
    import itertools

    modes = [(j, s) for j in range(len(k)) for s in (1, -1)]
    found = {}
    for t in itertools.product(modes, repeat=p):
        if np.all(np.abs(sum(s * k[j] for j, s in t)) < 1e-9):
            found[tuple(sorted(t))] = found.get(tuple(sorted(t)), 0) + 1
    return found


def _nonlinear(eta, k):
    """N_j: the derivative by conj(eta_j) of the cell average of -t/3 n^3 + v/4 n^4."""
    if len(k) == 3:
        A2 = 2.0 * sum(e.abs() ** 2 for e in eta)
        return torch.stack([3 * V * (A2 - eta[j].abs() ** 2) * eta[j] - 2 * T * (eta[(j + 1) % 3] * eta[(j + 2) % 3]).conj()
                            for j in range(3)])
    mode = {(j, 1): eta[j] for j in range(len(k))}
    mode.update({(j, -1): eta[j].conj() for j in range(len(k))})
    out = torch.zeros_like(eta)
    for p, c in ((3, -T / 3.0), (4, 0.25 * V)):
        for t, mult in _terms(k, p).items():
            for j in range(len(k)):
                m = t.count((j, -1))
                if m:
                    rest = list(t)
                    rest.remove((j, -1))
                    prod = mode[rest[0]]
                    for q in rest[1:]:
                        prod = prod * mode[q]
                    out[j] += c * mult * m * prod
    return out


def _solve(rhs, k, dt, dB):
    """eta_j = S_j^{-1} rhs_j with S_j = (1/dt + |k_j|^2 dB) I + |k_j|^2 Bx G_h^2."""
    out = []
    for j in range(len(k)):
        kap = float(k[j] @ k[j])
        s = 1.0 / dt + kap * dB + kap * BX * _symbol(k[j], tuple(rhs[j].shape), rhs.device) ** 2
        out.append(torch.fft.ifftn(torch.fft.fftn(rhs[j]) / s))
    return torch.stack(out)


def _exact_step(eta, k, dt, dB=DB):
    kap = torch.tensor([float(v @ v) for v in k], dtype=torch.float64, device=eta.device).reshape((-1,) + (1,) * (eta.dim() - 1))
    return _solve(eta / dt - kap * _nonlinear(eta, k), k, dt, dB)


def _exact_picard(eta_n, k, dt, iters, jacobian):
    """Picard iterations of one step on the triangular lattice, D_j = dN_j/d eta_j = 3 v A^2."""
    eta = eta_n
    for _ in range(iters):
        N = _nonlinear(eta, k)
        if not jacobian:
            eta = _solve(eta_n / dt - N, k, dt, DB)  # |k_j| = 1
            continue
        D = 3.0 * V * 2.0 * sum(e.abs() ** 2 for e in eta)
        b = eta_n / dt - (N - D * eta)
        mean = float(D.mean())
        new = []
        for j in range(3):
            # conjugate gradients on (1/dt + dB + D) I + Bx G_h^2, preconditioned with D's mean
            sym = 1.0 / dt + DB + mean + BX * _symbol(k[j], tuple(eta.shape[1:]), eta.device) ** 2
            x = eta[j].clone()
            r = b[j] - ((1.0 / dt + DB + D) * x + BX * _G(_G(x, k[j]), k[j]))
            z = torch.fft.ifftn(torch.fft.fftn(r) / sym)
            p, rz, stop = z.clone(), torch.sum(r.conj() * z).real, 1e-15 * torch.linalg.vector_norm(b[j])
            for _ in range(60):
                q = (1.0 / dt + DB + D) * p + BX * _G(_G(p, k[j]), k[j])
                a = rz / torch.sum(p.conj() * q).real
                x, r = x + a * p, r - a * q
                if torch.linalg.vector_norm(r) <= stop:
                    break
                z = torch.fft.ifftn(torch.fft.fftn(r) / sym)
                new_rz = torch.sum(r.conj() * z).real
                p, rz = z + new_rz / rz * p, new_rz
            new.append(x)
        eta = torch.stack(new)
    return eta


def _energy(eta, k, dB):
    """The triangular lattice's free energy."""
    m2 = [e.abs() ** 2 for e in eta]
    A2 = 2.0 * sum(m2)
    f = 0.5 * dB * A2 + 0.75 * V * A2 ** 2 - 1.5 * V * sum(m ** 2 for m in m2)
    f = f - 4.0 * T * (eta[0] * eta[1] * eta[2]).real
    f = f + BX * sum(_G(eta[j], k[j]).abs() ** 2 for j in range(3))
    return H * H * f.sum()


def _analysis(eta, k):
    """Rotation tensor, A and the adaptivity map of a hexagonal state."""
    phases = []
    for j in range(3):
        d = [torch.angle(torch.roll(eta[j], -1, 1 - a) * torch.roll(eta[j], 1, 1 - a).conj()) / (2 * H) for a in (0, 1)]
        phases.append(d)
    M = np.linalg.inv(sum(np.outer(v, v) for v in k))
    W = [M @ v for v in k]
    du = [[sum(W[j][i] * phases[j][d] for j in range(3)) for d in (0, 1)] for i in (0, 1)]
    omega = 0.5 * (du[0][1] - du[1][0])
    solid = torch.stack([e.abs() ** 2 >= 1e-12 for e in eta]).all(0)
    omega = torch.where(solid, omega, torch.zeros_like(omega))
    amp = torch.sqrt(2.0 * sum(e.abs() ** 2 for e in eta))
    g2 = sum(((torch.roll(amp, -1, d) - torch.roll(amp, 1, d)) / (2 * H)) ** 2 for d in (0, 1))
    half = torch.sin(0.5 * torch.asin(omega.abs().clamp(max=1.0)))
    kmax = max(math.sqrt(float(v @ v)) for v in k)
    h = (math.pi / (ADAPT["n"] * kmax) / half).clamp(ADAPT["h_int"], ADAPT["h_max"])
    h = torch.where(amp > ADAPT["A_min"], h, torch.full_like(h, ADAPT["h_max"]))
    h = torch.where(g2 >= ADAPT["eps"] ** 2, torch.full_like(h, ADAPT["h_int"]), h)
    return omega.unsqueeze(0), amp, h


def exact(case, seed):
    device = "cuda" if torch.cuda.is_available() else "cpu"
    k, _ = _lattice(case.get("lattice", "hex"))
    eta = _initial(case, seed, device)
    if case["kind"] == "step":
        for _ in range(case["n"]):
            if case["picard"] > 1 or case["jacobian"]:
                eta = _exact_picard(eta, k, case["dt"], case["picard"], case["jacobian"])
            else:
                eta = _exact_step(eta, k, case["dt"])
        return eta
    if case["kind"] == "batch":
        for _ in range(case["n"]):
            eta = [_exact_step(e, k, case["dt"]) for e in eta]
        return eta
    if case["kind"] == "rollout":
        eta.requires_grad_(True)
        dB = torch.tensor(DB, dtype=torch.float64, device=device, requires_grad=True)
        x = eta
        for _ in range(case["n"]):
            x = _exact_step(x, k, case["dt"], dB)
        loss = _loss(x, _energy(x, k, dB), _target(case, seed, device))
        loss.backward()
        return {"eta": x.detach(), "loss": loss.detach(), "grad": eta.grad, "grad_dB": dB.grad}
    e = eta.clone().requires_grad_(True)
    F = _energy(e, k, DB)
    F.backward()
    omega, amp, h = _analysis(eta, k)
    return {"F": F.detach(), "grad": e.grad, "dF": H * H * sum((v.abs() ** 2).sum() for v in eta), "omega": omega,
            "A": amp, "h": h}
