"""Performance cases of the library: what a program has it do through its public entry points.

A case is one call pattern at one size:

* ``run``       set a state, integrate (``run_steps`` or ``run_until``), read the state back;
* ``field``     one effective field of a device tensor (``h_eff``);
* ``vjp``       the transpose product of the field, with the Ms gradient (``h_eff_vjp``);
* ``gradient``  a differentiated run (``autograd.llg_loss`` and its backward pass);
* ``serve``     a batch of requests through the request loop (``serve.Server``).

``prepare`` makes what a program has in hand before the call (the mesh with its material, the inputs on the
GPU, the server), ``run`` is the call, ``work`` the bytes and operations it cannot do without and ``exact``
the same result in 64 bits by plain torch operations.  Materials and workloads are those of ``nm_inputs.py``;
every random quantity is drawn from the seed.

A mesh of precision F32 evaluates the field in FP32 and keeps an FP64 state, so the state carries the FP32
field's error: such runs return m in FP32, as a program that stores trajectories does.
"""
import math

import numpy as np
import torch

import paper_2411_11725_gb300 as nmgb
from paper_2411_11725_gb300.autograd import LossSpec, llg_loss
from paper_2411_11725_gb300.serve import Server

MU0 = 4e-7 * math.pi
GAMMA = MU0 * 1.76085963023e11

# name -> cell size, Ms, A, Ku, alpha, field terms, applied field (T), state (None: random directions; else the
# noise on a uniform one) and dt (the step the controller settles near, from which a run that continues a
# trajectory starts; with cell maps the step of the fixed-step runs)
MATERIALS = {
    # the RK4 cuboid: exchange, demag and a 20 mT field from a random state
    "cuboid": dict(dx=(2e-9, 2e-9, 2e-9), Ms=8e5, A=1.3e-11, Ku=0.0, alpha=0.1,
                   terms=nmgb.EXCH | nmgb.ZEE | nmgb.DEMAG, b=20e-3, noise=None, dt=2.5e-13),
    # the thin film of the validation runs: nearly uniform in the plane
    "film": dict(dx=(2.5e-9, 2.5e-9, 3e-9), Ms=8e5, A=1.3e-11, Ku=0.0, alpha=0.02,
                 terms=nmgb.EXCH | nmgb.ZEE | nmgb.DEMAG, b=30e-3, noise=1e-2, dt=3.3e-13),
    # the throughput cuboids: random state, easy axis along z
    "throughput": dict(dx=(3e-9, 3e-9, 3e-9), Ms=1e6, A=1.5e-11, Ku=5e5, alpha=0.1,
                       terms=nmgb.EXCH | nmgb.ANIS | nmgb.DEMAG, b=0.0, noise=None, dt=5e-13),
    # cell maps of Ms, A and Ku with vacuum cells, a uniform and a cell-wise applied field
    "maps": dict(dx=(2e-9, 2.5e-9, 3e-9), Ms=8e5, A=1.2e-11, Ku=1e5, alpha=0.2, terms=nmgb.ALL, b=50e-3,
                 noise=None, dt=2e-14),
    # the spin-wave guide of the inverse problem: Ms map, driven stripe, state along x
    "waveguide": dict(dx=(4e-9, 4e-9, 10e-9), Ms=1.4e5, A=3.5e-12, Ku=0.0, alpha=1e-3,
                      terms=nmgb.EXCH | nmgb.ZEE | nmgb.DEMAG, b=0.0, noise=5e-2, dt=2.5e-13),
}


def listed():
    return [
        # the smallest run of the tests and the benchmark: 100 fixed steps, all launches and latency
        dict(name="run_rk4_16x16x4", call="run", n1=16, n2=16, n3=4, material="cuboid", method="rk4", steps=100,
             dt=1e-14, basis=3, f64=False, until=False),
        # the validation film: adaptive steps to a given time
        dict(name="until_dp5_film_200x50x1", call="run", n1=200, n2=50, n3=1, material="film", method="dp5",
             steps=30, dt=3.3e-13, basis=3, f64=False, until=True),
        # odd sizes, cell-wise material with vacuum, uniform and cell fields
        dict(name="run_rk4_maps_131x67x5", call="run", n1=131, n2=67, n3=5, material="maps", method="rk4", steps=20,
             dt=2e-14, basis=3, f64=False, until=False),
        # the smallest of the throughput sweep, the largest shape of the serving stream
        dict(name="run_dp5_256x256x8", call="run", n1=256, n2=256, n3=8, material="throughput", method="dp5",
             steps=10, dt=6e-13, basis=3, f64=False, until=False),
        # the benchmark's headline mesh
        dict(name="run_dp5_1024x1024x32", call="run", n1=1024, n2=1024, n3=32, material="throughput", method="dp5",
             steps=3, dt=6e-13, basis=3, f64=False, until=False),
        # a large film on the 2D nodal basis
        dict(name="run_dp5_2d_1024x1024x1", call="run", n1=1024, n2=1024, n3=1, material="throughput", method="dp5",
             steps=6, dt=5e-13, basis=2, f64=False, until=False),
        # plain FP64
        dict(name="run_dp5_f64_128x128x4", call="run", n1=128, n2=128, n3=4, material="throughput", method="dp5",
             steps=4, dt=5e-13, basis=3, f64=True, until=False),
        # single field evaluations (energy minimisers, static problems): a small film and a large cuboid
        dict(name="field_100x40x1", call="field", n1=100, n2=40, n3=1, material="cuboid", basis=3, f64=False),
        dict(name="field_512x512x16", call="field", n1=512, n2=512, n3=16, material="throughput", basis=3, f64=False),
        # static inverse problems: transpose product and Ms gradient
        dict(name="vjp_256x256x8", call="vjp", n1=256, n2=256, n3=8, material="maps", basis=3, f64=False),
        # the waveguide's gradient: RK4 forward with samples, checkpoints, discrete adjoint
        dict(name="gradient_waveguide_256x64x1", call="gradient", n1=256, n2=64, n3=1, material="waveguide",
             steps=24, dt=2.5e-13, sample_every=4, checkpoint=8, f64=False),
        # eight requests of the serving stream's shapes in flight together
        dict(name="serve_8_requests", call="serve", requests=8, shapes=1234, t_ps=8.0),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    call = rng.choices(("run", "field", "vjp", "gradient", "serve"), (50, 18, 14, 12, 6))[0]
    if call == "serve":
        return dict(call=call, requests=rng.randint(3, 10), shapes=rng.randint(0, 10 ** 6),
                    t_ps=round(rng.uniform(3.0, 9.0), 3))
    if call == "gradient":
        n = (_log_int(rng, 12, 256), _log_int(rng, 12, 160), rng.choice((1, 1, 2, 3, 4)))
        return dict(call=call, n1=n[0], n2=n[1], n3=n[2], material="waveguide", steps=rng.randint(8, 24), dt=2.5e-13,
                    sample_every=rng.randint(1, 6), checkpoint=rng.randint(4, 32), f64=rng.random() < 0.15)
    f64 = rng.random() < 0.15
    most = 2 ** 20 if f64 else 2 ** 25  # cells
    while True:
        n = (_log_int(rng, 12, 1024), _log_int(rng, 12, 1024), _log_int(rng, 1, 32))
        if 200 <= n[0] * n[1] * n[2] <= (most if call == "run" else min(most, 2 ** 23)):
            break
    material = rng.choice(("cuboid", "film", "throughput", "throughput", "maps"))
    case = dict(call=call, n1=n[0], n2=n[1], n3=n[2], material=material, basis=3, f64=f64)
    if call == "run":
        if n[2] <= 4 and material != "maps" and rng.random() < 0.3:
            case["basis"] = 2
        method = "rk4" if material == "maps" else rng.choice(("dp5", "dp5", "dp5", "rk4"))
        nodes = (n[0] + 1) * (n[1] + 1) * (n[2] + 1)
        steps = int(max(2, min(60 if method == "rk4" else 12, (2e6 if f64 else 4e7) / nodes)))
        dt = MATERIALS[material]["dt"] if method == "dp5" or material == "maps" else 1e-14
        case.update(method=method, steps=steps, dt=dt, until=method == "dp5" and rng.random() < 0.3)
    elif call == "field" and material == "film":
        case["material"] = "cuboid"  # single evaluations and transpose products: states far from uniform
    elif call == "vjp":
        case["material"] = rng.choice(("throughput", "maps"))
    return case


# ---------------------------------------------------------------------------------------------- inputs
def _device():
    return torch.device("cuda" if torch.cuda.is_available() else "cpu")


def _unit(v):
    return v / v.norm(dim=-1, keepdim=True)


def _problem(case, seed):
    """Material (numbers or cell maps), applied fields and state of a case, from the seed alone."""
    mat = MATERIALS[case["material"]]
    n = (case["n1"], case["n2"], case["n3"])
    basis = case.get("basis", 3)
    nodes = (n[0] + 1, n[1] + 1, n[2] + 1 if basis == 3 else 1)
    rng = np.random.default_rng(seed)
    gen = torch.Generator(device=_device())
    gen.manual_seed(seed)
    p = dict(n=n, nodes=nodes, basis=basis, dx=mat["dx"], Ms=mat["Ms"], A=mat["A"], Ku=mat["Ku"], axis=(0.0, 0.0, 1.0),
             alpha=mat["alpha"], terms=mat["terms"], hc=None, hc_freq=0.0)
    if case["material"] == "maps":
        p["Ms"] = rng.uniform(4e5, 1.2e6, n)
        p["Ms"][rng.uniform(size=n) < 0.15] = 0.0
        p["A"] = rng.uniform(5e-12, 2e-11, n)
        p["Ku"] = rng.uniform(-3e5, 5e5, n)
        axis = rng.standard_normal(3)
        p["axis"] = tuple(axis / np.linalg.norm(axis))
        p["hc"] = rng.standard_normal(n + (3,)) * (5e-3 / MU0)
    elif case["material"] == "waveguide":
        # a design of the running optimisation: the initial map with changes of a few per cent
        p["Ms"] = 1.4e5 * (1.0 + 0.05 * rng.standard_normal(n))
        p["hc"] = np.zeros(n + (3,))
        p["hc"][:8, :, :, 1] = 1e-3 / MU0
        p["hc_freq"] = 2e9
    h = rng.standard_normal(3)
    p["hu"] = tuple(h / np.linalg.norm(h) * (mat["b"] / MU0))
    noise = torch.randn(nodes + (3,), generator=gen, dtype=torch.float64, device=_device())
    if mat["noise"] is None:
        m0 = noise
    else:
        if case["material"] == "waveguide":
            d = torch.tensor([1.0, 0.0, 0.0], dtype=torch.float64)
        else:
            psi = rng.uniform(0, 2 * math.pi)
            d = torch.tensor([math.cos(psi), math.sin(psi), 0.0], dtype=torch.float64)
        m0 = d.to(noise.device) + mat["noise"] * noise
    p["m0"] = _unit(m0)
    real = torch.float64 if case.get("f64") else torch.float32
    if case["call"] == "field":
        p["m0"] = p["m0"].to(real)
    elif case["call"] == "vjp":
        p["m0"] = p["m0"].to(real)
        p["v"] = torch.randn(nodes + (3,), generator=gen, dtype=torch.float64, device=_device()).to(real)
    elif case["call"] == "gradient":
        p["m0"] = p["m0"].to(real)
        p["Ms"] = torch.tensor(p["Ms"], device=_device()).to(real)
        # the mean of m_y^2 and m_z^2 in the right half of the guide
        p["weight"] = np.zeros(nodes + (3,))
        p["weight"][nodes[0] // 2:, :, :, 1:] = 1.0 / ((nodes[0] - nodes[0] // 2) * nodes[1] * nodes[2])
    return p


def _requests(case, seed):
    """Requests with the sizes and materials of the serving stream, each a few picoseconds long."""
    rng = np.random.default_rng(seed)
    shapes = np.random.default_rng(case["shapes"])  # (a case keeps its shapes from seed to seed)
    out = []
    for _ in range(case["requests"]):
        n = (int(shapes.choice([64, 128, 256])), int(shapes.choice([64, 128])), int(shapes.choice([1, 2, 4, 8])))
        h, d = rng.standard_normal(3), rng.standard_normal(3)
        m0 = d / np.linalg.norm(d) + 0.05 * rng.standard_normal(tuple(v + 1 for v in n) + (3,))
        out.append(dict(n=n, dx=(3e-9, 3e-9, 3e-9), m0=m0 / np.linalg.norm(m0, axis=-1, keepdims=True),
                        t_end=case["t_ps"] * 1e-12 * rng.uniform(0.6, 1.0), dt0=1e-13, Ms=rng.uniform(4e5, 1.2e6),
                        A=rng.uniform(5e-12, 2e-11), alpha=rng.uniform(0.01, 0.5),
                        h=tuple(h / np.linalg.norm(h) * rng.uniform(0, 100e-3) / MU0)))
    return out


def prepare(case, seed):
    if case["call"] == "serve":
        return dict(call="serve", server=Server(2 << 30, max_active=16), requests=_requests(case, seed))
    p = _problem(case, seed)
    mesh = nmgb.Mesh(p["n"], p["dx"], nmgb.F64 if case["f64"] else nmgb.F32, basis=p["basis"])
    state = dict(case, mesh=mesh, terms=p["terms"], m0=p["m0"])
    if case["call"] == "gradient":
        mesh.set_terms(p["terms"])
        mesh.set_zeeman(p["hu"], h_cell=p["hc"], cell_freq=p["hc_freq"])
        state["Ms"] = p["Ms"].requires_grad_()
        state["m0"] = p["m0"].requires_grad_()
        state["weight"] = p["weight"]
        state["spec"] = LossSpec(t_end=case["steps"] * case["dt"], A=p["A"], alpha=p["alpha"], gamma=GAMMA,
                                 method=nmgb.RK4, dt0=case["dt"], sample_dt=case["sample_every"] * case["dt"],
                                 checkpoint_every=case["checkpoint"])
        return state
    mesh.set_material(p["Ms"], p["A"], p["Ku"], p["axis"], p["alpha"], GAMMA)
    mesh.set_zeeman(p["hu"], h_cell=p["hc"], cell_freq=p["hc_freq"])
    mesh.set_terms(p["terms"])
    if case["call"] == "vjp":
        state["v"] = p["v"]
    return state


def run(state):
    call = state["call"]
    if call == "serve":
        server = state["server"]
        tags = [server.submit(**r) for r in state["requests"]]
        done = {r["tag"]: r for r in server.drain(len(tags))}
        return [torch.from_numpy(done[t]["m"]).float() for t in tags]
    mesh = state["mesh"]
    if call == "field":
        return mesh.h_eff(state["m0"], state["terms"])
    if call == "vjp":
        return mesh.h_eff_vjp(state["m0"], state["v"], state["terms"])
    if call == "gradient":
        loss = llg_loss(mesh, state["Ms"], state["m0"], state["weight"], state["spec"])
        return (loss.detach(),) + torch.autograd.grad(loss, (state["Ms"], state["m0"]))
    method = nmgb.DP54 if state["method"] == "dp5" else nmgb.RK4
    mesh.set_state(state["m0"], 0.0, state["dt"])
    if state["until"]:
        mesh.run_until(state["steps"] * state["dt"], method)
    else:
        mesh.run_steps(state["steps"], method)
    m, t, _ = mesh.get_state(device=True)
    return m.to(mesh.dtype), t


# ---------------------------------------------------------------------------------------------- work
def _pad(n):
    p = 1
    while p < 2 * n - 1:
        p *= 2
    return p


def _evaluation(n, basis, size):
    """(bytes, flops) of one field evaluation: m in, h out, the tensor spectrum and the material read once;
    the transforms of the three components at the padded length (pruned to the lines that hold data), the
    tensor product and the 27-point stencil."""
    P = [_pad(v) for v in n]
    nodes = (n[0] + 1) * (n[1] + 1) * (n[2] + 1 if basis == 3 else 1)
    half = [v // 2 + 1 for v in P]
    lg = [math.log2(v) if v > 1 else 0.0 for v in P]
    lines = 2.5 * P[0] * lg[0] * n[1] * n[2] + 5 * half[0] * (P[1] * lg[1] * n[2] + P[1] * P[2] * lg[2])
    flops = 2 * 3 * lines + 30 * half[0] * P[1] * P[2] + nodes * (27 if basis == 3 else 9) * 12
    return size * (6 * nodes + 6 * half[0] * half[1] * half[2]), flops


def work(case):
    if case["call"] == "serve":
        total = [0.0, 0.0]
        for r in _requests(case, 0):
            b, f = _evaluation(r["n"], 3, 4)
            total[0] += 48 * r["m0"].size / 3 + 20 * 6 * b
            total[1] += 20 * 6 * f
        return {"bytes": total[0], "flops": total[1]}
    n, size, basis = (case["n1"], case["n2"], case["n3"]), 8 if case["f64"] else 4, case.get("basis", 3)
    nodes = (n[0] + 1) * (n[1] + 1) * (n[2] + 1 if basis == 3 else 1)
    cells = n[0] * n[1] * n[2]
    b, f = _evaluation(n, basis, size)
    if case["call"] == "field":
        return {"bytes": b, "flops": f}
    if case["call"] == "vjp":  # the field, its transpose and the Ms gradient's demag fields of m and of v
        return {"bytes": 2 * b + size * cells, "flops": 3 * f}
    if case["call"] == "gradient":  # per step and stage: the field forward, its transpose and the Ms gradient
        e = 4 * case["steps"]
        return {"bytes": e * 3 * b + 2 * size * (3 * nodes + cells), "flops": e * 4 * f}
    e = case["steps"] * (6 if case["method"] == "dp5" else 4)
    return {"bytes": e * b + case["steps"] * 48 * nodes, "flops": e * f}


# ---------------------------------------------------------------------------------------------- 64 bits
def _angle(u, v):
    return torch.where(v == 0, torch.zeros_like(u), torch.atan(u / torch.where(v == 0, torch.ones_like(v), v)))


def _newell_f(x, y, z):
    R = torch.sqrt(x * x + y * y + z * z)
    tiny = torch.finfo(x.dtype).tiny
    a = 0.5 * y * (z * z - x * x) * torch.asinh(y / torch.sqrt((x * x + z * z).clamp_min(tiny)))
    b = 0.5 * z * (y * y - x * x) * torch.asinh(z / torch.sqrt((x * x + y * y).clamp_min(tiny)))
    c = x * y * z * _angle(y * z, x * R)
    return a * (x * x + z * z > 0) + b * (x * x + y * y > 0) - c + (2 * x * x - y * y - z * z) * R / 6


def _newell_g(x, y, z):
    R = torch.sqrt(x * x + y * y + z * z)
    tiny = torch.finfo(x.dtype).tiny

    def root(u, v):
        return torch.sqrt((u * u + v * v).clamp_min(tiny))

    return (x * y * z * torch.asinh(z / root(x, y)) + y / 6 * (3 * z * z - y * y) * torch.asinh(x / root(y, z)) +
            x / 6 * (3 * z * z - x * x) * torch.asinh(y / root(x, z)) - z ** 3 / 6 * _angle(x * y, z * R) -
            0.5 * z * y * y * _angle(x * z, y * R) - 0.5 * z * x * x * _angle(y * z, x * R) - x * y * R / 3)


def _tensor(n, dx):
    """Demag tensor of cell offsets 0 <= d < n, (6, n1, n2, n3) for xx, yy, zz, xy, xz, yz: the closed form of
    Newell, Williams and Dunlop near the origin, where its differences still carry digits; farther out the
    dipole kernel integrated against the tent density of two cells' points, by Gauss-Legendre rules on both
    halves of the tent and by the three-point rule of the tent where the kernel is smooth."""
    dev = _device()
    d = torch.meshgrid(*[torch.arange(v, dtype=torch.float64, device=dev) * s for v, s in zip(n, dx)], indexing="ij")
    rho = torch.sqrt(d[0] ** 2 + d[1] ** 2 + d[2] ** 2) / max(dx)
    out = torch.zeros((6,) + n, dtype=torch.float64, device=dev)

    def quadrature(where, s, w):
        X = [v[where] for v in d]
        acc = [torch.zeros_like(X[0]) for _ in range(6)]
        for i in range(len(s)):
            x = X[0] + s[i] * dx[0]
            for j in range(len(s)):
                y = X[1] + s[j] * dx[1]
                for k in range(len(s)):
                    z = X[2] + s[k] * dx[2]
                    r2 = x * x + y * y + z * z
                    q = (w[i] * w[j] * w[k]) / (r2 * torch.sqrt(r2))
                    q3 = 3 * q / r2
                    acc[0] += q3 * x * x - q
                    acc[1] += q3 * y * y - q
                    acc[2] += q3 * z * z - q
                    acc[3] += q3 * x * y
                    acc[4] += q3 * x * z
                    acc[5] += q3 * y * z
        for c in range(6):
            out[c][where] = -dx[0] * dx[1] * dx[2] / (4 * math.pi) * acc[c]

    def tent(points):
        u, w = np.polynomial.legendre.leggauss(points)
        u, w = 0.5 * (u + 1), 0.5 * w
        return np.concatenate([u, -u]), np.concatenate([w * (1 - u), w * (1 - u)])

    near = rho < 5
    X = [v[near] for v in d]
    acc = [torch.zeros_like(X[0]) for _ in range(6)]
    for p in (-1, 0, 1):
        for q in (-1, 0, 1):
            for r in (-1, 0, 1):
                w = (2.0 if p == 0 else -1.0) * (2.0 if q == 0 else -1.0) * (2.0 if r == 0 else -1.0)
                # in units of the largest cell edge
                x, y, z = ((X[0] + p * dx[0]) / max(dx), (X[1] + q * dx[1]) / max(dx), (X[2] + r * dx[2]) / max(dx))
                acc[0] += w * _newell_f(x, y, z)
                acc[1] += w * _newell_f(y, x, z)
                acc[2] += w * _newell_f(z, y, x)
                acc[3] += w * _newell_g(x, y, z)
                acc[4] += w * _newell_g(x, z, y)
                acc[5] += w * _newell_g(y, z, x)
    vol = dx[0] * dx[1] * dx[2] / max(dx) ** 3
    for c in range(6):
        out[c][near] = acc[c] / (4 * math.pi * vol)
    quadrature((rho >= 5) & (rho < 12), *tent(6))
    quadrature((rho >= 12) & (rho < 40), *tent(3))
    a = math.sqrt(0.4)
    quadrature(rho >= 40, np.array([0.0, a, -a]), np.array([7 / 12, 5 / 24, 5 / 24]))
    return out


class _Field:
    """H_eff in 64 bits by plain torch operations on (n1, n2, n3, 3) tensors, differentiable."""

    def __init__(self, p):
        self.n, self.dx, self.terms, self.basis = p["n"], p["dx"], p["terms"], p["basis"]
        dev = _device()

        def cells(v):
            v = torch.as_tensor(v, dtype=torch.float64, device=dev)
            return v if v.dim() else v.reshape(1, 1, 1)

        self.Ms, self.A, self.Ku = cells(p["Ms"]), cells(p["A"]), cells(p["Ku"])
        self.e = torch.tensor(p["axis"], dtype=torch.float64, device=dev)
        self.hu = torch.tensor(p["hu"], dtype=torch.float64, device=dev)
        self.hc = None if p["hc"] is None else torch.as_tensor(p["hc"], dtype=torch.float64, device=dev)
        self.hc_freq = p["hc_freq"]
        self.alpha = p["alpha"]
        # element matrices of the trilinear basis, corner (i1, i2, i3) at index 4 i1 + 2 i2 + i3
        one = [np.array([[1.0, -1.0], [-1.0, 1.0]]) / v for v in self.dx]
        mass = [np.array([[2.0, 1.0], [1.0, 2.0]]) * v / 6 for v in self.dx]
        k = sum(np.kron(np.kron(one[0] if a == 0 else mass[0], one[1] if a == 1 else mass[1]),
                        one[2] if a == 2 else mass[2]) for a in range(3))
        self.stiff = torch.tensor(k, device=dev)
        self.mass8 = torch.tensor(np.kron(np.kron(mass[0], mass[1]), mass[2]), device=dev)
        if self.terms & nmgb.DEMAG:
            self._spectrum()

    def _spectrum(self):
        P = [_pad(v) for v in self.n]
        N = _tensor(self.n, self.dx)
        parity = ((1, 1, 1), (1, 1, 1), (1, 1, 1), (-1, -1, 1), (-1, 1, -1), (1, -1, -1))
        self.P, self.hat = P, []
        for c in range(6):
            f = N[c]
            for a in range(3):
                if P[a] == 1:
                    continue
                shape = list(f.shape)
                shape[a] = P[a] - 2 * self.n[a] + 1
                f = torch.cat([f, f.new_zeros(shape), parity[c][a] * f.narrow(a, 1, self.n[a] - 1).flip(a)], a)
            # real (even) or imaginary-free product of two odd directions: the spectrum is real
            self.hat.append(torch.fft.rfftn(f, dim=(2, 1, 0)).real.contiguous())
            del f

    def _demag(self, M):
        P, n = self.P, self.n
        sp = [torch.fft.rfftn(M[c], s=(P[2], P[1], P[0]), dim=(2, 1, 0)) for c in range(3)]
        xx, yy, zz, xy, xz, yz = self.hat
        out = []
        for row in ((xx, xy, xz), (xy, yy, yz), (xz, yz, zz)):
            s = sum(t * v for t, v in zip(row, sp))
            h = torch.fft.irfftn(s, s=(P[2], P[1], P[0]), dim=(2, 1, 0))
            out.append(-h[:n[0], :n[1], :n[2]])
        return out

    def __call__(self, m, t=0.0, Ms=None):
        Ms = self.Ms if Ms is None else Ms
        n = self.n
        if self.basis == 2:
            m = m.expand(-1, -1, n[2] + 1, -1)
        on = (Ms > 0).to(torch.float64)
        V8 = self.dx[0] * self.dx[1] * self.dx[2] / 8
        corners = [(slice(i, i + n[0]), slice(j, j + n[1]), slice(k, k + n[2])) for i in (0, 1) for j in (0, 1)
                   for k in (0, 1)]
        nodes = tuple(v + 1 for v in n)
        cell = torch.zeros(n, dtype=torch.float64, device=m.device)
        mass = torch.zeros(nodes, dtype=torch.float64, device=m.device)
        for s in corners:
            mass[s] = mass[s] + (MU0 * V8) * (Ms + cell)
        comp = [m[..., c] for c in range(3)]
        num = [torch.zeros(nodes, dtype=torch.float64, device=m.device) for _ in range(3)]
        if self.terms & nmgb.EXCH:
            for c in range(3):
                mc = [comp[c][s] for s in corners]
                for i in range(8):
                    # (rows of the element matrix sum to zero)
                    d = sum(float(self.stiff[i, j]) * (mc[j] - mc[i]) for j in range(8) if j != i)
                    num[c][corners[i]] = num[c][corners[i]] - 2 * (self.A * on) * d
        if self.terms & nmgb.ANIS:
            em = self.e[0] * comp[0] + self.e[1] * comp[1] + self.e[2] * comp[2]
            ec = [em[s] for s in corners]
            for i in range(8):
                d = 2 * (self.Ku * on) * sum(float(self.mass8[i, j]) * ec[j] for j in range(8))
                for c in range(3):
                    num[c][corners[i]] = num[c][corners[i]] + self.e[c] * d
        H = [0.0, 0.0, 0.0]
        if self.terms & nmgb.DEMAG:
            H = self._demag([Ms * 0.125 * sum(comp[c][s] for s in corners) for c in range(3)])
        if self.terms & nmgb.ZEE and self.hc is not None:
            f = math.sin(2 * math.pi * self.hc_freq * t) if self.hc_freq else 1.0
            H = [H[c] + f * self.hc[..., c] for c in range(3)]
        for c in range(3):
            if torch.is_tensor(H[c]):
                w = (MU0 * V8) * Ms * H[c]
                for s in corners:
                    num[c][s] = num[c][s] + w
        if self.basis == 2:
            mass = mass.sum(2, keepdim=True)
            num = [v.sum(2, keepdim=True) for v in num]
        self.on_node = mass > 0
        inv = torch.where(self.on_node, 1 / torch.where(self.on_node, mass, torch.ones_like(mass)),
                          torch.zeros_like(mass))
        hu = self.hu if self.terms & nmgb.ZEE else torch.zeros_like(self.hu)
        return torch.stack([inv * num[c] + hu[c] * self.on_node for c in range(3)], -1)

    def slope(self, m, t, Ms=None):
        h = self(m, t, Ms)
        a = torch.linalg.cross(m, h)
        k = a + self.alpha * torch.linalg.cross(m, a)
        return -GAMMA / (1 + self.alpha ** 2) * k * self.on_node[..., None]


_DP = ((1 / 5,), (3 / 40, 9 / 40), (44 / 45, -56 / 15, 32 / 9),
       (19372 / 6561, -25360 / 2187, 64448 / 6561, -212 / 729),
       (9017 / 3168, -355 / 33, 46732 / 5247, 49 / 176, -5103 / 18656),
       (35 / 384, 0.0, 500 / 1113, 125 / 192, -2187 / 6784, 11 / 84))
_DPC = (0.0, 1 / 5, 3 / 10, 4 / 5, 8 / 9, 1.0, 1.0)
_DPE = (35 / 384 - 5179 / 57600, 0.0, 500 / 1113 - 7571 / 16695, 125 / 192 - 393 / 640,
        -2187 / 6784 + 92097 / 339200, 11 / 84 - 187 / 2100, -1 / 40)


def _rk4_step(F, m, t, dt, Ms=None):
    k1 = F.slope(m, t, Ms)
    k2 = F.slope(m + 0.5 * dt * k1, t + 0.5 * dt, Ms)
    k3 = F.slope(m + 0.5 * dt * k2, t + 0.5 * dt, Ms)
    k4 = F.slope(m + dt * k3, t + dt, Ms)
    return _unit(m + dt / 6 * (k1 + 2 * k2 + 2 * k3 + k4))


def _dp5(F, m, dt, attempts=None, t_end=None, tol=1e-5):
    """Dormand-Prince 5(4) with a FSAL slope: `attempts` step attempts, or steps to t_end."""
    t, k1 = 0.0, F.slope(m, 0.0)
    if t_end is not None:
        dt = min(dt, t_end)
    while attempts is None or attempts > 0:
        k = [k1]
        for s in range(6):
            y = m + dt * sum(a * v for a, v in zip(_DP[s], k) if a)
            k.append(F.slope(y, t + _DPC[s + 1] * dt))
        e = dt * sum(c * v for c, v in zip(_DPE, k) if c)
        scale = tol + tol * torch.maximum(m.abs(), y.abs())
        on = F.on_node[..., None]
        err = math.sqrt(float(((e / scale) ** 2 * on).sum()) / (3 * float(F.on_node.sum())))
        factor = 5.0 if err == 0 else min(5.0, max(0.2, 0.9 * err ** -0.2))
        if err <= 1:
            t += dt
            m, k1 = _unit(y), k[6]
        dt *= factor
        if attempts is not None:
            attempts -= 1
        if t_end is not None:
            if t_end - t <= 1e-12 * t_end:
                break
            dt = min(dt, t_end - t)
    return m


def exact(case, seed):
    if case["call"] == "serve":
        out = []
        for r in _requests(case, seed):
            F = _Field(dict(r, basis=3, Ku=0.0, axis=(0.0, 0.0, 1.0), terms=nmgb.EXCH | nmgb.ZEE | nmgb.DEMAG,
                            hu=r["h"], hc=None, hc_freq=0.0))
            out.append(_dp5(F, torch.as_tensor(r["m0"], device=_device()), r["dt0"], t_end=r["t_end"]).cpu())
        return out
    p = _problem(case, seed)
    F = _Field(p)
    m0 = p["m0"].double()
    if case["call"] == "field":
        return F(m0)
    if case["call"] == "vjp":
        m0.requires_grad_()
        Ms = F.Ms.expand(p["n"]).clone().requires_grad_()
        return torch.autograd.grad((F(m0, 0.0, Ms) * p["v"].double()).sum(), (m0, Ms))
    if case["call"] == "gradient":
        Ms, m = F.Ms.clone().requires_grad_(), m0.requires_grad_()
        W = torch.as_tensor(p["weight"], device=m0.device)
        loss = 0.0
        for i in range(case["steps"]):
            m = _rk4_step(F, m, i * case["dt"], case["dt"], Ms)
            if (i + 1) % case["sample_every"] == 0:
                loss = loss + (W * m * m).sum()
        return (loss.detach(),) + torch.autograd.grad(loss, (Ms, m0))
    m = m0
    if case["method"] == "dp5":
        t_end = case["steps"] * case["dt"] if case["until"] else None
        m = _dp5(F, m, case["dt"], None if case["until"] else case["steps"], t_end)
    else:
        for i in range(case["steps"]):
            m = _rk4_step(F, m, i * case["dt"], case["dt"])
    # (the time follows from the error estimate, whose digits depend on the working precision)
    return m, None
