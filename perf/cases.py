"""Performance cases of the residual / Runge-Kutta library and its indicator network.

Every case is one call (or the few calls that belong together) that a program
using the package makes, on the repository's own workloads: the Taylor-Green
vortex with a random-phase velocity perturbation on a jittered lattice of
hexahedra, or of the tetrahedra, prisms or pyramids it splits into.  ``listed()``
names the usual ones, ``draw()`` gives more of the same ranges.

``exact()`` computes what ``run()`` returns in plain torch FP64 from the mesh
and the state alone (geometry and least squares by quadrature and a QR
factorisation of its own), for every case but the gated step, whose flags hang
on the indicator's BF16 roundings, and the training epoch, whose Adam steps
carry them on from batch to batch (its gradient has one).
"""
import math

import numpy as np
import torch

TWO_PI = 2.0 * math.pi
GAMMA, PRANDTL, CFL, LAMBDA, EPSILON, ALPHA = 1.4, 0.71, 0.5, 1000.0, 1e-6, 4.0 / 3.0
AMPLITUDE = 0.05   # rms of the velocity perturbation
LR, W_POS, W_NEG = 1e-3, 10.0, 0.5
DEVICE = "cuda" if torch.cuda.is_available() else "cpu"


# ------------------------------------------------------------------ cases
def _mesh_case(name, op, mesh, size, order, scheme, precision, mach, re=1600.0, integrator=0, walls=False, jitter=0.1,
               steps=1):
    nx, ny, nz = size
    c = {"op": op, "mesh": mesh, "nx": nx, "ny": ny, "nz": nz, "jitter": jitter, "order": order, "scheme": scheme,
         "precision": precision, "mach": mach, "re": re, "integrator": integrator, "walls": walls, "steps": steps}
    return c if name is None else {"name": name, **c}


def listed():
    return [
        # a small uniform P1 run between two diagnostics, as the history of a coarse run is written: launches and latency
        _mesh_case("steps_hex16_p1_fp64", "steps", "hex", (16, 16, 16), 1, 0, 0, 0.1, jitter=0.0, steps=10),
        # the plain FP64 form's step at Mach 1.25 (the labels of the gate, and the reference of every history)
        _mesh_case("step_hex80_p2_fp64", "step", "hex", (72, 80, 88), 2, 1, 0, 1.25),
        # the mixed form on a state that lives in pinned host memory, copied in and out on every call
        _mesh_case("host_hex64_p2_mixed", "host", "hex", (64, 64, 64), 2, 1, 1, 0.1),
        # the mixed form's step, the largest mesh
        _mesh_case("step_hex96_p2_mixed", "step", "hex", (96, 96, 96), 2, 1, 1, 1.25),
        # the learned form: features, network and gated reconstruction, flags evaluated on every step
        _mesh_case("gated_hex96_p2_mixed", "gated", "hex", (96, 96, 96), 2, 1, 1, 1.25),
        # tetrahedra
        _mesh_case("step_tet42_p2_mixed", "step", "tet", (40, 42, 45), 2, 1, 1, 0.1),
        # P3 with the five-stage integrator
        _mesh_case("step_hex40_p3_mixed_ssp54", "step", "hex", (40, 40, 40), 3, 1, 1, 1.25, integrator=1),
        # P4 in both forms, the residual on its own as an implicit or steady outer solver calls it
        _mesh_case("residual_hex24_p4_fp64", "residual", "hex", (24, 24, 24), 4, 1, 0, 1.25),
        _mesh_case("residual_hex32_p4_mixed", "residual", "hex", (32, 32, 32), 4, 1, 1, 1.25),
        # an inviscid box between slip walls
        _mesh_case("residual_walls36_p2_fp64", "residual", "hex", (33, 36, 39), 2, 1, 0, 0.5, re=0.0, walls=True),
        # one epoch of the indicator's training, the weights read back
        {"name": "train_131072_rows", "op": "train", "rows": 131072, "batch": 4096},
        # one snapshot of the training data (features, labels) and its logits, as the threshold is chosen from them
        _mesh_case("collect_hex50_p2_fp64", "collect", "hex", (48, 50, 52), 2, 1, 0, 1.25),
    ]


def _size(rng, low, high):
    """Lattice cells per direction, log-uniform in the total, the directions up to 30 % apart."""
    n = math.exp(rng.uniform(math.log(low), math.log(high))) ** (1.0 / 3.0)
    return tuple(max(10, int(round(n * rng.uniform(0.87, 1.15)))) for _ in range(3))


def draw(rng):
    kind = rng.choice(["p1", "p2_fp64", "p2_mixed", "host", "gated", "split", "p3", "p4", "walls", "train", "collect"])
    mach = rng.choice([0.1, 0.3, 0.5, 1.25])
    integrator = rng.randint(0, 1)
    if kind == "p1":
        prec = rng.randint(0, 1)
        mach = max(mach, 0.5) if prec else mach  # below, the dilatational dissipation is under the mixed form's resolution
        return _mesh_case(None, "steps", "hex", _size(rng, 1000, 150000), 1, 0, prec, mach, integrator=integrator,
                          steps=rng.randint(1, 12))
    if kind == "p2_fp64":
        return _mesh_case(None, rng.choice(["step", "residual"]), "hex", _size(rng, 1500, 250000), 2, rng.randint(0, 1),
                          0, mach, integrator=integrator)
    if kind == "p2_mixed":
        return _mesh_case(None, rng.choice(["step", "residual"]), "hex", _size(rng, 1500, 400000), 2, rng.randint(0, 1),
                          1, mach, integrator=integrator)
    if kind == "host":
        return _mesh_case(None, "host", "hex", _size(rng, 1500, 250000), 2, 1, rng.randint(0, 1), mach,
                          integrator=integrator, steps=rng.randint(1, 3))
    if kind == "gated":
        return _mesh_case(None, "gated", "hex", _size(rng, 20000, 400000), 2, 1, rng.choice([0, 1, 1]), mach,
                          integrator=integrator)
    if kind == "split":
        mesh = rng.choice(["tet", "tet", "prism", "pyramid"])
        prec = rng.randint(0, 1) if mesh == "tet" else 0
        mach = min(mach, 0.5) if mesh == "pyramid" else mach  # their reconstruction leaves the physical range above
        return _mesh_case(None, rng.choice(["step", "residual"]), mesh, _size(rng, 1000, 40000 if prec else 12000), 2, 1,
                          prec, mach, integrator=integrator)
    if kind == "p3":
        prec = rng.randint(0, 1)
        return _mesh_case(None, rng.choice(["step", "residual"]), "hex", _size(rng, 1500, 50000 if prec else 12000), 3,
                          rng.choice([0, 1, 1]), prec, mach, integrator=integrator)
    if kind == "p4":
        prec = rng.randint(0, 1)
        return _mesh_case(None, "residual", "hex", _size(rng, 1500, 25000 if prec else 10000), 4, rng.choice([0, 1, 1]),
                          prec, mach)
    if kind == "walls":
        order = rng.randint(1, 2)
        return _mesh_case(None, rng.choice(["step", "residual"]), "hex", _size(rng, 1500, 80000), order,
                          rng.randint(0, 1) if order == 2 else 0, 0, mach, re=0.0, walls=True)
    if kind == "train":
        rows = int(math.exp(rng.uniform(math.log(3000), math.log(250000))))
        if rng.random() < 0.4:
            return {"op": "grad", "rows": rows}
        return {"op": "train", "rows": rows, "batch": 8 * max(rng.randint(64, 1024), rows // 256)}
    return _mesh_case(None, "collect", "hex", _size(rng, 1500, 150000), 2, 1, 0, mach)


# ----------------------------------------------------------------- inputs
_HEX = np.array([[0, 0, 0], [1, 0, 0], [1, 1, 0], [0, 1, 0], [0, 0, 1], [1, 0, 1], [1, 1, 1], [0, 1, 1]])
_TETS = [[0, 1, 2, 6], [0, 5, 1, 6], [0, 2, 3, 6], [0, 3, 7, 6], [0, 4, 5, 6], [0, 7, 4, 6]]
_PRISMS = [[0, 1, 2, 4, 5, 6], [0, 2, 3, 4, 6, 7]]
_PYRAMIDS = [[0, 3, 7, 4, 8], [1, 5, 6, 2, 8], [0, 4, 5, 1, 8], [3, 2, 6, 7, 8], [0, 1, 2, 3, 8], [4, 7, 6, 5, 8]]
_PARTS = {"hex": [list(range(8))], "tet": _TETS, "prism": _PRISMS, "pyramid": _PYRAMIDS}  # node 8: the middle


def lattice(case):
    """(nodes [n, 3], cells [N, nodes per cell], box) of the case's mesh: a lattice over [0, 2 pi]^3 whose inner nodes
    are jittered, every hexahedron split into the case's elements."""
    n = np.array([case["nx"], case["ny"], case["nz"]])
    m = n + 1
    k, j, i = np.meshgrid(*[np.arange(v) for v in m[::-1]], indexing="ij")
    ijk = np.stack([i.ravel(), j.ravel(), k.ravel()], axis=1)
    nodes = TWO_PI * ijk / n
    if case["jitter"]:
        d = np.random.default_rng(3).uniform(-1.0, 1.0, nodes.shape) * (case["jitter"] * TWO_PI / n)
        inner = ((ijk > 0) & (ijk < n)).all(axis=1)
        nodes[inner] += d[inner]
    ck, cj, ci = np.meshgrid(*[np.arange(v) for v in n[::-1]], indexing="ij")
    base = np.stack([ci.ravel(), cj.ravel(), ck.ravel()], axis=1)
    o = base[:, None, :] + _HEX[None]
    hexes = o[..., 0] + m[0] * (o[..., 1] + m[1] * o[..., 2])
    if case["mesh"] == "pyramid":
        hexes = np.concatenate([hexes, len(nodes) + np.arange(len(hexes))[:, None]], axis=1)
        nodes = np.concatenate([nodes, nodes[hexes[:, :8]].mean(axis=1)])
    parts = np.array(_PARTS[case["mesh"]])
    box = np.full(3, TWO_PI)
    if case["walls"]:
        box[2] = 0.0
    return nodes, hexes[:, parts].reshape(-1, parts.shape[1]).astype(np.int64), box


def start_state(case, seed, nodes, cells):
    """[5, N] conserved Taylor-Green state at the cells' vertex means, with the seed's velocity perturbation, on the
    GPU in the caller's cell order."""
    x = _on_gpu(nodes)[_on_gpu(cells)].mean(dim=1)
    rng = np.random.default_rng(seed)
    d = torch.zeros_like(x)
    for c in range(3):
        ks = rng.integers(-3, 4, size=(8, 3)).astype(np.float64)
        ks[np.all(ks == 0, axis=1)] = [1, 0, 0]
        if case["walls"]:
            ks[:, 2] = 0.0
        d[:, c] = torch.sin(x @ _on_gpu(ks).T + _on_gpu(rng.uniform(0.0, TWO_PI, size=8))).sum(dim=1)
    d *= AMPLITUDE / torch.sqrt((d * d).sum(dim=1).mean())
    X, Y, Z = x.T
    u = torch.sin(X) * torch.cos(Y) * torch.cos(Z) + d[:, 0]
    v = -torch.cos(X) * torch.sin(Y) * torch.cos(Z) + d[:, 1]
    w = d[:, 2]
    p = 1.0 / (GAMMA * case["mach"] ** 2) + (torch.cos(2 * Z) + 2.0) * (torch.cos(2 * X) + torch.cos(2 * Y)) / 16.0
    rho = GAMMA * case["mach"] ** 2 * p
    return torch.stack([rho, rho * u, rho * v, rho * w, p / (GAMMA - 1.0) + 0.5 * rho * (u * u + v * v + w * w)])


def training_set(case, seed):
    """Feature rows (BF16 [n, 32]) and labels (float [n]): jumps and sensors with a long tail, the rows with the
    largest jumps troubled (about 4 %)."""
    g = torch.Generator(device=DEVICE).manual_seed(seed)
    n = case["rows"]
    size = torch.exp(1.2 * torch.randn(n, 1, generator=g, device=DEVICE) - 4.0)
    x = torch.randn(n, 32, generator=g, device=DEVICE) * size
    x[:, 24:] = x[:, 24:].abs() / (x[:, 24:].abs() + 0.05)
    y = (x[:, :24].abs().amax(dim=1) > 0.35).float()
    return x.to(torch.bfloat16).contiguous(), y


def initial_weights(seed):
    """The network's 6337 parameters before training: He-normal weights, zero biases."""
    th, rng = np.zeros(6337, np.float32), np.random.default_rng(seed)
    for at, n, var in ((0, 2048, 2.0 / 32), (2112, 4096, 2.0 / 64), (6272, 64, 1.0 / 64)):
        th[at:at + n] = rng.normal(0.0, math.sqrt(var), n)
    return th


def _on_gpu(a):
    return torch.from_numpy(np.ascontiguousarray(a)).to(DEVICE)


def prepare(case, seed):
    from paper_2609_07387_gb300 import gate, ucns

    if case["op"] in ("train", "grad"):
        X, y = training_set(case, seed)
        net = ucns.Net()
        net.set_params(initial_weights(seed))
        return {"case": case, "net": net, "X": X, "y": y}
    nodes, cells, box = lattice(case)
    mesh = ucns.Mesh(nodes, cells, box, ucns.Params(
        order=case["order"], scheme=case["scheme"], precision=case["precision"], gamma=GAMMA, Pr=PRANDTL, Re=case["re"],
        Mach=case["mach"], cfl=CFL, lam_central=LAMBDA, eps=EPSILON, alpha=ALPHA, integrator=case["integrator"]))
    U = start_state(case, seed, nodes, cells)[:, _on_gpu(mesh.perm)].contiguous()
    s = {"case": case, "mesh": mesh, "U": U}
    if case["op"] == "host":
        s["U"] = U.cpu().pin_memory()
    if case["op"] in ("gated", "collect"):
        s["net"] = gate.rule_network(0.0)  # the sum of the cell's jumps
    if case["op"] == "gated":
        z = s["net"].forward(mesh.gate_features(U)[0])
        mesh.gate_attach(s["net"], float(z.sort().values[int(0.98 * z.numel())]))  # flags one cell in fifty
        mesh.gate_enable(True)
    return s


def run(s):
    case, op = s["case"], s["case"]["op"]
    if op == "grad":
        return s["net"].grad(s["X"], s["y"], w_pos=W_POS, w_neg=W_NEG)
    if op == "train":
        s["net"].train(s["X"], s["y"], batch=case["batch"], lr=LR, w_pos=W_POS, w_neg=W_NEG)
        return s["net"].params()
    mesh, U = s["mesh"], s["U"]
    if op == "residual":
        return mesh.residual(U)
    if op == "steps":
        t = mesh.rk_steps(U, case["steps"])
        return {"U": U, **{k: np.float64(v) for k, v in (("t", t), *mesh.diagnostics(U).items())}}
    if op == "host":
        t = mesh.rk_steps_host(U, case["steps"])
        return {"U": U, "t": np.float64(t)}
    if op == "collect":
        X, _ = mesh.gate_features(U)
        return {"X": X, "dev": mesh.gate_labels(U), "z": s["net"].forward(X)}
    mesh.rk_step(U)
    return U


# ------------------------------------------------------- work, tolerances
def _modes(order):
    return (order + 1) * (order + 2) * (order + 3) // 6 - 1


def work(case):
    """Bytes: per stage the least-squares rows, stencil ids, geometry and state read, the state or residual written;
    flops: differences, contractions, indicators, point evaluations and fluxes (an FMA is two)."""
    if case["op"] in ("train", "grad"):
        n, steps = case["rows"], -(-case["rows"] // case.get("batch", case["rows"]))
        return {"bytes": n * 68 + steps * 6337 * 24, "flops": 3 * 2.0 * n * (32 * 64 + 64 * 64 + 64)}
    parts, faces = {"hex": (1, 6), "tet": (6, 4), "prism": (2, 5), "pyramid": (6, 5)}[case["mesh"]]
    N = case["nx"] * case["ny"] * case["nz"] * parts
    F = N * faces // 2
    order, w = case["order"], 4 if case["precision"] else 8
    K, nq = _modes(order), order * order
    M, nd = 2 * K, faces if case["scheme"] and order > 1 else 0
    KD = 9 if order == 4 else 3
    MD = 2 * KD
    share = 0.02 if case["op"] == "gated" else 1.0  # cells that take the directional candidates
    cell_bytes = K * M * w + M * 4 + 7 * w + 40
    cell_flops = 5.0 * (M + 2 * M * K)
    if nd:
        cell_bytes += share * nd * (KD * MD * w + MD * 4) + (K * (K + 1) // 2 * w if order > 2 else 0)
        cell_flops += share * 5.0 * (nd * (MD + 2 * KD * MD) + 2 * (K * K + nd * KD * KD) + 120)
    if case["op"] == "collect":  # features (BF16 rows) and labels, each with its reconstruction, then the logits
        return {"bytes": N * (2 * cell_bytes + 64 + 4 + 64 + 4), "flops": N * (1.5 * cell_flops + 2.0 * 6208)}
    gradients = 3 if case["re"] > 0 else 0
    point_flops = 20.0 * K + gradients * 10.0 * _modes(order - 1) + gradients * 10.0 + 358
    stage_bytes = N * (cell_bytes + 40) + F * (nq * 6 * w + 4 * w + 8)
    stage_flops = N * cell_flops + F * nq * point_flops
    stages = (5 if case["integrator"] else 3) * case["steps"] if case["op"] != "residual" else 1
    total = {"bytes": stages * stage_bytes, "flops": stages * stage_flops}
    if case["op"] == "gated":
        total["bytes"] += N * (64 + 64 + 2)
        total["flops"] += N * (5.0 * (M + 2 * M * K) + 2.0 * 6208)
    if case["op"] == "steps":
        total["bytes"] += N * (cell_bytes + 60)
        total["flops"] += N * cell_flops
    if case["op"] == "host":
        total["bytes"] += 2 * 40 * N
    return total


def tolerance(case):
    if case["op"] == "train":
        return {"rel": 5e-4, "max": 0.1}
    if case["op"] == "grad":  # a rounding to BF16 that falls the other way here and there
        return {"rel": 1e-5, "max": 2e-4}
    if case["op"] == "collect":  # BF16 features
        return {"rel": 1e-3, "max": 0.02}
    # against exact(), over the declared ranges: the residual is a difference of fluxes 10^2 (Mach 1.25) to 10^4 (Mach
    # 0.1) times its size, FP64 up to 8e-14 and 4e-13 off, mixed 4e-6 and 7e-6; a step adds dt times it to the state
    slow = case["mach"] < 1.0
    if case["op"] == "residual":
        if case["precision"]:
            return {"rel": 3e-5, "max": 5e-4} if slow else {"rel": 2e-5, "max": 2.5e-4}
        return {"rel": 1.5e-12, "max": 1.6e-11} if slow else {"rel": 3.5e-13, "max": 6e-12}
    if case["op"] == "steps":  # the dilatational dissipation among the outputs, small beside the solenoidal one
        return {"rel": 3e-7, "max": 5e-7} if case["precision"] else {"rel": 3e-14, "max": 5e-14}
    if case["precision"]:
        return {"rel": 4e-8, "max": 5e-7}
    return {"rel": 3e-15, "max": 3e-14}


# ------------------------------------------------- the same in plain FP64
_FACES = {
    "hex": [[0, 4, 7, 3], [1, 2, 6, 5], [0, 1, 5, 4], [3, 7, 6, 2], [0, 3, 2, 1], [4, 5, 6, 7]],
    "tet": [[0, 2, 1], [0, 1, 3], [1, 2, 3], [0, 3, 2]],
    "prism": [[0, 2, 1], [3, 4, 5], [0, 1, 4, 3], [1, 2, 5, 4], [2, 0, 3, 5]],
    "pyramid": [[0, 3, 2, 1], [0, 1, 4], [1, 2, 4], [2, 3, 4], [3, 0, 4]],
}


def _exponents(order):
    """The non-constant monomials of the basis, linear first."""
    return [(a, b, d - a - b) for d in range(1, order + 1) for a in range(d, -1, -1) for b in range(d - a, -1, -1)]


def _gauss(n):
    x, w = np.polynomial.legendre.leggauss(n)
    return 0.5 * (x + 1.0), 0.5 * w


def _cross(a, b):
    return torch.linalg.cross(a, b, dim=-1)


def _reference_map(mesh, p, s, t, u):
    """Position and Jacobian of the unit cube's point (s, t, u) in elements with corners p [N, n, 3]."""
    c = [p[:, k] for k in range(p.shape[1])]
    if mesh == "hex":
        def q(k, f, g):  # bilinear in (f, g) on four corners
            return (1 - f) * (1 - g) * c[k] + f * (1 - g) * c[k + 1] + f * g * c[k + 2] + (1 - f) * g * c[k + 3]
        low, top = q(0, s, t), q(4, s, t)
        ds = sum(w * ((1 - t) * (c[k + 1] - c[k]) + t * (c[k + 2] - c[k + 3])) for k, w in ((0, 1 - u), (4, u)))
        dt = sum(w * ((1 - s) * (c[k + 3] - c[k]) + s * (c[k + 2] - c[k + 1])) for k, w in ((0, 1 - u), (4, u)))
        return (1 - u) * low + u * top, (ds * _cross(dt, top - low)).sum(-1)
    if mesh == "prism":
        e1, e2, f1, f2 = c[1] - c[0], c[2] - c[1], c[4] - c[3], c[5] - c[4]
        low, top = c[0] + s * e1 + s * t * e2, c[3] + s * f1 + s * t * f2
        ds = (1 - u) * (e1 + t * e2) + u * (f1 + t * f2)
        dt = s * ((1 - u) * e2 + u * f2)
        return (1 - u) * low + u * top, (ds * _cross(dt, top - low)).sum(-1)
    if mesh == "pyramid":
        q = (1 - s) * (1 - t) * c[0] + s * (1 - t) * c[1] + s * t * c[2] + (1 - s) * t * c[3]
        qs = (1 - t) * (c[1] - c[0]) + t * (c[2] - c[3])
        qt = (1 - s) * (c[3] - c[0]) + s * (c[2] - c[1])
        return (1 - u) * q + u * c[4], ((1 - u) * qs * _cross((1 - u) * qt, c[4] - q)).sum(-1)
    six = ((c[1] - c[0]) * _cross(c[2] - c[0], c[3] - c[0])).sum(-1)
    return c[0] + s * (c[1] - c[0]) + s * t * (c[2] - c[1]) + s * t * u * (c[3] - c[2]), s * s * t * six


def _face_points(p, order):
    """Gauss points and area vectors [N, q, 3] of faces with corners p [N, 3 or 4, 3]."""
    c = [p[:, k] for k in range(p.shape[1])]
    if len(c) == 3 and order == 1:
        return ((c[0] + c[1] + c[2]) / 3.0)[:, None], (0.5 * _cross(c[1] - c[0], c[2] - c[0]))[:, None]
    g, w = _gauss(order)
    xs, ds = [], []
    for a, wa in zip(g, w):
        for b, wb in zip(g, w):
            if len(c) == 4:
                xs.append((1 - a) * (1 - b) * c[0] + a * (1 - b) * c[1] + a * b * c[2] + (1 - a) * b * c[3])
                da = (1 - b) * (c[1] - c[0]) + b * (c[2] - c[3])
                db = (1 - a) * (c[3] - c[0]) + a * (c[2] - c[1])
                ds.append(wa * wb * _cross(da, db))
            else:
                xs.append(c[0] + a * (c[1] - c[0]) + a * b * (c[2] - c[1]))
                ds.append(wa * wb * a * _cross(c[1] - c[0], c[2] - c[1]))
    return torch.stack(xs, 1), torch.stack(ds, 1)


def _monomials(x, exps, beta=(0, 0, 0)):
    """d^beta of the monomials at points x [..., 3] -> [..., len(exps)]."""
    out = []
    for e in exps:
        f, t = 1.0, None
        for d in range(3):
            for q in range(beta[d]):
                f *= e[d] - q
        if f == 0.0:
            out.append(torch.zeros_like(x[..., 0]))
            continue
        for d in range(3):
            if e[d] - beta[d]:
                g = x[..., d] ** (e[d] - beta[d])
                t = g if t is None else t * g
        out.append(torch.full_like(x[..., 0], f) if t is None else f * t)
    return torch.stack(out, -1)


class _Template:
    """The lattice's element adjacency: what lies across each local face of each of the parts a hexahedron splits into,
    as (lattice offset, part)."""

    def __init__(self, mesh):
        corner = [tuple(2 * v for v in h) for h in _HEX.tolist()] + [(1, 1, 1)]
        self.parts = [[corner[k] for k in part] for part in _PARTS[mesh]]
        self.faces = _FACES[mesh]
        owner = {}
        around = [(a, b, c) for a in (-1, 0, 1) for b in (-1, 0, 1) for c in (-1, 0, 1)]
        for o in around:
            for t in range(len(self.parts)):
                for f in self.faces:
                    owner.setdefault(frozenset(self.nodes(o, t)[k] for k in f), []).append((o, t))
        self.across = [[next(x for x in owner[frozenset(self.nodes((0, 0, 0), t)[k] for k in f)] if x != ((0, 0, 0), t))
                        for f in self.faces] for t in range(len(self.parts))]

    def nodes(self, o, t):
        return [tuple(n[d] + 2 * o[d] for d in range(3)) for n in self.parts[t]]

    def search(self, start, avoid, depth):
        """{(offset, part): face-graph distance from start}, never through `avoid`."""
        seen, front = {start: 0}, [start]
        for d in range(1, depth + 1):
            new = []
            for o, t in front:
                for do, tn in self.across[t]:
                    n = (tuple(o[q] + do[q] for q in range(3)), tn)
                    if n not in seen and n != avoid:
                        seen[n] = d
                        new.append(n)
            front = new
        return seen


class _Scheme:
    """The residual of a case in FP64, in the caller's cell order."""

    def __init__(self, case):
        self.case = case
        mesh, order = case["mesh"], case["order"]
        nodes, cells, box = lattice(case)
        self.template = T = _Template(mesh)
        self.n = (case["nx"], case["ny"], case["nz"])
        self.P = len(T.parts)
        self.N = len(cells)
        self.perm = self.morton(nodes, cells)
        corners = _on_gpu(nodes)[_on_gpu(cells)]
        self.box = _on_gpu(box)
        hexes = torch.arange(self.N // self.P, device=DEVICE)
        self.hex_at = torch.stack([hexes % self.n[0], hexes // self.n[0] % self.n[1],
                                   hexes // (self.n[0] * self.n[1])], 1)
        g, w = _gauss(3 if order < 3 else 5)
        xs, ws = [], []
        for a, wa in zip(g, w):
            for b, wb in zip(g, w):
                for c, wc in zip(g, w):
                    x, j = _reference_map(mesh, corners, a, b, c)
                    xs.append(x)
                    ws.append(wa * wb * wc * j)
        self.xq, wq = torch.stack(xs, 1), torch.stack(ws, 1)
        self.V = wq.sum(1)
        self.wq = wq / self.V[:, None]
        self.cen = (self.wq[..., None] * self.xq).sum(1)
        self.h = self.V ** (1.0 / 3.0)
        self.exps = _exponents(order)
        self.K = len(self.exps)
        local = (self.xq - self.cen[:, None]) / self.h[:, None, None]
        self.mean = (self.wq[..., None] * _monomials(local, self.exps)).sum(1)
        self.weno = case["scheme"] == 1 and order > 1
        if self.weno:
            self.si = torch.zeros(self.N, self.K, self.K, dtype=torch.float64, device=DEVICE)
            for beta in [(0, 0, 0)] + self.exps:
                if sum(beta):
                    D = _monomials(local, self.exps, beta)
                    self.si += (D * self.wq[..., None]).transpose(1, 2) @ D
        self.stencils()
        self.face_geometry(corners)

    @staticmethod
    def morton(nodes, cells):
        low, span = nodes.min(0), nodes.max(0) - nodes.min(0)
        s = np.zeros((len(cells), 3))
        for a in range(cells.shape[1]):
            s += nodes[cells[:, a]]
        q = np.clip((s / cells.shape[1] - low) / span * 2097151.0, 0.0, 2097151.0).astype(np.uint64)
        code = np.zeros(len(cells), dtype=np.uint64)
        for bit in range(21):
            for d in range(3):
                code |= ((q[:, d] >> np.uint64(bit)) & np.uint64(1)) << np.uint64(3 * bit + d)
        return torch.from_numpy(np.argsort(code, kind="stable")).to(DEVICE)

    def neighbours(self, o, t):
        """Ids of the part t of the hexahedra at offset o, -1 outside the box."""
        at, out = self.hex_at + torch.tensor(o, device=DEVICE), None
        for d in range(3):
            if self.box[d] > 0:
                at[:, d] %= self.n[d]
            else:
                bad = (at[:, d] < 0) | (at[:, d] >= self.n[d])
                out = bad if out is None else out | bad
        ids = (at[:, 0] + self.n[0] * (at[:, 1] + self.n[1] * at[:, 2])) * self.P + t
        return ids if out is None else torch.where(out, -1, ids)

    def choose(self, ranked, M):
        """Per hexahedron the first M of the candidates [(rank, offset, part)], by rank, then by id."""
        ids = torch.stack([self.neighbours(o, t) for _, o, t in ranked], 1)
        rank = torch.tensor([r for r, _, _ in ranked], device=DEVICE)
        key = torch.where(ids < 0, 1 << 60, (rank[None] << 40) + ids).sort(1).values[:, :M]
        return key & ((1 << 40) - 1)

    def shift(self, i, j):
        d = self.cen[j] - self.cen[i]
        return torch.where(self.box > 0, -self.box * torch.round(d / torch.where(self.box > 0, self.box, 1.0)), 0.0)

    def pinv(self, i, members, K):
        """[n, K, M]: P = A^+ diag(V_m) of the rows A_mk = int_{V_m} phi_k of cells i."""
        n, M = members.shape
        A = torch.empty(n, M, K, dtype=torch.float64, device=DEVICE)
        for m in range(M):
            j = members[:, m]
            x = (self.xq[j] + (self.shift(i, j) - self.cen[i])[:, None]) / self.h[i][:, None, None]
            A[:, m] = self.V[j][:, None] * ((self.wq[j][..., None] * _monomials(x, self.exps[:K])).sum(1) - self.mean[i, :K])
        Q, R = torch.zeros_like(A), torch.zeros(n, K, K, dtype=torch.float64, device=DEVICE)
        for k in range(K):  # Gram-Schmidt, each column orthogonalised twice
            v = A[:, :, k].clone()
            for _ in range(2 if k else 0):
                c = (Q[:, :, :k].transpose(1, 2) @ v[..., None])[..., 0]
                v -= (Q[:, :, :k] @ c[..., None])[..., 0]
                R[:, :k, k] += c
            R[:, k, k] = v.norm(dim=1)
            Q[:, :, k] = v / R[:, k, k][:, None]
        P = torch.linalg.solve_triangular(R, Q.transpose(1, 2), upper=True)
        return P * self.V[members][:, None]

    def stencils(self):
        T, order = self.template, self.case["order"]
        M, KD = 2 * self.K, 9 if order == 4 else 3
        self.sc = torch.empty(self.N, M, dtype=torch.int64, device=DEVICE)
        self.Pc = torch.empty(self.N, self.K, M, dtype=torch.float64, device=DEVICE)
        self.sd, self.Pd, self.valid = [], [], []
        for t in range(self.P):
            me = torch.arange(t, self.N, self.P, device=DEVICE)
            here, own = ((0, 0, 0), t), set(T.nodes((0, 0, 0), t))
            found = T.search(here, None, 4 if order == 4 else 3)
            order_of = sorted({(d, -len(own & set(T.nodes(*c)))) for c, d in found.items() if c != here})
            ranked = [(order_of.index((d, -len(own & set(T.nodes(*c))))), *c) for c, d in found.items() if c != here]
            self.sc[me] = self.choose(ranked, M)
            self.Pc[me] = self.pinv(me, self.sc[me], self.K)
            if not self.weno:
                continue
            for s, nb in enumerate(T.across[t]):
                ranked = [(d, *c) for c, d in T.search(nb, here, 2 if KD == 3 else 3).items()]
                there = self.neighbours(*nb) >= 0
                members = torch.where(there[:, None], self.choose(ranked, 2 * KD), self.sc[me][:, :2 * KD])
                if t == 0:
                    self.sd.append(torch.empty(self.N, 2 * KD, dtype=torch.int64, device=DEVICE))
                    self.Pd.append(torch.empty(self.N, KD, 2 * KD, dtype=torch.float64, device=DEVICE))
                    self.valid.append(torch.empty(self.N, dtype=torch.bool, device=DEVICE))
                self.sd[s][me], self.valid[s][me] = members, there
                self.Pd[s][me] = torch.where(there[:, None, None], self.pinv(me, members, KD), 0.0)

    def face_geometry(self, corners):
        T, order = self.template, self.case["order"]
        self.faces, area = [], torch.zeros(self.N, dtype=torch.float64, device=DEVICE)
        for t in range(self.P):
            me = torch.arange(t, self.N, self.P, device=DEVICE)
            for f, (o, tn) in zip(T.faces, T.across[t]):
                nb = self.neighbours(o, tn)
                x, dS = _face_points(corners[me][:, f], order)
                area[me] += dS.sum(1).norm(dim=1)
                keep = nb > me  # each inner face from its cell of the smaller id, whose corner order places the points
                self.faces.append((me[keep], nb[keep], x[keep], dS[keep]))
                if bool((nb < 0).any()):
                    out = nb < 0
                    self.faces.append((me[out], None, x[out], dS[out]))
        self.dtlen = 2.0 * self.V / area

    def reconstruct(self, U):
        """Coefficients [N, 5, K + 1] of the final polynomials in xi (entry 0: the constant term), the largest departure
        of a cell's weights from the linear ones, and the central polynomial's coefficients and indicators."""
        du = lambda ids: (U[:, ids] - U[:, :, None]).permute(1, 0, 2)  # noqa: E731
        a = du(self.sc) @ self.Pc.transpose(1, 2)
        c, dev, SI0 = a, None, None
        if self.weno:
            form = lambda b: ((b @ self.si[:, :b.shape[2], :b.shape[2]]) * b).sum(-1)  # noqa: E731
            b = [du(s) @ P.transpose(1, 2) for s, P in zip(self.sd, self.Pd)]
            ok = [v.double()[:, None] for v in self.valid]
            SI0, SI = form(a), [form(x) for x in b]
            count = sum(ok)
            lam0, lam = LAMBDA / (LAMBDA + count), 1.0 / (LAMBDA + count)
            tau = sum(v * (SI0 - s).abs() for v, s in zip(ok, SI)) / count
            w0 = lam0 * (1.0 + tau / (EPSILON + SI0))
            ws = [v * lam * (1.0 + tau / (EPSILON + s)) for v, s in zip(ok, SI)]
            total = w0 + sum(ws)
            w0, ws = w0 / total, [w / total for w in ws]
            dev = torch.stack([(w0 - lam0).abs()] + [(w - lam).abs() for w in ws]).amax(dim=(0, 2))
            c = (w0 / lam0)[..., None] * a
            for w, x in zip(ws, b):
                c[..., :x.shape[2]] += (w - w0 / lam0 * lam)[..., None] * x
        c0 = U.T - (c[..., 3:] * self.mean[:, None, 3:]).sum(-1)
        return torch.cat([c0[..., None], c], -1), dev, a, SI0

    def residual(self, U):
        coef = self.reconstruct(U)[0]
        R = torch.zeros_like(U)
        for own, nb, x, dS in self.faces:
            area = dS.norm(dim=-1)
            n = dS / area[..., None]
            UL, gL = self.at(coef, own, x)
            if nb is None:  # slip wall: the mirror image
                mn = (UL[..., 1:4] * n).sum(-1, keepdim=True)
                flux = _hllc(UL, torch.cat([UL[..., :1], UL[..., 1:4] - 2 * mn * n, UL[..., 4:]], -1), n)
                R[:, own] -= (flux * area[..., None]).sum(1).T / self.V[own]
                continue
            shift = self.shift(own, nb)
            UR, gR = self.at(coef, nb, x - shift[:, None])
            flux = _hllc(UL, UR, n)
            if self.case["re"] > 0:
                L = (self.cen[nb] + shift - self.cen[own]).norm(dim=1)
                g = 0.5 * (gL + gR) + (ALPHA / L)[:, None, None, None] * (UR - UL)[..., None] * n[..., None, :]
                flux = flux - _viscous(0.5 * (UL + UR), g, n, self.case)
            G = (flux * area[..., None]).sum(1).T
            R[:, own] -= G / self.V[own]
            R[:, nb] += G / self.V[nb]
        return R

    def at(self, coef, cell, x):
        """Values [n, q, 5] and gradients [n, q, 5, 3] of the cells' polynomials at x [n, q, 3]."""
        h = self.h[cell][:, None, None]
        xi = (x - self.cen[cell][:, None]) / h
        c = coef[cell].transpose(1, 2)
        U = c[:, :1] + _monomials(xi, self.exps) @ c[:, 1:]
        if self.case["re"] <= 0:
            return U, None
        g = [_monomials(xi, self.exps, beta) @ c[:, 1:] / h for beta in ((1, 0, 0), (0, 1, 0), (0, 0, 1))]
        return U, torch.stack(g, -1)

    def time_step(self, U):
        rho, m, E = U[0], U[1:4], U[4]
        q2 = (m * m).sum(0) / rho ** 2
        p = (GAMMA - 1.0) * (E - 0.5 * rho * q2)
        d = self.dtlen / (q2.sqrt() + (GAMMA * p / rho).sqrt())
        if self.case["re"] > 0:
            d = torch.minimum(d, rho * self.dtlen ** 2 * PRANDTL * self.case["re"] / (2.0 * GAMMA))
        return CFL * d.min()

    def step(self, U):
        dt = self.time_step(U)
        if self.case["integrator"] == 0:
            U1 = U + dt * self.residual(U)
            U2 = 0.75 * U + 0.25 * (U1 + dt * self.residual(U1))
            return U / 3.0 + 2.0 / 3.0 * (U2 + dt * self.residual(U2)), dt
        # SSP(5,4) of Spiteri and Ruuth, the published coefficients
        u1 = U + 0.391752226571890 * dt * self.residual(U)
        u2 = 0.444370493651235 * U + 0.555629506348765 * u1 + 0.368410593050371 * dt * self.residual(u1)
        u3 = 0.620101851488403 * U + 0.379898148511597 * u2 + 0.251891774271694 * dt * self.residual(u2)
        r3 = self.residual(u3)
        u4 = 0.178079954393132 * U + 0.821920045606868 * u3 + 0.544974750228521 * dt * r3
        return (0.517231671970585 * u2 + 0.096059710526147 * u3 + 0.063692468666290 * dt * r3 +
                0.386708617503269 * u4 + 0.226007483236906 * dt * self.residual(u4)), dt

    def diagnostics(self, U):
        g = self.reconstruct(U)[0][:, :4, 1:4] / self.h[:, None, None]
        u = U[1:4] / U[0]
        gu = (g[:, 1:] - u.T[..., None] * g[:, :1]) / U[0][:, None, None]
        w = torch.stack([gu[:, 2, 1] - gu[:, 1, 2], gu[:, 0, 2] - gu[:, 2, 0], gu[:, 1, 0] - gu[:, 0, 1]], 1)
        mu = 1.0 / self.case["re"] if self.case["re"] > 0 else 1.0
        total = self.V.sum()
        div = gu[:, 0, 0] + gu[:, 1, 1] + gu[:, 2, 2]
        return {"ke": float((self.V * 0.5 * U[0] * (u * u).sum(0)).sum() / total),
                "eps_s": float(mu * (self.V * (w * w).sum(1)).sum() / total),
                "eps_d": float(4.0 / 3.0 * mu * (self.V * div * div).sum() / total), "volume": float(total)}

    def features(self, U):
        """The indicator's 32 features [N, 32] of a hexahedral P2 mesh."""
        _, dev, a, SI = self.reconstruct(U)
        rho, u = U[0], U[1:4] / U[0]
        p = (GAMMA - 1.0) * (U[4] - 0.5 * rho * (u * u).sum(0))
        c = (GAMMA * p / rho).sqrt()
        q = 0.1 * torch.stack([rho, rho * c, rho * c, rho * c, rho * c * c], 1)
        gu = (a[:, 1:4, :3] - u.T[..., None] * a[:, :1, :3]) / (self.h * rho)[:, None, None]
        w = torch.stack([gu[:, 2, 1] - gu[:, 1, 2], gu[:, 0, 2] - gu[:, 2, 0], gu[:, 1, 0] - gu[:, 0, 1]], 1)
        flow = torch.stack([(u * u).sum(0).sqrt() / c,
                            self.h * (gu[:, 0, 0] + gu[:, 1, 1] + gu[:, 2, 2]).abs() / c,
                            self.h * w.norm(dim=1) / c], 1)
        jump = lambda f, ids: (f[ids] - f[:, None]) / f[:, None]  # noqa: E731
        return torch.cat([jump(rho, self.sc), jump(p, self.sc[:, :6]), SI / (SI + q * q), flow], 1), dev


def _hllc(UL, UR, n):
    """HLLC flux per unit area with Einfeldt's wave-speed bounds."""
    def side(U):
        r, u = U[..., 0], U[..., 1:4] / U[..., :1]
        p = (GAMMA - 1.0) * (U[..., 4] - 0.5 * r * (u * u).sum(-1))
        return r, u, p, (u * n).sum(-1), (GAMMA * p / r).sqrt()
    rL, uL, pL, nL, aL = side(UL)
    rR, uR, pR, nR, aR = side(UR)
    sL, sR = rL.sqrt(), rR.sqrt()
    ut = (sL[..., None] * uL + sR[..., None] * uR) / (sL + sR)[..., None]
    Ht = (sL * (UL[..., 4] + pL) / rL + sR * (UR[..., 4] + pR) / rR) / (sL + sR)
    at, tn = ((GAMMA - 1.0) * (Ht - 0.5 * (ut * ut).sum(-1))).sqrt(), (ut * n).sum(-1)
    SL, SR = torch.fmin(nL - aL, tn - at), torch.fmax(nR + aR, tn + at)
    mL, mR = rL * (SL - nL), rR * (SR - nR)
    S = (pR - pL + nL * mL - nR * mR) / (mL - mR)

    def flux(U, u, p, un):
        return torch.cat([U[..., :1] * un[..., None], U[..., 1:4] * un[..., None] + p[..., None] * n,
                          ((U[..., 4] + p) * un)[..., None]], -1)

    def star(U, r, u, p, un, m, Sk):
        f = (m / (Sk - S))[..., None]
        Us = torch.cat([f, f * (u + (S - un)[..., None] * n),
                        f * (U[..., 4] / r + (S - un) * (S + p / m))[..., None]], -1)
        return flux(U, u, p, un) + Sk[..., None] * (Us - U)
    F = torch.where((S >= 0)[..., None], star(UL, rL, uL, pL, nL, mL, SL), star(UR, rR, uR, pR, nR, mR, SR))
    F = torch.where((SL >= 0)[..., None], flux(UL, uL, pL, nL), F)
    return torch.where((SR < 0)[..., None], flux(UR, uR, pR, nR), F)


def _viscous(U, g, n, case):
    """Viscous flux through n from the face state and the conserved gradient g [..., 5, 3]."""
    mu = 1.0 / case["re"]
    kap = mu * GAMMA / (GAMMA - 1.0) / (GAMMA * case["mach"] ** 2) / PRANDTL
    r, u = U[..., :1], U[..., 1:4] / U[..., :1]
    gu = (g[..., 1:4, :] - u[..., None] * g[..., :1, :]) / r[..., None]
    ge = (g[..., 4, :] - U[..., 4:] / r * g[..., 0, :]) / r - (u[..., None] * gu).sum(-2)
    gT = (GAMMA - 1.0) * GAMMA * case["mach"] ** 2 * ge
    div = gu.diagonal(dim1=-2, dim2=-1).sum(-1, keepdim=True)
    t = mu * ((gu + gu.transpose(-1, -2)) * n[..., None, :]).sum(-1) - 2.0 / 3.0 * mu * div * n
    return torch.cat([torch.zeros_like(r), t, ((u * t).sum(-1) + kap * (gT * n).sum(-1))[..., None]], -1)


def _gradient(X, y, theta):
    """Gradient of the class-weighted cross-entropy in FP64, with the network's BF16 roundings (inputs, weights, first
    hidden layer and the gradients entering products)."""
    r = lambda v: v.float().to(torch.bfloat16).double()  # noqa: E731
    x, y, th = X.double(), y.double(), torch.from_numpy(theta).double().to(DEVICE)
    cut = [0, 2048, 2112, 6208, 6272, 6336, 6337]
    W1, b1, W2, b2, w3, b3 = (th[i:j] for i, j in zip(cut, cut[1:]))
    W1, W2, w3 = r(W1).view(64, 32), r(W2).view(64, 64), r(w3)
    a1 = x @ W1.T + b1
    h1 = r(a1.relu())
    a2 = h1 @ W2.T + b2
    h2 = a2.relu()
    dz = torch.where(y > 0.5, W_POS, W_NEG) * (torch.sigmoid(h2 @ w3 + b3) - y) / len(y)
    d2 = dz[:, None] * w3 * (a2 > 0)
    d1 = (r(d2) @ W2) * (a1 > 0)
    return torch.cat([(r(d1).T @ x).flatten(), d1.sum(0), (r(d2).T @ h1).flatten(), d2.sum(0), h2.T @ dz,
                      dz.sum()[None]])


def exact(case, seed):
    if case["op"] in ("gated", "train"):
        return None
    if case["op"] == "grad":
        return _gradient(*training_set(case, seed), initial_weights(seed))
    s = _Scheme(case)
    nodes, cells, _ = lattice(case)
    U = start_state(case, seed, nodes, cells)
    if case["op"] == "residual":
        return s.residual(U)[:, s.perm]
    if case["op"] == "collect":
        X, dev = s.features(U)
        return {"X": X[s.perm], "dev": dev[s.perm], "z": None}
    t = 0.0
    for _ in range(case["steps"]):
        U, dt = s.step(U)
        t += float(dt)
    if case["op"] == "steps":
        return {"U": U[:, s.perm], **{k: np.float64(v) for k, v in (("t", t), *s.diagnostics(U).items())}}
    if case["op"] == "host":
        return {"U": U[:, s.perm].cpu(), "t": np.float64(t)}
    return U[:, s.perm]
