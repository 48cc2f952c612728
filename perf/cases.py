"""Performance cases: the calls a user of this framework makes, through its public entry
points, over the range of sizes, precisions and options the framework is used at.

Families (the "kind" of a case):
  cavity    a cavity advanced by LBM.step and read back: the macroscopic fields on the
            device (net.targets: u / U0 and 2 T), or for FP64 contexts the populations in
            page-locked host arrays (LBM.get_populations_native)
  batch     a parameter sweep: many uneven cavities advanced together by Batch.step, the
            fields of every member read back
  warm      a cavity started from a predicted steady state (net.warm_start with rounds of
            the consistent initialisation), its fields read back
  conv      one 3x3x3 convolution of the warm-start network (net.conv3d_bf16): forward
            (bias, ReLU, BF16 out) or the input gradient (FP32 out)
  wgrad     the weight gradient of such a convolution (net.conv3d_wgrad_bf16)

The network's whole forward pass and training step return FP32 values behind eleven BF16
layers, where a change of summation order in one layer moves the last digits of all that
follow; its layers stand for it here one by one.

exact() restates every case in plain torch operations in 64 bits.
"""
import math
import random

import torch

import paper_1710_04751_gb300 as lbm
from paper_1710_04751_gb300 import net

DEVICE = "cuda"
U0 = 0.05
MA = U0 * math.sqrt(3.0)
PRECISIONS = {"fp64": 0, "fp32": 1, "fp16": 2, "bf16": 3}
STORED_BYTES = {"fp64": 8, "fp32": 4, "fp16": 2, "bf16": 2}
SMS = 152


def _cavity(name, grid, lattice, precision, Ra, Pr, steps):
    c = {"kind": "cavity", "nx": grid[0], "ny": grid[1], "nz": grid[2], "lattice": lattice,
         "precision": precision, "Ra": Ra, "Pr": Pr, "steps": steps}
    return dict(c, name=name) if name else c


def listed():
    return [
        # a small cavity advanced a few steps at a time, its fields read after each call (a
        # solver coupled to a caller's own loop): launches and host waits
        _cavity("cavity_24_fp32_10", (24, 24, 24), 15, "fp32", 1e3, 0.71, 10),
        # the FP64 verification run of the paper's smallest cavity, all populations read back
        _cavity("cavity_32_fp64_300", (32, 32, 32), 15, "fp64", 1e3, 0.71, 300),
        # the grid at which the warm start's training states are generated
        _cavity("cavity_64_fp32_100", (64, 64, 64), 15, "fp32", 1e4, 0.71, 100),
        # the paper's own (odd) grid, seven-velocity scalar
        _cavity("cavity_91_fp32_q7_100", (91, 91, 91), 7, "fp32", 1e4, 0.71, 100),
        # the benchmark's cavity, one residual interval
        _cavity("cavity_128_fp32_100", (128, 128, 128), 15, "fp32", 1e5, 0.71, 100),
        # the precision study's large cavity in 16-bit storage
        _cavity("cavity_256_fp16_20", (256, 256, 256), 15, "fp16", 1e6, 0.71, 20),
        # a sweep over uneven cavities, one graph of 100 steps
        {"name": "batch_16", "kind": "batch", "lattice": 15, "steps": 100,
         "grids": "32x32x32 96x96x96 48x48x48 64x64x64 64x64x64 32x32x32 48x48x48 96x96x96 "
                  "48x48x48 48x48x48 32x32x32 64x64x64 96x96x96 32x32x32 48x48x48 96x96x96"},
        # a 128^3 cavity started from a 64^3 prediction, as the warm-start evaluation does
        {"name": "warm_64_to_128", "kind": "warm", "m": 64, "nx": 128, "ny": 128, "nz": 128,
         "lattice": 15, "Ra": 1e5, "Pr": 0.71, "iterations": 50},
        # the network's widest input at full resolution (decoder, 96 -> 32 channels)
        {"name": "conv_fwd_64_96_32", "kind": "conv", "batch": 2, "n": 64, "cin": 96, "cout": 32,
         "mode": "bias_relu_bf16"},
        # its deepest level: many channels on a coarse grid, a short call
        {"name": "conv_fwd_16_128_128", "kind": "conv", "batch": 2, "n": 16, "cin": 128, "cout": 128,
         "mode": "bias_relu_bf16"},
        # input gradient of the middle level's 192 -> 64 layer
        {"name": "conv_dgrad_32_64_192", "kind": "conv", "batch": 2, "n": 32, "cin": 64, "cout": 192,
         "mode": "f32"},
        # weight gradient of the 96 -> 32 layer
        {"name": "conv_wgrad_64_96_32", "kind": "wgrad", "batch": 2, "n": 64, "cin": 96, "cout": 32},
    ]


# ---- draws -----------------------------------------------------------------------------

MOST_BYTES = 5.0e10   # of the cavities' state traffic in a pass (the largest listed ones)
MOST_FLOPS = 1.0e11   # of a convolution


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _ra(rng, n):
    """A Rayleigh number the edge length resolves."""
    return float("%.3g" % (10.0 ** rng.uniform(3.0, 3.0 + 2.0 * math.log10(max(n, 16) / 16.0))))


def _box(rng, lo, hi):
    """A cube, or a box with sides of its own."""
    n = _log_int(rng, lo, hi)
    if rng.random() < 0.4:
        return n, n, n
    return n, max(8, int(n * rng.uniform(0.5, 1.4))), max(8, int(n * rng.uniform(0.5, 1.4)))


def _draw_cavity(rng):
    precision = rng.choice(["fp32", "fp32", "fp32", "fp64", "fp16", "bf16"])
    lattice = rng.choice([15, 7])
    hi = {"fp64": 48, "fp32": 160, "fp16": 224, "bf16": 224}[precision]
    box = _box(rng, 16 if precision in ("fp32", "fp64") else 32, hi)
    steps = {"fp64": 100, "fp32": rng.choice([10, 100, 100, _log_int(rng, 1, 100)]), "fp16": 20, "bf16": 20}[precision]
    per = _node_bytes(lattice, precision) * box[0] * box[1] * box[2]
    return _cavity(None, box, lattice, precision, _ra(rng, box[0]), rng.choice([0.71, 1.0, 7.0]),
                   max(1, min(steps, int(MOST_BYTES / per))))


def _draw_batch(rng):
    grids, nodes = [], 0
    for _ in range(rng.randint(4, 20)):
        g = _box(rng, 16, 96)
        if nodes + g[0] * g[1] * g[2] > 4_000_000:
            break
        nodes += g[0] * g[1] * g[2]
        grids.append("%dx%dx%d" % g)
    return {"kind": "batch", "lattice": rng.choice([15, 7]), "steps": 50, "grids": " ".join(grids)}


def _draw_warm(rng):
    n = _log_int(rng, 40, 128)
    return {"kind": "warm", "m": rng.choice([32, 48, 64]), "nx": n, "ny": n, "nz": n,
            "lattice": rng.choice([15, 7]), "Ra": _ra(rng, n), "Pr": rng.choice([0.71, 1.0, 7.0]),
            "iterations": rng.choice([10, 20, 50])}


def _draw_layer(rng, couts, most):
    """Sizes of a convolution on a power-of-two grid, within `most` operations."""
    while True:
        n = rng.choice([8, 16, 16, 32, 32, 64])
        c = {"batch": rng.randint(1, 4), "n": n, "cin": 32 * rng.randint(1, 8), "cout": rng.choice(couts)}
        if 2e8 <= _conv_flops(c) <= most:
            return c


def draw(rng):
    kind = rng.choice(["cavity", "cavity", "cavity", "batch", "warm", "conv", "conv", "wgrad"])
    if kind == "cavity":
        return _draw_cavity(rng)
    if kind == "batch":
        return _draw_batch(rng)
    if kind == "warm":
        return _draw_warm(rng)
    if kind == "conv":
        couts = [16, 24, 32, 32, 48, 64, 64, 96, 128, 192, 256]
        return dict(_draw_layer(rng, couts, MOST_FLOPS), kind="conv", mode=rng.choice(["bias_relu_bf16", "f32"]))
    return dict(_draw_layer(rng, [16, 24, 32, 48, 64, 64, 96, 128, 256], MOST_FLOPS), kind="wgrad")


# ---- inputs ----------------------------------------------------------------------------

def _smooth_fields(grid, seed):
    """Smooth fields of a differentially heated cavity, FP64: (u_x, u_y, u_z) vanishing at
    the walls (amplitude a fraction of U0) and T between the faces, random mode weights."""
    nx, ny, nz = grid
    r = random.Random(seed)
    X = ((torch.arange(nx, device=DEVICE, dtype=torch.float64) + 0.5) / nx).view(1, 1, nx)
    Y = ((torch.arange(ny, device=DEVICE, dtype=torch.float64) + 0.5) / ny).view(1, ny, 1)
    Z = ((torch.arange(nz, device=DEVICE, dtype=torch.float64) + 0.5) / nz).view(nz, 1, 1)
    pi = math.pi
    ux = torch.zeros((nz, ny, nx), device=DEVICE, dtype=torch.float64)
    uy, uz = torch.zeros_like(ux), torch.zeros_like(ux)
    T = (X - 0.5).expand(nz, ny, nx).clone()
    sy = torch.sin(pi * Y) ** 2
    for m in (1, 2):
        a = U0 * r.uniform(0.05, 0.2) / m
        ux -= a * torch.sin(m * pi * X) ** 2 * torch.sin(2 * m * pi * Z) * sy
        uz += a * torch.sin(2 * m * pi * X) * torch.sin(m * pi * Z) ** 2 * sy
        uy += 0.1 * a * torch.sin(pi * X) ** 2 * torch.sin(2 * pi * Y) * torch.sin(m * pi * Z) ** 2
        T += r.uniform(0.05, 0.15) / m * torch.sin(m * pi * X) * torch.cos(m * pi * Z) * (1 + 0.3 * torch.cos(pi * Y))
    return ux, uy, uz, T


def _grid(case):
    return case["nx"], case["ny"], case["nz"]


def _members(case):
    """The sweep's members: grid, Ra (resolved by the grid), Pr."""
    r = random.Random(7)
    out = []
    for g in case["grids"].split():
        grid = tuple(int(v) for v in g.split("x"))
        out.append({"grid": grid, "Ra": _ra(r, grid[0]), "Pr": r.choice([0.71, 1.0, 7.0])})
    return out


def _layer(case, seed):
    """Operands of a convolution layer: activations behind a ReLU, He-normal weights, and
    for the gradients an output gradient behind a ReLU's mask; all BF16."""
    g = torch.Generator(device=DEVICE).manual_seed(seed)
    B, n, cin, cout = case["batch"], case["n"], case["cin"], case["cout"]

    def normal(*shape):
        return torch.randn(shape, generator=g, device=DEVICE, dtype=torch.float32)

    if case["kind"] == "wgrad":
        X = normal(B, n ** 3, cin).relu_().to(torch.bfloat16)
        dZ = (1e-3 * normal(B * n ** 3, cout)).to(torch.bfloat16)
        dZ *= normal(B * n ** 3, cout) > 0
        return X, dZ
    if case["mode"] == "f32":
        X = (1e-3 * normal(B, n ** 3, cin)).to(torch.bfloat16)
        X *= normal(B, n ** 3, cin) > 0
    else:
        X = normal(B, n ** 3, cin).relu_().to(torch.bfloat16)
    ldw = (27 * cin + 63) // 64 * 64
    W = torch.zeros((cout, ldw), device=DEVICE, dtype=torch.bfloat16)
    W[:, :27 * cin] = (math.sqrt(2.0 / (27 * cin)) * normal(cout, 27 * cin)).to(torch.bfloat16)
    bias = 0.1 * normal(cout)
    return X, W, bias


def _kp(case):
    return (27 * case["cin"] + 63) // 64 * 64


def _splits(case):
    """About two CTAs per SM over the 128-row tiles of dW^T, at least one K block each."""
    tiles = (_kp(case) + 127) // 128
    return max(1, min(2 * SMS // tiles, (case["batch"] * case["n"] ** 3 + 63) // 64))


def _prediction(case, seed):
    """A network's prediction on its m^3 grid: u / U0 and 2 T, FP32, with small errors."""
    m = case["m"]
    ux, uy, uz, T = _smooth_fields((m, m, m), seed)
    p = torch.stack([ux / U0, uy / U0, uz / U0, 2 * T], dim=-1).reshape(m ** 3, 4)
    g = torch.Generator(device=DEVICE).manual_seed(seed)
    noise = torch.randn(p.shape, generator=g, device=DEVICE, dtype=torch.float32)
    return (p.to(torch.float32) + 1e-3 * noise).contiguous()


def prepare(case, seed):
    kind = case["kind"]
    if kind == "cavity":
        sim = lbm.LBM(_grid(case), case["lattice"], Ra=case["Ra"], Pr=case["Pr"], Ma=MA,
                      precision=PRECISIONS[case["precision"]], seed=seed)
        ux, uy, uz, T = _smooth_fields(_grid(case), seed)
        sim.set_fields(ux, uy, uz, T)
        state = {"kind": kind, "sim": sim, "steps": case["steps"], "host": None}
        if case["precision"] == "fp64":
            nx, ny, nz = _grid(case)
            state["host"] = [torch.empty((q, nz, ny, nx), dtype=torch.float64, pin_memory=True).numpy()
                             for q in (15, case["lattice"])]
        return state
    if kind == "batch":
        b = lbm.Batch(_members(case), lattice=case["lattice"], Ma=MA, seed=seed)
        for i, g in enumerate(b.grids):
            b.member(i).set_fields(*_smooth_fields(g, seed + i))
        return {"kind": kind, "batch": b, "steps": case["steps"], "members": [b.member(i) for i in range(b.count)]}
    if kind == "warm":
        sim = lbm.LBM(_grid(case), case["lattice"], Ra=case["Ra"], Pr=case["Pr"], Ma=MA, seed=seed)
        return {"kind": kind, "sim": sim, "pred": _prediction(case, seed), "m": case["m"],
                "iterations": case["iterations"]}
    if kind == "conv":
        X, W, bias = _layer(case, seed)
        relu = case["mode"] == "bias_relu_bf16"
        out = torch.empty((case["batch"] * case["n"] ** 3, case["cout"]), device=DEVICE,
                          dtype=torch.bfloat16 if relu else torch.float32)
        return {"kind": kind, "X": X, "W": W, "bias": bias if relu else None, "n": case["n"], "out": out,
                "mode": net.CONV_BIAS_RELU_BF16 if relu else net.CONV_F32}
    X, dZ = _layer(case, seed)
    return {"kind": kind, "X": X, "dZ": dZ, "n": case["n"], "splits": _splits(case),
            "dWT": torch.empty((_kp(case), case["cout"]), device=DEVICE, dtype=torch.float32)}


def run(state):
    kind = state["kind"]
    if kind == "cavity":
        sim = state["sim"]
        sim.step(state["steps"])
        if state["host"] is not None:
            return list(sim.get_populations_native(*state["host"]))
        return net.targets(sim)
    if kind == "batch":
        state["batch"].step(state["steps"])
        return [net.targets(m) for m in state["members"]]
    if kind == "warm":
        net.warm_start(state["sim"], state["pred"], state["m"], state["iterations"])
        return net.targets(state["sim"])
    if kind == "conv":
        net.conv3d_bf16(state["X"], state["n"], state["W"], state["out"], mode=state["mode"], bias=state["bias"])
        return state["out"]
    state["dWT"].zero_()
    net.conv3d_wgrad_bf16(state["X"], state["n"], state["dZ"], state["dWT"], splits=state["splits"])
    return state["dWT"]


# ---- the work of a pass ----------------------------------------------------------------

def _node_bytes(lattice, precision):
    """Bytes of one node update: every stored value read once and written once."""
    return 2 * ((15 + lattice) * STORED_BYTES[precision] + (4 if STORED_BYTES[precision] == 2 else 0))


def _node_flops(lattice):
    return 470 if lattice == 15 else 360


def _conv_flops(c):
    return 2.0 * c["batch"] * c["n"] ** 3 * 27 * c["cin"] * c["cout"]


def work(case):
    kind = case["kind"]
    if kind in ("cavity", "warm"):
        nodes = case["nx"] * case["ny"] * case["nz"]
        steps = case.get("steps", case.get("iterations"))
        precision = case.get("precision", "fp32")
        out = (15 + case["lattice"]) * 8 if precision == "fp64" else 16
        return {"bytes": nodes * (steps * _node_bytes(case["lattice"], precision) + out),
                "flops": nodes * steps * _node_flops(case["lattice"])}
    if kind == "batch":
        nodes = sum(m["grid"][0] * m["grid"][1] * m["grid"][2] for m in _members(case))
        return {"bytes": nodes * (case["steps"] * _node_bytes(case["lattice"], "fp32") + 16),
                "flops": nodes * case["steps"] * _node_flops(case["lattice"])}
    M = case["batch"] * case["n"] ** 3
    cin, cout = case["cin"], case["cout"]
    if kind == "conv":
        b = M * cin * 2 + 27 * cin * cout * 2 + M * cout * (2 if case["mode"] == "bias_relu_bf16" else 4)
    else:
        b = M * (cin + cout) * 2 + 27 * cin * cout * 4
    return {"bytes": b, "flops": _conv_flops(case)}


# ---- the same in plain torch operations, 64 bits ---------------------------------------

E = [(0, 0, 0), (1, 0, 0), (-1, 0, 0), (0, 1, 0), (0, -1, 0), (0, 0, 1), (0, 0, -1)] + [
    (x, y, z) for z in (1, -1) for y in (1, -1) for x in (1, -1)]
MONOMIALS = [(0, 0, 0), (1, 0, 0), (0, 1, 0), (0, 0, 1), (1, 1, 0), (1, 0, 1), (0, 1, 1), (2, 0, 0), (0, 2, 0),
             (0, 0, 2), (1, 2, 0), (2, 1, 0), (2, 0, 1), (1, 1, 1), (2, 2, 0)]
MONOMIALS7 = MONOMIALS[:4] + MONOMIALS[7:10]


def _moment_matrix(q):
    """Row b: the monomial b of every velocity, so that matrix @ populations = raw moments."""
    rows = [[float(e[0] ** p[0] * e[1] ** p[1] * e[2] ** p[2]) for e in E[:q]]
            for p in (MONOMIALS if q == 15 else MONOMIALS7)]
    return torch.tensor(rows, dtype=torch.float64, device=DEVICE)


def _combine(matrix, v):
    return (matrix @ v.reshape(v.shape[0], -1)).reshape((matrix.shape[0],) + v.shape[1:])


def _raw_moments(k0, k1, k2, k4, u):
    """Raw moments (order of MONOMIALS) from central moments about u: zeroth k0, first k1
    (x, y, z), second k2 (xy, xz, yz, xx, yy, zz), vanishing third ones, xxyy k4."""
    x, y, z = u
    kx, ky, kz = k1
    xy, xz, yz, xx, yy, zz = k2
    return torch.stack([
        k0, kx + x * k0, ky + y * k0, kz + z * k0,
        xy + x * ky + y * kx + x * y * k0, xz + x * kz + z * kx + x * z * k0, yz + y * kz + z * ky + y * z * k0,
        xx + 2 * x * kx + x * x * k0, yy + 2 * y * ky + y * y * k0, zz + 2 * z * kz + z * z * k0,
        x * yy + 2 * y * xy + 2 * x * y * ky + y * y * kx + x * y * y * k0,
        y * xx + 2 * x * xy + 2 * x * y * kx + x * x * ky + x * x * y * k0,
        z * xx + 2 * x * xz + 2 * x * z * kx + x * x * kz + x * x * z * k0,
        x * yz + y * xz + z * xy + x * y * kz + x * z * ky + y * z * kx + x * y * z * k0,
        k4 + x * x * yy + y * y * xx + 4 * x * y * xy + 2 * x * y * y * kx + 2 * x * x * y * ky + x * x * y * y * k0])


class _Cavity64:
    """The cascaded central-moment model of the cavity at unit higher-order rates."""

    def __init__(self, grid, q, Ra, Pr):
        nx = grid[0]
        self.q, self.grid = q, grid
        nu = math.sqrt(Pr / Ra) * U0 * nx
        cs = 1.0 / 3.0 if q == 15 else 0.25
        self.cs, self.gbeta = cs, U0 * U0 / nx
        self.om_nu, self.om_phi = 1.0 / (3.0 * nu + 0.5), 1.0 / (nu / Pr / cs + 0.5)
        w7 = cs * cs / 8.0 if q == 15 else 0.0
        w1 = 0.5 * (cs - cs * cs) if q == 15 else 0.5 * cs
        self.wg = [1.0 - 6.0 * w1 - 8.0 * w7] + [w1] * 6 + [w7] * 8
        self.Mf, self.Mg = _moment_matrix(15), _moment_matrix(q)
        self.Mf_inv, self.Mg_inv = torch.linalg.inv(self.Mf), torch.linalg.inv(self.Mg)
        self.opp = [E.index((-a, -b, -c)) for a, b, c in E]

    def _scalar(self, phi, k1, u):
        zero, s = torch.zeros_like(phi), self.cs * phi
        m = _raw_moments(phi, k1, (zero, zero, zero, s, s, s), self.cs * self.cs * phi, u)
        if self.q == 7:
            m = m[[MONOMIALS.index(p) for p in MONOMIALS7]]
        return _combine(self.Mg_inv, m)

    def equilibria(self, rho, u, T):
        zero, s = torch.zeros_like(rho), rho / 3.0
        m = _raw_moments(rho, (zero, zero, zero), (zero, zero, zero, s, s, s), rho / 9.0, u)
        return _combine(self.Mf_inv, m), self._scalar(T, (zero, zero, zero), u)

    def fields(self, F, G):
        T, rho = G.sum(0), F.sum(0)
        j = _combine(self.Mf[1:4], F)
        return rho, [j[0] / rho, j[1] / rho, (j[2] - 0.5 * self.gbeta * T) / rho], T

    def _pull(self, F, G):
        nx, ny, nz = self.grid
        idx = [torch.arange(n, device=F.device).view(s) for n, s in ((nx, (1, 1, nx)), (ny, (1, ny, 1)), (nz, (nz, 1, 1)))]

        def out(axis, e):  # nodes whose source along the axis lies beyond a wall
            return idx[axis] == (0 if e > 0 else (nx, ny, nz)[axis] - 1)

        f, g = torch.empty_like(F), torch.empty_like(G)
        for a, (ex, ey, ez) in enumerate(E):
            walls = [out(d, e) for d, e in enumerate((ex, ey, ez)) if e]
            v = torch.roll(F[a], (ez, ey, ex), (0, 1, 2))
            for w in walls:
                v = torch.where(w, F[self.opp[a]], v)
            f[a] = v
            if a >= self.q:
                continue
            v = torch.roll(G[a], (ez, ey, ex), (0, 1, 2))
            if ey:  # adiabatic walls: specular reflection
                v = torch.where(out(1, ey), torch.roll(G[E.index((ex, -ey, ez))], (ez, 0, ex), (0, 1, 2)), v)
            if ez:
                v = torch.where(out(2, ez), torch.roll(G[E.index((ex, ey, -ez))], (0, ey, ex), (0, 1, 2)), v)
            if ey and ez:
                v = torch.where(out(1, ey) & out(2, ez), torch.roll(G[E.index((ex, -ey, -ez))], (0, 0, ex), (0, 1, 2)), v)
            if ex:  # heated faces: anti-bounce-back
                Tw = -0.5 if ex > 0 else 0.5
                v = torch.where(out(0, ex), 2.0 * self.wg[a] * Tw - G[self.opp[a]], v)
            g[a] = v
        return f, g

    def step(self, F, G):
        f, g = self._pull(F, G)
        gm = _combine(self.Mg[:4], g)
        T = gm[0]
        Fz = self.gbeta * T
        m = _combine(self.Mf[:10], f)
        rho, jx, jy, jz, mxy, mxz, myz, mxx, myy, mzz = m
        u = [jx / rho, jy / rho, (jz + 0.5 * Fz) / rho]
        x, y, z = u
        c = 1.0 - self.om_nu
        kxx, kyy, kzz = mxx - 2 * x * jx + rho * x * x, myy - 2 * y * jy + rho * y * y, mzz - 2 * z * jz + rho * z * z
        A, B, tr = c * (kxx - kyy), c * (kxx + kyy - 2 * kzz), rho
        zz = (tr - B) / 3.0
        xx, yy = 0.5 * (tr - zz + A), 0.5 * (tr - zz - A)
        k2 = (c * (mxy - x * jy - y * jx + rho * x * y), c * (mxz - x * jz - z * jx + rho * x * z),
              c * (myz - y * jz - z * jy + rho * y * z), xx, yy, zz)
        zero = torch.zeros_like(rho)
        F = _combine(self.Mf_inv, _raw_moments(rho, (zero, zero, 0.5 * Fz), k2, xx * yy / rho, u))
        d = 1.0 - self.om_phi
        G = self._scalar(T, [d * (gm[1 + i] - u[i] * T) for i in range(3)], u)
        return F, G

    def targets(self, F, G):
        _, u, T = self.fields(F, G)
        return torch.stack([u[0] / U0, u[1] / U0, u[2] / U0, 2.0 * T], dim=-1).reshape(-1, 4)


def _exact_cavity(grid, lattice, Ra, Pr, steps, seed, whole):
    sim = _Cavity64(grid, lattice, Ra, Pr)
    ux, uy, uz, T = _smooth_fields(grid, seed)
    F, G = sim.equilibria(torch.ones_like(T), [ux, uy, uz], T)
    for _ in range(steps):
        F, G = sim.step(F, G)
    return [F, G] if whole else sim.targets(F, G)


def _resample(pred, m, grid):
    """Trilinear, cell-centred, clamped at the walls: [m^3][4] -> [4][nz][ny][nx]."""
    v = pred.to(torch.float64).reshape(m, m, m, 4)
    for axis, n in ((0, grid[2]), (1, grid[1]), (2, grid[0])):
        s = ((torch.arange(n, device=v.device, dtype=torch.float64) + 0.5) * m / n - 0.5).clamp(0, m - 1)
        lo = s.floor().long().clamp(max=m - 2)
        w = (s - lo).view([-1 if d == axis else 1 for d in range(4)])
        v = v.index_select(axis, lo) * (1 - w) + v.index_select(axis, lo + 1) * w
    return v.permute(3, 0, 1, 2).contiguous()


def _exact_warm(case, seed):
    sim = _Cavity64(_grid(case), case["lattice"], case["Ra"], case["Pr"])
    p = _resample(_prediction(case, seed), case["m"], _grid(case))
    u, T = [U0 * p[0], U0 * p[1], U0 * p[2]], 0.5 * p[3]
    F, G = sim.equilibria(torch.ones_like(T), u, T)
    for _ in range(case["iterations"]):
        F, G = sim.step(F, G)
        rho, uc, Tc = sim.fields(F, G)
        Fe, Ge = sim.equilibria(rho, uc, Tc)
        F, G = F - Fe, G - Ge
        Fe, Ge = sim.equilibria(rho, u, T)
        F, G = F + Fe, G + Ge
    return sim.targets(F, G)


def _shifted(X, case):
    """(tap, X shifted by the tap) of zero-padded activations, as [B n^3][cin] FP64."""
    B, n, cin = case["batch"], case["n"], case["cin"]
    P = torch.zeros((B, n + 2, n + 2, n + 2, cin), dtype=torch.float64, device=X.device)
    P[:, 1:-1, 1:-1, 1:-1] = X.double().reshape(B, n, n, n, cin)
    for tap in range(27):
        kz, ky, kx = tap // 9, tap // 3 % 3, tap % 3
        yield tap, P[:, kz:kz + n, ky:ky + n, kx:kx + n].reshape(-1, cin)


def exact(case, seed):
    kind = case["kind"]
    if kind == "cavity":
        return _exact_cavity(_grid(case), case["lattice"], case["Ra"], case["Pr"], case["steps"], seed,
                             case["precision"] == "fp64")
    if kind == "batch":
        return [_exact_cavity(m["grid"], case["lattice"], m["Ra"], m["Pr"], case["steps"], seed + i, False)
                for i, m in enumerate(_members(case))]
    if kind == "warm":
        return _exact_warm(case, seed)
    cin, cout = case["cin"], case["cout"]
    if kind == "conv":
        X, W, bias = _layer(case, seed)
        y = torch.zeros((case["batch"] * case["n"] ** 3, cout), dtype=torch.float64, device=X.device)
        for tap, S in _shifted(X, case):
            y += S @ W[:, tap * cin:(tap + 1) * cin].double().T
        return (y + bias.double()).relu_() if case["mode"] == "bias_relu_bf16" else y
    X, dZ = _layer(case, seed)
    out = torch.zeros((_kp(case), cout), dtype=torch.float64, device=X.device)
    for tap, S in _shifted(X, case):
        out[tap * cin:(tap + 1) * cin] = S.T @ dZ.double()
    return out
