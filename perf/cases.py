"""The workloads that the framework's speed is measured on, and what they return in 64 bits.

Every case goes through the public classes: lb.Solver / lb.Batch (one lattice, a sweep of
lattices), lb3d.Solver3D (the three-dimensional box), lb.Net (the network of the learned
stepper) and the single-layer calls lb.conv3x3*.  A case is a plain dict; its "kind" says which.
One pass of a simulation advances it by some steps from a developed state (a restart: moving
fluid, stressed polymer, noisy director) and takes the state out, as a run between two snapshots
does; one pass of the network is an inference, or a forward and a backward pass.

exact() computes the same in FP64 from the paper's equations (central differences, Heun, D2Q9 /
D3Q19 BGK with the Guo force, the cosine kernel), in plain torch.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2209_14889_gb300 import lb, lb3d

PHYSICS = dict(tau=0.8, rho0=1.0, K=(2e-3, 1e-3, 1e-3, 1e-3), lambda_steps=50.0, Dp=0.05, alpha=-0.9, beta=1.0,
               xi=1.1, Gamma=1.0, kappa=0.001, P_cap=0.99, ericksen=1, director_angle=0.0)
PHYSICS_3D = dict(tau=0.8, rho0=1.0, K=(2e-3, 1e-3, 1e-3, 1e-3, 5e-4), eta_p=0.05, Dp=0.05, alpha=-0.9, beta=1.0,
                  xi=1.1, Gamma=1.0, kappa=0.001, P_cap=0.99, ericksen=1, director=(1.0, 0.0, 0.0))

# the network's layers: name, input and output channels, activation
LAYERS = [("e0a", 16, 32, True), ("e0b", 32, 32, True), ("e1a", 32, 64, True), ("e1b", 64, 64, True),
          ("e2a", 64, 96, True), ("e2b", 96, 96, True), ("bta", 96, 128, True), ("btb", 128, 128, True),
          ("d2a", 224, 96, True), ("d2b", 96, 96, True), ("d1a", 160, 64, True), ("d1b", 64, 64, True),
          ("d0a", 96, 32, True), ("d0b", 32, 32, True), ("head", 32, 16, False)]
LAYER_LEVEL = [0, 0, 1, 1, 2, 2, 3, 3, 2, 2, 1, 1, 0, 0, 0]


# ------------------------------------------------------------------------------------ cases

def listed():
    return [
        # the method's small validation run: one ring dragged through a 64^2 box, ten readouts
        dict(name="ring_64", kind="lattice", nx=64, ny=64, steps=100, rings=1, nodes=32, radius=6.0),
        # the paper's own experiment (App. C): scalar model, 250^2 closed box, the droplet dragged by the trap
        dict(name="paper_box_250", kind="lattice", nx=250, ny=250, steps=100, rings=1, nodes=157, radius=12.5,
             scalar=True, walls=True),
        # an ordinary run on a lattice that fits no tile, two rings, strong stress diffusion (three sub-steps)
        dict(name="ring_ragged_333x190", kind="lattice", nx=333, ny=190, steps=50, rings=2, nodes=96, radius=12.0,
             Dp=0.55, substeps=3, theta=0.6),
        # the headline workload: 1024^2, one ring of 256 nodes, one readout period
        dict(name="ring_1024", kind="lattice", nx=1024, ny=1024, steps=10, rings=1, nodes=256, radius=24.0, Dp=0.1,
             lambda_steps=200.0),
        # a large domain with many swimmers: 4096^2, sixteen rings
        dict(name="rings_4096", kind="lattice", nx=4096, ny=4096, steps=10, rings=16, nodes=128, radius=12.0, Dp=0.1,
             lambda_steps=200.0),
        # the reduced-precision storage form (FP16 populations, BF16 stress) of a large domain
        dict(name="half_state_2048", kind="lattice", nx=2048, ny=2048, steps=10, rings=4, nodes=128, radius=12.0,
             Dp=0.1, lambda_steps=200.0, half=True),
        # a parameter sweep: twenty lattices of uneven size and physics advanced as one batch
        dict(name="sweep_20", kind="sweep", count=20, side_min=128, side_max=512, steps=30),
        # three dimensions: a small ragged box, as in a validation run, and the measured cube
        dict(name="box3d_45x38x30", kind="box3d", nx=45, ny=38, nz=30, steps=40),
        dict(name="box3d_256", kind="box3d", nx=256, ny=256, nz=256, steps=5),
        # the learned stepper's network: one inference, and the gradients of one training batch
        dict(name="unet_infer_256", kind="infer", batch=1, height=256, width=256),
        dict(name="unet_gradients_4x256", kind="gradients", batch=4, height=256, width=256),
        # one convolution layer by itself, forward with activation and both gradients, on an odd image
        dict(name="conv_layer_75x100", kind="conv", batch=3, height=75, width=100, ci=96, co=64),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["lattice"] * 6 + ["sweep", "box3d", "box3d", "infer", "gradients", "conv"])
    if kind == "lattice":
        scalar = rng.random() < 0.25
        half = not scalar and rng.random() < 0.2
        walls = not half and rng.random() < 0.25
        nx, ny = _log(rng, 48, 2500), _log(rng, 48, 2500)
        radius = rng.uniform(4.0, min(24.0, min(nx, ny) / 4 - 7.0))
        room = (nx // int(2 * radius + 24)) * (ny // int(2 * radius + 24))
        Dp = rng.choice([0.01, 0.05, 0.1, 0.2])
        sub = 0
        if not (half or walls) and rng.random() < 0.25:
            Dp, sub = 0.6, 3
        return dict(kind=kind, nx=nx, ny=ny, steps=10 * rng.randint(1, 5), rings=1 if walls else rng.randint(0, max(1, min(12, room))),
                    nodes=max(16, int(2 * math.pi * radius / 0.78)), radius=round(radius, 2), scalar=scalar, half=half,
                    walls=walls, Dp=Dp, substeps=sub, theta=round(rng.uniform(0.0, 1.5), 2),
                    lambda_steps=round(rng.uniform(20.0, 500.0), 1))
    if kind == "sweep":
        return dict(kind=kind, count=rng.randint(4, 20), side_min=64, side_max=rng.randint(128, 512), steps=10 * rng.randint(1, 3))
    if kind == "box3d":
        return dict(kind=kind, nx=_log(rng, 16, 220), ny=_log(rng, 12, 220), nz=_log(rng, 8, 220),
                    steps=rng.randint(2, 10), ericksen=rng.random() < 0.8)
    if kind == "conv":
        return dict(kind=kind, batch=rng.randint(1, 4), height=_log(rng, 9, 256), width=_log(rng, 9, 256),
                    ci=16 * rng.randint(1, 10), co=16 * rng.randint(1, 8))
    return dict(kind=kind, batch=rng.randint(1, 4), height=8 * _log(rng, 4, 32), width=8 * _log(rng, 4, 32))


def _physics(case):
    w = dict(PHYSICS, Dp=case.get("Dp", 0.05), lambda_steps=case.get("lambda_steps", 50.0),
             director_angle=case.get("theta", 0.0))
    if case.get("scalar"):
        # Tables I, II and IV in lattice units: C = 0.01 Pa, eta_p = 0.1 Pa s, D_p = 1e-13 m^2/s, tau = 1.25
        C = 2e-5
        w.update(K=(C, 0.0, C, C / 2), ericksen=0, model=1, tau=1.25, eta_p=25.0, Dp=case.get("Dp", 5e-4))
    w.update(nx=case["nx"], ny=case["ny"], every=10, steps=case["steps"], noise=None,
             diffusion_substeps=case.get("substeps", 0), walls_x=int(bool(case.get("walls"))),
             walls_y=int(bool(case.get("walls"))))
    return w


def _rings(case, seed):
    """Rings on a loose grid (one alone: at the middle, moved by a fraction of a cell), each a circle."""
    rng = np.random.Generator(np.random.PCG64(seed))
    nx, ny, r, n = case["nx"], case["ny"], case["radius"], case["rings"]
    pitch = int(2 * r + 24)
    cells = [(i, j) for j in range(max(1, ny // pitch)) for i in range(max(1, nx // pitch))]
    pick = rng.permutation(len(cells))[:n]
    out = []
    for k in pick:
        i, j = cells[k]
        cx, cy = ((i + 0.5) * pitch, (j + 0.5) * pitch) if n > 1 else (nx / 2.0, ny / 2.0)
        cx, cy = cx + rng.uniform(-0.5, 0.5), cy + rng.uniform(-0.5, 0.5)
        a = rng.uniform(0, 2 * math.pi) + 2 * math.pi * np.arange(case["nodes"]) / case["nodes"]
        X = np.stack([cx + r * np.cos(a), cy + r * np.sin(a)], axis=1)
        g = dict(X=X, k_spring=0.1, eps_angle=0.01, l_eq=float(np.hypot(*(X[1] - X[0]))), pull_force=5e-4,
                 pull_angle=float(rng.uniform(0, math.pi / 2)), trap=None)
        if case.get("walls"):      # held and dragged by the trap (App. C), on the droplet's constants (Table II)
            g.update(k_spring=0.5, eps_angle=0.3125, pull_force=0.0,
                     trap=dict(k=0.05, dx=min(100.0, nx / 5.0), dy=0.0, t_eq=30.0, pull=25000.0, width=30.0))
        out.append(g)
    return out


def _sweep_members(case, seed):
    """Members as in the batched recipe: side, ring, pull, diffusion (with sub-steps above 0.2), relaxation."""
    rng = np.random.Generator(np.random.PCG64(case["side_max"] * 1000 + case["count"]))   # sizes: the case's, not the seed's
    sides = [s for s in (64, 96, 128, 192, 256, 384, 512) if case["side_min"] <= s <= case["side_max"]]
    out = []
    for k in range(case["count"]):
        side = int(sides[k % len(sides)])
        r = float(rng.uniform(4.0, min(32.0, side / 4 - 7)))
        Dp = float(math.exp(rng.uniform(math.log(1e-3), math.log(1.0))))
        out.append(dict(nx=side, ny=side, steps=case["steps"], rings=1, radius=r, Dp=Dp,
                        nodes=int(min(256, max(32, round(2 * math.pi * r / 0.78)))),
                        substeps=int(math.ceil(Dp / 0.2)) if Dp > 0.2 else 0, lambda_steps=float(rng.uniform(20, 500))))
    return [(c, seed * 100 + k) for k, c in enumerate(out)]


def _dev():
    return torch.device("cuda" if torch.cuda.is_available() else "cpu")


def _waves(shape, count, amplitude, gen):
    """`count` smooth random fields: a few Fourier modes each (FP64)."""
    dev = gen.device
    ax = [torch.arange(n, dtype=torch.float64, device=dev) * (2 * math.pi / n) for n in shape]
    out = []
    for _ in range(count):
        f = torch.zeros(shape, dtype=torch.float64, device=dev)
        for _ in range(4):
            q = torch.randint(-3, 4, (len(shape),), generator=gen, device=dev).tolist()
            phase, amp = (torch.rand(2, dtype=torch.float64, generator=gen, device=dev)).tolist()
            arg = phase * 2 * math.pi
            for d, n in enumerate(shape):
                arg = arg + (q[d] * ax[d]).reshape([-1 if e == d else 1 for e in range(len(shape))])
            f += (0.3 + amp) * torch.cos(arg)
        out.append(amplitude * f)
    return torch.stack(out)


D2Q9 = [(0, 0), (1, 0), (0, 1), (-1, 0), (0, -1), (1, 1), (-1, 1), (-1, -1), (1, -1)]
W9 = [4 / 9] + [1 / 9] * 4 + [1 / 36] * 4
OPP9 = [0, 3, 4, 1, 2, 7, 8, 5, 6]


def _restart_state(case, seed):
    """The stored state [14, ny, nx] FP32: shifted populations of a moving fluid, stress, P - P_ref."""
    gen = torch.Generator(device=_dev()).manual_seed(seed)
    shape = (case["ny"], case["nx"])
    modulus = 2e-5 if case.get("scalar") else 2e-3
    drho, ux, uy = _waves(shape, 3, 2e-3, gen)
    drho = 0.1 * drho
    stress = _waves(shape, 3, 0.05 * modulus, gen)
    noise = torch.rand((2,) + shape, dtype=torch.float64, generator=gen, device=gen.device) * 0.1 - 0.05
    if case.get("scalar"):
        noise.zero_()
    pops = [w * (drho + 3 * (c[0] * ux + c[1] * uy) + 4.5 * (c[0] * ux + c[1] * uy) ** 2 - 1.5 * (ux * ux + uy * uy))
            for c, w in zip(D2Q9, W9)]
    return torch.cat([torch.stack(pops), stress, noise]).float().contiguous()


def _p_ref(w):
    Peq = math.sqrt(-w["alpha"] / w["beta"])
    return [float(np.float32(Peq * f(w["director_angle"]))) for f in (math.cos, math.sin)]


def _solver(case, seed):
    w = _physics(case)
    w["rings"] = _rings(case, seed)
    s = lb.Solver.from_workload(w, precision=lb.LB_FP16_BF16 if case.get("half") else lb.LB_FP32)
    state = _restart_state(case, seed)
    if case.get("half"):
        ref = _p_ref(w)
        for n in range(9):
            s.write_field("pop%d" % n, state[n].contiguous())
        for n, f in enumerate(("sxx", "syy", "sxy")):
            s.write_field(f, state[9 + n].contiguous())
        for n, f in enumerate(("Px", "Py")):
            s.write_field(f, (state[12 + n].double() + ref[n]).float())
    else:
        s.write_state(state)
    s.sync()
    X0 = np.concatenate([g["X"] for g in w["rings"]]) if w["rings"] else np.zeros((0, 2))
    return s, state, X0


def _net_params(seed):
    """He-scaled weights and small biases, one flat FP32 array in the network's order."""
    rng = np.random.Generator(np.random.PCG64(seed))
    parts = []
    for _, ci, co, act in LAYERS:
        sd = math.sqrt(2.0 / (9 * ci)) if act else 0.1 * math.sqrt(1.0 / (9 * ci))
        parts.append(rng.normal(0.0, sd, 9 * co * ci))
        parts.append(rng.normal(0.0, 0.05, co))
    return np.concatenate(parts).astype(np.float32)


def _net_inputs(case, seed):
    """Seven smooth noisy fields and an indicator, eight unused channels; targets likewise (FP32)."""
    gen = torch.Generator(device=_dev()).manual_seed(seed)
    B, H, W = case["batch"], case["height"], case["width"]
    x = torch.zeros((B, H, W, 16), dtype=torch.float64, device=gen.device)
    t = torch.zeros_like(x)
    for b in range(B):
        x[b, :, :, :8] = _waves((H, W), 8, 0.6, gen).permute(1, 2, 0)
        t[b, :, :, :7] = _waves((H, W), 7, 0.6, gen).permute(1, 2, 0) + 0.2
    x[..., :8] += 0.3 * torch.randn(x[..., :8].shape, dtype=torch.float64, generator=gen, device=gen.device)
    return x.to(torch.bfloat16).contiguous(), t.float().contiguous()


def _conv_inputs(case, seed):
    gen = torch.Generator(device=_dev()).manual_seed(seed)
    B, H, W, ci, co = (case[k] for k in ("batch", "height", "width", "ci", "co"))
    r = lambda *s: torch.randn(s, dtype=torch.float32, generator=gen, device=gen.device)  # noqa: E731
    x = torch.nn.functional.leaky_relu(r(B, H, W, ci) + 0.2, 0.1).to(torch.bfloat16)
    w = (r(9, co, ci) * math.sqrt(2.0 / (9 * ci))).to(torch.bfloat16)
    return x, w, 0.1 * r(co), (r(B, H, W, co) + 0.1).to(torch.bfloat16)


def prepare(case, seed):
    kind = case["kind"]
    if kind == "lattice":
        s, state, X0 = _solver(case, seed)
        return dict(case=case, s=s, out=state, X0=X0)
    if kind == "sweep":
        members = [(_solver(c, sd), c) for c, sd in _sweep_members(case, seed)]
        solvers = [m[0][0] for m in members]
        return dict(case=case, s=solvers, out=[m[0][1] for m in members], X0=[m[0][2] for m in members],
                    batch=lb.Batch(solvers))
    if kind == "box3d":
        w = _physics_3d(case)
        w["noise"] = _noise_3d(case, seed).cpu().numpy()
        return dict(case=case, s=lb3d.Solver3D.from_workload(w),
                    out=torch.empty((13, case["nz"], case["ny"], case["nx"]), dtype=torch.float32, device="cuda"))
    if kind == "conv":
        return dict(case=case, inputs=_conv_inputs(case, seed))
    net = lb.Net(case["batch"], case["height"], case["width"], seed=0)
    net.set_params(_net_params(seed))
    x, t = _net_inputs(case, seed)
    return dict(case=case, net=net, x=x, t=t)


def _motion(case, nodes, X0):
    """How far each node has moved (minimum image), FP32: what the Return and the deflection are made of."""
    box = np.array([case["nx"], case["ny"]], dtype=np.float64)
    d = nodes - X0
    return (d - box * np.round(d / box)).astype(np.float32)


def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "lattice":
        s, rings = state["s"], case["rings"]
        s.step(case["steps"])
        if case.get("half"):
            out = {k: s.readout(k) for k in lb.FIELDS}
        else:
            f = s.read_state(state["out"])
            out = {"populations": f[:9], "stress": f[9:12], "polarisation": f[12:]}
        if rings:
            out["motion"] = _motion(case, s.nodes(), state["X0"])
            out["restoring force"] = s.series_latest(1)[0, 6:].reshape(-1, 4)[:, :2].astype(np.float32)
        return out
    if kind == "sweep":
        state["batch"].step(case["steps"])
        out = {}
        for k, s in enumerate(state["s"]):
            f = s.read_state(state["out"][k])
            out["%d" % k] = [f[:9], f[9:12], f[12:]]
        out["restoring force"] = np.concatenate([s.series_latest(1)[0, 6:8] for s in state["s"]]).astype(np.float32)
        return out
    if kind == "box3d":
        s, out = state["s"], state["out"]
        s.step(case["steps"])
        for k, f in enumerate(lb3d.SCALARS):
            s.readout_device(f, out[k].data_ptr(), out[k].numel())
        return {"drho": out[0], "u": out[1:4], "stress": out[4:10], "polarisation": out[10:]}
    if kind == "conv":
        x, w, b, gz = state["inputs"]
        y = lb.conv3x3(x, w, b, act=True, out_f32=False)
        return [y, lb.conv3x3_dgrad(gz, w), *lb.conv3x3_wgrad(x, gz)]
    net = state["net"]
    y = net.forward(state["x"])
    if kind == "infer":
        return y
    # mean square over the seven used channels, its gradient back through the network
    g = (y - state["t"]) * (2.0 / (7 * y[..., 0].numel()))
    g[..., 7:] = 0.0
    net.backward(g)
    return {"y": y, "gradients": _by_layer(net.grads())}


def _by_layer(flat):
    """The parameters' gradients, one piece for each layer (its weights, then its bias)."""
    out, at = {}, 0
    for name, ci, co, _ in LAYERS:
        n = 9 * ci * co + co
        out[name] = flat[at:at + n]
        at += n
    return out


def work(case):
    """The state in and out once a step (as the solver stores it); the network's and the layer's
    inputs, weights and results once, and their multiply-adds."""
    kind = case["kind"]
    if kind == "lattice":
        n = case["nx"] * case["ny"] * case["steps"]
        return {"bytes": n * (96 if case.get("scalar") else 56 if case.get("half") else 112),
                "flops": n * (600 if case.get("scalar") else 1000)}
    if kind == "sweep":
        n = sum(c["nx"] * c["ny"] for c, _ in _sweep_members(case, 0)) * case["steps"]
        return {"bytes": n * 112, "flops": n * 1000}
    if kind == "box3d":
        n = case["nx"] * case["ny"] * case["nz"] * case["steps"]
        return {"bytes": n * 224, "flops": n * 2400}
    if kind == "conv":
        n, ci, co = case["batch"] * case["height"] * case["width"], case["ci"], case["co"]
        return {"bytes": 2 * n * 2 * (ci + co) + 9 * ci * co * 8, "flops": 3 * 18.0 * n * ci * co}
    n = case["batch"] * case["height"] * case["width"]
    layer = [18.0 * ci * co * n / 4 ** lev for (_, ci, co, _), lev in zip(LAYERS, LAYER_LEVEL)]
    par = sum(9 * ci * co + co for _, ci, co, _ in LAYERS)
    if kind == "infer":
        return {"bytes": n * 16 * 6 + par * 2, "flops": sum(layer)}
    return {"bytes": n * 16 * 14 + par * 8, "flops": 3 * sum(layer) - layer[0]}


# ------------------------------------------------------------------------------------ FP64

def exact(case, seed):
    kind = case["kind"]
    with torch.no_grad():
        if kind == "lattice":
            return _exact_lattice(case, seed)
        if kind == "sweep":
            got = [_exact_lattice(c, sd) for c, sd in _sweep_members(case, seed)]
            out = {"%d" % k: [r["populations"], r["stress"], r["polarisation"]] for k, r in enumerate(got)}
            out["restoring force"] = np.concatenate([r["restoring force"].reshape(-1) for r in got])
            return out
        if kind == "box3d":
            return _exact_3d(case, seed)
    if kind == "conv":
        return _exact_conv(case, seed)
    return _exact_net(case, seed)


class _Grid:
    """Neighbours and central differences on fields [..., ny, nx]: periodic, or with half-way walls on
    both axes whose ghost cells mirror the cell inside (negated where sign = -1)."""

    def __init__(self, walls):
        self.walls = walls

    def nb(self, f, axis, step, sign=1.0):
        r = torch.roll(f, -step, axis)
        if self.walls:
            edge = -1 if step > 0 else 0
            r.select(axis, edge).copy_(sign * f.select(axis, edge))
        return r

    def dx(self, f, sign=1.0):
        return 0.5 * (self.nb(f, -1, 1, sign) - self.nb(f, -1, -1, sign))

    def dy(self, f, sign=1.0):
        return 0.5 * (self.nb(f, -2, 1, sign) - self.nb(f, -2, -1, sign))

    def lap(self, f):
        return self.nb(f, -1, 1) + self.nb(f, -1, -1) + self.nb(f, -2, 1) + self.nb(f, -2, -1) - 4 * f


def _invert(P, ratio_and_slope, guess):
    k = guess
    for _ in range(8):
        r, d = ratio_and_slope(k)
        k = torch.clamp(k - (r - P) / d, min=1e-3)
    return k


def _stiffness(w, P):
    """C~(P) of App. B: nine planes, from |P| = I1(k) / I0(k) (capped) and the angle of P."""
    K11, K12, K22, K66 = w["K"]
    S, dK, X = 3 * K11 + 2 * K12 + 4 * K66 + 3 * K22, K11 - K22, K11 - 2 * K12 - 4 * K66 + K22
    Pm = torch.sqrt(P[0] ** 2 + P[1] ** 2)
    if X == 0.0 and dK == 0.0:
        r2 = r4 = torch.zeros_like(Pm)
    else:
        pc = torch.clamp(Pm, 1e-3, w["P_cap"])

        def ratio(k):
            r = torch.special.i1e(k) / torch.special.i0e(k)
            return r, 1 - r / k - r * r
        k = _invert(pc, ratio, pc * (2 - pc * pc) / (1 - pc * pc))
        r1 = ratio(k)[0]
        r2 = 1 - 2 * r1 / k
        r4 = r2 - 6 / k * (r1 - 4 * r2 / k)
    th = torch.atan2(P[1], P[0])
    c2, s2, c4, s4 = torch.cos(2 * th), torch.sin(2 * th), torch.cos(4 * th), torch.sin(4 * th)
    C11 = (S + 4 * r2 * dK * c2 + r4 * X * c4) / 8
    C12 = (K11 + 6 * K12 - 4 * K66 + K22 - r4 * X * c4) / 8
    C13 = (r4 * X * s4 + 2 * r2 * dK * s2) / 4
    C22 = C11 - r2 * dK * c2
    C23 = (2 * r2 * dK * s2 - r4 * X * s4) / 4
    C33 = (K11 - 2 * K12 + 4 * K66 + K22 - r4 * X * c4) / 4
    return [[C11, C12, C13], [C12, C22, C23], [C13 / 2, C23 / 2, C33]]


def _node_forces(g, X, t):
    """-dU/dR of springs, bending, pull and trap for one ring; X [n, 2] unwrapped."""
    n = X.shape[0]
    q = torch.roll(X, -1, 0) - X
    p = torch.roll(X, 1, 0) - X
    lq, lp = q.norm(dim=1, keepdim=True), p.norm(dim=1, keepdim=True)
    T = g["k_spring"] * (lq - g["l_eq"]) * q / lq
    f = T - torch.roll(T, 1, 0)
    c = (p * q).sum(1, keepdim=True) / (lp * lq)
    dp, dq = q / (lp * lq) - c * p / lp ** 2, p / (lp * lq) - c * q / lq ** 2
    f = f + g["eps_angle"] * (dp + dq - torch.roll(dp, -1, 0) - torch.roll(dq, 1, 0))
    pull = [g["pull_force"] * fn(g["pull_angle"]) / n for fn in (math.cos, math.sin)]
    tr = g["trap"]
    if tr:
        sig = lambda c0: 1 / (1 + math.exp(min(700.0, -8 * (t - c0) / tr["width"])))  # noqa: E731
        soft = lambda z: max(z, 0.0) + math.log1p(math.exp(-abs(z)))  # noqa: E731
        a, end = 8 / tr["width"], tr["t_eq"] + tr["pull"]
        k = tr["k"] * sig(tr["width"] / 2) * (1 - sig(end + tr["width"] / 2))
        s = (soft(a * (t - tr["t_eq"])) - soft(a * (t - end))) / (a * tr["pull"])
        com = X.mean(0).tolist()
        pull = [pull[d] + k * (g["centre"][d] + tr[("dx", "dy")[d]] * s - com[d]) / n for d in (0, 1)]
    return f + torch.tensor(pull, dtype=torch.float64, device=X.device)


def _support(X, ny, nx):
    """Cells (flat) and cosine-kernel weights of the 4 x 4 support of every node: [n, 16] each."""
    o = torch.arange(-1, 3, device=X.device)
    base = torch.floor(X).long()
    cx, cy = base[:, :1] + o, base[:, 1:] + o
    phi = lambda d: 0.25 * (1 + torch.cos(math.pi * d / 2))  # noqa: E731
    wx, wy = phi(X[:, :1] - cx), phi(X[:, 1:] - cy)
    cell = (cy % ny)[:, :, None] * nx + (cx % nx)[:, None, :]
    return cell.reshape(len(X), 16), (wy[:, :, None] * wx[:, None, :]).reshape(len(X), 16)


def _interp(f, X):
    cell, wt = _support(X, f.shape[1], f.shape[2])
    return (f.reshape(2, -1)[:, cell] * wt).sum(2).T


def _exact_lattice(case, seed):
    w, rings = _physics(case), _rings(case, seed)
    state = _restart_state(case, seed).double()
    dev, ny, nx = state.device, case["ny"], case["nx"]
    g = _Grid(bool(case.get("walls")))
    wn = torch.tensor(W9, dtype=torch.float64, device=dev).reshape(9, 1, 1)
    c9 = torch.tensor(D2Q9, dtype=torch.float64, device=dev)
    h = state[:9] + wn * w["rho0"]
    sig = state[9:12].clone()
    ref = _p_ref(w)
    ref_planes = torch.tensor(ref, dtype=torch.float64, device=dev).reshape(2, 1, 1)
    P = state[12:] + ref_planes
    X0 = [torch.tensor(r["X"], dtype=torch.float64, device=dev) for r in rings]
    X = [x.clone() for x in X0]
    for r, x in zip(rings, X0):
        r["centre"] = x.mean(0).tolist()
    eta = w.get("eta_p") or w["lambda_steps"] * (3 * w["K"][0] + 2 * w["K"][1] + 4 * w["K"][3] + 3 * w["K"][2]) / 8
    sub = w["diffusion_substeps"]
    scalar = bool(case.get("scalar"))
    frest = None

    def field_h(P):
        return (w["alpha"] + w["beta"] * (P * P).sum(0)) * P - w["kappa"] * g.lap(P)

    def rhs(sig, P, u, psi, om):
        C = _stiffness(w, P)
        gx, gy, lap = g.dx(sig), g.dy(sig), g.lap(sig)
        J = torch.stack([2 * om * sig[2], -2 * om * sig[2], om * (sig[1] - sig[0])])
        e = [psi[k] - sig[k] / eta for k in range(3)]
        Ce = torch.stack([C[i][0] * e[0] + C[i][1] * e[1] + C[i][2] * e[2] for i in range(3)])
        ds = -(u[0] * gx + u[1] * gy) - J + Ce + (0.0 if sub else w["Dp"]) * lap
        if scalar:
            return ds, torch.zeros_like(P)
        adv = u[0] * g.dx(P) + u[1] * g.dy(P)
        rot = torch.stack([om * P[1], -om * P[0]])
        stretch = torch.stack([psi[0] * P[0] + psi[2] * P[1], psi[2] * P[0] + psi[1] * P[1]])
        return ds, -adv - rot + w["xi"] * stretch - w["Gamma"] * field_h(P)

    for t in range(case["steps"]):
        fp = torch.stack([g.dx(sig[0]) + g.dy(sig[2]), g.dx(sig[2]) + g.dy(sig[1])])
        F = fp.clone()
        if w["ericksen"]:
            hm = field_h(P)
            Gx, Gy = g.dx(P), g.dy(P)
            grad = (Gx, Gy)
            sE = [[-0.5 * (P[i] * hm[j] - hm[i] * P[j]) + 0.5 * w["xi"] * (P[i] * hm[j] + hm[i] * P[j])
                   - w["kappa"] * (grad[i] * grad[j]).sum(0) for j in (0, 1)] for i in (0, 1)]
            F += torch.stack([g.dx(sE[i][0], -1.0) + g.dy(sE[i][1], -1.0) for i in (0, 1)])
        for r, x in zip(rings, X):
            f = _node_forces(r, x, float(t))
            cell, wt = _support(x, ny, nx)
            for d in (0, 1):
                F[d].reshape(-1).index_add_(0, cell.reshape(-1), (f[:, d:d + 1] * wt).reshape(-1))
        if rings and t % w["every"] == 0:
            frest = torch.stack([_interp(fp, x).sum(0) for x in X])
        rho = h.sum(0)
        u = (torch.einsum("na,nyx->ayx", c9, h) + 0.5 * F) / rho
        uu, uF = (u * u).sum(0), (u * F).sum(0)
        hs = torch.empty_like(h)
        for n, (cx, cy) in enumerate(D2Q9):
            cu, cF = cx * u[0] + cy * u[1], cx * F[0] + cy * F[1]
            heq = W9[n] * rho * (1 + 3 * cu + 4.5 * cu * cu - 1.5 * uu)
            src = (1 - 0.5 / w["tau"]) * W9[n] * (3 * (cF - uF) + 9 * cu * cF)
            hs[n] = h[n] - (h[n] - heq) / w["tau"] + src
        for n, (cx, cy) in enumerate(D2Q9):
            h[n] = torch.roll(hs[n], (cy, cx), (0, 1))
            if g.walls:       # what would have come through a wall is the opposite one, sent back
                back = hs[OPP9[n]]
                if cx:
                    at = 0 if cx > 0 else nx - 1
                    h[n][:, at] = back[:, at]
                if cy:
                    at = 0 if cy > 0 else ny - 1
                    h[n][at] = back[at]
        dxu, dyu = g.dx(u, -1.0), g.dy(u, -1.0)
        psi = [dxu[0], dyu[1], 0.5 * (dxu[1] + dyu[0])]
        om = 0.5 * (dxu[1] - dyu[0])
        ds0, dP0 = rhs(sig, P, u, psi, om)
        ds1, dP1 = rhs(sig + ds0, P + dP0, u, psi, om)
        sig = sig + 0.5 * (ds0 + ds1)
        P = P + 0.5 * (dP0 + dP1)
        for _ in range(sub):
            D = w["Dp"] / sub
            d0 = D * g.lap(sig)
            sig = sig + 0.5 * (d0 + D * g.lap(sig + d0))
        for k, x in enumerate(X):
            v0 = _interp(u, x)
            X[k] = x + 0.5 * (v0 + _interp(u, x + v0))
    if case.get("half"):
        # rho and u of the last state take its forces
        out = dict(zip(lb.FIELDS, [None, None, None, sig[0], sig[1], sig[2], P[0], P[1]]))
    else:
        out = {"populations": h - wn * w["rho0"], "stress": sig, "polarisation": P - ref_planes}
    if rings:
        out["motion"] = torch.cat([x - x0 for x, x0 in zip(X, X0)]).cpu().numpy()
        out["restoring force"] = frest.cpu().numpy()
    return out


# three dimensions

D3Q19 = [(0, 0, 0), (1, 0, 0), (-1, 0, 0), (0, 1, 0), (0, -1, 0), (0, 0, 1), (0, 0, -1), (1, 1, 0), (-1, -1, 0),
         (1, -1, 0), (-1, 1, 0), (1, 0, 1), (-1, 0, -1), (1, 0, -1), (-1, 0, 1), (0, 1, 1), (0, -1, -1), (0, 1, -1),
         (0, -1, 1)]
W19 = [1 / 3] + [1 / 18] * 6 + [1 / 36] * 12
SYM = [[0, 5, 4], [5, 1, 3], [4, 3, 2]]      # index of (i, j) in (xx, yy, zz, yz, xz, xy)
PAIRS = [(0, 0), (1, 1), (2, 2), (1, 2), (0, 2), (0, 1)]


def _physics_3d(case):
    return dict(PHYSICS_3D, nx=case["nx"], ny=case["ny"], nz=case["nz"], every=10, fext=None,
                ericksen=int(case.get("ericksen", True)))


def _noise_3d(case, seed):
    gen = torch.Generator(device=_dev()).manual_seed(seed)
    shape = (3, case["nz"], case["ny"], case["nx"])
    return torch.rand(shape, dtype=torch.float64, generator=gen, device=gen.device) * 0.1 - 0.05


def _contract_3d(w, P, X):
    """C : X with C the average of the rotated K^x over the Fisher density of mean P (X: six planes)."""
    K11, K12, K22, K66, K23 = w["K"]
    a5 = 0.5 * (K22 - K23)
    a3, a4, a2 = K23, K66 - a5, K12 - K23
    a1 = K11 - 2 * a2 - a3 - 4 * a4 - 2 * a5
    Pm = torch.sqrt((P * P).sum(0))
    pc = torch.clamp(Pm, 1e-3, w["P_cap"])
    n = P / Pm

    def ratio(k):
        return 1 / torch.tanh(k) - 1 / k, 1 / (k * k) - 1 / torch.sinh(k) ** 2
    k = _invert(pc, ratio, pc * (3 - pc * pc) / (1 - pc * pc))
    L = ratio(k)[0]
    m2 = 1 - 2 * L / k
    m3 = 1 / torch.tanh(k) - 3 * m2 / k
    m4 = 1 - 4 * m3 / k
    A, B = 0.5 * (1 - m2), 0.5 * (3 * m2 - 1)
    e3 = (A - B + m4) / 8
    e2 = A - 5 * e3
    e1 = B - 7 * e2
    Xn = torch.stack([sum(X[SYM[i][j]] * n[j] for j in range(3)) for i in range(3)])
    nXn, tr = (n * Xn).sum(0), X[0] + X[1] + X[2]
    out = []
    for c, (i, j) in enumerate(PAIRS):
        d = 1.0 if i == j else 0.0
        nn, sym = n[i] * n[j], n[i] * Xn[j] + n[j] * Xn[i]
        m4x = e1 * nn * nXn + e2 * (nn * tr + 2 * sym + d * nXn) + e3 * (d * tr + 2 * X[c])
        m2ij = A * d + B * nn
        out.append(a1 * m4x + a2 * (m2ij * tr + d * (A * tr + B * nXn)) + a3 * d * tr
                   + a4 * (4 * A * X[c] + 2 * B * sym) + 2 * a5 * X[c])
    return torch.stack(out)


def _exact_3d(case, seed):
    w = _physics_3d(case)
    noise = _noise_3d(case, seed)
    dev = noise.device
    Peq = math.sqrt(-w["alpha"] / w["beta"])
    P = noise + Peq * torch.tensor(w["director"], dtype=torch.float64, device=dev).reshape(3, 1, 1, 1)
    d = lambda f, a: 0.5 * (torch.roll(f, -1, -1 - a) - torch.roll(f, 1, -1 - a))  # noqa: E731
    lap = lambda f: sum(torch.roll(f, s, -1 - a) for a in range(3) for s in (1, -1)) - 6 * f  # noqa: E731
    shape = noise.shape[1:]
    h = torch.tensor(W19, dtype=torch.float64, device=dev).reshape(19, 1, 1, 1).expand((19,) + shape) * w["rho0"]
    h = h.contiguous()
    sig = torch.zeros((6,) + shape, dtype=torch.float64, device=dev)

    def field_h(P):
        return (w["alpha"] + w["beta"] * (P * P).sum(0)) * P - w["kappa"] * lap(P)

    def moments():
        F = torch.stack([sum(d(sig[SYM[i][j]], j) for j in range(3)) for i in range(3)])
        if w["ericksen"]:
            hm = field_h(P)
            grad = [d(P, a) for a in range(3)]
            for i in range(3):
                for j in range(3):
                    F[i] += d(-0.5 * (P[i] * hm[j] - hm[i] * P[j]) + 0.5 * w["xi"] * (P[i] * hm[j] + hm[i] * P[j])
                              - w["kappa"] * (grad[i] * grad[j]).sum(0), j)
        rho = h.sum(0)
        u = torch.stack([sum(c[a] * h[n] for n, c in enumerate(D3Q19) if c[a]) + 0.5 * F[a] for a in range(3)]) / rho
        return F, rho, u

    def rhs(sig, P, u, G):
        om = lambda i, j: 0.5 * (G[i][j] - G[j][i])  # noqa: E731
        psi = torch.stack([0.5 * (G[i][j] + G[j][i]) for i, j in PAIRS])
        ds = _contract_3d(w, P, psi - sig / w["eta_p"]) + w["Dp"] * lap(sig) - sum(u[a] * d(sig, a) for a in range(3))
        for c, (i, j) in enumerate(PAIRS):
            for k in range(3):
                ds[c] -= om(i, k) * sig[SYM[k][j]] - sig[SYM[i][k]] * om(k, j)
        dP = -sum(u[a] * d(P, a) for a in range(3)) - w["Gamma"] * field_h(P)
        for i in range(3):
            for k in range(3):
                dP[i] += -om(i, k) * P[k] + w["xi"] * psi[SYM[i][k]] * P[k]
        return ds, dP

    for _ in range(case["steps"]):
        F, rho, u = moments()
        uu, uF = (u * u).sum(0), (u * F).sum(0)
        for n, c in enumerate(D3Q19):
            cu, cF = sum(c[a] * u[a] for a in range(3)), sum(c[a] * F[a] for a in range(3))
            heq = W19[n] * rho * (1 + 3 * cu + 4.5 * cu * cu - 1.5 * uu)
            src = (1 - 0.5 / w["tau"]) * W19[n] * (3 * (cF - uF) + 9 * cu * cF)
            h[n] = torch.roll(h[n] - (h[n] - heq) / w["tau"] + src, (c[2], c[1], c[0]), (0, 1, 2))
        G = [d(u, i) for i in range(3)]
        ds0, dP0 = rhs(sig, P, u, G)
        ds1, dP1 = rhs(sig + ds0, P + dP0, u, G)
        sig, P = sig + 0.5 * (ds0 + ds1), P + 0.5 * (dP0 + dP1)
    _, rho, u = moments()
    return {"drho": rho - w["rho0"], "u": u, "stress": sig, "polarisation": P}


# the network

def _conv64(x, w, b, act):
    """x [B, C, H, W], w [9, Co, Ci] with tap 3 (dy + 1) + dx + 1."""
    k = w.reshape(3, 3, w.shape[1], w.shape[2]).permute(2, 3, 0, 1)
    y = torch.nn.functional.conv2d(x, k, b, padding=1)
    return torch.nn.functional.leaky_relu(y, 0.1) if act else y


def _exact_conv(case, seed):
    x, w, b, gz = (v.double() for v in _conv_inputs(case, seed))
    x, gz = x.permute(0, 3, 1, 2), gz.permute(0, 3, 1, 2)
    y = _conv64(x, w, b, True).permute(0, 2, 3, 1).contiguous()
    x.requires_grad_(True), w.requires_grad_(True), b.requires_grad_(True)
    gx, gw, gb = torch.autograd.grad(_conv64(x, w, b, False), (x, w, b), gz)
    return [y, gx.permute(0, 2, 3, 1).contiguous(), gw, gb]


def _exact_net(case, seed):
    x, t = _net_inputs(case, seed)
    x, t = x.double().permute(0, 3, 1, 2), t.double()
    flat = torch.tensor(_net_params(seed), device=x.device).double()
    flat.requires_grad_(case["kind"] == "gradients")
    at, par = 0, {}
    for name, ci, co, act in LAYERS:
        n = 9 * ci * co
        par[name] = (flat[at:at + n].reshape(9, co, ci), flat[at + n:at + n + co], act)
        at += n + co
    layer = lambda name, v: _conv64(v, *par[name])  # noqa: E731
    pool = lambda v: torch.nn.functional.avg_pool2d(v, 2)  # noqa: E731
    up = lambda v: torch.nn.functional.interpolate(v, scale_factor=2, mode="nearest")  # noqa: E731
    e0 = layer("e0b", layer("e0a", x))
    e1 = layer("e1b", layer("e1a", pool(e0)))
    e2 = layer("e2b", layer("e2a", pool(e1)))
    bt = layer("btb", layer("bta", pool(e2)))
    d2 = layer("d2b", layer("d2a", torch.cat([up(bt), e2], 1)))
    d1 = layer("d1b", layer("d1a", torch.cat([up(d2), e1], 1)))
    d0 = layer("d0b", layer("d0a", torch.cat([up(d1), e0], 1)))
    y = layer("head", d0).permute(0, 2, 3, 1)
    if case["kind"] == "infer":
        return y.contiguous()
    g = (y.detach() - t) * (2.0 / (7 * y[..., 0].numel()))
    g[..., 7:] = 0.0
    (gf,) = torch.autograd.grad(y, flat, g)
    return {"y": y.detach().contiguous(), "gradients": _by_layer(gf.cpu().numpy())}
