"""The performance cases: what users of the solver have it do, each a whole call of the public API.

A flow case is one solve from an initial state: the state goes in, `steps` time steps run, the
macroscopic fields come out; the population store is the caller's own buffer, so the updated state
is at hand as well.  Sizes and parameters are those of the configurations, tests and benchmark of
this repository (Kolmogorov flow, Taylor-Green vortex, porous channels, Shan-Chen droplet,
Orszag-Tang vortex, Rayleigh-Taylor instability, batched porous channels, the neural operator of the
warm start), with seeded variations of the initial state.  exact() is the same mathematics in FP64
with plain torch.
"""
import ctypes
import math

import torch

from paper_1905_10182_gb300 import Solver
from paper_1905_10182_gb300 import _native as nat

DEV = "cuda"
TYPES = {"fp32": torch.float32, "fp16": torch.float16, "bf16": torch.bfloat16}


# ------------------------------------------------------------------------------------- cases
def listed():
    return [
        # parity-sized study: a small periodic box, many steps, where launches and latency count
        dict(name="kolmogorov_32_fp32", kind="kolmogorov", nx=32, ny=32, nz=32, storage="fp32", steps=100, nu=0.05),
        # an ordinary box at 16-bit storage, sizes that are no powers of two
        dict(name="tgv_100x72x90_bf16", kind="tgv", nx=100, ny=72, nz=90, storage="bf16", steps=60, nu=1e-3),
        # one porous channel (walls, solid mask), odd sizes
        dict(name="porous_93x47x81_fp32", kind="porous", nx=93, ny=47, nz=81, storage="fp32", steps=60, nu=0.05),
        # 16-bit storage on a large box
        dict(name="kolmogorov_256_fp16", kind="kolmogorov", nx=256, ny=256, nz=256, storage="fp16", steps=40, nu=0.05),
        # the forced benchmark path: static droplet with the Shan-Chen force
        dict(name="droplet_128_fp32", kind="droplet", nx=128, ny=128, nz=128, storage="fp32", steps=40, nu=1.0 / 6.0),
        # the same physics at 16-bit storage on an uneven box that fits in L2
        dict(name="droplet_96x80x112_fp16", kind="droplet", nx=96, ny=80, nz=112, storage="fp16", steps=40, nu=1.0 / 6.0),
        # magnetic field (Orszag-Tang vortex)
        dict(name="orszag_tang_128", kind="mhd", nx=128, ny=128, nz=128, storage="fp32", steps=40, nu=0.005),
        # two-phase colour gradient (Rayleigh-Taylor, walls)
        dict(name="rayleigh_taylor_64x256x64", kind="cg", nx=64, ny=256, nz=64, storage="fp32", steps=30, nu=0.005),
        # many uneven channels advanced together, the steady solves of the warm start
        dict(name="batch_porous_40", kind="batch", count=40, steps=100),
        # the benchmark's default workload, the largest box
        dict(name="tgv_512_fp32", kind="tgv", nx=512, ny=512, nz=512, storage="fp32", steps=16, nu=1e-4),
        # inference of the warm start at its study's configuration
        dict(name="operator_forward_64", kind="forward", D=64, modes=12, batch=4),
        # one optimisation step of its training
        dict(name="operator_train_64", kind="train", D=64, modes=12, batch=4),
    ]


def draw(rng):
    kind = rng.choice(["kolmogorov", "tgv", "tgv", "porous", "droplet", "droplet", "mhd", "cg", "batch", "forward", "train"])
    if kind == "batch":
        return dict(kind=kind, count=round(math.exp(rng.uniform(math.log(4), math.log(64)))), steps=2 * rng.randint(20, 50))
    if kind in ("forward", "train"):
        return dict(kind=kind, D=rng.choice([32, 48, 64]), modes=rng.choice([8, 12]), batch=rng.randint(1, 4))
    top = {"mhd": 160, "cg": 120}.get(kind, 320)
    edge = math.exp(rng.uniform(math.log(28), math.log(top)))
    nx, ny, nz = (max(16, round(edge * rng.uniform(0.7, 1.4))) for _ in range(3))
    storage = "fp32" if kind in ("mhd", "cg", "porous") else rng.choice(["fp32", "fp16", "bf16" if kind != "droplet" else "fp16"])
    steps = 2 * rng.randint(8, 40)
    while nx * ny * nz * steps > 6e8 and steps > 8:
        steps -= 2
    nu = {"mhd": 0.005, "cg": 0.005, "droplet": 1.0 / 6.0, "porous": 0.05}.get(kind, round(rng.uniform(1e-3, 0.1), 4))
    return dict(kind=kind, nx=nx, ny=ny, nz=nz, storage=storage, steps=steps, nu=nu)


def nodes(case):
    return case["nx"] * case["ny"] * case["nz"]


def work(case):
    k = case["kind"]
    if k in ("forward", "train"):
        return operator_work(case)
    if k == "batch":
        n = sum(d["nx"] * d["ny"] * d["nz"] for d in batch_domains(case, 0))
        # populations read and written once a step, fields out at the end
        return {"bytes": n * (216 * case["steps"] + 16), "flops": 600 * n * case["steps"]}
    n, size = nodes(case), 4 if case["storage"] == "fp32" else 2
    # populations read and written once a step (two colours, 21 magnetic ones), initial fields in, fields out
    per = {"mhd": 2 * 4 * 48, "cg": 2 * 4 * 54}.get(k, 2 * 27 * size)
    ends = {"mhd": 28 + 40, "cg": 8 + 24}.get(k, 32)
    return {"bytes": n * (per * case["steps"] + ends), "flops": (1300 if k == "cg" else 600) * n * case["steps"]}


# ------------------------------------------------------------------------------------- inputs
def generator(seed):
    return torch.Generator(device=DEV).manual_seed(int(seed) + 20261)


def uniform(gen, lo, hi, shape=(1,)):
    return lo + (hi - lo) * torch.rand(shape, generator=gen, device=DEV, dtype=torch.float64)


def axes(nx, ny, nz):
    ar = [torch.arange(n, device=DEV, dtype=torch.float64) for n in (nx, ny, nz)]
    return ar[0][None, None, :], ar[1][None, :, None], ar[2][:, None, None]


def spheres(gen, nx, ny, nz, fraction, walls):
    """Solid spheres of radius 3 to 8 put at random until the solid fraction is reached (periodic in x and z)."""
    x, y, z = axes(nx, ny, nz)
    mask = torch.zeros((nz, ny, nx), dtype=torch.bool, device=DEV)
    par = torch.rand((400, 4), generator=gen, device=DEV, dtype=torch.float64).cpu().tolist()
    room, volume = fraction * nx * ny * nz, 0.0
    for a, b, c, r in par:
        if volume >= room:
            break
        r = 3 + 5 * r
        cx, cz = a * nx, c * nz
        cy = r + b * max(0.0, ny - 2 * r)
        dx = (x - cx).abs()
        dz = (z - cz).abs()
        mask |= torch.minimum(dx, nx - dx) ** 2 + (y - cy) ** 2 + torch.minimum(dz, nz - dz) ** 2 <= r * r
        volume += 4.19 * r ** 3
    return mask.to(torch.uint8)


def flow_inputs(case, seed):
    """rho, u (4 fields), and what the kind needs besides, all FP32 as a user hands them over."""
    nx, ny, nz, kind = case["nx"], case["ny"], case["nz"], case["kind"]
    gen = generator(seed)
    x, y, z = axes(nx, ny, nz)
    kx, ky, kz = (2 * math.pi / n for n in (nx, ny, nz))
    f = torch.zeros((4, nz, ny, nx), device=DEV)
    f[0] = 1.0
    more = {}
    ph = uniform(gen, 0, 2 * math.pi, (3,))
    amp = uniform(gen, 0.8, 1.2).item()
    if kind == "tgv":
        u0 = 0.05 * amp
        X, Y, Z = kx * x + ph[0], ky * y + ph[1], kz * z + ph[2]
        f[1] = u0 * torch.sin(X) * torch.cos(Y) * torch.cos(Z)
        f[2] = -u0 * torch.cos(X) * torch.sin(Y) * torch.cos(Z)
        f[0] = 1 + 3 * u0 * u0 / 16 * (torch.cos(2 * X) + torch.cos(2 * Y)) * (torch.cos(2 * Z) + 2)
    elif kind == "kolmogorov":
        f[1] = 5e-3 * amp * torch.sin(ky * y + 0 * x + 0 * z) + 5e-4 * torch.sin(kz * z + ph[0])
        f[2] = 5e-4 * torch.sin(kx * x + ph[1])
        f[3] = 5e-4 * torch.sin(kx * x + ky * y + ph[2])
        more["force"] = ("kolmogorov", (1e-5 * amp,))
    elif kind == "porous":
        more["mask"] = spheres(gen, nx, ny, nz, 0.12, True)
        more["force"] = ("uniform", (5e-6 * amp, 0.0, 0.0))
        h = (y + 0.5) * (ny - 0.5 - y) * 4 / ny ** 2
        f[1] = 0.01 * amp * h
        f[3] = 0.002 * h * torch.sin(kx * x + ph[0])
    elif kind == "droplet":
        radius = min(nx, ny, nz) * 0.1875 * amp
        r = torch.sqrt((x - nx / 2 - ph[0]) ** 2 + (y - ny / 2 - ph[1]) ** 2 + (z - nz / 2 + ph[2]) ** 2)
        f[0] = 0.5 * (2.4 + 0.13) - 0.5 * (2.4 - 0.13) * torch.tanh(r - radius)
        more["force"] = ("shan_chen", (-5.5,))
    elif kind == "mhd":
        u0 = 0.0203 * amp
        X, Y, Z = kx * x + ph[0], ky * y + ph[1], kz * z + ph[2]
        f[1] = 2 * u0 * torch.sin(Y)
        f[2] = 2 * u0 * torch.sin(X)
        b = torch.zeros((3, nz, ny, nx), device=DEV)
        b[0] = 0.8 * u0 * (-2 * torch.sin(2 * Y) + torch.sin(Z))
        b[1] = 0.8 * u0 * (2 * torch.sin(X) + torch.sin(Z))
        b[2] = 0.8 * u0 * (torch.sin(X) + torch.sin(Y))
        more["b"] = b
    elif kind == "cg":
        heavy = y + 0.5 > ny / 2 + 0.05 * nx * amp * (torch.cos(kx * x + ph[0]) + torch.cos(kz * z + ph[1]))
        more["red"] = torch.where(heavy, 3.0, 0.0).to(torch.float32).contiguous()
        more["blue"] = torch.where(heavy, 0.0, 1.0).to(torch.float32).contiguous()
        more["prm"] = dict(rho_r0=3.0, rho_b0=1.0, nu_r=case["nu"], nu_b=case["nu"], A=1e-4, beta=0.7,
                           g=(0.0, -0.04 ** 2 / nx, 0.0))
    return f, more


def batch_domains(case, seed):
    """Sizes come from the case alone, so that every seed's batch is the same amount of work."""
    out = []
    for k in range(case["count"]):
        h = (k * 2654435761 + 97) % (1 << 32)
        nx, ny, nz = 32 + h % 65, 32 + (h >> 8) % 17, 32 + (h >> 16) % 65
        out.append(dict(nx=nx, ny=ny, nz=nz, nu=0.01 + 0.09 * ((h >> 5) % 1000) / 1000, fraction=0.2 * ((h >> 11) % 100) / 100,
                        fx=1e-6 + 9e-6 * ((h >> 3) % 1000) / 1000, seed=int(seed) * 1009 + k))
    return out


def batch_inputs(d):
    gen = generator(d["seed"])
    x, y, z = axes(d["nx"], d["ny"], d["nz"])
    mask = spheres(gen, d["nx"], d["ny"], d["nz"], d["fraction"], True)
    f = torch.zeros((4, d["nz"], d["ny"], d["nx"]), device=DEV)
    f[0] = 1.0
    f[1] = 0.02 * (y + 0.5) * (d["ny"] - 0.5 - y) * 4 / d["ny"] ** 2 * (1 + 0.1 * uniform(gen, -1, 1))
    return mask, f


def operator_shapes(case, width=32, layers=4, ch=4):
    m = case["modes"]
    shapes = [("P", (width, ch)), ("p", (width,))]
    for k in range(layers):
        shapes += [("Wm%d" % k, (m, 2 * m, 2 * m, width, width, 2)), ("Wc%d" % k, (width, width)), ("b%d" % k, (width,))]
    return shapes + [("Q", (ch, width)), ("q", (ch,))]


def operator_inputs(case, seed):
    """Parameters of a fan-in-scaled draw; features and targets like those of the porous channels."""
    gen = generator(seed)
    parts = []
    for name, shape in operator_shapes(case):
        n = math.prod(shape)
        r = torch.rand(n, generator=gen, device=DEV)
        if name.startswith("Wm"):
            parts.append(r / 32 ** 2)
        elif len(shape) == 1:
            parts.append(0.2 * r - 0.1)
        else:
            parts.append((2 * r - 1) / math.sqrt(shape[-1]))
    D, B = case["D"], case["batch"]
    a = torch.empty((B, 4, D, D, D), device=DEV)
    t = torch.empty_like(a)
    x, y, z = axes(D, D, D)
    for k in range(B):
        mask = spheres(gen, D, D, D, 0.1, True)
        par = uniform(gen, 0.1, 1.0, (8,))
        a[k, 0] = mask
        a[k, 1], a[k, 2] = par[0], par[1]
        a[k, 3] = (y + 0.5) / D
        flow = (y + 0.5) * (D - 0.5 - y) * 4 / D ** 2 * (1 - mask)
        t[k, 0] = par[2] * flow
        t[k, 1] = 0.1 * flow * torch.sin(2 * math.pi * x / D + 6 * par[3])
        t[k, 2] = 0.1 * flow * torch.cos(2 * math.pi * z / D + 6 * par[4])
        t[k, 3] = 0.05 * torch.sin(2 * math.pi * (x + 2 * z) / D + 6 * par[5])
    return torch.cat(parts), a, t


def operator_work(case, W=32, L=4, ch=4):
    """One pass over the activations that the definition needs: the features and each layer's input and
    mode matrices read, each layer's output written (activations FP32), the transforms' and maps' operations."""
    D, m, B = case["D"], case["modes"], case["batch"]
    S, modes = D ** 3, 4 * m ** 3
    act = 4.0 * B * W * S
    par = 4.0 * sum(math.prod(s) for _, s in operator_shapes(case))
    forward = 4.0 * B * ch * S * 2 + 2 * L * act + par
    dft = 2.0 * B * W * 2 * (S * 2 * m + 2 * D * D * m * 4 * m + 4 * D * m * 2 * m * 2 * m)
    flops = L * (dft + 2.0 * B * W * W * S + 8.0 * B * W * W * modes) + 4.0 * B * W * ch * S
    if case["kind"] == "forward":
        return {"bytes": forward, "flops": flops}
    # backward reads each layer's activations and writes their gradient; Adam reads p, g, m, v and writes p, m, v
    return {"bytes": forward + 3 * L * act + 7 * par, "flops": 3 * flops}


# ------------------------------------------------------------------------------------- the calls
def check(status, what):
    if status != nat.LBM_OK:
        raise RuntimeError("%s: %s" % (what, nat.status_name(status)))


class Handle:
    """A handle of the C ABI that goes with its owner."""

    def __init__(self, h, destroy):
        self.h, self.destroy = h, destroy

    def __del__(self):
        self.destroy(self.h)


def stream():
    return ctypes.c_void_p(torch.cuda.current_stream().cuda_stream)


def prepare(case, seed):
    kind = case["kind"]
    if kind == "batch":
        return prepare_batch(case, seed)
    if kind in ("forward", "train"):
        return prepare_operator(case, seed)
    nx, ny, nz = case["nx"], case["ny"], case["nz"]
    f, more = flow_inputs(case, seed)
    store = torch.zeros(27 * nodes(case) * (4 if case["storage"] == "fp32" else 2), dtype=torch.uint8, device=DEV)
    s = Solver(nx, ny, nz, nu=case["nu"], walls_y=kind in ("porous", "cg"), mask=more.get("mask"), storage=case["storage"], store=store)
    if "force" in more:
        s.set_force(*more["force"])
    state = dict(case=case, solver=s, fields=f, more=more, store=store.view(TYPES[case["storage"]]).view(27, nz, ny, nx),
                 out=torch.empty((4, nz, ny, nx), device=DEV))
    if kind in ("mhd", "cg"):
        state["extra"] = torch.empty((6 if kind == "mhd" else 2, nz, ny, nx), device=DEV)
    return state


def prepare_batch(case, seed):
    L = nat.lib()
    doms = batch_domains(case, seed)
    arr = (nat.LbmDomain * len(doms))()
    keep, fields, outs = [], [], []
    for a, d in zip(arr, doms):
        mask, f = batch_inputs(d)
        a.nx, a.ny, a.nz, a.nu, a.walls_y, a.mask = d["nx"], d["ny"], d["nz"], d["nu"], 1, mask.data_ptr()
        a.force[0] = d["fx"]
        keep.append(mask)
        fields.append(f)
        outs.append(torch.empty_like(f))
    h = ctypes.c_void_p()
    check(L.lbm_batch_create(arr, len(doms), 1.0, stream(), ctypes.byref(h)), "lbm_batch_create")
    check(L.lbm_batch_set_shape(h, 64, 8, 2), "lbm_batch_set_shape")  # the shape that tuning reports for such batches
    return dict(case=case, batch=Handle(h, L.lbm_batch_destroy), fields=fields, outs=outs)


def prepare_operator(case, seed):
    L = nat.lib()
    theta, a, t = operator_inputs(case, seed)
    h = ctypes.c_void_p()
    check(L.lbm_no_create(case["D"], 32, case["modes"], 4, 4, 4, case["batch"], 1, stream(), ctypes.byref(h)), "lbm_no_create")
    net = Handle(h, L.lbm_no_destroy)
    check(L.lbm_no_params(h, theta.data_ptr(), 1), "lbm_no_params")
    state = dict(case=case, net=net, a=a, t=t)
    if case["kind"] == "forward":
        state["out"] = torch.empty_like(a)
    else:
        state["grads"], state["params"] = torch.empty_like(theta), theta
    return state


def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "batch":
        return run_batch(state)
    if kind in ("forward", "train"):
        return run_operator(state)
    s, f, out, L = state["solver"], state["fields"], state["out"], nat.lib()
    if kind == "cg":
        s.set_colour_gradient(state["more"]["red"], state["more"]["blue"], **state["more"]["prm"])
    else:
        s.set_state(f[0], f[1], f[2], f[3])
    if kind == "mhd":
        b = state["more"]["b"]
        s.set_magnetic(case["nu"], (b[0], b[1], b[2]))
    s.step(case["steps"])
    s.macroscopic(out[0], out[1], out[2], out[3])
    got = {"rho": out[0], "u": out[1:], "populations": state["store"]}
    if kind == "mhd":
        e = state["extra"]
        check(L.lbm_magnetic(s.handle, *(e[k].data_ptr() for k in range(6))), "lbm_magnetic")
        got["b"], got["j"] = e[:3], e[3:]
    elif kind == "cg":
        e = state["extra"]
        check(L.lbm_colour_densities(s.handle, e[0].data_ptr(), e[1].data_ptr()), "lbm_colour_densities")
        got["red"], got["blue"] = e[0], e[1]
    return got


def run_batch(state):
    L, h = nat.lib(), state["batch"].h
    for k, f in enumerate(state["fields"]):
        check(L.lbm_batch_set_state(h, k, *(f[j].data_ptr() for j in range(4))), "lbm_batch_set_state")
    check(L.lbm_batch_step(h, state["case"]["steps"]), "lbm_batch_step")
    for k, o in enumerate(state["outs"]):
        check(L.lbm_batch_macroscopic(h, k, *(o[j].data_ptr() for j in range(4))), "lbm_batch_macroscopic")
    return state["outs"]


def run_operator(state):
    L, h, case = nat.lib(), state["net"].h, state["case"]
    if case["kind"] == "forward":
        check(L.lbm_no_forward(h, case["batch"], state["a"].data_ptr(), state["out"].data_ptr()), "lbm_no_forward")
        return state["out"]
    loss = ctypes.c_double()
    check(L.lbm_no_train_step(h, case["batch"], state["a"].data_ptr(), state["t"].data_ptr(), 1e-4, ctypes.byref(loss)), "lbm_no_train_step")
    check(L.lbm_no_grads(h, state["grads"].data_ptr()), "lbm_no_grads")
    check(L.lbm_no_params(h, state["params"].data_ptr(), 0), "lbm_no_params")
    return {"grads": state["grads"], "params": state["params"]}


# ------------------------------------------------------------------------------------- in 64 bits
# Populations are (3, 3, 3, nz, ny, nx) by velocity (cx, cy, cz) + 1, or by moment order.
VEL = ([(0, 0, 0), (1, 0, 0), (-1, 0, 0), (0, 1, 0), (0, -1, 0), (0, 0, 1), (0, 0, -1)]
       + [(a, b, 0) for b in (1, -1) for a in (1, -1)] + [(a, 0, c) for c in (1, -1) for a in (1, -1)]
       + [(0, b, c) for c in (1, -1) for b in (1, -1)] + [(a, b, c) for c in (1, -1) for b in (1, -1) for a in (1, -1)])


def weight(c):
    return math.prod((1 / 6, 2 / 3, 1 / 6)[k + 1] for k in c)


def at(P, c):
    return P[c[0] + 1, c[1] + 1, c[2] + 1]


def raw_moments(P):
    K = P.clone()
    for axis in range(3):
        m, o, p = (K.select(axis, j).clone() for j in range(3))
        K.select(axis, 0).copy_(m + o + p)
        K.select(axis, 1).copy_(p - m)
        K.select(axis, 2).copy_(p + m)
    return K


def shift(K, u):
    """Raw moments to moments about u, in place."""
    for axis in range(3):
        k0, k1, k2 = (K.select(axis, j) for j in range(3))
        k2.copy_(k2 - 2 * u[axis] * k1 + u[axis] ** 2 * k0)
        k1.copy_(k1 - u[axis] * k0)
    return K


def populations(K, u):
    """Central moments back to populations, in place."""
    for axis in range(3):
        k0, k1, k2 = (K.select(axis, j) for j in range(3))
        m2 = k2 + 2 * u[axis] * k1 + u[axis] ** 2 * k0
        m1 = k1 + u[axis] * k0
        m0 = k0.clone()
        k0.copy_((m2 - m1) / 2)
        k1.copy_(m0 - m2)
        k2.copy_((m2 + m1) / 2)
    return K


def equilibrium(rho, u):
    s = (1, 0, 1 / 3)
    K = torch.stack([torch.stack([torch.stack([rho * (s[a] * s[b] * s[c]) for c in range(3)]) for b in range(3)]) for a in range(3)])
    return populations(K, u)


def collide(P, F, omega, extra=None):
    """The post-collision populations; F: 3 fields or numbers; extra(rho, u): populations added to the equilibrium."""
    K = raw_moments(P)
    rho = K[0, 0, 0].clone()
    u = [(K[1, 0, 0] + F[0] / 2) / rho, (K[0, 1, 0] + F[1] / 2) / rho, (K[0, 0, 1] + F[2] / 2) / rho]
    shift(K, u)
    zero = torch.zeros_like(rho)
    E = None if extra is None else shift(raw_moments(extra(rho, u)), u)
    k7, k8 = K[2, 0, 0] - K[0, 2, 0], K[2, 0, 0] - K[0, 0, 2]
    off = [K[1, 1, 0] * (1 - omega), K[1, 0, 1] * (1 - omega), K[0, 1, 1] * (1 - omega)]
    k7, k8, k9 = k7 * (1 - omega), k8 * (1 - omega), rho.clone()
    if E is not None:
        off = [o + omega * e for o, e in zip(off, (E[1, 1, 0], E[1, 0, 1], E[0, 1, 1]))]
        k7 = k7 + omega * (E[2, 0, 0] - E[0, 2, 0])
        k8 = k8 + omega * (E[2, 0, 0] - E[0, 0, 2])
        k9 = k9 + E[2, 0, 0] + E[0, 2, 0] + E[0, 0, 2]
    K.zero_()
    K[0, 0, 0] = rho
    K[2, 2, 0] = K[2, 0, 2] = K[0, 2, 2] = rho / 9
    K[2, 2, 2] = rho / 27
    for axis in range(3):
        b = [0, 0, 0]
        b[axis] = 1
        h = zero + F[axis]
        K[tuple(b)] = h / 2
        for o in range(3):
            if o != axis:
                c = list(b)
                c[o] = 2
                K[tuple(c)] = h / 6
        K[tuple(1 if k == axis else 2 for k in range(3))] = h / 18
    if E is not None:
        K += E
    K[1, 1, 0], K[1, 0, 1], K[0, 1, 1] = off
    K[2, 0, 0], K[0, 2, 0], K[0, 0, 2] = (k9 + k7 + k8) / 3, (k9 - 2 * k7 + k8) / 3, (k9 + k7 - 2 * k8) / 3
    return populations(K, u)


def blocked_links(mask, walls, shape):
    """{c: where the node x - c is solid or behind a y wall}; None where all is periodic."""
    if mask is None and not walls:
        return None
    out = {}
    for c in VEL:
        b = torch.zeros(shape, dtype=torch.bool, device=DEV) if mask is None else torch.roll(mask, (c[2], c[1], c[0]), (0, 1, 2)).clone()
        if walls and c[1] == 1:
            b[:, 0] = True
        if walls and c[1] == -1:
            b[:, -1] = True
        out[c] = b
    return out


def stream_all(P, blocked):
    out = torch.empty_like(P)
    for c in VEL:
        v = torch.roll(at(P, c), (c[2], c[1], c[0]), (0, 1, 2))
        if blocked is not None:
            v = torch.where(blocked[c], at(P, tuple(-k for k in c)), v)
        at(out, c).copy_(v)
    return out


def stencil(X, blocked):
    """sum_i w_i c_i X(x + c_i); behind a wall, X(x)."""
    g = [torch.zeros_like(X) for _ in range(3)]
    for c in VEL[1:]:
        v = torch.roll(X, (-c[2], -c[1], -c[0]), (0, 1, 2))
        if blocked is not None:
            v = torch.where(blocked[tuple(-k for k in c)], X, v)
        for axis in range(3):
            if c[axis]:
                g[axis] += c[axis] * weight(c) * v
    return g


def deviations(P, solid=None):
    out = torch.stack([at(P, c) - weight(c) for c in VEL])
    if solid is not None:
        out[:, solid] = 0.0
    return out


def fields_of(P, F, solid=None):
    K = raw_moments(P)
    rho = K[0, 0, 0]
    u = torch.stack([(k + f / 2) / rho for k, f in zip((K[1, 0, 0], K[0, 1, 0], K[0, 0, 1]), F)])
    if solid is not None:
        rho, u = torch.where(solid, 1.0, rho), torch.where(solid, 0.0, u)
    return rho, u


def exact(case, seed):
    kind = case["kind"]
    with torch.no_grad():
        if kind == "batch":
            return exact_batch(case, seed)
        if kind in ("forward", "train"):
            return exact_operator(case, seed)
        if nodes(case) > 4e7:
            return None  # the FP64 state and its temporaries take too long
        return {"mhd": exact_mhd, "cg": exact_cg}.get(kind, exact_flow)(case, seed)


def exact_flow(case, seed):
    f, more = flow_inputs(case, seed)
    f = f.double()
    ny = case["ny"]
    walls = case["kind"] == "porous"
    solid = more["mask"].bool() if "mask" in more else None
    blocked = blocked_links(solid, walls, f.shape[1:])
    omega = 1 / (3 * case["nu"] + 0.5)
    kind, prm = more.get("force", ("none", ()))

    def force(P):
        if kind == "uniform":
            return prm
        if kind == "kolmogorov":
            return (prm[0] * torch.sin(2 * math.pi * torch.arange(ny, device=DEV, dtype=torch.float64) / ny)[None, :, None], 0.0, 0.0)
        if kind == "shan_chen":
            psi = 1 - torch.exp(-P.sum((0, 1, 2)))
            return [-prm[0] * psi * g for g in stencil(psi, None)]
        return (0.0, 0.0, 0.0)

    rho, u = f[0], [f[1], f[2], f[3]]
    if solid is not None:
        rho, u = torch.where(solid, 1.0, rho), [torch.where(solid, 0.0, v) for v in u]
    P = equilibrium(rho, u)
    for _ in range(case["steps"]):
        P = stream_all(collide(P, force(P), omega), blocked)
        if solid is not None:
            P[..., solid] = torch.tensor([weight((a, b, c)) for a in (-1, 0, 1) for b in (-1, 0, 1) for c in (-1, 0, 1)],
                                         device=DEV, dtype=torch.float64).view(3, 3, 3, 1)
    rho, u = fields_of(P, force(P), solid)
    return {"rho": rho, "u": u, "populations": deviations(P, solid)}


def exact_batch(case, seed):
    out = []
    for d in batch_domains(case, seed):
        mask, f = batch_inputs(d)
        f = f.double()
        solid = mask.bool()
        blocked = blocked_links(solid, True, f.shape[1:])
        omega, F = 1 / (3 * d["nu"] + 0.5), (d["fx"], 0.0, 0.0)
        P = equilibrium(torch.where(solid, 1.0, f[0]), [torch.where(solid, 0.0, f[k]) for k in (1, 2, 3)])
        for _ in range(case["steps"]):
            P = stream_all(collide(P, F, omega), blocked)
            P[..., solid] = 1 / 27
        rho, u = fields_of(P, F, solid)
        out.append(torch.cat([rho[None], u]))
    return out


def cross(a, b):
    return [a[1] * b[2] - a[2] * b[1], a[2] * b[0] - a[0] * b[2], a[0] * b[1] - a[1] * b[0]]


def exact_mhd(case, seed):
    """D3Q7 vector populations h[velocity][component], coupled to the fluid by j x b."""
    f, more = flow_inputs(case, seed)
    f, b = f.double(), more["b"].double()
    omega, om = 1 / (3 * case["nu"] + 0.5), 1 / (4 * case["nu"] + 0.5)
    kappa = 4 * om
    seven = VEL[:7]

    def h_eq(b, u):
        out = []
        for c in seven:
            w = 0.25 if c == (0, 0, 0) else 0.125
            uc, bc = sum(k * v for k, v in zip(c, u)), sum(k * v for k, v in zip(c, b))
            out.append(torch.stack([w * (b[a] + 4 * (uc * b[a] - bc * u[a])) for a in range(3)]))
        return torch.stack(out)

    def node(P, h):
        K = raw_moments(P)
        rho, m = K[0, 0, 0], [K[1, 0, 0], K[0, 1, 0], K[0, 0, 1]]
        b = h.sum(0)
        lam = [h[1] - h[2], h[3] - h[4], h[5] - h[6]]  # by axis of the velocity, then component
        E = [lam[1][2] - lam[2][1], lam[2][0] - lam[0][2], lam[0][1] - lam[1][0]]
        s = [m[a] - 0.5 * kappa * e for a, e in enumerate(cross(E, b))]
        bb = (b * b).sum(0)
        sb = torch.where(bb > 0, (s[0] * b[0] + s[1] * b[1] + s[2] * b[2]) / bb.clamp_min(1e-300), 0.0)
        u = [sb * b[a] / rho + (s[a] - sb * b[a]) / (rho + kappa * bb) for a in range(3)]
        j = [-kappa * (E[a] - 2 * v) for a, v in enumerate(cross(u, b))]
        return rho, u, b, j, cross(j, b)

    u = [f[1], f[2], f[3]]
    P, h = equilibrium(f[0], u), h_eq(b, u)
    for _ in range(case["steps"]):
        rho, u, b, j, F = node(P, h)
        h = h + om * (h_eq(b, u) - h)
        h = torch.stack([torch.roll(h[k], (c[2], c[1], c[0]), (1, 2, 3)) for k, c in enumerate(seven)])
        P = stream_all(collide(P, F, omega), None)
    rho, u, b, j, F = node(P, h)
    return {"rho": rho, "u": torch.stack(u), "populations": deviations(P), "b": b, "j": torch.stack(j)}


def exact_cg(case, seed):
    """Red and blue populations with the enhanced equilibrium, the surface tension and the recolouring."""
    _, more = flow_inputs(case, seed)
    rr, rb, q = more["red"].double(), more["blue"].double(), more["prm"]
    blocked = blocked_links(None, True, rr.shape)
    ab = 8 / 27
    ar = 1 - (1 - ab) * q["rho_b0"] / q["rho_r0"]
    shell = [sum(k * k for k in c) for c in VEL]

    def phi_w(s, alpha):
        return alpha if s == 0 else (1 - alpha) * (2 / 19, 1 / 38, 1 / 152)[s - 1]

    def order(rr, rb):
        a, b = rr / q["rho_r0"], rb / q["rho_b0"]
        return (a - b) / (a + b)

    def alpha_of(phi):
        return 0.5 * (1 + phi) * ar + 0.5 * (1 - phi) * ab

    alpha = alpha_of(order(rr, rb))
    R, B = (torch.empty((3, 3, 3) + tuple(rr.shape), device=DEV, dtype=torch.float64) for _ in range(2))
    for c, s in zip(VEL, shell):
        at(R, c).copy_(rr * phi_w(s, alpha))
        at(B, c).copy_(rb * phi_w(s, alpha))

    def force(rho):
        return [(rho - 0.5 * (q["rho_r0"] + q["rho_b0"])) * g for g in q["g"]]

    for _ in range(case["steps"]):
        rr, rb = R.sum((0, 1, 2)), B.sum((0, 1, 2))
        rho, phi = rr + rb, order(rr, rb)
        gp, gr = ([3 * g for g in stencil(X, blocked)] for X in (phi, rho))
        alpha = alpha_of(phi)
        nu = 1 / (0.5 * (1 + phi) / q["nu_r"] + 0.5 * (1 - phi) / q["nu_b"])

        def extra(rho, u):
            D = torch.empty_like(R)
            ug = sum(a * b for a, b in zip(u, gr))
            for c, s in zip(VEL, shell):
                cu, cg = (sum(k * v for k, v in zip(c, w)) for w in (u, gr))
                Phi = -3 * nu * ug if s == 0 else (16.0, 4.0, 1.0)[s - 1] * nu * cu * cg / 24
                at(D, c).copy_(rho * (phi_w(s, alpha) - weight(c)) + Phi)
            return D

        P = collide(R + B, force(rho), 1 / (3 * nu + 0.5), extra)
        g2 = sum(g * g for g in gp)
        there = g2 > 0
        gn = g2.sqrt()
        safe2, safe = torch.where(there, g2, 1.0), torch.where(there, gn, 1.0)
        R, B = torch.empty_like(P), torch.empty_like(P)
        for c, s in zip(VEL, shell):
            cg = sum(k * v for k, v in zip(c, gp)) if s else torch.zeros_like(g2)
            bi = (-10 / 27, 2 / 27, 1 / 54, 1 / 216)[s]
            tension = torch.where(there, 0.5 * q["A"] * gn * (weight(c) * cg * cg / safe2 - bi), 0.0)
            fs = at(P, c) + tension
            cos = torch.where(there, cg / (safe * math.sqrt(max(s, 1))), 0.0)
            r = rr / rho * fs + q["beta"] * rr * rb / rho * cos * phi_w(s, alpha)
            at(R, c).copy_(r)
            at(B, c).copy_(fs - r)
        R, B = stream_all(R, blocked), stream_all(B, blocked)
    rr, rb = R.sum((0, 1, 2)), B.sum((0, 1, 2))
    rho, u = fields_of(R + B, force(rr + rb))
    return {"rho": rho, "u": u, "populations": torch.stack([at(R, c) for c in VEL]), "red": rr, "blue": rb}


def exact_operator(case, seed):
    theta, a, t = operator_inputs(case, seed)
    theta, a, t = theta.double(), a.double(), t.double()
    D, m = case["D"], case["modes"]
    kept = torch.tensor(list(range(m)) + list(range(D - m, D)), device=DEV)
    train = case["kind"] == "train"
    with torch.enable_grad():
        theta.requires_grad_(train)
        par, off = {}, 0
        for name, shape in operator_shapes(case):
            n = math.prod(shape)
            par[name] = theta[off:off + n].view(shape)
            off += n

        def dense(W, h, b):
            return torch.einsum("oc,bczyx->bozyx", W, h) + b[None, :, None, None, None]

        h = dense(par["P"], a, par["p"])
        for k in range(4):
            X = torch.fft.rfftn(h, dim=(2, 3, 4))[:, :, kept][:, :, :, kept][..., :m]
            W = torch.complex(par["Wm%d" % k][..., 0].contiguous(), par["Wm%d" % k][..., 1].contiguous())
            Y = torch.einsum("xyzoc,bczyx->bozyx", W, X)
            full = torch.zeros(h.shape[:4] + (D // 2 + 1,), dtype=Y.dtype, device=DEV)
            zz, yy = torch.meshgrid(kept, kept, indexing="ij")
            full = full.index_put((torch.arange(h.shape[0], device=DEV)[:, None, None, None, None],
                                   torch.arange(32, device=DEV)[None, :, None, None, None], zz[None, None, :, :, None],
                                   yy[None, None, :, :, None], torch.arange(m, device=DEV)[None, None, None, None, :]), Y)
            z = torch.fft.irfftn(full, s=(D, D, D), dim=(2, 3, 4)) + dense(par["Wc%d" % k], h, par["b%d" % k])
            h = torch.nn.functional.gelu(z) if k < 3 else z
        out = dense(par["Q"], h, par["q"])
        if not train:
            return out
        g, = torch.autograd.grad(((out - t) ** 2).mean(), theta)
    # Adam's first step moves every parameter by the rate in the direction of its gradient's sign: where a
    # gradient is below its own rounding there is no value for it in 64 bits
    return {"grads": g, "params": None}
