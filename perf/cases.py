"""The work a user of this library has it do, as cases that can be timed and compared.

A case is one pass of one of three programs, written with the public entry points:

  step     advance a flow by a block of time steps, then take the density and velocity
           fields on the device (how a simulation runs between two outputs);
  report   the invariants and the fields of a state that is in hand (monitoring);
  adjoint  an outlet-flux loss and its gradients with respect to the per-node force and
           the relaxation time (one iteration of an optimisation).

The flows are the ones the library is used on: the plane channel, random sphere packs,
the vessel tree, the lid-driven cavity and the inlet/outlet duct, with the storage formats
FP64, FP32 and FP16 and the collision models. ``exact`` is the same flow in plain FP64
torch on compact node lists (one gather index per node and direction), without the library.
"""
import math
import types

import numpy as np
import torch
import torch.utils.checkpoint

from paper_1611_02445_gb300 import inputs, lbm
from paper_1611_02445_gb300.autograd import outlet_flux_loss

# D3Q19 in the library's direction numbering: velocities, opposites, weights.
C = np.array([(0, 0, 0), (1, 0, 0), (0, 1, 0), (-1, 0, 0), (0, -1, 0), (0, 0, 1), (0, 0, -1),
              (1, 1, 0), (-1, 1, 0), (-1, -1, 0), (1, -1, 0), (1, 0, 1), (1, 0, -1), (-1, 0, 1),
              (-1, 0, -1), (0, 1, 1), (0, 1, -1), (0, -1, 1), (0, -1, -1)])
OPP = [int(np.flatnonzero((C == -c).all(axis=1))[0]) for c in C]
W = np.array([1 / 3] + [1 / 18] * 6 + [1 / 36] * 12)
VALUE_BYTES = {"f64": 8, "f32": 4, "f16s": 2}
LID_FACE = 5   # z = nz


def _step(name, flow, nx, ny, nz, dtype, steps, eq=0, coll=0):
    return {"name": name, "kind": "step", "flow": flow, "nx": nx, "ny": ny, "nz": nz, "dtype": dtype,
            "steps": steps, "eq": eq, "coll": coll}


def listed():
    return [
        # the smallest call: a 32^3 plane channel (walls y = 0 and ny - 1, periodic x and z),
        # as used to validate a set-up; one step fills less than the GPU
        _step("channel_32_f64", "channel", 32, 32, 32, "f64", 50),
        # a small ragged channel section with Zou-He velocity inlet and pressure outlet, the
        # boundary scheme of the method; no axis is a multiple of the tile
        _step("duct_ragged_f64", "duct", 126, 61, 67, "f64", 50),
        # porous medium at full size in each storage format: the headline workload
        _step("pack_256_f64", "pack", 256, 256, 256, "f64", 20),
        _step("pack_256_f32", "pack", 256, 256, 256, "f32", 20),
        _step("pack_256_f16s", "pack", 256, 256, 256, "f16s", 20),
        # sparse vessel tree in a large box: few tiles kept, inlet and outlet nodes inside
        _step("tree_1024_f32", "tree", 1024, 512, 512, "f32", 60),
        # dense lid-driven cavity, incompressible LBGK, ragged size: full tiles, moving wall
        _step("cavity_190_incompr_f64", "cavity", 190, 190, 190, "f64", 20, eq=lbm.EQ_INCOMPR),
        # the MRT collision, in FP64 on a porous medium and in FP32 on a cavity
        _step("pack_128_mrt_f64", "pack", 128, 128, 128, "f64", 20, coll=lbm.COLL_MRT),
        _step("cavity_128_mrt_f32", "cavity", 128, 128, 128, "f32", 30, coll=lbm.COLL_MRT),
        # the adjoint on the 128^3 pack in FP32 storage, and a smaller one in FP64
        {"name": "adjoint_128_f32", "kind": "adjoint", "n": 128, "dtype": "f32", "steps": 200, "every": 50},
        {"name": "adjoint_80_f64", "kind": "adjoint", "n": 80, "dtype": "f64", "steps": 60, "every": 20},
        # monitoring a state: total mass and momentum, and both fields
        {"name": "report_160_f64", "kind": "report", "n": 160, "dtype": "f64"},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["step"] * 7 + ["adjoint"] * 2 + ["report"])
    if kind == "adjoint":
        n = 4 * _log_int(rng, 6, 32)
        steps = _log_int(rng, 20, 200)
        dtype = rng.choice(["f64", "f32"])
        if dtype == "f64":
            n = min(n, 96)
            steps = min(steps, 60)
        return {"kind": "adjoint", "n": n, "dtype": dtype, "steps": steps, "every": rng.randint(5, 60)}
    if kind == "report":
        return {"kind": "report", "n": 4 * _log_int(rng, 6, 40), "dtype": rng.choice(["f64", "f32", "f16s"])}
    flow = rng.choice(["channel", "duct", "pack", "pack", "pack", "tree", "cavity", "cavity"])
    dtype = rng.choice(["f64", "f64", "f32", "f32", "f16s"])
    steps = rng.randint(5, 60)
    eq = coll = 0
    if flow == "tree":
        nx = 8 * _log_int(rng, 20, 96)
        ny, nz = nx // 2 + rng.randint(-9, 9), nx // 2 + rng.randint(-9, 9)
    else:
        side = _log_int(rng, 24, 224)
        nx, ny, nz = (max(16, int(side * rng.uniform(0.7, 1.3))) for _ in range(3))
        if flow in ("channel", "pack"):   # usually periodic, which takes whole tiles
            nx, ny, nz = (d if rng.random() < 0.3 else d // 4 * 4 for d in (nx, ny, nz))
        if flow in ("pack", "cavity") and rng.random() < 0.4:
            eq, coll = rng.choice([(lbm.EQ_INCOMPR, lbm.COLL_BGK), (lbm.EQ_QCOMPR, lbm.COLL_MRT)])
        if nx * ny * nz > 6_000_000:
            steps = min(steps, 20)
        if coll and dtype == "f64":
            steps = min(steps, 15)
    return {"kind": "step", "flow": flow, "nx": nx, "ny": ny, "nz": nz, "dtype": dtype, "steps": steps,
            "eq": eq, "coll": coll}


# ------------------------------------------------------------------------- geometry
def _device():
    return torch.device("cuda" if torch.cuda.is_available() else "cpu")


def _sphere_pack(nx, ny, nz, porosity, seed, radius=8.0):
    """Overlapping solid spheres with uniform random centres in a periodic box, as many as
    give the porosity on average."""
    dev = _device()
    gen = torch.Generator().manual_seed(seed)
    count = max(1, round(-math.log(porosity) * nx * ny * nz / (4.0 / 3.0 * math.pi * radius ** 3)))
    dims = torch.tensor([nx, ny, nz], dtype=torch.float64)
    centres = (torch.rand(count, 3, generator=gen, dtype=torch.float64) * dims).to(dev)
    ext = math.ceil(radius) + 1
    o = torch.arange(-ext, ext + 1, device=dev)
    off = torch.stack(torch.meshgrid(o, o, o, indexing="ij"), -1).reshape(-1, 3)
    nt = torch.full((nz * ny * nx,), lbm.FLUID, dtype=torch.uint8, device=dev)
    for c in centres.split(256):
        node = torch.floor(c).long()[:, None, :] + off[None]
        inside = ((node - c[:, None, :]) ** 2).sum(-1) <= radius * radius
        x, y, z = node[inside].unbind(-1)
        nt[x % nx + nx * (y % ny + ny * (z % nz))] = lbm.SOLID
    return nt.reshape(nz, ny, nx)


def _flow(case, seed):
    """Node types, periodic mask and parameters of a step case's flow."""
    nx, ny, nz = case["nx"], case["ny"], case["nz"]
    rng = np.random.default_rng(seed)
    p = types.SimpleNamespace(periodic=0, tau=0.7, g=(0.0, 0.0, 0.0), u_in=None, rho_out=1.0, lid=None,
                              zou_he=False, rho0=1.0, u0=(0.0, 0.0, 0.0))
    vary = rng.uniform(0.8, 1.2)
    whole = [not d % 4 for d in (nx, ny, nz)]   # only such axes can be periodic
    if case["flow"] == "channel":
        nt = torch.from_numpy(inputs.poiseuille_channel(nx, ny, nz)).to(_device())
        p.periodic = (1 if whole[0] else 0) | (4 if whole[2] else 0)
        p.tau, p.g, p.u0 = 0.8, (1e-6 * vary, 0.0, 0.0), (1e-4 * vary, 0.0, 0.0)
    elif case["flow"] == "pack":
        nt = _sphere_pack(nx, ny, nz, 0.35, seed)
        p.periodic = sum(1 << a for a in range(3) if whole[a])
        p.g = (1e-5 * vary, 0.0, 0.0)
    elif case["flow"] == "tree":
        nt = torch.from_numpy(inputs.vessel_tree(nx, ny, nz, seed=seed, root_radius=24.0 * nx / 1024)).to(_device())
        p.tau, p.u_in = 0.6, (0.05 * vary, 0.0, 0.0)
    elif case["flow"] == "cavity":
        nt = torch.full((nz, ny, nx), lbm.FLUID, dtype=torch.uint8, device=_device())
        p.tau, p.lid = 0.6, (0.05 * vary, 0.01 * (vary - 1.0), 0.0)
    else:   # duct along x: walls y = 0 and ny - 1, inlet x = 0, outlet x = nx - 1
        nt = torch.full((nz, ny, nx), lbm.FLUID, dtype=torch.uint8, device=_device())
        nt[:, :, 0], nt[:, :, -1] = lbm.INLET, lbm.OUTLET
        nt[:, 0, :] = nt[:, -1, :] = lbm.SOLID
        p.tau, p.u_in, p.zou_he = 0.8, (0.04 * vary, 0.0, 0.0), True
        p.u0 = p.u_in
    return nt, p


def _force(n, seed, dtype):
    """Per-node x force of an adjoint case: 1e-5 plus noise of 1e-7."""
    gen = torch.Generator().manual_seed(seed + 1)
    g = 1e-5 + 1e-7 * torch.randn(n, n, n, generator=gen, dtype=torch.float64)
    return g.to(dtype)


def _tau(seed, dtype):
    return torch.tensor(0.8 + 0.01 * (seed % 7), dtype=dtype)


def _populations(nt, seed):
    """Random populations near the weights (a state in motion), dense [19, nz, ny, nx]."""
    gen = torch.Generator(device=nt.device).manual_seed(seed + 2)
    r = torch.rand((19,) + tuple(nt.shape), generator=gen, device=nt.device, dtype=torch.float64)
    return torch.from_numpy(W).to(nt.device)[:, None, None, None] * (1.0 + 0.05 * (2.0 * r - 1.0))


# ----------------------------------------------------------------------- a user's program
def prepare(case, seed):
    s = types.SimpleNamespace(kind=case["kind"], case=case)
    if case["kind"] == "adjoint":
        n = case["n"]
        s.lattice = lbm.Lattice(_sphere_pack(n, n, n, 0.4, seed), case["dtype"], 7)
        # the program's own parameters, in the precision of its storage
        dtype = torch.float64 if case["dtype"] == "f64" else torch.float32
        s.force = _force(n, seed, dtype).cuda().requires_grad_()
        s.tau = _tau(seed, dtype).requires_grad_()
        return s
    out = torch.float64 if case["dtype"] == "f64" else torch.float32
    s.out_f64 = case["dtype"] == "f64"
    if case["kind"] == "report":
        n = case["n"]
        nt = _sphere_pack(n, n, n, 0.35, seed)
        s.lattice = lbm.Lattice(nt, case["dtype"], 7)
        s.lattice.set_params(0.7, (1e-5, 0.0, 0.0))
        s.lattice.set_f(_populations(nt, seed).cpu().numpy())
    else:
        nt, p = _flow(case, seed)
        s.lattice = lbm.Lattice(nt, case["dtype"], p.periodic)
        s.lattice.set_params(p.tau, p.g, None, p.u_in, p.rho_out)
        if case["eq"] or case["coll"]:
            s.lattice.set_model(case["eq"], case["coll"])
        if p.lid:
            s.lattice.set_lid(LID_FACE, p.lid)
        if p.zou_he:
            s.lattice.set_bc(lbm.BC_ZOU_HE, 0, 1)
        s.lattice.init_equilibrium(p.rho0, p.u0)
    s.rho = torch.empty(tuple(nt.shape), dtype=out, device="cuda")
    s.u = torch.empty((3,) + tuple(nt.shape), dtype=out, device="cuda")
    return s


def run(s):
    if s.kind == "adjoint":
        s.force.grad = s.tau.grad = None
        loss = outlet_flux_loss(s.force.double(), s.tau.double(), s.lattice, s.case["steps"], s.case["n"] - 1,
                                s.case["every"])
        loss.backward()
        return {"loss": loss.detach().to(s.force.dtype), "force_grad": s.force.grad, "tau_grad": s.tau.grad}
    if s.kind == "step":
        s.lattice.step(s.case["steps"])
        lbm.lbm_macroscopic(s.lattice.ctx, s.rho, s.u, s.out_f64)
        return {"rho": s.rho, "u": s.u}
    mass, momentum = s.lattice.reduce()
    lbm.lbm_macroscopic(s.lattice.ctx, s.rho, s.u, s.out_f64)
    return {"mass": mass, "momentum": momentum, "rho": s.rho, "u": s.u}


def _nodes(case):
    """Non-solid nodes, from the sizes alone (packs at their porosity, trees at the usual
    share of their box)."""
    if case["kind"] != "step":
        return (0.4 if case["kind"] == "adjoint" else 0.35) * case["n"] ** 3
    box = case["nx"] * case["ny"] * case["nz"]
    if case["flow"] == "pack":
        return 0.35 * box
    if case["flow"] == "tree":
        return 0.0064 * box
    if case["flow"] in ("channel", "duct"):
        return box * (case["ny"] - 2) / case["ny"]
    return float(box)


def work(case):
    n, b = _nodes(case), VALUE_BYTES[case["dtype"]]
    if case["kind"] == "adjoint":
        # a step reads and writes the populations once; a reverse step reads a state and
        # the adjoint and writes the adjoint (in the arithmetic precision) and the gradient
        a = 8 if case["dtype"] == "f64" else 4
        per_step = 2 * 38 * b + 19 * b + 38 * a + 16
        return {"bytes": n * case["steps"] * per_step, "flops": n * case["steps"] * (2 * 250 + 350)}
    out = 8 if case["dtype"] == "f64" else 4
    if case["kind"] == "report":
        return {"bytes": 2 * n * 19 * b + 4 * out * case["n"] ** 3, "flops": 2 * n * 60}
    box = case["nx"] * case["ny"] * case["nz"]
    per_node = 250 if not case["coll"] else 500
    return {"bytes": n * case["steps"] * 38 * b + n * 19 * b + 4 * out * box,
            "flops": n * (case["steps"] * per_node + 60)}


# ------------------------------------------------------- the same in plain FP64 torch
class _Plain:
    """Compact node lists of a geometry: for every direction the node a population is
    pulled from, or -1 for a bounced link."""

    def __init__(self, nt, periodic):
        self.shape = tuple(nt.shape)
        self.on = (nt != lbm.SOLID).reshape(-1).nonzero().squeeze(1)
        self.type = nt.reshape(-1)[self.on]
        ids = torch.full((nt.numel(),), -1, dtype=torch.long, device=nt.device)
        ids[self.on] = torch.arange(self.on.numel(), device=nt.device)
        ids = ids.reshape(self.shape)
        self.src = []
        for c in C:
            r = torch.roll(ids, tuple(int(v) for v in c[::-1]), (0, 1, 2))
            for a in range(3):
                if c[a] and not (periodic >> a) & 1:
                    r.select(2 - a, 0 if c[a] > 0 else -1).fill_(-1)   # r is a copy: c has a shift
            self.src.append(r.reshape(-1)[self.on].clone())
        nx, ny = self.shape[2], self.shape[1]
        self.x, self.z = self.on % nx, self.on // (nx * ny)
        self.bounce = [v < 0 for v in self.src]
        self.src = [v.clamp_min(0) for v in self.src]

    def pull(self, f):
        return [torch.where(self.bounce[i], f[OPP[i]], f[i][self.src[i]]) for i in range(19)]

    def dense(self, v):
        out = torch.zeros(math.prod(self.shape), dtype=v.dtype, device=v.device)
        out[self.on] = v
        return out.reshape(self.shape)


def _dot(c, v):
    """c . v for a lattice velocity c and three components (tensors or numbers)."""
    out = 0.0
    for a in range(3):
        if c[a]:
            out = out + (v[a] if c[a] > 0 else -v[a])
    return out


def _moments(f):
    return sum(f), [sum((f[i] if C[i][a] > 0 else -f[i]) for i in range(19) if C[i][a]) for a in range(3)]


def _equilibrium(rho, u, incompressible):
    a = 1.0 if incompressible else rho
    uu = 1.5 * sum(v * v for v in u)
    out = []
    for i in range(19):
        cu = _dot(C[i], u)
        out.append(W[i] * (rho + a * (3.0 * cu + 4.5 * cu * cu - uu)))
    return out


def _guo(u, F):
    uF = sum(a * b for a, b in zip(u, F))
    return [W[i] * (3.0 * (_dot(C[i], F) - uF) + 9.0 * _dot(C[i], u) * _dot(C[i], F)) for i in range(19)]


def _mrt(tau):
    """D3Q19 moment basis (d'Humieres et al. 2002) and its relaxation rates."""
    x, y, z = C.T.astype(float)
    cc = x * x + y * y + z * z
    pxx, pww = 3 * x * x - cc, y * y - z * z
    m = np.array([x * 0 + 1, 19 * cc - 30, (21 * cc * cc - 53 * cc + 24) / 2, x, (5 * cc - 9) * x, y,
                  (5 * cc - 9) * y, z, (5 * cc - 9) * z, pxx, (3 * cc - 5) * pxx, pww, (3 * cc - 5) * pww,
                  x * y, y * z, x * z, (y * y - z * z) * x, (z * z - x * x) * y, (x * x - y * y) * z])
    v = 1.0 / tau
    s = np.array([1, 1.19, 1.4, 1, 1.2, 1, 1.2, 1, 1.2, v, 1.4, v, 1.4, v, v, v, 1.98, 1.98, 1.98])
    return m, s


def _zou_he(v, nodes, inward, u, rho_out, incompressible):
    """Completes the populations of boundary nodes on an x face (inward normal +1 or -1)
    with velocity u, or with density rho_out and no tangential velocity if u is None."""
    w = [t[nodes] for t in v]
    normal = [int(c[0]) * inward for c in C]
    b = sum(w[i] * (1 if normal[i] == 0 else 2) for i in range(19) if normal[i] <= 0)
    if u is not None:
        un = u[0] * inward
        scale = 1.0 if incompressible else b / (1.0 - un)
        j = [scale * t + 0.0 * b for t in u]
    else:
        j = [(rho_out - b) * inward, 0.0 * b, 0.0 * b]
    jn = j[0] * inward
    for i in range(19):
        if normal[i] <= 0:
            continue
        side = [a for a in (1, 2) if C[i][a]]
        val = w[OPP[i]] + jn / 3.0
        if side:
            a, t = side[0], int(C[i][side[0]])
            tangential = sum(w[k] * int(C[k][a]) for k in range(19) if normal[k] == 0 and C[k][a])
            val = w[OPP[i]] + (jn + t * j[a]) / 6.0 - t * (0.5 * tangential - j[a] / 3.0)
        v[i] = v[i].index_put((nodes,), val)


def _collide(v, tau, F, incompressible=False, mrt=None):
    rho, j = _moments(v)
    u = [a + 0.5 * b for a, b in zip(j, F)]
    if not incompressible:
        u = [a / rho for a in u]
    eq, G = _equilibrium(rho, u, incompressible), _guo(u, F)
    if mrt is None:
        return [v[i] + (eq[i] - v[i]) / tau + (1.0 - 0.5 / tau) * G[i] for i in range(19)]
    m, s = mrt
    norm = (m * m).sum(1)
    out = [t.clone() for t in eq]
    for k in range(19):
        neq = sum(m[k, i] * (v[i] - eq[i]) for i in range(19) if m[k, i])
        src = sum(m[k, i] * G[i] for i in range(19) if m[k, i])
        r = ((1.0 - s[k]) * neq + (1.0 - 0.5 * s[k]) * src) / norm[k]
        for i in range(19):
            if m[k, i]:
                out[i] = out[i] + m[k, i] * r
    return out


def _fields(plain, f, F, incompressible=False):
    rho, j = _moments(f)
    u = [a - 0.5 * b for a, b in zip(j, F)]
    if not incompressible:
        u = [a / rho for a in u]
    return plain.dense(rho), torch.stack([plain.dense(t) for t in u])


def _exact_step(case, seed):
    nt, p = _flow(case, seed)
    plain = _Plain(nt, p.periodic)
    inc, one = case["eq"] == lbm.EQ_INCOMPR, torch.ones(plain.on.numel(), dtype=torch.float64, device=nt.device)
    f = _equilibrium(p.rho0 * one, [t * one for t in p.u0], inc)
    mrt = _mrt(p.tau) if case["coll"] == lbm.COLL_MRT else None
    inlet = (plain.type == lbm.INLET).nonzero().squeeze(1)
    outlet = (plain.type == lbm.OUTLET).nonzero().squeeze(1)
    lid = plain.z == plain.shape[0] - 1
    for _ in range(case["steps"]):
        v = plain.pull(f)
        if p.lid:
            for i in range(19):
                if C[i][2] < 0:   # the link crosses the top face
                    v[i] = v[i] + (lid & plain.bounce[i]).double() * (6.0 * W[i] * _dot(C[i], p.lid))
        if p.zou_he:
            _zou_he(v, inlet, 1, p.u_in, None, inc)
            _zou_he(v, outlet, -1, None, p.rho_out, inc)
        f = _collide(v, p.tau, p.g, inc, mrt)
        if p.u_in and not p.zou_he:
            for nodes, rho_out in ((inlet, None), (outlet, p.rho_out)):
                w = [t[nodes] for t in v]
                rho, j = _moments(w)
                u = [t + 0.0 * rho for t in p.u_in] if rho_out is None else [t / rho for t in j]
                eq = _equilibrium(rho if rho_out is None else rho_out + 0.0 * rho, u, inc)
                for i in range(19):
                    f[i][nodes] = eq[i]
    rho, u = _fields(plain, f, p.g, inc)
    return {"rho": rho, "u": u}


def _exact_report(case, seed):
    n, F = case["n"], (1e-5, 0.0, 0.0)
    nt = _sphere_pack(n, n, n, 0.35, seed)
    plain = _Plain(nt, 7)
    f = [t.reshape(-1)[plain.on] for t in _populations(nt, seed)]
    rho, u = _fields(plain, f, F)
    momentum = (u * rho).sum((1, 2, 3))
    return {"mass": rho.sum(), "momentum": momentum.cpu().numpy(), "rho": rho, "u": u}


def _exact_adjoint(case, seed):
    n, T = case["n"], case["steps"]
    dtype = torch.float64 if case["dtype"] == "f64" else torch.float32
    nt = _sphere_pack(n, n, n, 0.4, seed)
    plain = _Plain(nt, 7)
    force = _force(n, seed, dtype).to(nt.device, torch.float64).reshape(-1)[plain.on].requires_grad_()
    tau = _tau(seed, dtype).to(nt.device, torch.float64).requires_grad_()
    zero = torch.zeros_like(force)
    f = _equilibrium(zero + 1.0, [zero] * 3, False)

    def advance(force, tau, *f):
        return tuple(_collide(plain.pull(f), tau, (force, 0.0, 0.0)))

    for _ in range(T):
        f = torch.utils.checkpoint.checkpoint(advance, force, tau, *f, use_reentrant=False)
    rho, j = _moments(f)
    loss = ((j[0] - 0.5 * force) / rho)[plain.x == n - 1].mean()
    loss.backward()
    return {"loss": loss.detach(), "force_grad": plain.dense(force.grad), "tau_grad": tau.grad}


def exact(case, seed):
    if case["kind"] == "adjoint":
        return _exact_adjoint(case, seed)
    return _exact_report(case, seed) if case["kind"] == "report" else _exact_step(case, seed)
