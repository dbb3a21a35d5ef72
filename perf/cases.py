"""The work that users of this library have it do, as cases to be timed.

A case is a dict of plain values; `prepare` makes what a program holds before
the call (handle, device arrays, network), `run` is one pass through the
public entry points, `work` the bytes and operations the pass cannot do
without, `exact` its outputs in 64 bits by plain torch.  The kinds of work
("op"):

  kv        one operator application y = K(E) v, the call a user's own Krylov
            method makes, FP64 and FP32;
  kv_multi  the same for several load cases at once;
  design    a SIMP iteration without its solve: filter, modulus, compliance
            and sensitivities, filter transpose, OC update (a program that
            brings its own solver calls exactly these);
  vcycle    one multigrid V-cycle as a preconditioner;
  unet      the network's forward pass on a node grid (the learned initial
            guess and correction);
  unet_grad its loss and parameter gradient (training);
  simp      a whole SIMP iteration with the mixed-precision solver;
  gmg       a whole solve with multigrid, its hierarchy set up for the new
            moduli as every SIMP iteration needs it;
  batch     many uneven small designs solved together.

Meshes are those of the named workloads (24x12x12, 120x60x30, 55x55x165,
256x128x150, 100x50x50 with eight loads, 64 uneven instances) and the
network's training grids; `draw` spreads over the ranges between them.
The three whole solves run to a relative residual of 1e-10, so that their
displacements are determined by the inputs to well below 1e-9: at the usual
1e-8 two equally correct solvers differ by more than FP64 outputs are compared
to.  Iteration counts are no outputs for the same reason.
"""
from __future__ import annotations

import math

import numpy as np
import torch
import torch.nn.functional as F

from paper_2604_18020_gb300 import learned, mfto, workloads as W

DEV = "cuda"
LEVELS = 4          # levels of the network
BASE = 14           # its channels on the finest grid
KV_ITERS_PER_LENGTH = 10   # Jacobi-CG iterations per element of the longest axis, roughly

# elements of the largest mesh that draw() gives each kind of work
MOST = {"kv": 4_915_200, "kv_multi": 300_000, "design": 4_915_200, "vcycle": 1_000_000,
        "unet": 264 * 136 * 152, "unet_grad": 136 * 72 * 72, "simp": 250_000, "gmg": 600_000,
        "batch": 64}


def listed():
    return [
        # the smallest call: the unit-test cantilever, where latency counts
        {"name": "kv_f64_24x12x12", "op": "kv", "form": "f64", "problem": "cantilever",
         "nx": 24, "ny": 12, "nz": 12},
        # FP64 operator on the torsion bar (odd sizes): plain PCG and every
        # refinement residual apply it
        {"name": "kv_f64_55x55x165", "op": "kv", "form": "f64", "problem": "torsion",
         "nx": 55, "ny": 55, "nz": 165},
        # FP32 operator on the largest mesh
        {"name": "kv_f32_256x128x150", "op": "kv", "form": "f32", "problem": "cantilever",
         "nx": 256, "ny": 128, "nz": 150},
        # eight load cases at once
        {"name": "kv_multi_f32_100x50x50", "op": "kv_multi", "form": "f32",
         "problem": "cantilever", "nx": 100, "ny": 50, "nz": 50, "nrhs": 8},
        # the design update of the benchmark mesh, and of the largest mesh
        {"name": "design_120x60x30", "op": "design", "nx": 120, "ny": 60, "nz": 30,
         "rmin": 1.5, "penal": 3.0, "volfrac": 0.3},
        {"name": "design_256x128x150", "op": "design", "nx": 256, "ny": 128, "nz": 150,
         "rmin": 1.5, "penal": 3.0, "volfrac": 0.12},
        # the preconditioner on the benchmark mesh
        {"name": "vcycle_120x60x30", "op": "vcycle", "problem": "cantilever",
         "nx": 120, "ny": 60, "nz": 30},
        # the network on the larger of its training meshes, and its gradient
        # on the smaller one
        {"name": "unet_128x64x64", "op": "unet", "nx": 128, "ny": 64, "nz": 64},
        {"name": "unet_grad_64x32x32", "op": "unet_grad", "nx": 64, "ny": 32, "nz": 32},
        # whole calls: the benchmark's SIMP iteration, a multigrid solve of the
        # torsion bar, 64 uneven designs in one batch
        {"name": "simp_mixed_120x60x30", "op": "simp", "problem": "cantilever",
         "nx": 120, "ny": 60, "nz": 30},
        {"name": "gmg_solve_55x55x165", "op": "gmg", "problem": "torsion",
         "nx": 55, "ny": 55, "nz": 165},
        {"name": "batch_solve_64", "op": "batch", "count": 64, "kmin": 8, "kmax": 24,
         "instances": 5},
    ]


def _mesh_sizes(rng, lo, hi):
    """nx, ny, nz with about exp(U(log lo, log hi)) elements (at most hi) and
    aspect ratios between a cube and 4:1:1, in either orientation; sizes fall
    on odd values as often as on even ones."""
    n = math.exp(rng.uniform(math.log(lo), math.log(hi)))
    ax, ay = math.exp(rng.uniform(0.0, math.log(4.0))), math.exp(rng.uniform(0.0, math.log(2.0)))
    s = (n / (ax * ay)) ** (1.0 / 3.0)
    dims = [max(4, round(s * ax)), max(4, round(s * ay)), max(4, round(s))]
    if rng.random() < 0.3:
        dims.reverse()
    while dims[0] * dims[1] * dims[2] > hi:
        dims[dims.index(max(dims))] -= 1
    return dict(zip(("nx", "ny", "nz"), dims))


def draw(rng):
    op = rng.choice(["kv", "kv", "kv_multi", "design", "design", "vcycle", "unet", "unet_grad",
                     "simp", "gmg", "batch"])
    if op == "kv":
        return {"op": op, "form": rng.choice(["f64", "f32"]),
                "problem": rng.choice(["cantilever", "torsion"]),
                **_mesh_sizes(rng, 3_456, MOST[op])}
    if op == "kv_multi":
        return {"op": op, "form": rng.choice(["f64", "f32", "f32"]), "problem": "cantilever",
                "nrhs": rng.randint(2, 8), **_mesh_sizes(rng, 3_456, MOST[op])}
    if op == "design":
        return {"op": op, "rmin": rng.choice([1.35, 1.5, 1.5, 2.0]),
                "penal": rng.choice([1.5, 3.0, 3.0, 3.5, 4.5]),
                "volfrac": rng.choice([0.12, 0.2, 0.3]), **_mesh_sizes(rng, 3_456, MOST[op])}
    if op == "vcycle":
        return {"op": op, "problem": rng.choice(["cantilever", "torsion"]),
                **_mesh_sizes(rng, 3_456, MOST[op])}
    if op in ("unet", "unet_grad"):
        return {"op": op, **_mesh_sizes(rng, 8_000, MOST[op] // 3)}
    if op == "simp":
        return {"op": op, "problem": rng.choice(["cantilever", "torsion"]),
                **_mesh_sizes(rng, 3_456, MOST[op])}
    if op == "gmg":
        return {"op": op, "problem": rng.choice(["cantilever", "torsion"]),
                **_mesh_sizes(rng, 20_000, MOST[op])}
    return {"op": op, "count": rng.randint(8, MOST[op]), "kmin": rng.randint(4, 10),
            "kmax": rng.randint(12, 24), "instances": rng.randrange(1000)}


# ------------------------------------------------------------------ inputs

def _problem(case):
    make = W.torsion if case.get("problem") == "torsion" else W.cantilever
    return make(case["nx"], case["ny"], case["nz"])


def _gen(seed):
    return torch.Generator(device=DEV).manual_seed(seed)


def _uniform(n, g, lo=-1.0, hi=1.0):
    return torch.rand(n, dtype=torch.float64, device=DEV, generator=g) * (hi - lo) + lo


def _smooth(nx, ny, nz, g):
    """A smooth random field in [0, 1], [nz, ny, nx]."""
    x = torch.rand((1, 1, nz, ny, nx), dtype=torch.float64, device=DEV, generator=g)
    k = 5 if min(nx, ny, nz) >= 8 else 3
    for _ in range(2):
        x = F.avg_pool3d(F.pad(x, (k // 2,) * 6, mode="replicate"), k, 1)
    x = x[0, 0]
    return (x - x.amin()) / (x.amax() - x.amin()).clamp_min(1e-12)


def _design(nx, ny, nz, g):
    """Densities like a SIMP iterate on its way: solid flanges along the
    beam's top and bottom, a web of graded and nearly void regions between."""
    rho = (1.6 * _smooth(nx, ny, nz, g) - 0.3).clamp(0.02, 1.0)
    t = max(1, ny // 8)
    rho[:, :t, :] = rho[:, :t, :].clamp_min(0.9)
    rho[:, ny - t:, :] = rho[:, ny - t:, :].clamp_min(0.9)
    return rho.reshape(-1).contiguous()


def _modulus(rho, penal=3.0):
    return 1e-9 + (1.0 - 1e-9) * rho ** penal


def _bending(nx, ny, nz, g):
    """A displacement field of the shape a loaded cantilever takes, with
    rough variation of a few percent of an element's strain."""
    z, y, x = torch.meshgrid(*(torch.arange(n + 1, dtype=torch.float64, device=DEV)
                               for n in (nz, ny, nx)), indexing="ij")
    t = x / nx
    uy = -(nx / 10.0) * t * t * (3.0 - t)
    ux = (nx / 10.0) * (y - ny / 2) * (6.0 * t - 3.0 * t * t) / nx
    uz = 0.02 * (z - nz / 2) * (1.0 - t)
    u = torch.stack([ux, uy, uz], dim=-1)
    u += 0.05 * _uniform(u.numel(), g).reshape(u.shape)
    u[:, :, 0, :] = 0.0
    return u.reshape(-1).contiguous()


def _network_input(dims, case, g):
    """Density and load channels as the library feeds them: a design on the
    real nodes, a residual scaled to its largest entry, zero padding."""
    D, H, Wd = dims
    nx, ny, nz = case["nx"], case["ny"], case["nz"]
    x = torch.zeros((4, D, H, Wd), dtype=torch.float64, device=DEV)
    x[0, :nz + 1, :ny + 1, :nx + 1] = (1.6 * _smooth(nx + 1, ny + 1, nz + 1, g)
                                       - 0.3).clamp(0.02, 1.0)
    for c in range(3):
        r = torch.randn((nz + 1, ny + 1, nx + 1), dtype=torch.float64, device=DEV, generator=g)
        x[1 + c, :nz + 1, :ny + 1, :nx + 1] = r / r.abs().max()
    return x.float().contiguous()


def prepare(case, seed):
    g = _gen(seed)
    op = case["op"]
    if op in ("unet", "unet_grad"):
        dims = mfto.nn_grid(case["nx"], case["ny"], case["nz"], LEVELS)
        vox = dims[0] * dims[1] * dims[2]
        net = learned.load(max_voxels=vox, max_train_voxels=vox if op == "unet_grad" else 0)
        s = {"case": case, "net": net, "dims": dims, "x": _network_input(dims, case, g)}
        if op == "unet":
            s["out"] = torch.empty((3,) + dims, dtype=torch.float32, device=DEV)
        else:
            s["target"] = torch.stack([_smooth(dims[2], dims[1], dims[0], g)
                                       for _ in range(3)]).float().contiguous()
            mask = torch.zeros((3,) + dims, dtype=torch.float32, device=DEV)
            mask[:, :case["nz"] + 1, :case["ny"] + 1, 1:case["nx"] + 1] = 1.0
            s["mask"] = mask
        return s
    if op == "batch":
        problems = W.uneven_instances(case["count"], case["instances"], case["kmin"],
                                      case["kmax"])
        meshes = [(p.mesh.nelx, p.mesh.nely, p.mesh.nelz) for p in problems]
        b = mfto.Batch(meshes, [p.fixed for p in problems],
                       mfto.default_params(rtol=1e-10))
        b.set_ir_mode(mfto.IR_CONTINUE)
        rho = [_design(*m, g) for m in meshes]
        return {"case": case, "b": b, "E": _modulus(torch.cat(rho)),
                "F": torch.tensor(np.concatenate([p.f for p in problems]), device=DEV),
                "U": torch.zeros(b.n_dof, dtype=torch.float64, device=DEV)}
    if op == "design":
        nx, ny, nz = case["nx"], case["ny"], case["nz"]
        p = W.cantilever(nx, ny, nz)
        h = mfto.Handle(nx, ny, nz, p.fixed,
                        mfto.default_params(volfrac=case["volfrac"], rmin=case["rmin"],
                                            penal=case["penal"]))
        rho = _design(nx, ny, nz, g)
        s = {"case": case, "h": h, "rho": rho, "u": _bending(nx, ny, nz, g)}
        for k in ("rho_phys", "E", "dc_phys", "dc", "rho_new"):
            s[k] = torch.empty_like(rho)
        return s
    p = _problem(case)
    m = p.mesh
    if op in ("kv", "kv_multi"):
        nrhs = case.get("nrhs", 1)
        dt = torch.float64 if case["form"] == "f64" else torch.float32
        h = mfto.Handle(m.nelx, m.nely, m.nelz, p.fixed, mfto.default_params(max_rhs=nrhs))
        if op == "kv" and case["form"] == "f32":
            h.kv_autotune()
        v = _uniform(nrhs * m.n_dof, g).to(dt)
        return {"case": case, "h": h, "form": mfto.FORMS[case["form"]], "fixed": p.fixed,
                "E": _uniform(m.n_elem, g, 0.01, 1.0).to(dt), "v": v, "y": torch.empty_like(v)}
    rho = _design(m.nelx, m.nely, m.nelz, g)
    f = torch.tensor(p.f, device=DEV)
    if op == "simp":
        h = mfto.Handle(m.nelx, m.nely, m.nelz, p.fixed,
                        mfto.default_params(volfrac=p.volfrac, rmin=p.rmin, rtol=1e-10))
        h.set_solver(mfto.FORM_F32, 0.1)
        h.set_ir_mode(mfto.IR_CONTINUE)
        h.kv_autotune()
        return {"case": case, "h": h, "rho0": rho, "rho": rho.clone(), "f": f,
                "u": torch.zeros(m.n_dof, dtype=torch.float64, device=DEV),
                "rho_phys": torch.empty_like(rho)}
    h = mfto.Handle(m.nelx, m.nely, m.nelz, p.fixed, mfto.default_params(rtol=1e-10))
    h.kv_autotune()
    s = {"case": case, "h": h, "E": _modulus(rho)}
    if op == "vcycle":
        h.gmg_setup(s["E"])
        r = _uniform(m.n_dof, g)
        r[torch.tensor(W.fixed_dofs(p.fixed), device=DEV)] = 0.0
        return {**s, "r": r.float(), "z": torch.empty(m.n_dof, dtype=torch.float32, device=DEV)}
    return {**s, "f": f, "u": torch.zeros(m.n_dof, dtype=torch.float64, device=DEV)}


def run(s):
    case = s["case"]
    op = case["op"]
    if op == "kv":
        s["h"].kv(s["E"], s["v"], s["y"], form=s["form"])
        return s["y"]
    if op == "kv_multi":
        s["h"].kv_multi(s["E"], s["v"], s["y"], case["nrhs"], form=s["form"])
        return s["y"]
    if op == "design":
        h = s["h"]
        h.filter(s["rho"], s["rho_phys"])
        h.simp_modulus(s["rho_phys"], s["E"])
        c = h.compliance_sens(s["rho_phys"], s["u"], s["dc_phys"])
        h.filter(s["dc_phys"], s["dc"], transpose=True)
        st = h.oc_update(s["rho"], s["dc"], s["rho_new"])
        return {"rho_phys": s["rho_phys"], "E": s["E"], "dc_phys": s["dc_phys"], "dc": s["dc"],
                "rho_new": s["rho_new"], "compliance": c, "volume": st.volume,
                "change": st.change, "lambda": st.lambda_}
    if op == "vcycle":
        s["h"].gmg_vcycle(s["r"], s["z"])
        return s["z"]
    if op == "unet":
        s["net"].forward(s["x"], s["out"], s["dims"])
        return s["out"]
    if op == "unet_grad":
        loss, grad = s["net"].gradient(s["x"], s["target"], s["mask"], s["dims"])
        return {"loss": loss, "grad": grad}
    if op == "simp":
        s["rho"].copy_(s["rho0"])     # every pass starts from the same design
        s["u"].zero_()
        st = s["h"].simp_step(s["rho"], s["u"], s["f"], s["rho_phys"])
        return {"rho": s["rho"], "u": s["u"], "rho_phys": s["rho_phys"],
                "compliance": st.compliance, "volume": st.volume, "grayness": st.grayness}
    if op == "gmg":
        s["u"].zero_()
        s["h"].gmg_setup(s["E"])
        s["h"].gmg_solve(s["E"], s["f"], s["u"])
        return s["u"]
    s["U"].zero_()
    s["b"].solve(s["E"], s["F"], s["U"], inner_tol=0.1)
    return s["U"]


# -------------------------------------------------------------------- work

def _counts(case):
    nx, ny, nz = case["nx"], case["ny"], case["nz"]
    n = nx * ny * nz
    nodes = (nx + 1) * (ny + 1) * (nz + 1)
    return n, nodes, 3 * nodes


def _network_flops(vox):
    flops = 0.0
    for _, ci, co, k, level in _layers():
        flops += 2.0 * vox / 8 ** level * k ** 3 * ci * co
    return flops


def work(case):
    """Bytes: inputs once, outputs once.  Operations: 1,152 per element and
    application of the operator (the dense 24 x 24 element product); solves
    count the operator applications of Jacobi-CG or V-cycle CG at these sizes,
    roughly."""
    op = case["op"]
    if op in ("unet", "unet_grad"):
        D, H, Wd = mfto.nn_grid(case["nx"], case["ny"], case["nz"], LEVELS)
        vox = D * H * Wd
        params = 4.0 * 1_118_785
        if op == "unet":
            return {"bytes": 4.0 * 7 * vox + params / 2, "flops": _network_flops(vox)}
        return {"bytes": 4.0 * 10 * vox + 1.5 * params, "flops": 3 * _network_flops(vox)}
    if op == "batch":
        n = dofs = flops = 0.0
        for p in W.uneven_instances(case["count"], case["instances"], case["kmin"],
                                    case["kmax"]):
            n += p.mesh.n_elem
            dofs += p.mesh.n_dof
            flops += 1152.0 * p.mesh.n_elem * KV_ITERS_PER_LENGTH * p.mesh.nelx
        return {"bytes": 8.0 * (n + 2 * dofs), "flops": flops}
    n, nodes, dofs = _counts(case)
    if op in ("kv", "kv_multi"):
        size = 8.0 if case["form"] == "f64" else 4.0
        nrhs = case.get("nrhs", 1)
        return {"bytes": size * (n + 2 * dofs * nrhs) + nodes, "flops": 1152.0 * n * nrhs}
    if op == "design":
        # rho, u in; five element fields out; two filters, the element
        # energies and one volume evaluation
        terms = len(mfto.filter_stencil(case["rmin"])[1])
        return {"bytes": 8.0 * (6 * n + dofs), "flops": n * (4.0 * terms + 1152.0 + 8.0)}
    if op == "vcycle":
        return {"bytes": 4.0 * (n + 3 * dofs) + nodes, "flops": 6 * 1152.0 * n}
    length = max(case["nx"], case["ny"], case["nz"])
    if op == "simp":
        return {"bytes": 8.0 * (3 * n + 2 * dofs),
                "flops": 1152.0 * n * KV_ITERS_PER_LENGTH * length}
    return {"bytes": 8.0 * (n + 2 * dofs), "flops": 1152.0 * n * 7 * 40}


# ------------------------------------------------------------------- exact

def _corners():
    return [(l & 1, (l >> 1) & 1, l >> 2) for l in range(8)]


def _unit_stiffness(nu=0.3):
    """24 x 24 stiffness of the unit trilinear hexahedron (2 x 2 x 2 Gauss
    points), local DOF 3 (a + 2 b + 4 c) + component."""
    lam, mu = nu / ((1 + nu) * (1 - 2 * nu)), 1 / (2 * (1 + nu))
    Dm = np.diag([2 * mu] * 3 + [mu] * 3)
    Dm[:3, :3] += lam
    K = np.zeros((24, 24))
    pts = (0.5 - 0.5 / math.sqrt(3.0), 0.5 + 0.5 / math.sqrt(3.0))
    for p in ((x, y, z) for x in pts for y in pts for z in pts):
        B = np.zeros((6, 24))
        for l, corner in enumerate(_corners()):
            shape = [t if a else 1 - t for a, t in zip(corner, p)]
            slope = [1.0 if a else -1.0 for a in corner]
            d = [slope[0] * shape[1] * shape[2], shape[0] * slope[1] * shape[2],
                 shape[0] * shape[1] * slope[2]]
            for c in range(3):
                B[c, 3 * l + c] = d[c]
            for row, (i, j) in ((3, (0, 1)), (4, (1, 2)), (5, (2, 0))):
                B[row, 3 * l + i], B[row, 3 * l + j] = d[j], d[i]
        K += B.T @ Dm @ B / 8
    return K


def _at(corner, v, nz, ny, nx):
    a, b, c = corner
    return v[c:c + nz, b:b + ny, a:a + nx]


def _exact_kv(E, v, fixed, nx, ny, nz):
    K = torch.tensor(_unit_stiffness(), device=DEV)
    fd = torch.tensor(W.fixed_dofs(fixed), device=DEV)
    E4 = E.double().reshape(nz, ny, nx, 1)
    pv = torch.where(fd, 0.0, v.double()).reshape(nz + 1, ny + 1, nx + 1, 3)
    y = torch.zeros_like(pv)
    for l, cl in enumerate(_corners()):
        acc = 0.0
        for m, cm in enumerate(_corners()):
            acc = acc + _at(cm, pv, nz, ny, nx) @ K[3 * l:3 * l + 3, 3 * m:3 * m + 3].T
        _at(cl, y, nz, ny, nx).add_(E4 * acc)
    return torch.where(fd, v.double(), y.reshape(-1))


def _exact_filter(x, rmin):
    """Unnormalised cone filter of a [nz, ny, nx] field."""
    R = math.ceil(rmin) - 1
    nz, ny, nx = x.shape
    xp = F.pad(x, (R,) * 6)
    y = torch.zeros_like(x)
    for dz in range(-R, R + 1):
        for dy in range(-R, R + 1):
            for dx in range(-R, R + 1):
                w = rmin - math.sqrt(dx * dx + dy * dy + dz * dz)
                if w > 0:
                    y += w * xp[R + dz:R + dz + nz, R + dy:R + dy + ny, R + dx:R + dx + nx]
    return y


def _exact_design(s):
    case = s["case"]
    nx, ny, nz, p = case["nx"], case["ny"], case["nz"], case["penal"]
    n = nx * ny * nz
    rho = s["rho"].reshape(nz, ny, nx)
    W1 = _exact_filter(torch.ones_like(rho), case["rmin"])
    rho_phys = _exact_filter(rho, case["rmin"]) / W1
    E = _modulus(rho_phys, p)
    K = torch.tensor(_unit_stiffness(), device=DEV)
    u = s["u"].reshape(nz + 1, ny + 1, nx + 1, 3)
    ce = torch.zeros_like(rho)
    for l, cl in enumerate(_corners()):
        acc = 0.0
        for m, cm in enumerate(_corners()):
            acc = acc + _at(cm, u, nz, ny, nx) @ K[3 * l:3 * l + 3, 3 * m:3 * m + 3].T
        ce += (_at(cl, u, nz, ny, nx) * acc).sum(-1)
    dc_phys = -p * rho_phys ** (p - 1) * (1.0 - 1e-9) * ce
    dc = _exact_filter(dc_phys / W1, case["rmin"])
    lo, hi = (rho - 0.2).clamp_min(0.0), (rho + 0.2).clamp_max(1.0)
    a = rho * ((-dc).clamp_min(0.0) * n).sqrt()
    l1, l2, new = 0.0, 1e9, rho
    while (l2 - l1) / (l1 + l2) > 1e-10:
        lam = 0.5 * (l1 + l2)
        new = torch.maximum(lo, torch.minimum(hi, a / math.sqrt(lam)))
        if float(new.sum()) > case["volfrac"] * n:
            l1 = lam
        else:
            l2 = lam
    return {"rho_phys": rho_phys.reshape(-1), "E": E.reshape(-1), "dc_phys": dc_phys.reshape(-1),
            "dc": dc.reshape(-1), "rho_new": new.reshape(-1), "compliance": float((E * ce).sum()),
            "volume": float(new.mean()), "change": float((new - rho).abs().max()),
            "lambda": 0.5 * (l1 + l2)}


def _layers():
    """(name, c_in, c_out, kernel, level) of every convolution, in order."""
    ch = [BASE * 2 ** l for l in range(LEVELS)]
    out, prev = [], 4
    for l in range(LEVELS):
        out += [(f"e{l}a", prev, ch[l], 3, l), (f"e{l}b", ch[l], ch[l], 3, l)]
        prev = ch[l]
    for l in range(LEVELS - 2, -1, -1):
        out += [(f"d{l}a", prev + ch[l], ch[l], 3, l), (f"d{l}b", ch[l], ch[l], 3, l)]
        prev = ch[l]
    return out + [("out", ch[0], 3, 1, 0)]


def _exact_network(s, gradient):
    """Forward pass (and loss and gradient) with the weights rounded to BF16,
    as the network defines them."""
    flat = torch.tensor(s["net"].get_params(), device=DEV).bfloat16().double()
    flat.requires_grad_(gradient)
    at, par = 0, {}
    for name, ci, co, k, _ in _layers():
        nw = co * ci * k ** 3
        par[name] = (flat[at:at + nw].reshape(co, ci, k, k, k), flat[at + nw:at + nw + co])
        at += nw + co

    def conv(name, x):
        w, b = par[name]
        return F.conv3d(x, w, b, padding=w.shape[-1] // 2)

    def block(name, x):
        return F.relu(conv(name + "b", F.relu(conv(name + "a", x))))

    x, skips = s["x"].double()[None], []
    for l in range(LEVELS - 1):
        x = block(f"e{l}", x)
        skips.append(x)
        x = F.avg_pool3d(x, 2)
    x = block(f"e{LEVELS - 1}", x)
    for l in range(LEVELS - 2, -1, -1):
        x = block(f"d{l}", torch.cat([F.interpolate(x, scale_factor=2, mode="nearest"),
                                      skips[l]], 1))
    out = conv("out", x)[0]
    if not gradient:
        return out
    loss = (((out - s["target"].double()) * s["mask"].double()) ** 2).sum() / s["mask"].sum()
    loss.backward()
    return {"loss": float(loss), "grad": flat.grad}


def exact(case, seed):
    """None for a V-cycle and the whole solves (no closed form, or minutes of
    work in plain torch) and for networks on grids of over a million voxels."""
    op = case["op"]
    if op in ("vcycle", "simp", "gmg", "batch"):
        return None
    if op in ("unet", "unet_grad"):
        dims = mfto.nn_grid(case["nx"], case["ny"], case["nz"], LEVELS)
        if dims[0] * dims[1] * dims[2] > 1_000_000:
            return None
    s = prepare(case, seed)
    if op in ("unet", "unet_grad"):
        return _exact_network(s, op == "unet_grad")
    if op == "design":
        return _exact_design(s)
    nrhs = case.get("nrhs", 1)
    return torch.cat([_exact_kv(s["E"], v, s["fixed"], case["nx"], case["ny"], case["nz"])
                      for v in s["v"].reshape(nrhs, -1)])
