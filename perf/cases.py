"""Measured cases: the matrix-free operators and solves of the melt-pool model as a program calls them.

Each case is one call through the public classes (Context, Mesh, DofMap, Operator, MeltPoolStep) on
inputs made on the GPU from a seed.  The ranges are those of the library's own workloads and
tests: uniform meshes from a few thousand cells up to 128^3, adaptive octrees with three levels, one
to eight right-hand sides, fp64, double-float and fp32 arithmetic, forward and adjoint.
"""
import math

import torch

from paper_2501_18781_gb300 import Context, DofMap, MeltPoolStep, Mesh, Operator

# Ti-6Al-4V (liquid / gas), SI units
RHO_L, RHO_G, MU_L, MU_G = 4087.0, 4.087, 3.5e-3, 3.5e-5
CP_L, CP_G, K_L, K_G = 1130.0, 11.3, 28.63, 0.02863
T_BOIL, H_V, MOLAR, P_AMB = 3133.0, 8.84e6, 4.78e-2, 101325.0
T_SOLIDUS, T_LIQUIDUS = 1933.0, 2200.0
BOX = 6e-4                       # edge of the laser box [m]
HEAT_DT, SPOT, T_BASE, T_REF = 1e-5, 50e-6, 500.0, 500.0
BOTTOM = 1 << 4                  # Dirichlet z-
WALLS = 0b011111                 # Dirichlet on every face but z+
MELT_FLAGS = 1 | 2 | 4           # three-phase properties, Darcy damping, trace-corrected stress
A_LIQUID, A_GAS = 1000.0, 1.0    # level-set coefficient of the Helmholtz operator


def listed():
    return [
        # the smallest call: one fp64 Helmholtz apply on 16^3 cells (latency and launches)
        {"name": "helmholtz_apply_16_f64", "op": "helmholtz", "call": "apply", "nx": 16, "ny": 16, "nz": 16,
         "arith": "f64", "nrhs": 1},
        # a whole small solve: Jacobi-CG with its iterations replayed as a CUDA graph
        {"name": "helmholtz_cg_16", "op": "helmholtz", "call": "cg", "nx": 16, "ny": 16, "nz": 16,
         "arith": "f64", "nrhs": 1},
        # the implicit heat step's operator at its largest size, fp64-accurate (outer residuals)
        {"name": "heat_apply_128_df64", "op": "heat", "call": "apply", "nx": 128, "ny": 128, "nz": 128,
         "arith": "df64", "nrhs": 1},
        # the same operator in fp32 (inner iterations, smoother) on an odd-sized box
        {"name": "heat_apply_125x97x111_f32", "op": "heat", "call": "apply", "nx": 125, "ny": 97, "nz": 111,
         "arith": "f32", "nrhs": 1},
        # the adjoint direction: transpose of the convective heat operator with a conductivity per Gauss point
        {"name": "adjoint_apply_64_df64", "op": "adjoint", "call": "apply", "nx": 64, "ny": 64, "nz": 64,
         "arith": "df64", "nrhs": 1},
        # velocity-pressure operator inside the flow preconditioner, with the melt-pool terms
        {"name": "meltpool_oseen_apply_64_f32", "op": "oseen", "call": "apply", "nx": 64, "ny": 64, "nz": 64,
         "arith": "f32", "melt": True, "nrhs": 1},
        # two-phase velocity-pressure operator, fp64-accurate (outer residuals of the flow solve)
        {"name": "oseen_apply_64_df64", "op": "oseen", "call": "apply", "nx": 64, "ny": 64, "nz": 64,
         "arith": "df64", "melt": False, "nrhs": 1},
        # the same on the fp64 pipes, odd and ragged box
        {"name": "oseen_apply_33x40x27_f64", "op": "oseen", "call": "apply", "nx": 33, "ny": 40, "nz": 27,
         "arith": "f64", "melt": False, "nrhs": 1},
        # level-set reinitialisation on an adaptive octree, eight right-hand sides in one call, fp32
        {"name": "reinit_octree_8rhs_f32", "op": "reinit", "call": "apply", "base": 20, "levels": 3, "shape": 1,
         "arith": "f32", "nrhs": 8},
        # the same operator fp64-accurate (outer residuals of the batched solve)
        {"name": "reinit_octree_8rhs_df64", "op": "reinit", "call": "apply", "base": 12, "levels": 3, "shape": 2,
         "arith": "df64", "nrhs": 8},
        # the mixed-precision heat solve: fp32 Chebyshev-CG inside, fp64-accurate outside
        {"name": "heat_solve_96_mixed", "op": "heat", "call": "mixed", "nx": 96, "ny": 96, "nz": 96,
         "arith": "df64", "nrhs": 1},
        # one step of the whole melt-pool algorithm (advection, reinitialisation, heat, flow)
        {"name": "meltpool_step_40", "op": "step", "call": "step", "nx": 40, "ny": 40, "nz": 40,
         "arith": "df64", "nrhs": 1},
    ]


def _size(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _box(rng, lo, hi):
    """Three extents in lo..hi, spread over their logarithm and at most a factor of two apart."""
    n = _size(rng, lo, hi)
    return {k: max(lo, min(hi, int(round(n * rng.uniform(0.7, 1.4))))) for k in ("nx", "ny", "nz")}


def draw(rng):
    kind = rng.choice(["helmholtz", "heat", "heat", "adjoint", "oseen", "oseen", "reinit", "reinit", "cg", "mixed", "step"])
    arith = rng.choice(["f64", "df64", "f32"])
    if kind == "helmholtz":
        return {"op": "helmholtz", "call": "apply", **_box(rng, 8, 48), "arith": arith, "nrhs": rng.choice([1, 1, 3])}
    if kind == "heat":
        return {"op": "heat", "call": "apply", **_box(rng, 16, 128), "arith": arith, "nrhs": 1}
    if kind == "adjoint":
        return {"op": "adjoint", "call": "apply", **_box(rng, 12, 64), "arith": arith, "nrhs": 1}
    if kind == "oseen":
        return {"op": "oseen", "call": "apply", **_box(rng, 10, 64), "arith": arith, "melt": rng.random() < 0.5, "nrhs": 1}
    if kind == "reinit":
        levels = rng.randint(1, 3)
        return {"op": "reinit", "call": "apply", "base": rng.randint(4, 12 if levels == 3 else 20), "levels": levels,
                "shape": rng.randint(3, 99), "arith": arith, "nrhs": rng.randint(1, 8)}
    if kind == "cg":
        return {"op": "helmholtz", "call": "cg", **_box(rng, 8, 24), "arith": "f64", "nrhs": 1}
    if kind == "mixed":
        return {"op": "heat", "call": "mixed", **_box(rng, 24, 96), "arith": "df64", "nrhs": 1}
    n = _size(rng, 12, 40)
    return {"op": "step", "call": "step", "nx": n, "ny": n, "nz": n, "arith": "df64", "nrhs": 1}


# ------------------------------------------------------------------------------ inputs

def _generator(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed) * 7919 + 17)
    return g


def _uniform(g, n, lo=-1.0, hi=1.0):
    return lo + (hi - lo) * torch.rand(n, generator=g, dtype=torch.float64, device="cuda")


def _span(case):
    """(cells per axis, cell edge, lower corner) of the uniform box: the longest edge is the unit cube's
    or, for the laser-driven operators, the 600 um box's."""
    n = (case["nx"], case["ny"], case["nz"])
    laser = case["op"] in ("heat", "adjoint", "step")
    h = (BOX if laser else 1.0) / max(n)
    return n, h, (-0.5 * BOX,) * 3 if laser else (0.0,) * 3


def _lattice(case):
    """Coordinates of the Q2 nodes in DoF order (x fastest) and the upper corner of the box."""
    n, h, lo = _span(case)
    ax = [lo[d] + 0.5 * h * torch.arange(2 * n[d] + 1, dtype=torch.float64, device="cuda") for d in range(3)]
    z, y, x = torch.meshgrid(ax[2], ax[1], ax[0], indexing="ij")
    return x.reshape(-1), y.reshape(-1), z.reshape(-1), [lo[d] + n[d] * h for d in range(3)]


def _dirichlet(case, faces):
    n, _, _ = _span(case)
    m = torch.zeros((2 * n[2] + 1, 2 * n[1] + 1, 2 * n[0] + 1), dtype=torch.bool, device="cuda")
    for bit, (axis, end) in enumerate(((2, 0), (2, -1), (1, 0), (1, -1), (0, 0), (0, -1))):
        if (faces >> bit) & 1:
            m.select(axis, end)[...] = True
    return m.reshape(-1)


def _convection(x, y, z, lo, hi, g):
    """Divergence-free velocity, tangential on every wall, largest magnitude one: the curl of a seeded
    trigonometric vector potential times the bubble of the box."""
    waves = ((1, 1, 1), (1, 2, 1), (2, 1, 1), (1, 1, 2))
    a = _uniform(g, 12).reshape(3, 4).tolist()
    t = _uniform(g, 12, 0.0, 2.0 * math.pi).reshape(3, 4).tolist()
    xi = [(v - lo[d]) / (hi[d] - lo[d]) for d, v in enumerate((x, y, z))]
    s, c = [torch.sin(math.pi * v) for v in xi], [torch.cos(math.pi * v) for v in xi]
    bub = s[0] * s[1] * s[2]
    db = [math.pi * c[0] * s[1] * s[2], math.pi * s[0] * c[1] * s[2], math.pi * s[0] * s[1] * c[2]]
    curl = {}
    for cc in range(3):
        pot = torch.zeros_like(x)
        dpot = [torch.zeros_like(x) for _ in range(3)]
        for m, k in enumerate(waves):
            arg = 2.0 * math.pi * (k[0] * xi[0] + k[1] * xi[1] + k[2] * xi[2]) + t[cc][m]
            pot += a[cc][m] * torch.sin(arg)
            co = a[cc][m] * 2.0 * math.pi * torch.cos(arg)
            for d in range(3):
                dpot[d] += k[d] * co
        for d in range(3):
            curl[cc, d] = bub * dpot[d] + pot * db[d]
    b = torch.stack([curl[2, 1] - curl[1, 2], curl[0, 2] - curl[2, 0], curl[1, 0] - curl[0, 1]])
    return b / b.square().sum(0).max().sqrt()


def _hot_spot(x, y, z, hi, g):
    """Absolute temperature under a laser spot near the centre of the top face."""
    dx, dy = _uniform(g, 2, -20e-6, 20e-6).tolist()
    x0, y0 = 0.5 * (hi[0] - 0.5 * BOX) + dx, 0.5 * (hi[1] - 0.5 * BOX) + dy
    r2 = (x - x0) ** 2 + (y - y0) ** 2 + (z - hi[2]) ** 2
    return T_BASE + 2633.0 * torch.exp(-2.0 * r2 / SPOT ** 2)


def _fields(case, seed):
    """The nodal fields of a uniform-mesh operator and, for applies, its source vectors (fp64)."""
    g = _generator(seed)
    n, h, lo = _span(case)
    x, y, z, hi = _lattice(case)
    nd = x.numel()
    op, f = case["op"], {}
    size = nd
    if op == "helmholtz":
        c = _uniform(g, 3, -0.05, 0.05).tolist()
        d = 0.3 * min(hi) - torch.sqrt(sum((v - 0.5 * hi[i] - c[i]) ** 2 for i, v in enumerate((x, y, z))))
        f["phi"] = torch.tanh(d / (4.0 * h))
    elif op == "heat":
        f["t_prev"] = _hot_spot(x, y, z, hi, g)
    elif op == "adjoint":
        f["t_prev"] = _hot_spot(x, y, z, hi, g)
        f["beta"] = _convection(x, y, z, lo, hi, g).reshape(-1)
        f["k_qpoint"] = K_L * (1.25 + 0.25 * _uniform(g, 27 * n[0] * n[1] * n[2]))
    else:
        t1, t2 = _uniform(g, 2, 0.0, 2.0 * math.pi).tolist()
        zs = 0.5 * hi[2] + 0.05 * torch.sin(2.0 * math.pi * x + t1) * torch.sin(2.0 * math.pi * y + t2)
        f["phi"] = torch.tanh((zs - z) / (4.0 * h))
        f["beta"] = _convection(x, y, z, lo, hi, g).reshape(-1)
        if case["melt"]:
            r2 = sum((v - 0.5 * hi[i]) ** 2 for i, v in enumerate((x, y, z)))
            f["t_prev"] = 1500.0 + 2100.0 * torch.exp(-2.0 * r2 / 0.2 ** 2)
        size = 3 * nd + (n[0] + 1) * (n[1] + 1) * (n[2] + 1)
    if case["call"] == "apply":
        # Krylov vectors: nothing in the rows of fixed values
        src = _uniform(g, case["nrhs"] * size)
        if op in ("heat", "adjoint"):
            src[_dirichlet(case, BOTTOM)] = 0.0
        elif op == "oseen":
            src[:3 * nd].reshape(3, nd)[:, _dirichlet(case, WALLS)] = 0.0
        f["src"] = src.float() if case["arith"] == "f32" else src
    elif case["call"] == "cg":
        f["b"] = _uniform(g, size)
    else:
        # load of the lumped heat content of theta = T - T_ref with 1 % noise, fixed bottom
        w = []
        for m in n:
            v = torch.full((2 * m + 1,), 2.0 / 3.0, dtype=torch.float64, device="cuda")
            v[0::2] = 1.0 / 3.0
            v[0] = v[-1] = 1.0 / 6.0
            w.append(v)
        mass = (h ** 3 * w[2][:, None, None] * w[1][None, :, None] * w[0][None, None, :]).reshape(-1)
        f["b"] = RHO_L * CP_L / HEAT_DT * mass * (f["t_prev"] - T_REF + 10.0 * _uniform(g, size))
        f["b"][_dirichlet(case, BOTTOM)] = 0.0
    return f


def _sphere_distance(g):
    """Pseudo-distance function to a sphere whose radius varies by up to 5 % with the direction."""
    k = _uniform(g, 18, -3.0, 3.0).reshape(6, 3).tolist()
    t, a = _uniform(g, 6, 0.0, 2.0 * math.pi).tolist(), _uniform(g, 6).tolist()
    norm = sum(abs(v) for v in a)

    def distance(x, y, z):
        dx, dy, dz = x - 0.5, y - 0.5, z - 0.5
        r = torch.sqrt(dx * dx + dy * dy + dz * dz).clamp_min(1e-300)
        s = sum(a[m] * torch.cos((k[m][0] * dx + k[m][1] * dy + k[m][2] * dz) / r + t[m]) for m in range(6))
        return 0.3 * (1.0 + 0.05 * s / norm) - r
    return distance


def _octree(case):
    """Band-refined, 2:1-balanced leaves around the case's deformed sphere: (levels on the finest grid
    [x, y, z], leaves as int32 rows, distance function)."""
    base, levels = case["base"], case["levels"]
    nf = base << levels
    eps = 2.0 / nf
    dist = _sphere_distance(_generator(case["shape"]))
    up = lambda v, s: v.repeat_interleave(s, 0).repeat_interleave(s, 1).repeat_interleave(s, 2)
    lev = torch.zeros((nf, nf, nf), dtype=torch.float32, device="cuda")
    for l in range(levels):
        s, n = 1 << (levels - l), base << l
        c = (torch.arange(n, dtype=torch.float64, device="cuda") + 0.5) / n
        X, Y, Z = torch.meshgrid(c, c, c, indexing="ij")
        mark = (lev[::s, ::s, ::s] == l) & (dist(X, Y, Z).abs() < 4.0 * eps + 0.5 * math.sqrt(3.0) / n)
        lev = torch.maximum(lev, up(mark.float() * (l + 1), s))
    pool = torch.nn.functional.max_pool3d
    while True:
        dil, changed = pool(lev[None], 3, 1, 1)[0], False
        for l in range(levels - 1):
            s = 1 << (levels - l)
            need = (lev[::s, ::s, ::s] == l) & (pool(dil[None], s, s)[0] >= l + 2)
            if bool(need.any()):
                lev, changed = torch.maximum(lev, up(need.float() * (l + 1), s)), True
        if not changed:
            break
    rows = []
    for l in range(levels + 1):
        s = 1 << (levels - l)
        ijk = (lev[::s, ::s, ::s] == l).nonzero()
        rows.append(torch.cat([torch.full_like(ijk[:, :1], l), ijk], 1))
    return lev.to(torch.int64), torch.cat(rows).to(torch.int32), dist


def _step_state(case, seed):
    """Two time levels of velocity, temperature and level set of a wavy melt surface under the laser."""
    g = _generator(seed)
    n, h, lo = _span(case)
    x, y, z, hi = _lattice(case)
    t1, t2 = _uniform(g, 2, 0.0, 2.0 * math.pi).tolist()
    xi, eta = (x - lo[0]) / (hi[0] - lo[0]), (y - lo[1]) / (hi[1] - lo[1])
    zs = lo[2] + (hi[2] - lo[2]) * (0.6 + 0.03 * torch.sin(2.0 * math.pi * xi + t1) * torch.sin(2.0 * math.pi * eta + t2))
    xc, yc = 0.5 * (lo[0] + hi[0]), 0.5 * (lo[1] + hi[1])
    r2 = (x - xc) ** 2 + (y - yc) ** 2 + (z - zs) ** 2
    T = T_BASE + 3100.0 * torch.exp(-2.0 * r2 / SPOT ** 2)
    u = _convection(x, y, z, lo, hi, g).reshape(-1)
    return dict(u=u, u_prev=0.9 * u, T=T, T_prev=T_BASE + 0.97 * (T - T_BASE),
                phi=torch.tanh((zs - z) / (4.0 * h)), phi_prev=torch.tanh((zs - z + 0.5 * h) / (4.0 * h)))


# ------------------------------------------------------------------------------ the call

def _oseen_params(case):
    _, h, _ = _span(case)
    sigma = 2.0 / h                  # time step of half a cell at unit speed
    p = dict(sigma=sigma, rho_l=RHO_L, rho_g=RHO_G, mu_l=MU_L, mu_g=MU_G, eps=2.0 * h)
    if case["melt"]:
        p.update(rho_s=RHO_L, mu_s=MU_L, t_solidus=T_SOLIDUS, t_liquidus=T_LIQUIDUS, darcy_c=1e4 * sigma, darcy_b=1.0,
                 oseen_flags=MELT_FLAGS)
    return p


def prepare(case, seed):
    ctx = Context(0)
    op_kind, call = case["op"], case["call"]
    if op_kind == "reinit":
        lev, leaves, dist = _octree(case)
        base, levels = case["base"], case["levels"]
        nf = base << levels
        dm = DofMap(Mesh.octree(ctx, base, levels, leaves.cpu().numpy()), 2, 0)
        phi = _octree_phi(case, _OctreeLattice(lev, case), dist, seed)
        op = Operator(ctx, "reinit", [dm], eps=2.0 / nf, dtau=0.5 / nf, coef_mode=1)
        op.set_field("phi", phi)
        src = _uniform(_generator(seed), case["nrhs"] * phi.numel())
        f = {"src": src.float() if case["arith"] == "f32" else src}
    else:
        n, h, lo = _span(case)
        mesh = Mesh.uniform(ctx, list(n), lo, [lo[d] + n[d] * h for d in range(3)])
        if op_kind == "step":
            maps = [DofMap(mesh, 2, WALLS), DofMap(mesh, 1, 0), DofMap(mesh, 2, 0), DofMap(mesh, 2, BOTTOM)]
            step = MeltPoolStep(
                ctx, maps,
                evaporation=dict(mass_flux="knight", p_ambient=P_AMB, latent_heat=H_V, molar_mass=MOLAR, t_boil=T_BOIL,
                                 sticking=1.0, gas_constant=8.314),
                laser=dict(power=200.0, radius=SPOT, absorptivity=0.35, focus=(0.0, 0.0, 0.0), direction=(0.0, 0.0, -1.0)),
                gravity=(0.0, 0.0, -9.81), dt=1e-8, eps=2.0 * h, rho_l=RHO_L, rho_g=RHO_G, mu_l=MU_L, mu_g=MU_G,
                rhocp_l=RHO_L * CP_L, rhocp_g=RHO_G * CP_G, k_l=K_L, k_g=K_G, oseen_flags=MELT_FLAGS, rho_s=RHO_L,
                mu_s=MU_L, t_solidus=T_SOLIDUS, t_liquidus=T_LIQUIDUS, darcy_c=1e12, darcy_b=1.0, alpha0=1.493,
                alpha1=5.5e-4, t_alpha=1928.0, alpha_res=0.01, reinit_steps=2, dtau=0.5 * h, tol=1e-12, flow_tol=1e-12,
                maxit=500, reinit_mixed=1, flow_velocity_steps=5, flow_schur_maxit=30, flow_schur_tol=0.1)
            return {"case": case, "step": step, "state": _step_state(case, seed)}
        f = _fields(case, seed)
        if op_kind == "helmholtz":
            op = Operator(ctx, "helmholtz", [DofMap(mesh, 2, 0)], mass_coef=1.0, a_liquid=A_LIQUID, a_gas=A_GAS,
                          eps=2.0 * h, coef_mode=1)
        elif op_kind == "oseen":
            op = Operator(ctx, "oseen", [DofMap(mesh, 2, WALLS), DofMap(mesh, 1, 0)], **_oseen_params(case))
        else:
            op = Operator(ctx, "heat", [DofMap(mesh, 2, BOTTOM)], rhocp=RHO_L * CP_L, dt=HEAT_DT, k0=K_L, t_boil=T_BOIL,
                          coef_mode=1)
        for name in ("phi", "t_prev", "beta", "k_qpoint"):
            if name in f:
                op.set_field(name, f[name])
    op.autotune()
    return {"case": case, "op": op, **{k: f[k] for k in ("src", "b") if k in f}}


def run(state):
    case = state["case"]
    if case["call"] == "step":
        out, _ = state["step"].advance(state["state"])
        return {k: out[k] for k in ("u", "p", "T", "phi")}
    op = state["op"]
    if case["call"] == "apply":
        return op.apply(state["src"], nrhs=case["nrhs"], transpose=case["op"] == "adjoint",
                        arith="df64" if case["arith"] == "df64" else None)
    if case["call"] == "cg":
        return op.solve(state["b"], solver="cg", precond="jacobi", tol=1e-12, use_graph=True)[0]
    return op.solve(state["b"], solver="defect_correction", precond="chebyshev", cheby_degree=4, tol=1e-12,
                    use_graph=True, fp64_arith="df64")[0]


def work(case):
    """Each input read once, each output written once; operations as the sum-factorised cell needs
    them (a multiply-add counts as two).  Solves: the data of the call and the operations of one
    application per factor of ten of the residual."""
    word = 4 if case["arith"] == "f32" else 8
    r = case["nrhs"]
    if case["op"] == "reinit":
        # about 12 n^2 leaves in the band per level-surface area, 7.3 free nodes per leaf
        nf = case["base"] << case["levels"]
        leaves = 24.0 * nf * nf
        return {"bytes": word * 7.3 * leaves * (2 * r + 1) + 108 * leaves, "flops": 2000.0 * leaves * r}
    n, _, _ = _span(case)
    cells = n[0] * n[1] * n[2]
    nodes = (2 * n[0] + 1) * (2 * n[1] + 1) * (2 * n[2] + 1)
    pnodes = (n[0] + 1) * (n[1] + 1) * (n[2] + 1)
    if case["op"] == "step":
        return {"bytes": 8.0 * (10 * nodes + 5 * nodes + pnodes), "flops": 12.0 * cells * (5929 + 3 * 2000)}
    if case["op"] == "oseen":
        fields = nodes * (5 if case["melt"] else 4)
        return {"bytes": float(word) * (2 * (3 * nodes + pnodes) + fields), "flops": 5929.0 * cells}
    flops = 1539.0 if case["op"] != "adjoint" else 1539.0 + 27 * 7
    fields = nodes if case["op"] != "adjoint" else 3 * nodes + 27 * cells
    times = 1 if case["call"] == "apply" else 12
    return {"bytes": float(word) * (2 * r * nodes + fields), "flops": flops * cells * r * times}


# ------------------------------------------------------------------------------ the same in plain torch, 64 bits

def _tables():
    """Q2 shape values N[q, i], reference gradients G[d][q, i], Q1 values P[q, i] and weights at the 27
    Gauss points (x fastest)."""
    s = math.sqrt(15.0) / 10.0
    x = torch.tensor([0.5 - s, 0.5, 0.5 + s], dtype=torch.float64)
    w = torch.tensor([5.0, 8.0, 5.0], dtype=torch.float64) / 18.0
    n1 = torch.stack([(2 * x - 1) * (x - 1), 4 * x * (1 - x), x * (2 * x - 1)], 1)
    d1 = torch.stack([4 * x - 3, 4 - 8 * x, 4 * x - 1], 1)
    p1 = torch.stack([1 - x, x], 1)
    k3 = lambda a, b, c: torch.kron(torch.kron(c.contiguous(), b.contiguous()), a.contiguous()).cuda()
    N, G = k3(n1, n1, n1), [k3(d1, n1, n1), k3(n1, d1, n1), k3(n1, n1, d1)]
    return N, G, k3(p1, p1, p1), k3(w[:, None], w[:, None], w[:, None]).reshape(-1)


def _cells(n, degree):
    """Node numbers of every cell of a uniform lattice (cells and local nodes x fastest)."""
    k, R = degree, [degree * m + 1 for m in n]
    ar = lambda m: torch.arange(m, device="cuda")
    cell = (k * ar(n[0]))[None, None, :] + R[0] * (k * ar(n[1]))[None, :, None] + R[0] * R[1] * (k * ar(n[2]))[:, None, None]
    loc = ar(k + 1)[None, None, :] + R[0] * ar(k + 1)[None, :, None] + R[0] * R[1] * ar(k + 1)[:, None, None]
    return cell.reshape(-1, 1) + loc.reshape(1, -1)


class _Scalar:
    """y = A x of a scalar cell operator: value coefficient m, diffusion k, convection c (forward or
    transposed) or direction field nrm, per cell and Gauss point."""

    def __init__(self, m, h, k=None, conv=None, nrm=None, transpose=False):
        self.N, self.G, _, self.w = _tables()
        self.m, self.h, self.k, self.conv, self.nrm, self.tr = m, h, k, conv, nrm, transpose

    def cell(self, U):
        N, G, w, h = self.N, self.G, self.w, self.h
        u = U @ N.T
        g = [U @ G[d].T / h for d in range(3)]
        f = self.m * u
        if self.nrm is not None:
            s = self.k * sum(self.nrm[d] * g[d] for d in range(3))
            F = [s * self.nrm[d] for d in range(3)]
        else:
            F = [self.k * g[d] for d in range(3)]
        if self.conv is not None:
            if self.tr:
                F = [F[d] + self.conv[d] * u for d in range(3)]
            else:
                f = f + sum(self.conv[d] * g[d] for d in range(3))
        jxw = w * h ** 3
        return (jxw * f) @ N + sum((jxw / h * F[d]) @ G[d] for d in range(3))


def _uniform_scalar(case, f):
    """(apply function, number of nodes) of the case's scalar operator on its uniform mesh."""
    n, h, _ = _span(case)
    N, _, _, _ = _tables()
    idx = _cells(n, 2)
    nd = (2 * n[0] + 1) * (2 * n[1] + 1) * (2 * n[2] + 1)
    if case["op"] == "helmholtz":
        H = (0.5 * (1.0 + f["phi"][idx] @ N.T)).clamp(0.0, 1.0)
        A, fixed = _Scalar(1.0, h, A_GAS + (A_LIQUID - A_GAS) * H), None
    else:
        fixed = _dirichlet(case, BOTTOM)
        if case["op"] == "heat":
            A = _Scalar(RHO_L * CP_L / HEAT_DT, h, K_L * (1.0 + 0.5 * (f["t_prev"][idx] @ N.T) / T_BOIL))
        else:
            b = f["beta"].reshape(3, -1)
            A = _Scalar(RHO_L * CP_L / HEAT_DT, h, f["k_qpoint"].reshape(-1, 27),
                        conv=[RHO_L * CP_L * (b[d][idx] @ N.T) for d in range(3)], transpose=True)

    def apply(x):
        xm = x if fixed is None else torch.where(fixed, 0.0, x)
        y = torch.zeros_like(x).index_add_(0, idx.reshape(-1), A.cell(xm[idx]).reshape(-1))
        return y if fixed is None else torch.where(fixed, x, y)
    return apply, nd


def _exact_oseen(case, f):
    n, h, _ = _span(case)
    N, G, P, w = _tables()
    iu, ip = _cells(n, 2), _cells(n, 1)
    nu = (2 * n[0] + 1) * (2 * n[1] + 1) * (2 * n[2] + 1)
    p = _oseen_params(case)
    fixed = _dirichlet(case, WALLS)
    H = (0.5 * (1.0 + f["phi"][iu] @ N.T)).clamp(0.0, 1.0)
    mass, nrm = 0.0, None
    if case["melt"]:
        fs = ((T_LIQUIDUS - f["t_prev"][iu] @ N.T) / (T_LIQUIDUS - T_SOLIDUS)).clamp(0.0, 1.0)
        hs = 3.0 * fs * fs - 2.0 * fs ** 3
        rho = 1.0 / (H / (hs * p["rho_s"] + (1.0 - hs) * RHO_L) + (1.0 - H) / RHO_G)
        mu = H * (hs * p["mu_s"] + (1.0 - hs) * MU_L) + (1.0 - H) * MU_G
        mass = H * p["darcy_c"] * fs * fs / ((1.0 - fs) ** 3 + p["darcy_b"])
        gp = [f["phi"][iu] @ G[d].T / h for d in range(3)]
        size = torch.sqrt(sum(v * v for v in gp))
        nrm = [torch.where(size < 1e-12 / h, 0.0, v / size) for v in gp]
    else:
        rho = 1.0 / (H / RHO_L + (1.0 - H) / RHO_G)
        mu = H * MU_L + (1.0 - H) * MU_G
    mass = mass + p["sigma"] * rho
    beta = [f["beta"].reshape(3, -1)[d][iu] @ N.T for d in range(3)]
    x = f["src"].double()
    u = x[:3 * nu].reshape(3, nu)
    um = torch.where(fixed, 0.0, u)
    jxw = w * h ** 3
    U = [um[d][iu] for d in range(3)]
    uq = [v @ N.T for v in U]
    g = [[v @ G[e].T / h for e in range(3)] for v in U]
    pq = x[3 * nu:][ip] @ P.T
    div = g[0][0] + g[1][1] + g[2][2]
    out = torch.zeros_like(x)
    for d in range(3):
        val = mass * uq[d] + rho * sum(beta[e] * g[d][e] for e in range(3))
        R = (jxw * val) @ N
        for e in range(3):
            flux = mu * (g[d][e] + g[e][d])
            if nrm is not None:
                flux = flux - 2.0 * mu * div * nrm[d] * nrm[e]
            if d == e:
                flux = flux - pq
            R += (jxw / h * flux) @ G[e]
        y = torch.zeros(nu, dtype=torch.float64, device="cuda").index_add_(0, iu.reshape(-1), R.reshape(-1))
        out[d * nu:(d + 1) * nu] = torch.where(fixed, u[d], y)
    out[3 * nu:].index_add_(0, ip.reshape(-1), ((-jxw * div) @ P).reshape(-1))
    return out


class _OctreeLattice:
    """The Q2 nodes of an octree on the lattice of half the finest cell edge: the free nodes in DoF
    order, and for each hanging node the coarser leaf whose interpolant gives its value."""

    def __init__(self, lev, case):
        L, nf = case["levels"], lev.shape[0]
        self.L, self.M = L, 2 * nf + 1
        M = self.M
        low = lev.permute(2, 1, 0).contiguous()          # [z, y, x]
        for axis in range(3):                            # coarsest leaf that touches each lattice point
            shape = list(low.shape)
            shape[axis] = M
            out = low.new_empty(shape)
            a = low.movedim(axis, 0)
            o = out.movedim(axis, 0)
            o[1::2] = a
            o[0], o[-1] = a[0], a[-1]
            o[2:-1:2] = torch.minimum(a[:-1], a[1:])
            low = out
        self.low, self.lev = low, lev
        self.leaf = []
        node = torch.zeros(M * M * M, dtype=torch.bool, device="cuda")
        ar = torch.arange(3, device="cuda")
        loc = ar[None, None, :] + M * ar[None, :, None] + M * M * ar[:, None, None]
        self.loc = loc.reshape(1, -1)
        for l in range(L + 1):
            s = 1 << (L - l)
            ijk = (lev[::s, ::s, ::s] == l).nonzero()
            anchor = 2 * s * (ijk[:, 0] + M * ijk[:, 1] + M * M * ijk[:, 2])
            idx = anchor[:, None] + s * self.loc
            self.leaf.append((s / nf, idx))
            node[idx.reshape(-1)] = True
        step = (1 << (L - low.reshape(-1)))
        at = torch.arange(M * M * M, device="cuda")
        xyz = (at % M, (at // M) % M, at // (M * M))
        on = (xyz[0] % step == 0) & (xyz[1] % step == 0) & (xyz[2] % step == 0)
        self.free = (node & on).nonzero().reshape(-1)
        self.hang = []
        rest = node & ~on
        for l in range(L):
            s = 1 << (L - l)
            p = (rest & (low.reshape(-1) == l)).nonzero().reshape(-1)
            if not p.numel():
                continue
            c = torch.stack([p % M, (p // M) % M, p // (M * M)])
            cell, found = torch.zeros_like(c), torch.zeros_like(p, dtype=torch.bool)
            for o in range(8):                           # a leaf of that level on whose closure the point lies
                t = torch.stack([(c[d] - ((o >> d) & 1)) // 2 for d in range(3)]).clamp_(0, nf - 1)
                hit = ~found & (lev[t[0], t[1], t[2]] == l)
                cell, found = torch.where(hit, t, cell), found | hit
            a = cell // s * (2 * s)
            xi = (c - a).double() / (2.0 * s)
            w = [torch.stack([(2 * v - 1) * (v - 1), 4 * v * (1 - v), v * (2 * v - 1)], 1) for v in xi]
            w27 = (w[2][:, :, None, None] * w[1][:, None, :, None] * w[0][:, None, None, :]).reshape(-1, 27)
            self.hang.append((p, (a[0] + M * a[1] + M * M * a[2])[:, None] + s * self.loc, w27))

    def coords(self):
        h = 1.0 / (self.M - 1)
        M = self.M
        return [v.double() * h for v in (self.free % M, (self.free // M) % M, self.free // (M * M))]

    def extend(self, x):
        v = torch.zeros(self.M ** 3, dtype=torch.float64, device="cuda")
        v[self.free] = x
        for p, idx, w in self.hang:
            v[p] = (v[idx] * w).sum(1)
        return v

    def condense(self, v):
        for p, idx, w in reversed(self.hang):
            v.index_add_(0, idx.reshape(-1), (w * v[p][:, None]).reshape(-1))
            v[p] = 0.0
        return v[self.free]


def _octree_phi(case, lat, dist, seed):
    """Level set of the sphere moved by up to a quarter of the finest cell edge, the distance kept to a
    band of 16 such edges (beyond it the level set is constant and has no normal)."""
    nf = case["base"] << case["levels"]
    d = dist(*lat.coords()) * nf + _uniform(_generator(seed + 101), 1, -0.25, 0.25)
    return torch.tanh((d / 4.0).clamp(-4.0, 4.0))


def _exact_reinit(case, seed):
    lev, _, dist = _octree(case)
    lat = _OctreeLattice(lev, case)
    nf = case["base"] << case["levels"]
    phi = _octree_phi(case, lat, dist, seed)
    src = _uniform(_generator(seed), case["nrhs"] * phi.numel())
    phi = lat.extend(phi)
    src = (src.float() if case["arith"] == "f32" else src).double().reshape(case["nrhs"], -1)
    _, G, _, _ = _tables()
    ops = []
    for h, idx in lat.leaf:
        g = [phi[idx] @ G[d].T / h for d in range(3)]
        size = torch.sqrt(sum(v * v for v in g))
        nrm = [torch.where(size < 1e-12 / h, 0.0, v / size) for v in g]
        ops.append((idx, _Scalar(2.0 * nf, h, 2.0 / nf, nrm=nrm)))
    out = []
    for r in range(case["nrhs"]):
        v = lat.extend(src[r])
        y = torch.zeros_like(v)
        for idx, A in ops:
            y.index_add_(0, idx.reshape(-1), A.cell(v[idx]).reshape(-1))
        out.append(lat.condense(y))
    return torch.cat(out)


def _diagonal(case, f):
    """Diagonal of the symmetric uniform-mesh operator, cell by cell."""
    n, h, _ = _span(case)
    N, G, _, w = _tables()
    idx = _cells(n, 2)
    if case["op"] == "helmholtz":
        m, k = 1.0, A_GAS + (A_LIQUID - A_GAS) * (0.5 * (1.0 + f["phi"][idx] @ N.T)).clamp(0.0, 1.0)
    else:
        m, k = RHO_L * CP_L / HEAT_DT, K_L * (1.0 + 0.5 * (f["t_prev"][idx] @ N.T) / T_BOIL)
    D = m * h ** 3 * (w @ N.square()) + (k * w * h) @ sum(g.square() for g in G)
    d = torch.zeros((2 * n[0] + 1) * (2 * n[1] + 1) * (2 * n[2] + 1), dtype=torch.float64, device="cuda")
    d.index_add_(0, idx.reshape(-1), D.expand(idx.shape).reshape(-1))
    return d if case["op"] == "helmholtz" else torch.where(_dirichlet(case, BOTTOM), 1.0, d)


def exact(case, seed):
    if case["call"] == "step":
        return None          # the coupled step has no direct form that ends in seconds
    if case["op"] == "reinit":
        return _exact_reinit(case, seed)
    f = _fields(case, seed)
    if case["op"] == "oseen":
        return _exact_oseen(case, f)
    apply, nd = _uniform_scalar(case, f)
    if case["call"] == "apply":
        return torch.cat([apply(x) for x in f["src"].double().reshape(case["nrhs"], nd)])
    b, dinv = f["b"], 1.0 / _diagonal(case, f)
    x = torch.zeros_like(b)
    r = b.clone()
    for _ in range(4):       # Jacobi-CG to rounding, restarted from the true residual
        z = dinv * r
        p, rz = z.clone(), torch.dot(r, z)
        goal = 1e-14 * b.norm()
        for it in range(1500):
            q = apply(p)
            a = rz / torch.dot(p, q)
            x += a * p
            r -= a * q
            if it % 10 == 9 and bool(r.norm() <= goal):
                break
            z = dinv * r
            new = torch.dot(r, z)
            p = z + (new / rz) * p
            rz = new
        r = b - apply(x)
        if bool(r.norm() <= 1e-13 * b.norm()):
            break
    return x
