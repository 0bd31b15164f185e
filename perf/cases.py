"""Performance cases of the library: the work that its users have it do, through the public binding
(paper_2511_21713_gb300.pbfb), from the smallest calls to whole solves.

listed() names the cases, draw(rng) gives further ones of the same ranges, prepare(case, seed) makes
what a program holds before the call, run(state) is one pass, work(case) counts what a pass cannot do
without, and exact(case, seed) gives the results in plain 64-bit torch where there is a closed
discrete definition (the boundary operators, the element sums, the energy, the flux).

Kinds of case ("op"):
  layer     one boundary operator, V or K, on one surface (verification, post-processing)
  operator  the coupled operator on a whole vector: the Newton residual's product
  assembly  Jacobian and load of the nonlinear term and one relaxation-factor evaluation: what a
            Newton step does besides its linear solve
  energy    the solvation energy of a solution
  inverse   the dense single-layer inverse of a surface, built once per molecule and ionic strength
  flux      the flux on the molecular surface of the formulation that meshes the solute too
  solve     a whole nonlinear solve on a mesh that the program keeps
  request   a molecule seen for the first time: mesh, charges, solve, release
"""
import functools
import math

import numpy as np
import torch

from paper_2511_21713_gb300 import inputs, pbfb

PRECISION = {"fp64": pbfb.FP64, "mixed": pbfb.MIXED, "float2": pbfb.FLOAT2}
SCHEME = {"linear": pbfb.LINEAR, "t3": pbfb.T3, "hs": pbfb.HS, "t5": pbfb.T5, "t7": pbfb.T7}

# Launch shapes a program has from an earlier autotuner run on the multi-charge sphere.
TUNED = {"treecode": 2, "ff_kernel": 4, "ff_blocks_per_sm": 16, "spmv_lanes": 4}


def listed():
    return [
        # the smallest boundary product: one layer of the single-charge sphere (500 triangles)
        dict(name="layer_smallest", op="layer", nu=5, layers=4, which="m", layer="V", precision="float2", ionic=0.15),
        # a float64 check of the Yukawa double layer on a mid-sized outer surface
        dict(name="layer_yukawa_fp64", op="layer", nu=9, layers=4, which="s", layer="K", precision="fp64", ionic=0.3),
        # the float64 path's operator product (default precision of a solve)
        dict(name="operator_fp64", op="operator", nu=13, layers=9, precision="fp64", ionic=0.1),
        # the mixed path's residual product at the size of the multi-charge sphere
        dict(name="operator_float2", op="operator", nu=20, layers=17, precision="float2", ionic=0.1),
        # a Newton step's assembly at the size of the multi-charge sphere
        dict(name="assembly_mixed", op="assembly", nu=20, layers=17, precision="mixed", scheme="hs", ionic=0.1),
        # solvation energy of a solution, 200 charges
        dict(name="energy", op="energy", nu=16, layers=12, charges=200, ionic=0.1),
        # preconditioner block of a new ionic strength
        dict(name="inverse_yukawa", op="inverse", nu=14, layers=4, which="s", ionic=0.2),
        # flux on the molecular surface, solute meshed (post-processing of each such solve)
        dict(name="flux_solute", op="flux", nu=8, layers=6, core_layers=6, charges=40, precision="float2", ionic=0.1),
        # the single-charge sphere in plain float64 (3528 vertices)
        dict(name="solve_fp64_small", op="solve", shape="sphere", nu=5, layers=13, charges=1, precision="fp64",
             ionic=0.15, tuned=False),
        # the multi-charge sphere, mixed precision, shapes from a tuning file, charges as host buffers
        dict(name="solve_mixed_sphere", op="solve", shape="sphere", nu=20, layers=17, charges=200, precision="mixed",
             ionic=0.1, tuned=True),
        # a highly charged double helix, mixed precision, built-in shapes
        dict(name="solve_mixed_helix", op="solve", shape="helix", nu=28, layers=10, base_pairs=24, precision="mixed",
             ionic=0.15, tuned=False),
        # a served request for an unseen molecule of ordinary size
        dict(name="request_new", op="request", shape="sphere", nu=12, layers=10, charges=60, precision="mixed",
             ionic=0.25),
    ]


def draw(rng):
    """One more case of the listed ones' ranges: sizes log-uniform in triangles (20 nu^2)."""

    def nu(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    ionic = round(math.exp(rng.uniform(math.log(0.01), math.log(1.0))), 4)
    op = rng.choice(["layer", "layer", "operator", "operator", "assembly", "energy", "inverse", "flux", "solve",
                     "solve", "request"])
    if op == "layer":
        precision = rng.choice(["fp64", "float2"])
        return dict(op=op, nu=nu(4, 14 if precision == "fp64" else 22), layers=rng.randint(3, 5),
                    which=rng.choice("ms"), layer=rng.choice("VK"), precision=precision, ionic=ionic)
    if op == "operator":
        precision = rng.choice(["fp64", "float2"])
        return dict(op=op, nu=nu(4, 13 if precision == "fp64" else 20), layers=rng.randint(4, 14),
                    precision=precision, ionic=ionic)
    if op == "assembly":
        return dict(op=op, nu=nu(4, 20), layers=rng.randint(4, 17), precision=rng.choice(["fp64", "mixed", "mixed"]),
                    scheme=rng.choice(["hs", "hs", "t3", "t5", "t7"]), ionic=ionic)
    if op == "energy":
        return dict(op=op, nu=nu(5, 20), layers=rng.randint(4, 12), charges=nu(1, 200), ionic=ionic)
    if op == "inverse":
        return dict(op=op, nu=nu(4, 18), layers=3, which=rng.choice("ms"), ionic=ionic)
    if op == "flux":
        return dict(op=op, nu=nu(4, 9), layers=rng.randint(4, 7), core_layers=rng.randint(3, 7), charges=nu(1, 80),
                    precision=rng.choice(["fp64", "float2"]), ionic=ionic)
    if op == "solve":
        if rng.random() < 0.3:
            return dict(op=op, shape="sphere", nu=nu(4, 7), layers=rng.randint(6, 13), charges=nu(1, 100),
                        precision="fp64", ionic=ionic, tuned=False)
        shape = rng.choice(["sphere", "helix"])
        more = dict(charges=nu(1, 200)) if shape == "sphere" else dict(base_pairs=rng.randint(8, 20))
        return dict(op=op, shape=shape, nu=nu(6, 20), layers=rng.randint(7, 14), precision="mixed", ionic=ionic,
                    tuned=rng.random() < 0.5, **more)
    return dict(op=op, shape="sphere", nu=nu(5, 16), layers=rng.randint(5, 11), charges=nu(1, 150), precision="mixed",
                ionic=ionic)


# ------------------------------------------------------------------------------------- inputs

@functools.lru_cache(maxsize=4)
def _shell(nu, layers, a, outer):
    return inputs.spherical_shell(nu, a, outer, layers)


def _molecule(case, seed):
    """The host arrays of a case's molecule: an inputs.Case."""
    T, eps_out = 300.0, 80.0
    nq = case.get("charges", 1)
    if case.get("shape") == "helix":
        return inputs.double_helix(n_bp=case["base_pairs"], nu=case["nu"], layers=case["layers"], seed=3000 + seed,
                                   n_interior=62 * case["base_pairs"], ionic=case["ionic"])
    if case["op"] == "flux":
        q, z = inputs.ball_charges(nq, 9.0, nq // 2, seed)
        return inputs.solute_sphere_case(nu=case["nu"], a=12.0, R=24.0, layers=case["layers"],
                                         core_layers=case["core_layers"], q_xyz=q, q_z=z, eps_in=2.0, eps_out=eps_out,
                                         ionic=case["ionic"], T=T)
    small = nq == 1  # the single-charge sphere
    a, outer, eps_in = (4.0, 10.0, 4.0) if small else (12.0, 24.0, 2.0)
    if small:
        r = np.random.default_rng(seed)
        q, z = r.uniform(-0.5, 0.5, (1, 3)), np.array([5.0])
    else:
        q, z = inputs.ball_charges(nq, 10.0, int(0.45 * nq), seed)
    if case["op"] == "inverse":  # no vector goes in: the surface itself differs from seed to seed
        a, outer = (float(v * np.random.default_rng(seed).uniform(0.9, 1.1)) for v in (a, outer))
    xyz, tets, gm, gs = _shell(case["nu"], case["layers"], a, outer)
    kappa = inputs.kappa_from_ionic_strength(case["ionic"], eps_out, T)
    return inputs.Case(case["op"], xyz, tets, gm, gs, q, z, eps_in, eps_out, kappa, T)


def _fields(mol, seed):
    """Potentials and fluxes like a solution's: u decays from a few kT/e over the shell, with the
    roughness of charges below the surface."""
    r = np.random.default_rng(seed)
    rad = np.linalg.norm(mol.xyz, axis=1)
    inner = np.linalg.norm(mol.xyz[mol.gm_tris[0]], axis=1).min()
    wave = np.cos(mol.xyz @ (r.normal(size=(3, 3)) / inner).T + r.uniform(0, 6.28, 3)).sum(axis=1)
    u = 3.0 * np.exp(-0.25 * np.maximum(rad - inner, 0.0)) * wave
    du = 0.3 * u * r.normal(size=u.size) + 0.05 * r.normal(size=u.size)
    vm, vs = np.unique(mol.gm_tris), np.unique(mol.gs_tris)
    lam_m = 0.5 * u[vm] * (1.0 + 0.1 * r.normal(size=vm.size))
    lam_s = -0.2 * u[vs] * (1.0 + 0.1 * r.normal(size=vs.size))
    return u, du, lam_m, lam_s


def _cuda(a):
    return torch.as_tensor(np.ascontiguousarray(a, np.float64), device="cuda")


def _layer_input(case, mol, seed):
    u, _, lam_m, lam_s = _fields(mol, seed)
    if case["layer"] == "V":
        return lam_m if case["which"] == "m" else lam_s
    return u[np.unique(mol.gm_tris if case["which"] == "m" else mol.gs_tris)]


def _which(case):
    return pbfb.GAMMA_M if case["which"] == "m" else pbfb.GAMMA_S


def prepare(case, seed):
    mol = _molecule(case, seed)
    op = case["op"]
    s = dict(case=case, mol=mol)
    if op == "request":  # host arrays only
        s["opts"] = pbfb.default_opts(precision=PRECISION[case["precision"]])
        return s
    m = s["mesh"] = pbfb.Mesh.from_case(mol)
    if op == "solve":
        s["opts"] = pbfb.default_opts(precision=PRECISION[case["precision"]])
        if case["tuned"]:
            m.apply_tuning(TUNED)
        s["x"] = torch.empty(m.n, dtype=torch.float64, device="cuda")
        return s
    m.set_params(mol.eps_in, mol.eps_out, mol.kappa, mol.T, PRECISION[case.get("precision", "fp64")])
    u, du, lam_m, lam_s = _fields(mol, seed)
    if op == "layer":
        s["x"] = _cuda(_layer_input(case, mol, seed))
        s["y"] = torch.empty_like(s["x"])
    elif op == "operator":
        s["x"] = _cuda(np.concatenate([u, lam_m, lam_s]))
        s["y"] = torch.empty_like(s["x"])
        m.assemble(pbfb.HS, _cuda(u), None)
    elif op == "assembly":
        r = np.random.default_rng(seed + 1)
        s["u"], s["du"] = _cuda(u), _cuda(du)
        s["c"] = _cuda(0.1 * r.normal(size=m.n))
        s["p"] = _cuda(0.1 * r.normal(size=m.n))
        s["N"] = torch.empty(m.n_v, dtype=torch.float64, device="cuda")
    elif op == "energy":
        m.charges_set(mol.q_xyz, mol.q_z)
        x = np.concatenate([u, lam_m, lam_s])
        s["xL"], s["xNL"] = _cuda(x), _cuda(-0.1 * np.concatenate([u + du, lam_m, lam_s]))
    elif op == "inverse":
        n = m.n_m if case["which"] == "m" else m.n_s
        s["V"] = torch.empty(n, n, dtype=torch.float32, device="cuda")
        s["inv"] = torch.empty(n, n, dtype=torch.float32, device="cuda")
    elif op == "flux":
        m.charges_set(mol.q_xyz, mol.q_z)
        s["x"] = _cuda(np.concatenate([u, 0.0 * lam_m, 0.0 * lam_s]))
        s["lam"] = torch.empty(m.n_m, dtype=torch.float64, device="cuda")
    return s


def run(s):
    case, mol, op = s["case"], s["mol"], s["case"]["op"]
    if op == "request":
        m = pbfb.Mesh.from_case(mol)
        m.charges_set(mol.q_xyz, mol.q_z)
        x, res = m.solve(mol.eps_in, mol.eps_out, mol.kappa, mol.T, s["opts"])
        m.close()
        return {"x": x, "total": res["total"]}
    m = s["mesh"]
    if op == "layer":
        m.bem_apply(_which(case), 0 if case["layer"] == "V" else 1, s["x"], s["y"])
        return s["y"]
    if op == "operator":
        m.apply(s["x"], s["y"])
        return s["y"]
    if op == "assembly":
        m.assemble(SCHEME[case["scheme"]], s["u"], s["N"])
        return {"N": s["N"], "dots": m.omega_eval(SCHEME[case["scheme"]], s["u"], s["du"], s["c"], s["p"], [1.0])}
    if op == "energy":
        return m.energy(s["xL"], s["xNL"])
    if op == "inverse":
        m.single_layer_dense(_which(case), False, s["V"])  # also makes the next call build the inverse anew
        m.single_layer_dense(_which(case), True, s["inv"])
        return {"V": s["V"], "inverse": s["inv"]}
    if op == "flux":
        m.gamma_m_flux(s["x"], 1, s["lam"])
        return s["lam"]
    m.charges_set(mol.q_xyz, mol.q_z)
    res = m.solve_device(mol.eps_in, mol.eps_out, mol.kappa, mol.T, s["x"], s["opts"])
    return {"x": s["x"], "total": res["total"]}


# ------------------------------------------------------------------------------------- work

def _sizes(case):
    nu, layers = case["nu"], case["layers"]
    nt = 20 * nu * nu
    ns = 10 * nu * nu + 2
    shells = layers + 1 + (case.get("core_layers", 0))
    return dict(nt=nt, nq=6 * nt, ns=ns, nv=ns * shells, tets=3 * nt * layers, n=ns * shells + 2 * ns)


def work(case):
    """Operations of one float32-counted pair of quadrature points (an FMA is 2): 20 with the Laplace
    kernel (single and double layer together), 28 with the Yukawa kernel, 1 root and 1 exponential
    not counted; one layer alone 14 and 20.  A solve: its Newton steps times two far fields of the
    residual (both surfaces), as many relaxation-factor evaluations and assemblies, and five operator
    products of the linear solver per step."""
    z, op = _sizes(case), case["op"]
    pairs = float(z["nq"]) ** 2
    both = 48.0 * pairs
    slots = 15.0 * z["nv"] + 80.0 * z["ns"]
    vec = 8.0 * z["n"]
    point = 80.0  # per quadrature point of a tet: root sums, exponential, Jacobian and load
    if op == "layer":
        return {"bytes": 16.0 * z["ns"] + 40.0 * z["nq"], "flops": (14.0 if case["which"] == "m" else 20.0) * pairs}
    if op == "operator":
        return {"bytes": 12.0 * slots + 2 * vec + 80.0 * z["nq"], "flops": both + 2.0 * slots}
    if op == "assembly":
        return {"bytes": 2 * 24.0 * z["tets"] + 8.0 * slots + 5 * vec, "flops": 2 * 14 * point * z["tets"]}
    if op == "energy":
        return {"bytes": 24.0 * z["tets"] + 80.0 * z["nq"] + 2 * vec,
                "flops": 30.0 * z["nq"] * case["charges"] + 14 * 40.0 * z["tets"]}
    if op == "inverse":
        return {"bytes": 8.0 * z["ns"] ** 2, "flops": 12.0 * pairs + 1.0 * z["ns"] ** 3}
    if op == "flux":
        return {"bytes": 80.0 * z["nq"], "flops": 11 * 14.0 * pairs}
    steps = 6.0
    flops = steps * ((1 + 5) * (both + 2.0 * slots) + 3 * 14 * point * z["tets"])
    if op == "request":
        flops += 150.0 * 600.0 * 60.0 * z["nt"]  # near-field rules: about 60 pairs a triangle, 600 points a pair
    return {"bytes": steps * (6 * 12.0 * slots + 20 * vec), "flops": flops}


# ------------------------------------------------------------------------------------- 64 bits
# The discrete quantities in plain float64 torch: 6-point triangle rule over all pairs of triangles,
# Sauter-Schwab rules (5 points per variable) for touching pairs, 16-fold subdivision for close ones.

_B1, _B2 = 0.44594849091596488632, 0.09157621350977074346
_W1, _W2 = 0.22338158967801146570, 0.10995174365532186764


def _dev():
    return "cuda" if torch.cuda.is_available() else "cpu"


def _t(a, dtype=torch.float64):
    return torch.as_tensor(np.asarray(a), dtype=dtype, device=_dev())


def _tri6():
    b = [[1 - 2 * c if i == k else c for i in range(3)] for c in (_B1, _B2) for k in range(3)]
    return _t(b), _t([_W1] * 3 + [_W2] * 3)


def _sub96():
    b6, w6 = _tri6()
    pts = []
    for i in range(4):
        for j in range(4 - i):
            tris = [((i, j), (i + 1, j), (i, j + 1))]
            if i + j < 3:
                tris.append(((i + 1, j), (i + 1, j + 1), (i, j + 1)))
            for t in tris:
                pts.append(b6 @ _t([[1 - (p + q) / 4, p / 4, q / 4] for p, q in t]))
    return torch.cat(pts), w6.repeat(16) / 16.0


def _touching_rule(kind):
    x, w = np.polynomial.legendre.leggauss(5)
    x, w = 0.5 * (x + 1), 0.5 * w
    xi, a, b, c = (v.reshape(-1) for v in np.meshgrid(x, x, x, x, indexing="ij"))
    W = np.einsum("i,j,k,l->ijkl", w, w, w, w).reshape(-1)
    if kind == "identical":
        half = [((xi, xi * (1 - a + a * b)), (xi * (1 - a * b * c), xi * (1 - a))),
                ((xi, xi * a * (1 - b + b * c)), (xi * (1 - a * b), xi * a * (1 - b))),
                ((xi * (1 - a * b * c), xi * a * (1 - b * c)), (xi, xi * a * (1 - b)))]
        maps = [(m, xi ** 3 * a ** 2 * b) for h in half for m in (h, h[::-1])]
    elif kind == "edge":
        j1, j2 = xi ** 3 * a ** 2, xi ** 3 * a ** 2 * b
        maps = [(((xi, xi * a * c), (xi * (1 - a * b), xi * a * (1 - b))), j1),
                (((xi, xi * a), (xi * (1 - a * b * c), xi * a * b * (1 - c))), j2),
                (((xi * (1 - a * b), xi * a * (1 - b)), (xi, xi * a * b * c)), j2),
                (((xi * (1 - a * b * c), xi * a * b * (1 - c)), (xi, xi * a)), j2),
                (((xi * (1 - a * b * c), xi * a * (1 - b * c)), (xi, xi * a * b)), j2)]
    else:
        j = xi ** 3 * b
        maps = [(((xi, xi * a), (xi * b, xi * b * c)), j), (((xi * b, xi * b * c), (xi, xi * a)), j)]
    hat = lambda p: np.stack([1 - p[0], p[0] - p[1], p[1]], -1)  # noqa: E731
    bx = np.concatenate([hat(m[0]) for m, _ in maps])
    by = np.concatenate([hat(m[1]) for m, _ in maps])
    return _t(bx), _t(by), _t(np.concatenate([W * j for _, j in maps]))


class _Surface:
    def __init__(self, xyz, tris, kappa):
        tris = np.asarray(tris, np.int64)
        self.verts = np.unique(tris)
        self.n, self.nt, self.kappa = self.verts.size, tris.shape[0], kappa
        self.tl = _t(np.searchsorted(self.verts, tris), torch.int64)
        self.P = _t(xyz[tris])
        cr = torch.linalg.cross(self.P[:, 1] - self.P[:, 0], self.P[:, 2] - self.P[:, 0])
        nn = cr.norm(dim=1)
        self.area, self.nrm = 0.5 * nn, cr / nn[:, None]
        self.b6, self.w6 = _tri6()
        self.q = torch.einsum("qa,tad->tqd", self.b6, self.P).reshape(-1, 3)
        self.w = (self.area[:, None] * self.w6).reshape(-1)
        self.n6 = self.nrm.repeat_interleave(6, 0)
        self._pairs()

    def kernels(self, x, y, n):
        d = x - y
        r = d.square().sum(-1).sqrt()
        e = torch.exp(-self.kappa * r) / (4 * math.pi)
        return e / r, (n * d).sum(-1) * (1 + self.kappa * r) * e / r ** 3

    def _pairs(self):
        """Ordered pairs of triangles that do not take the 6 x 6 rule, with corrV and corrK (3 x 3 each)."""
        P, tl = self.P, self.tl
        h = torch.stack([(P[:, (k + 1) % 3] - P[:, k]).square().sum(-1).sqrt() for k in range(3)]).amax(0)
        cen = (P[:, 0] + P[:, 1] + P[:, 2]) / 3.0
        found = {k: [] for k in ("identical", "edge", "vertex", "near")}
        step = max(1, 20_000_000 // self.nt)
        for t0 in range(0, self.nt, step):
            t = torch.arange(t0, min(self.nt, t0 + step), device=P.device)
            shared = (tl[t][:, None, :, None] == tl[None, :, None, :]).sum((2, 3))
            d = cen[t][:, None] - cen[None]
            near = d.square().sum(-1) < (2.0 * torch.maximum(h[t][:, None], h[None])).square()
            for name, mask in (("identical", shared == 3), ("edge", shared == 2), ("vertex", shared == 1),
                               ("near", (shared == 0) & near)):
                a, b = mask.nonzero(as_tuple=True)
                found[name].append(torch.stack([a + t0, b]))
        self.pt, self.ps, self.cV, self.cK = [], [], [], []
        for name, f in found.items():
            t, s = torch.cat(f, 1)
            if name == "near":
                bt, wt = _tri6()
                bs, ws = _sub96()
                bx, by = bt.repeat_interleave(96, 0), bs.repeat(6, 1)
                w, scale = (wt[:, None] * ws).reshape(-1), 1.0
            else:
                bx, by, w = _touching_rule(name)
                scale = 4.0
            for k in range(0, t.numel(), 8192):
                self._correct(name, t[k:k + 8192], s[k:k + 8192], bx, by, w, scale)
        self.pt, self.ps = torch.cat(self.pt), torch.cat(self.ps)
        self.cV, self.cK = torch.cat(self.cV), torch.cat(self.cK)

    def _correct(self, name, t, s, bx, by, w, scale):
        idt = torch.arange(3, device=t.device).expand(t.numel(), 3)
        ot, os_ = idt, idt  # vertex orders of the rule
        if name in ("edge", "vertex"):
            same = self.tl[t][:, :, None] == self.tl[s][:, None, :]
            it = same.any(2).int()
            partner = same.int().argmax(2)
            if name == "edge":
                a = it.argmax(1)
                c = it.argmin(1)
                b = 3 - a - c
                pa, pb = partner.gather(1, a[:, None])[:, 0], partner.gather(1, b[:, None])[:, 0]
                ot, os_ = torch.stack([a, b, c], 1), torch.stack([pa, pb, 3 - pa - pb], 1)
            else:
                a = it.argmax(1)
                pa = partner.gather(1, a[:, None])[:, 0]
                ot, os_ = (a[:, None] + idt) % 3, (pa[:, None] + idt) % 3
        pick = lambda P, o: torch.gather(P, 1, o[:, :, None].expand(-1, -1, 3))  # noqa: E731
        Pt, Ps, ns = pick(self.P[t], ot), pick(self.P[s], os_), self.nrm[s]
        sl = torch.zeros(t.numel(), 3, 3, dtype=torch.float64, device=t.device)
        dl = torch.zeros_like(sl)
        for k in range(0, w.numel(), 640):
            x = torch.einsum("ka,mad->mkd", bx[k:k + 640], Pt)
            y = torch.einsum("ka,mad->mkd", by[k:k + 640], Ps)
            g, e = self.kernels(x, y, ns[:, None])
            bb = (w[k:k + 640, None, None] * bx[k:k + 640, :, None] * by[k:k + 640, None, :]).reshape(-1, 9)
            sl += (g @ bb).reshape(-1, 3, 3)
            dl += (e @ bb).reshape(-1, 3, 3)
        jac = (scale * self.area[t] * self.area[s])[:, None, None]
        # rule order -> stored order
        back = lambda M: torch.zeros_like(M).scatter(  # noqa: E731
            1, ot[:, :, None].expand(-1, -1, 3), torch.zeros_like(M).scatter(2, os_[:, None, :].expand(-1, 3, -1), M))
        sl, dl = back(sl * jac), back(dl * jac)
        q = self.q.reshape(-1, 6, 3)
        g, e = self.kernels(q[t][:, :, None], q[s][:, None], self.nrm[s][:, None, None])
        skip = (t == s)[:, None, None] & torch.eye(6, dtype=torch.bool, device=t.device)
        W = self.w.reshape(-1, 6)
        W = W[t][:, :, None] * W[s][:, None]
        g, e = torch.where(skip, 0.0, g * W), torch.where(skip, 0.0, e * W)
        self.cV.append(sl - torch.einsum("mqp,qa,pb->mab", g, self.b6, self.b6))
        self.cK.append(dl - torch.einsum("mqp,qa,pb->mab", e, self.b6, self.b6))
        self.pt.append(t)
        self.ps.append(s)

    def _rows(self):
        """Blocks of whole triangles: point range and the regular rule's g and dg/dn against all points."""
        step = 6 * max(1, 60_000_000 // self.q.shape[0] // 6)
        for i0 in range(0, self.q.shape[0], step):
            i1 = min(self.q.shape[0], i0 + step)
            g, e = self.kernels(self.q[i0:i1, None], self.q[None], self.n6[None])
            k = torch.arange(i0, i1, device=g.device)
            g[k - i0, k] = 0.0
            e[k - i0, k] = 0.0
            yield i0, i1, g, e

    def apply(self, V=None, K=None):
        """V v + K k for P1 coefficients (either may be None)."""
        hat = lambda c: torch.einsum("qa,ta->tq", self.b6, c[self.tl]).reshape(-1) * self.w  # noqa: E731
        pot = torch.zeros_like(self.w)
        for i0, i1, g, e in self._rows():
            if V is not None:
                pot[i0:i1] += g @ hat(V)
            if K is not None:
                pot[i0:i1] += e @ hat(K)
        y = torch.zeros(self.n, dtype=torch.float64, device=pot.device)
        y.index_add_(0, self.tl.reshape(-1), torch.einsum("tq,qa->ta", (pot * self.w).reshape(-1, 6), self.b6).reshape(-1))
        for v, c in ((V, self.cV), (K, self.cK)):
            if v is not None:
                y.index_add_(0, self.tl[self.pt].reshape(-1), torch.einsum("mab,mb->ma", c, v[self.tl[self.ps]]).reshape(-1))
        return y

    def dense_V(self):
        V = torch.zeros(self.n * self.n, dtype=torch.float64, device=self.P.device)
        for i0, i1, g, _ in self._rows():
            t0, t1 = i0 // 6, i1 // 6
            g = (g * self.w[i0:i1, None] * self.w[None]).reshape(t1 - t0, 6, self.nt, 6)
            loc = torch.einsum("tqsp,qa,pb->tasb", g, self.b6, self.b6)
            at = self.tl[t0:t1].reshape(-1, 1) * self.n + self.tl.reshape(1, -1)
            V.index_add_(0, at.reshape(-1), loc.reshape(-1))
        at = self.tl[self.pt][:, :, None] * self.n + self.tl[self.ps][:, None, :]
        V.index_add_(0, at.reshape(-1), self.cV.reshape(-1))
        return V.reshape(self.n, self.n)

    def mass(self, v):
        """M v with the P1 mass matrix."""
        c = v[self.tl]
        y = torch.zeros(self.n, dtype=torch.float64, device=v.device)
        y.index_add_(0, self.tl.reshape(-1), (self.area[:, None] / 12.0 * (c + c.sum(1, keepdim=True))).reshape(-1))
        return y

    def test(self, f):
        """<f, psi_i> of point values f by the 6-point rule."""
        y = torch.zeros(self.n, dtype=torch.float64, device=f.device)
        y.index_add_(0, self.tl.reshape(-1), torch.einsum("tq,qa->ta", (f * self.w).reshape(-1, 6), self.b6).reshape(-1))
        return y


class _Shell:
    """Element sums on the tets of Omega_i, 14-point rule."""

    def __init__(self, mol):
        tets = mol.tets if mol.tet_region is None else mol.tets[mol.tet_region == 1]
        self.tets = _t(tets, torch.int64)
        X = _t(mol.xyz)[self.tets]
        E = X[:, 1:] - X[:, :1]
        det = torch.linalg.det(E)
        self.vol = det.abs() / 6.0
        g = torch.linalg.inv(E).transpose(1, 2)
        self.grad = torch.cat([-g.sum(1, keepdim=True), g], 1)
        a1, a2, c3 = 0.09273525031089122640, 0.31088591926330060980, 0.04550370412564964949
        l = [[1 - 3 * a if i == k else a for i in range(4)] for a in (a1, a2) for k in range(4)]
        l += [[0.5 - c3 if i in (p, q) else c3 for i in range(4)] for p in range(3) for q in range(p + 1, 4)]
        self.l = _t(l)
        self.w = _t([0.07349304311636194954] * 4 + [0.11268792571801585080] * 4 + [0.04254602077708146644] * 6)
        self.nv, self.coef = mol.xyz.shape[0], mol.eps_out * mol.kappa ** 2

    def at(self, u):
        return u[self.tets] @ self.l.T

    def load(self, f):
        """eps_s kappa^2 int f v_i for values f at the points."""
        y = torch.zeros(self.nv, dtype=torch.float64, device=f.device)
        loc = self.coef * self.vol[:, None] * ((f * self.w) @ self.l)
        return y.index_add_(0, self.tets.reshape(-1), loc.reshape(-1))

    def stiffness(self, u, eps):
        y = torch.zeros_like(u)
        flux = torch.einsum("ta,tad->td", u[self.tets], self.grad)
        loc = eps * self.vol[:, None] * torch.einsum("tad,td->ta", self.grad, flux)
        return y.index_add_(0, self.tets.reshape(-1), loc.reshape(-1))


def _F(scheme, u):
    """F, F' and F'' of the nonlinear term."""
    if scheme == "hs":
        return torch.sinh(u), torch.cosh(u), torch.sinh(u)
    top = {"linear": 1, "t3": 3, "t5": 5, "t7": 7}[scheme]
    term = lambda k: u ** k / math.factorial(k)  # noqa: E731
    F = sum(term(k) for k in range(1, top + 1, 2))
    Fp = sum(term(k - 1) for k in range(1, top + 1, 2))
    Fpp = sum((term(k - 2) for k in range(3, top + 1, 2)), torch.zeros_like(u))
    return F, Fp, Fpp


def exact(case, seed):
    op = case["op"]
    if op in ("solve", "request"):
        return None
    mol = _molecule(case, seed)
    u, du, lam_m, lam_s = _fields(mol, seed)
    kT = inputs.KB_KCAL * mol.T
    lB = inputs.COULOMB_KCAL_A / kT
    surface = lambda which: _Surface(mol.xyz, mol.gm_tris if which == "m" else mol.gs_tris,  # noqa: E731
                                     0.0 if which == "m" else mol.kappa)
    if op == "layer":
        x = _t(_layer_input(case, mol, seed))
        return surface(case["which"]).apply(**{case["layer"]: x})
    if op == "operator":
        S, M, Y = _Shell(mol), surface("m"), surface("s")
        u, lm, ls = _t(u), _t(lam_m), _t(lam_s)
        vm, vs = _t(M.verts, torch.int64), _t(Y.verts, torch.int64)
        yu = S.stiffness(u, mol.eps_out) + S.load(torch.cosh(S.at(u)) * S.at(u))
        yu.index_add_(0, vm, mol.eps_in * M.mass(lm))
        yu.index_add_(0, vs, -mol.eps_out * Y.mass(ls))
        return torch.cat([yu, 0.5 * M.mass(u[vm]) + M.apply(V=-lm, K=u[vm]),
                          0.5 * Y.mass(u[vs]) + Y.apply(V=ls, K=-u[vs])])
    if op == "assembly":
        S = _Shell(mol)
        r = np.random.default_rng(seed + 1)
        n = S.nv + lam_m.size + lam_s.size
        c, p = _t(0.1 * r.normal(size=n)), _t(0.1 * r.normal(size=n))
        F, _, _ = _F(case["scheme"], S.at(_t(u)))
        d = S.at(_t(du))
        G, Gp, Gpp = _F(case["scheme"], S.at(_t(u)) + d)
        pad = lambda v: torch.cat([v, torch.zeros(n - S.nv, dtype=v.dtype, device=v.device)])  # noqa: E731
        res, rp, rpp = c - pad(S.load(G)), -pad(S.load(Gp * d)), -pad(S.load(Gpp * d * d))
        dots = torch.stack([(p + rp) @ res, (p + rp) @ p, (p + rp) @ rp, res @ rpp, p @ rpp, res @ res, p @ res, p @ p])
        return {"N": S.load(F), "dots": dots[None]}
    if op == "energy":
        M, S = surface("m"), _Shell(mol)
        vm, q, z = _t(M.verts, torch.int64), _t(mol.q_xyz), _t(mol.q_z)
        hat = lambda v: torch.einsum("qa,ta->tq", M.b6, v[M.tl]).reshape(-1) * M.w  # noqa: E731
        g, e = M.kernels(q[:, None], M.q[None], M.n6[None])
        uN = -0.1 * (_t(u) + _t(du))
        E = [0.5 * kT * (z @ (g @ hat(lam) - e @ hat(v[vm])))
             for v, lam in ((_t(u), _t(lam_m)), (uN, -0.1 * _t(lam_m)))]
        uq = S.at(_t(u) + uN)
        ion = (S.vol * ((uq * torch.sinh(uq) - 2 * torch.cosh(uq) + 2) @ S.w)).sum()
        dG = kT * S.coef / (8 * math.pi * lB) * ion
        return torch.stack([E[0] + E[1] + dG, E[0], E[1], dG])
    if op == "inverse":
        V = surface(case["which"]).dense_V()
        V = 0.5 * (V + V.T)
        return {"V": V, "inverse": torch.linalg.inv(V)}
    M = surface("m")  # flux
    um = _t(u)[_t(M.verts, torch.int64)]
    pot = (_t(mol.q_z) / (M.q[:, None] - _t(mol.q_xyz)[None]).norm(dim=-1)).sum(1)
    rhs = 0.5 * M.mass(um) + M.apply(K=um) - lB / mol.eps_in * M.test(pot)
    return torch.linalg.solve(M.dense_V(), rhs)
