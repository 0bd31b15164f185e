"""The far fields by pairs of triangles (float64 and float-float) at the sizes where their tiles,
groups, step parts and point shares change, and at the ends of the Yukawa kernel's range.

The two precisions share the pair formulas but neither kernel, tile layout nor exponential; the
one-target-per-thread float-float sum shares no pair formula with either.  Tolerance: the float-float
coordinates are rounded to 2^-47 of the diameter, the nearest quadrature points of these surfaces are
1/200 of it apart, and 1/r^3 triples the relative error: 3 * 200 * 2^-47 = 4e-12 on the nearest pairs,
which carry at most a tenth of a row (half of them: the rest cancels in sign) -- 4e-13 of the largest
entry, taken as 1e-12.
"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu
TOL = 1e-12


def _layers(m, which, precision_tunings, seed):
    import torch
    from paper_2511_21713_gb300 import pbfb
    n = m.n_m if which == pbfb.GAMMA_M else m.n_s
    x = torch.as_tensor(np.random.default_rng(seed).standard_normal(n) + 0.5, device="cuda")
    out = {}
    for key, (params, precision, tuning) in precision_tunings.items():
        m.apply_tuning(tuning)
        m.set_params(*params, precision)
        for op in (0, 1):
            y = torch.full((n,), np.nan, dtype=torch.float64, device="cuda")
            m.bem_apply(which, op, x, y)
            out[key, op] = y.cpu().numpy()
    m.apply_tuning({})
    return out


# triangles: 20 (one ragged tile), 80, 180 (point shares, step parts), 2880 (step parts), 3920, 13,520
# (several tiles per group in both precisions)
@pytest.mark.parametrize("nu", [1, 2, 3, 12, 14, 26])
def test_pair_far_fields_agree(nu):
    from paper_2511_21713_gb300 import inputs, pbfb
    case = inputs.sphere_case(nu=nu, a=4.0, R=6.0, layers=1)
    m = pbfb.Mesh.from_case(case)
    params = (case.eps_in, case.eps_out, case.kappa, case.T)
    kinds = {"fp64": (params, pbfb.FP64, {}), "ff": (params, pbfb.FLOAT2, {}),
             "ff few tasks": (params, pbfb.FLOAT2, dict(ff_kernel=4, ff_blocks_per_sm=1)),
             "ff many tasks": (params, pbfb.FLOAT2, dict(ff_kernel=3, ff_blocks_per_sm=64)),
             "ff one target": (params, pbfb.FLOAT2, dict(ff_kernel=1))}
    for which in (pbfb.GAMMA_M, pbfb.GAMMA_S):
        ys = _layers(m, which, kinds, 7 + nu)
        for (key, op), y in ys.items():
            ref = ys["fp64", op]
            assert np.isfinite(y).all()
            assert np.abs(y - ref).max() <= TOL * np.abs(ref).max(), (which, op, key)
    m.close()


# kappa: below the scaled kernel's range (float64 form), near its end, past the exponential's cut
# (kappa r up to 100 and 2400, where far contributions vanish)
@pytest.mark.parametrize("kappa", [1e-12, 1e-9, 1.01e-8, 1e-4, 10.0, 200.0])
def test_yukawa_range(kappa):
    from paper_2511_21713_gb300 import inputs, pbfb
    case = inputs.sphere_case(nu=4, a=4.0, R=6.0, layers=1, kappa=kappa)
    m = pbfb.Mesh.from_case(case)
    params = (case.eps_in, case.eps_out, kappa, case.T)
    ys = _layers(m, pbfb.GAMMA_S, {"fp64": (params, pbfb.FP64, {}), "ff": (params, pbfb.FLOAT2, {})}, 3)
    for op in (0, 1):
        a, b = ys["ff", op], ys["fp64", op]
        assert np.isfinite(a).all() and np.isfinite(b).all()
        assert np.abs(a - b).max() <= TOL * np.abs(b).max(), (kappa, op)
    m.close()


# the near-field rules (every pair class) with a kernel of almost no decay, of ordinary decay, and one that
# decays within a triangle (kappa h = 20); the float64 parity bound of the boundary operators, 1e-11
@pytest.mark.parametrize("kappa", [1e-9, 0.2, 8.0])
def test_corrections_over_kappa(kappa):
    import torch
    from oracle import bem
    from paper_2511_21713_gb300 import inputs, pbfb
    case = inputs.sphere_case(nu=3, a=4.0, R=6.0, layers=1, kappa=kappa)
    V, K = bem.assemble(bem.Surface(case.xyz, case.gs_tris), kappa)
    m = pbfb.Mesh.from_case(case)
    m.set_params(case.eps_in, case.eps_out, kappa, case.T, pbfb.FP64)
    x = np.random.default_rng(5).standard_normal(m.n_s)
    for op, A in ((0, V), (1, K)):
        y = torch.zeros(m.n_s, dtype=torch.float64, device="cuda")
        m.bem_apply(pbfb.GAMMA_S, op, torch.as_tensor(x, device="cuda"), y)
        ref = A @ x
        assert np.abs(y.cpu().numpy() - ref).max() <= 1e-11 * np.abs(ref).max(), (kappa, op)
    m.close()
