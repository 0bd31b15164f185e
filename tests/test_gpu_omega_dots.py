"""The relaxation factor's dots one by one: float-float loads of F(w), F'(w) du and F''(w) du^2 against float64's, each held
to its own size.  u and du are positive, c is 0 and p positive, so that r, r' and r'' have one sign and every product one
sign: a dot is its own sum of magnitudes, however small it is beside the others.

Tolerance: a point's value takes about ten float-float roundings of 2^-46, which the second orbit's negative weight can
raise by alpha / beta = 4.6; a dot multiplies two loads: 2 * 10 * 4.6 * 2^-46 = 1.3e-12, taken as 2e-12."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu
TOL = 2e-12


def dev(a):
    import torch
    return torch.as_tensor(np.ascontiguousarray(a, np.float64), device="cuda")


# vertices on both sides of the two-lanes-a-vertex rule (19,456 unknowns)
@pytest.mark.parametrize("nu,layers", [(2, 1), (14, 10)])
@pytest.mark.parametrize("scheme", ["HS", "T3", "T5", "T7"])
def test_each_dot_at_its_own_size(nu, layers, scheme):
    from paper_2511_21713_gb300 import inputs, pbfb
    case = inputs.sphere_case(nu=nu, a=4.0, R=8.0, layers=layers)
    m = pbfb.Mesh.from_case(case)
    rng = np.random.default_rng(nu)
    om = [0.25, 1.0, 2.0]
    for scale in (0.0, 1e-20, 1e-4, np.log(2.0) / 512, 0.7, 5.0, 55.0):
        u = scale * (0.5 + 0.5 * rng.random(m.n_v))
        du = 0.01 * (scale + 1e-3) * (0.5 + 0.5 * rng.random(m.n_v))
        zero = np.zeros(m.n)
        out = {}
        for prec in (pbfb.FP64, pbfb.MIXED):
            # float64's sinh is exact to 1e-16 absolutely: for the small fields its reference is T7 (F'' u^7 / 7! away)
            sch = pbfb.T7 if prec == pbfb.FP64 and scheme == "HS" and scale < 0.01 else getattr(pbfb, scheme)
            m.set_params(case.eps_in, case.eps_out, case.kappa, case.T, prec)
            a = m.omega_eval(sch, dev(u), dev(du), dev(zero), dev(zero), om)
            # p well below r', so that (p + r').p is r'.p
            p = zero.copy()
            if prec == pbfb.FP64:
                size = 1e-6 * np.sqrt(a[0, 2] / m.n_v)
                out["p"] = size * (0.5 + 0.5 * np.cos(np.arange(m.n_v)) ** 2)
            p[:m.n_v] = out["p"]
            out[prec] = a, m.omega_eval(sch, dev(u), dev(du), dev(zero), dev(p), om)
        (a0, b0), (a1, b1) = out[pbfb.FP64], out[pbfb.MIXED]
        for col in (0, 2, 3, 5):  # r'.r, r'.r', r.r'', r.r
            assert (a0[:, col] > 0).all()
            assert (np.abs(a1[:, col] - a0[:, col]) <= TOL * a0[:, col]).all(), (scale, col)
        for col in (1, 4, 6):  # r'.p, p.r'', p.r
            assert (b0[:, col] < 0).all()
            assert (np.abs(b1[:, col] - b0[:, col]) <= TOL * -b0[:, col]).all(), (scale, col)
    m.close()
