"""Range of the float64 element loops (assemble, omega_eval in PBFB_FP64)."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def dev(a):
    import torch
    return torch.as_tensor(np.ascontiguousarray(a, np.float64), device="cuda")


# e^800 and (1e60)^7 are past float64: the rule's weights are positive, so loads and Jacobian are infinite with F's and
# F''s sign, on one side of the orbit sums' range (700) as on the other; just inside it everything is finite
@pytest.mark.parametrize("scheme,past", [("HS", 800.0), ("HS", np.inf), ("T3", np.inf), ("T7", 1e60)])
def test_values_past_the_range_stay_infinite(scheme, past):
    from paper_2511_21713_gb300 import inputs, pbfb
    case = inputs.sphere_case(nu=2, a=4.0, R=6.0, layers=2)
    m = pbfb.Mesh.from_case(case)
    m.set_params(case.eps_in, case.eps_out, case.kappa, case.T, pbfb.FP64)
    zero = dev(np.zeros(m.n))

    def evaluate(u):
        N = dev(np.zeros(m.n_v))
        m.assemble(getattr(pbfb, scheme), dev(u), N)
        rp, col, val = m.fem_rows()
        fem = np.concatenate([val[a:b][col[a:b] < m.n_v] for a, b in zip(rp[:-1], rp[1:])])
        # the load again, at u = 0 + 1 du: r.r with r = -N(du), and at u + 1 * 0
        r = [m.omega_eval(getattr(pbfb, scheme), dev(x), dev(y), zero, zero, [1.0])[0, 5]
             for x, y in ((np.zeros(m.n_v), u), (u, np.zeros(m.n_v)))]
        return N.cpu().numpy(), fem, r

    for sign in (1.0, -1.0):
        N, J, r = evaluate(np.full(m.n_v, sign * past))
        assert (N == sign * np.inf).all() and (J == np.inf).all() and r == [np.inf, np.inf]
    inside = np.full(m.n_v, 699.0)
    N, J, _ = evaluate(inside)
    assert np.isfinite(N).all() and np.isfinite(J).all()
    m.close()


# the two forms meet at 700: a field across it against one scaled to either side, entry by entry; a point's exponent
# of 700 carries 14 roundings of 2^-53, 700 * 14 * 2^-53 = 1.1e-12 of a value
def test_both_forms_agree_at_the_edge_of_the_range():
    from paper_2511_21713_gb300 import inputs, pbfb
    case = inputs.sphere_case(nu=3, a=4.0, R=6.0, layers=2)
    m = pbfb.Mesh.from_case(case)
    m.set_params(case.eps_in, case.eps_out, case.kappa, case.T, pbfb.FP64)
    rng = np.random.default_rng(3)
    base = 690.0 + 9.0 * rng.random(m.n_v)
    out = []
    for u in (base, base + 2.0):  # below 700; partly above
        N = dev(np.zeros(m.n_v))
        m.assemble(pbfb.HS, dev(u), N)
        out.append((N.cpu().numpy() * np.exp(-300.0), m.fem_rows()[2] * np.exp(-300.0)))
    # sinh u and cosh u are e^u / 2 here, so that both scale by e^2
    for a, b in zip(*out):
        big = np.abs(a) > np.abs(a).max() * 1e-12  # the rest is the stiffness
        assert np.abs(b[big] / a[big] / np.exp(2.0) - 1.0).max() <= 2 * 1.1e-12
    m.close()
