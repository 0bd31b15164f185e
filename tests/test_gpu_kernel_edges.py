"""The inner PCG's forms, the winding numbers, the Coulomb sums and the dense single layer at the sizes where
their blocks, chunks and forms change."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def dev(a):
    import torch
    return torch.as_tensor(np.ascontiguousarray(a, np.float64), device="cuda")


# FEM rows: 24, 36 (most blocks of the cluster idle), 552 (a ragged warp), 11,772 / 11,808 (the float64 cluster
# form's last size, and past it), 15,862 / 16,240 (float32's), 72,036 / 80,212 (both block sizes of the
# grid-wide form), 149,812 / 155,574 (its last size, and past it; on 152 SMs).
# One GMRES step gives the preconditioned vector up to a factor; a few PCG steps before convergence, so every
# form gives the same iterate up to rounding: rows of at most about 30 terms, 7 steps, a tenfold growth per form
# and unit roundoff u: 2000 u, times 5 for the dot products' part = 1e4 u.
@pytest.mark.parametrize("nu,layers", [(1, 1), (1, 2), (3, 5), (14, 5), (7, 23), (12, 10), (9, 19), (20, 17), (27, 10),
                                       (24, 25), (24, 26)])
def test_inner_pcg_forms_agree(nu, layers):
    from paper_2511_21713_gb300 import inputs, pbfb
    case = inputs.sphere_case(nu=nu, a=4.0, R=8.0, layers=layers)
    m = pbfb.Mesh.from_case(case)
    assert m.n_v == (10 * nu * nu + 2) * (layers + 1)
    m.set_params(case.eps_in, case.eps_out, case.kappa, case.T)
    m.clear_jacobian()
    b = dev(np.random.default_rng(nu).standard_normal(m.n))
    for steps in (1, 7):
        z = {}
        for key, tuning in dict(sell=dict(pcg_lanes=1), f64=dict(pcg_precision=1), f32=dict(pcg_precision=2)).items():
            m.apply_tuning(tuning)
            x = dev(np.zeros(m.n))
            with pytest.raises(pbfb.PbfbError) as e:
                m.gmres(b, x, 1e-14, maxit=1, precond=pbfb.BLOCK, inner_iters=steps)
            assert e.value.code == 3
            y = x.cpu().numpy()[:m.n_v]
            z[key] = y / np.linalg.norm(y)
        assert np.linalg.norm(z["f64"] - z["sell"]) <= 1e4 * 2.0 ** -53, steps
        assert np.linalg.norm(z["f32"] - z["sell"]) <= 1e4 * 2.0 ** -24, steps
    m.close()


# a block takes 64 charges and a chunk of the triangles; the refused charge is the last one
@pytest.mark.parametrize("nq", [1, 64, 65, 1300])
@pytest.mark.parametrize("nu", [1, 7])
def test_charges_inside_check(nq, nu):
    from paper_2511_21713_gb300 import inputs, pbfb
    case = inputs.sphere_case(nu=nu, a=4.0, R=6.0, layers=1)
    m = pbfb.Mesh.from_case(case)
    rng = np.random.default_rng(nq)
    q = rng.standard_normal((nq, 3))
    q *= 3.0 / np.linalg.norm(q, axis=1)[:, None] * rng.random((nq, 1))
    m.charges_set(q, rng.standard_normal(nq))
    P = np.asarray(case.xyz)[np.asarray(case.gm_tris)[5]]
    # the face's plane test: 1e-12 of the product of the distances; a point off it by more belongs to a side
    n = np.cross(P[1] - P[0], P[2] - P[0])
    n /= np.linalg.norm(n) * np.sign(n @ P[0])
    c = P.mean(axis=0)
    for p, w in ((c, 0.5), (P[1], 0.5), (c + 1e-6 * n, 0.0), (2.0 * c, 0.0), (100.0 * c, 0.0)):
        bad = q.copy()
        bad[-1] = p
        with pytest.raises(pbfb.PbfbError) as e:
            m.charges_set(bad, np.ones(nq))
        assert e.value.code == 1
        assert f"charge {nq - 1} " in str(e.value) and f"winding number {w:.3f}" in str(e.value).replace("-0.000", "0.000")
    q[-1] = c - 1e-6 * n
    m.charges_set(q, np.ones(nq))
    m.close()


# the sums over the charges run in chunks (1300 of them: several per block); they are linear in the charges, so
# parts of the set add up to the whole: regrouped sums of float64 numbers, 1e-12 of the parts' magnitudes
@pytest.mark.parametrize("nu", [1, 5, 14])
def test_reaction_energies_add_up(nu):
    from paper_2511_21713_gb300 import inputs, pbfb
    case = inputs.sphere_case(nu=nu, a=4.0, R=6.0, layers=1)
    m = pbfb.Mesh.from_case(case)
    m.set_params(case.eps_in, case.eps_out, case.kappa, case.T)
    rng = np.random.default_rng(nu)
    q, z = 2.0 * (rng.random((1300, 3)) - 0.5), rng.standard_normal(1300)
    xL, xNL = (dev(0.1 * rng.standard_normal(m.n)) for _ in range(2))

    def energy(k):
        m.charges_set(q[k], z[k])
        return m.energy(xL, xNL)[1:3]
    parts = [energy(k) for k in (slice(0, 1), slice(1, 4), slice(4, 300), slice(300, 1300))]
    assert (np.abs(energy(slice(None)) - sum(parts)) <= 1e-12 * (1.0 + sum(map(np.abs, parts)))).all()
    m.close()


# triangles: 20, 1280 (one chunk), 1620, 3920 (several); columns of the float64 operator, symmetrised, against the
# float32 matrix: float32 weights and kernel values, sums of at most 36 * 36 of them in a few pieces: 16 * 2^-24
@pytest.mark.parametrize("nu", [1, 8, 9, 14])
def test_dense_single_layer_columns(nu):
    import torch
    from paper_2511_21713_gb300 import inputs, pbfb
    case = inputs.sphere_case(nu=nu, a=4.0, R=6.0, layers=1)
    m = pbfb.Mesh.from_case(case)
    m.set_params(case.eps_in, case.eps_out, case.kappa, case.T)
    for which, n in ((pbfb.GAMMA_M, m.n_m), (pbfb.GAMMA_S, m.n_s)):
        D = torch.zeros((n, n), dtype=torch.float32, device="cuda")
        m.single_layer_dense(which, 0, D)
        assert torch.equal(D, D.T)
        D = D.cpu().numpy().astype(np.float64)
        k = np.unique(np.r_[0, n // 3, n - 1])
        V = np.empty((n, k.size))
        for j, kj in enumerate(k):
            x, y = dev(np.zeros(n)), dev(np.zeros(n))
            x[kj] = 1.0
            m.bem_apply(which, 0, x, y)
            V[:, j] = y.cpu().numpy()
        S = 0.5 * (V[k] + V[k].T)
        assert np.abs(D[np.ix_(k, k)] - S).max() <= 2.0 ** -20 * np.abs(V).max()
        # V itself is symmetric up to the quadrature of near pairs
        assert np.abs(D[:, k] - V).max() <= 1e-3 * np.abs(V).max()
    m.close()


# float-float element kernels against the float64 ones, over the table's range: u near 0, at and between table
# points, past the first 512 of them (|u| > ln 2), up to the end of the float-float range (60) and past it, zeros,
# tiny and huge values; vertices on both sides of the two-lanes-a-vertex rule (19,456 unknowns), one and several
# omegas.  Each sum has 24 tets of 14 points, a product of a few roundings of 2^-47 each: 1e-12 of the sum of
# magnitudes, which is at most the largest entry where all terms have a sign.
@pytest.mark.parametrize("nu,layers", [(2, 1), (9, 20), (14, 10)])
@pytest.mark.parametrize("scheme", ["HS", "T3", "T7"])
def test_float_float_elements(nu, layers, scheme):
    from paper_2511_21713_gb300 import inputs, pbfb
    case = inputs.sphere_case(nu=nu, a=4.0, R=8.0, layers=layers)
    m = pbfb.Mesh.from_case(case)
    rng = np.random.default_rng(nu)
    for scale in (0.0, 1e-20, 1e-4, np.log(2.0) / 512, 0.7, 5.0, 59.0, 70.0):
        u = scale * rng.random(m.n_v)
        u[::7] = scale
        du = 0.01 * (scale + 1e-3) * rng.random(m.n_v)
        c, p = rng.standard_normal(m.n), rng.standard_normal(m.n)
        out = {}
        for prec in (pbfb.FP64, pbfb.MIXED):
            # float64's sinh is exact to 1e-16 absolutely: for the small fields its reference is T7 (u^9 / 9! away)
            sch = pbfb.T7 if prec == pbfb.FP64 and scheme == "HS" and scale < 0.01 else getattr(pbfb, scheme)
            m.set_params(case.eps_in, case.eps_out, case.kappa, case.T, prec)
            N = dev(np.zeros(m.n_v))
            m.assemble(sch, dev(u), N)
            om = [m.omega_eval(sch, dev(u), dev(du), dev(c), dev(p), o) for o in ([0.5], [0.0, 0.25, 0.5, 1.0, 2.0])]
            out[prec] = N.cpu().numpy(), m.fem_rows()[2], om
        (N0, J0, o0), (N1, J1, o1) = out[pbfb.FP64], out[pbfb.MIXED]
        assert np.abs(N1 - N0).max() <= 1e-12 * np.abs(N0).max() + 1e-300
        assert np.abs(J1 - J0).max() <= 1e-12 * np.abs(J0).max()
        for a, b in zip(o0, o1):
            # every dot is at most |p + r'| or |r| times another: bounded by the batch's largest squares
            assert np.isfinite(a).all()
            assert np.abs(a - b).max() <= 1e-12 * np.abs(a).max() * np.sqrt(m.n)
        assert np.allclose(o1[0][0], o1[1][2], rtol=1e-13, atol=1e-13 * np.abs(o1[1]).max())
    m.close()


# the flux's vector steps take 256 threads to 4096 vertices and 1024 above: 12, 4002 and 4412 vertices.  The flux of a
# solution of V lam = rhs: V lam, from the operator itself, gives rhs back to CG's 1e-13 of its norm, plus the far
# field's rounding (1e-14 a product)
@pytest.mark.parametrize("nu", [1, 20, 21])
def test_flux_residual(nu):
    from paper_2511_21713_gb300 import inputs, pbfb
    case = inputs.sphere_case(nu=nu, a=4.0, R=6.0, layers=1)
    m = pbfb.Mesh.from_case(case)
    m.set_params(case.eps_in, case.eps_out, case.kappa, case.T, pbfb.FLOAT2)
    rng = np.random.default_rng(nu)
    x, lam, V, K = dev(rng.standard_normal(m.n)), dev(np.zeros(m.n_m)), dev(np.zeros(m.n_m)), dev(np.zeros(m.n_m))
    m.gamma_m_flux(x, 0, lam)
    u = x[dev(m.surface_vertices(pbfb.GAMMA_M)).long()].contiguous()
    m.bem_apply(pbfb.GAMMA_M, 0, lam, V)
    m.bem_apply(pbfb.GAMMA_M, 1, u, K)
    tri = np.searchsorted(np.unique(case.gm_tris), np.asarray(case.gm_tris))
    P, un = np.asarray(case.xyz)[np.asarray(case.gm_tris)], u.cpu().numpy()
    area = 0.5 * np.linalg.norm(np.cross(P[:, 1] - P[:, 0], P[:, 2] - P[:, 0]), axis=1)
    mass = np.zeros(m.n_m)
    for a in range(3):  # rows of the mass matrix: area / 12 (1 + [a = b])
        np.add.at(mass, tri[:, a], area / 12.0 * (un[tri].sum(axis=1) + un[tri[:, a]]))
    rhs = 0.5 * mass + K.cpu().numpy()
    assert np.linalg.norm(V.cpu().numpy() - rhs) <= 5e-13 * np.linalg.norm(rhs)
    m.close()
