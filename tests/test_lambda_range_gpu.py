"""The leading eigenvalue of gamma chi~ over the range of magnitudes its inputs reach: atoms at low
temperature give |lambda| up to 1e9, at high temperature down to 1e-13, against LAPACK.  Where the second
largest modulus is below half of the largest, the iteration settles (0.5^64 < 2e-6, then 24 steps
more), and the bound is the eigenvalue check's stated 1e-8."""
import numpy as np
import pytest

from oracle import df_oracle as O
from paper_1507_00895_gb300 import inputs as I

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def df():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_1507_00895_gb300 import build
    build.build_lib()
    from paper_1507_00895_gb300 import df as dfm
    return dfm


def check(lam, ok, gammas, chi):
    seen = 0
    assert np.all(np.isfinite(lam))
    for c, g in enumerate(gammas):
        for q in range(chi.shape[2]):
            ev = np.linalg.eigvals(g[0] * chi[0, :, q][None, :])
            ev = ev[np.argsort(-np.abs(ev))]
            assert (abs(lam[c, 0, q]) >= 1.0) == (abs(ev[0]) >= 1.0), (c, q)
            if abs(ev[1]) > 0.5 * abs(ev[0]):
                continue
            seen += 1
            assert ok[c, 0, q] == 1, (c, q)
            assert abs(lam[c, 0, q] - ev[0]) <= 1e-8 * abs(ev[0]), (c, q, lam[c, 0, q], ev[0])
    assert seen


@pytest.mark.parametrize("n_w", [8, 48, 96])
@pytest.mark.parametrize("p", [-12, -9, -6, -3, 3, 6, 9, 12])
def test_scaled_vertex(df, n_w, p):
    w = I.random_nonsymmetric(n_w, 0, 1, 16, seed=300 + n_w, scale=0.7)
    w.gamma_uu[:] += 3.0 * np.linspace(0.5, 1.0, n_w)[:, None]       # a dominant rank-one part
    w.gamma_ud[:] *= 0.2
    w = w.scaled(10.0 ** p)
    with df.DualFermion.from_workload(w, eig_mode=2) as d:
        d.bubble()
        d.bse(3)
        lam, ok = d.get_lambda()
        check(lam, ok, O.channel_vertices(w.gamma_uu, w.gamma_ud), d.get_chi())


@pytest.mark.parametrize("U,beta,n_w", [(2.0, 35.0, 64), (2.0, 40.0, 64), (2.0, 60.0, 64), (2.0, 50.0, 128),
                                        (1.0, 200.0, 64), (0.1, 0.01, 16)])
def test_half_filled_atom_at_both_ends_of_temperature(df, U, beta, n_w):
    w = I.half_filled_atom("t", 2, 8, U=U, beta=beta, n_w=n_w, m_max=0)
    with df.DualFermion.from_workload(w, eig_mode=1) as d:
        d.bubble()
        d.bse(3)
        lam, ok = d.get_lambda()
        if beta == 200.0:                # every pair of moduli within 1%: no system settles
            assert np.all(np.isfinite(lam)) and np.all(np.abs(lam) >= 1.0)
        else:
            check(lam, ok, O.channel_vertices(w.gamma_uu, w.gamma_ud), d.get_chi())
    with df.DualFermion.from_workload(w, eig_mode=1) as d:
        assert d.iterate(1)[2] == (df.DF_WARN_LADDER_RADIUS if U >= 1.0 else df.DF_OK)


def test_radius_order_far_outside_the_radius(df):
    # every ladder of W = 0 has |lambda| between 1.4e4 and 7.2e7: all take the low-order evaluation
    w = I.half_filled_atom("t", 2, 4, U=2.0, beta=35.0, n_w=64, m_max=0)
    st = O.run_workload(w, n_iter=1, radius_order=2)
    with df.DualFermion.from_workload(w, eig_mode=2, radius_order=2) as d:
        d.iterate(1)
        sig = d.get_sigma()
    assert np.max(np.abs(sig - st.sigmas[0])) < 1e-10 * np.max(np.abs(st.sigmas[0]))


def test_start_vector_that_is_nearly_annihilated(df):
    # chi~ = -1/16 everywhere (1D, N_k = 2, t = 0, g = Delta = 1, beta = 4), and gamma takes the uniform
    # start vector to 2^-22 h1, that to 2^-44 h2 and 2^-66 h3, whose eigenvalue 1 is the only one that is not 0:
    # growths of 2^-22 three times and then 1
    h = 0.5 * np.array([[1, 1, 1, 1], [1, -1, 1, -1], [1, 1, -1, -1], [1, -1, -1, 1]], float)
    e = 2.0 ** -22
    A = e * (np.outer(h[1], h[0]) + np.outer(h[2], h[1]) + np.outer(h[3], h[2])) + np.outer(h[3], h[3])
    g = np.ones(4, complex)
    gam = (-16.0 * A).astype(complex)[None]
    with df.DualFermion(dim=1, nk=2, t=0.0, tp=0.0, beta=4.0, mu=0.0, n_w=4, m_max=0, g=g, delta=g,
                        gamma_d=gam, gamma_m=2.0 ** 40 * gam, eig_mode=2) as d:
        d.bubble()
        assert np.array_equal(d.get_chi(), np.full((1, 4, 2), -1.0 / 16.0, complex))
        d.bse(3)
        lam, ok = d.get_lambda()
    assert np.all(ok == 1)
    assert np.max(np.abs(lam[0] - 1.0)) < 1e-8 and np.max(np.abs(lam[1] * 2.0 ** -40 - 1.0)) < 1e-8


def test_zero_vertex(df):
    g = np.ones(4, complex)
    gam = np.zeros((1, 4, 4), complex)
    with df.DualFermion(dim=1, nk=2, t=0.0, tp=0.0, beta=4.0, mu=0.0, n_w=4, m_max=0, g=g, delta=g,
                        gamma_d=gam, gamma_m=gam, eig_mode=2) as d:
        assert d.iterate(1)[2] == df.DF_OK
        lam, ok = d.get_lambda()
    assert np.all(lam == 0.0) and np.all(ok == 1)


def test_product_at_the_end_of_the_fp32_range(df):
    # chi~ = -T G0~^2 = -2^127 (g = 2^63, Delta = 1 / g: G0~ = -g / 2) and gamma = -2^126 diag(1, 1/4): lambda = 2^253
    g = np.full(2, 2.0 ** 63, complex)
    d_ = np.full(2, 2.0 ** -63, complex)
    gam = np.diag([-(2.0 ** 126), -(2.0 ** 124)]).astype(complex)[None]
    for up in (1.0, 2.0, 1.75):
        with df.DualFermion(dim=1, nk=2, t=0.0, tp=0.0, beta=0.125, mu=0.0, n_w=2, m_max=0, g=g, delta=d_,
                            gamma_d=up * gam, gamma_m=gam, eig_mode=2) as d:
            d.bubble()
            chi = d.get_chi()
            d.bse(3)
            lam, ok = d.get_lambda()
        assert np.all(chi == chi[0, 0, 0]) and chi[0, 0, 0] == -(2.0 ** 127)
        ref = up * gam[0, 0, 0] * chi[0, 0, 0]
        assert np.max(np.abs(lam[0] - ref)) < 1e-8 * abs(ref), (lam[0], ref)


@pytest.mark.parametrize("n_w", [8, 48, 128])
@pytest.mark.parametrize("p,q", [(-290, 0), (-60, 40), (45, -45), (60, 60), (250, 20), (41, 39)])
def test_vertex_and_bubble_far_from_one(df, n_w, p, q):
    """gamma by 2^p and beta by 2^-q (chi~ has the prefactor T): lambda is scaled by 2^(p + q), FP64's
    eigenvalues with it, wherever gamma's or chi~'s FP32 words would lie."""
    w = I.random_nonsymmetric(n_w, 0, 1, 4, seed=500 + n_w, scale=0.7)
    w.gamma_uu[:] += 3.0 * np.linspace(0.5, 1.0, n_w)[:, None]
    w.gamma_ud[:] *= 0.2
    lam = []
    for a, b in ((0, 0), (p, q)):
        v = w.scaled(2.0 ** a)
        v.beta = w.beta * 2.0 ** -b
        with df.DualFermion.from_workload(v, eig_mode=2) as d:
            d.bubble()
            chi = d.get_chi()
            d.bse(3)
            lam.append(d.get_lambda())
    ref = lam[0][0] * 2.0 ** p * 2.0 ** q
    assert np.array_equal(lam[0][1], lam[1][1])
    m = lam[0][1] == 1
    assert np.any(m)
    assert np.max(np.abs(lam[1][0] - ref)[m] / np.abs(ref)[m]) < 1e-8
