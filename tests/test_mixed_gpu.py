"""Mixed-precision ladder solves (DF_FP32_IR) against the CPU oracle.

FP32 factorisation + one correction with an extended-precision residual, and
per-ladder error control: a ladder whose predicted error rho^2 exceeds
ladder_tol (1e-9) is solved again by the FP64 LU.  Stated tolerance of the
refined mixed path (the bound for refined mixed-precision results): Sigma~
and every ladder-kernel (channel, W) plane within 1e-8 of the oracle,
normwise.
"""
import numpy as np
import pytest

from oracle import df_oracle as O
from paper_1507_00895_gb300 import inputs as I

pytestmark = pytest.mark.gpu

TOL_KERNEL = 1e-8
TOL_SIGMA = 1e-8


@pytest.fixture(scope="module")
def df():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_1507_00895_gb300 import build
    build.build_lib()
    from paper_1507_00895_gb300 import df as dfm
    return dfm


def nrel(a, b):
    return float(np.max(np.abs(a - b)) / max(np.max(np.abs(b)), 1e-300))


def erel(a, b, floor=1e-6):
    """Largest elementwise relative difference over the elements of b above floor * max |b|."""
    m = np.abs(b) > floor * np.max(np.abs(b))
    return float(np.max(np.abs(a - b)[m] / np.abs(b)[m]))


def oracle_first_pass(w):
    eps = O.dispersion(w.dim, w.nk, w.t, w.tp)
    g0 = O.bare_dual_g(w.g, w.delta, eps)
    gd, gm = O.channel_vertices(w.gamma_uu, w.gamma_ud)
    st = O.LoopState(g0_ext=g0, sigma=np.zeros((w.n_w, w.N), complex))
    O.one_iteration(st, gd, gm, w.n_w, w.m_max, w.beta, w.dim, w.nk)
    kd = st.gd_diag - 0.5 * O.second_order_diag(gd, st.chi)
    km = 3.0 * (st.gm_diag - 0.5 * O.second_order_diag(gm, st.chi))
    return st, np.stack([kd, km])


CASES = [
    ("square16_b5", dict(nk=4, n_w=2, m_max=0)),          # n_w=2 padded to 4
    ("square16_b5", dict(nk=8, n_w=6, m_max=1)),          # ragged pad
    ("paper_u20", dict(nk=8, n_w=16, m_max=1)),
    ("square32_tp", dict(nk=8, n_w=30, m_max=2)),
    ("square16_b5", dict()),                              # 16^2, n_w=32
]


@pytest.mark.parametrize("name,kw", CASES)
def test_mixed_first_pass(df, name, kw):
    w = I.workload(name, **kw)
    st, kref = oracle_first_pass(w)
    with df.DualFermion.from_workload(w, precision=df.DF_FP32_IR) as d:
        d.bubble()
        d.bse(3)
        kern = d.get_kernel()
        for c in range(2):
            for a in range(w.n_bos):
                assert nrel(kern[c, a], kref[c, a]) < TOL_KERNEL, (c, a)
        d.sigma()
        assert nrel(d.get_sigma(), st.sigma) < TOL_SIGMA


def test_mixed_square32_tp_full_size(df):
    # the benchmark workload: 30,720 ladders of order 64, cond up to ~1e6
    w = I.workload("square32_tp")
    st, kref = oracle_first_pass(w)
    with df.DualFermion.from_workload(w, precision=df.DF_FP32_IR) as d:
        d.bubble()
        d.bse(3)
        kern = d.get_kernel()
        worst = max(nrel(kern[c, a], kref[c, a]) for c in range(2) for a in range(w.n_bos))
        assert worst < TOL_KERNEL, worst
        worst_rho2, back = d.ladder_stats()
        d.sigma()
        err = nrel(d.get_sigma(), st.sigma)
        print(f"square32_tp mixed: worst kernel plane {worst:.2e}, Sigma~ {err:.2e}, "
              f"handed back {back} of {2 * w.n_bos * w.N}, worst rho^2 {worst_rho2:.1e}")
        assert err < TOL_SIGMA
        assert erel(d.get_sigma(), st.sigma) < TOL_SIGMA
        assert back < 0.05 * 2 * w.n_bos * w.N


def test_mixed_matches_fp64_gpu_over_iterations(df):
    # teacher-free comparison of the two GPU paths on the convergent paper workload
    w = I.workload("paper_u20", nk=16, n_w=48, m_max=1)
    with df.DualFermion.from_workload(w) as d64, \
            df.DualFermion.from_workload(w, precision=df.DF_FP32_IR) as d32:
        i64, r64, _ = d64.iterate(25, tol=1e-12)
        i32, r32, _ = d32.iterate(25, tol=1e-12)
        assert r64 <= 1e-12 and r32 <= 1e-12
        assert nrel(d32.get_sigma(), d64.get_sigma()) < TOL_SIGMA


LARGE = [
    ("cubic16_crit", dict(nk=4, n_w=96, m_max=1)),         # the 3D workload's order
    ("square16_b5", dict(nk=4, n_w=66, m_max=1)),          # 2n threads not a warp multiple
    ("paper_u20", dict(nk=4, n_w=128, m_max=0)),           # the largest order
]


@pytest.mark.parametrize("sweep", [0, 1])
@pytest.mark.parametrize("name,kw", LARGE)
def test_mixed_large_orders_first_pass(df, name, kw, sweep):
    # 64 < n_w <= 128: FP32 Gauss-Jordan inverse (on the tensor cores, sweep 0, or the
    # CUDA cores, sweep 1) + one double-float-residual correction
    w = I.workload(name, **kw)
    st, kref = oracle_first_pass(w)
    with df.DualFermion.from_workload(w, precision=df.DF_FP32_IR, mixed_sweep=sweep) as d:
        d.bubble()
        d.bse(3)
        kern = d.get_kernel()
        for c in range(2):
            for a in range(w.n_bos):
                assert nrel(kern[c, a], kref[c, a]) < TOL_KERNEL, (c, a)
        d.sigma()
        assert nrel(d.get_sigma(), st.sigma) < TOL_SIGMA


def test_mixed_large_order_over_iterations(df):
    # the 3D critical workload's order, three passes, against the GPU FP64 path
    w = I.workload("cubic16_crit", nk=4, n_w=96, m_max=2)
    with df.DualFermion.from_workload(w) as d64, \
            df.DualFermion.from_workload(w, precision=df.DF_FP32_IR) as d32:
        d64.iterate(3)
        d32.iterate(3)
        assert nrel(d32.get_sigma(), d64.get_sigma()) < TOL_SIGMA


def test_mixed_error_control_hands_back(df):
    # ladder_tol below any attainable rho^2: every ladder is solved again by the
    # FP64 LU, and the kernel equals the FP64 path's bit for bit
    w = I.workload("square32_tp", nk=8, n_w=40, m_max=1)
    with df.DualFermion.from_workload(w) as d64:
        d64.bubble()
        d64.bse(3)
        k64 = d64.get_kernel()
    with df.DualFermion.from_workload(w, precision=df.DF_FP32_IR, ladder_tol=1e-300) as d:
        d.bubble()
        d.bse(3)
        worst, back = d.ladder_stats()
        assert back == 2 * w.n_bos * w.N and worst > 0.0
        assert np.array_equal(d.get_kernel(), k64)
    # the default bound: a few ill-conditioned ladders are handed back, the rest
    # keep their mixed results, within the stated bound of the FP64 path
    with df.DualFermion.from_workload(w, precision=df.DF_FP32_IR) as d:
        d.bubble()
        d.bse(3)
        worst, back = d.ladder_stats()
        assert 0.0 < worst and back < 0.05 * 2 * w.n_bos * w.N
        kmix = d.get_kernel()
        for c in range(2):
            for a in range(w.n_bos):
                assert nrel(kmix[c, a], k64[c, a]) < TOL_KERNEL, (c, a)


def test_mixed_error_control_reports_without_fallback(df):
    # ladder_fallback = 0: a ladder above ladder_tol keeps its mixed result and the
    # pass reports DF_ERR_REFINE_STALL
    w = I.workload("square32_tp", nk=4, n_w=16, m_max=1)
    with df.DualFermion.from_workload(w, precision=df.DF_FP32_IR, ladder_tol=1e-300, ladder_fallback=0) as d:
        with pytest.raises(df.DFError) as e:
            d.iterate(1)
        assert e.value.status == df.DF_ERR_REFINE_STALL
    w = I.workload("cubic16_crit", nk=4, n_w=96, m_max=0)   # the large-order kernel
    with df.DualFermion.from_workload(w, precision=df.DF_FP32_IR, ladder_tol=1e-300, ladder_fallback=0) as d:
        with pytest.raises(df.DFError) as e:
            d.iterate(1)
        assert e.value.status == df.DF_ERR_REFINE_STALL


@pytest.mark.parametrize("n_w", [12, 80])
def test_mixed_ill_conditioned_ladder_is_handed_back(df, n_w):
    # one ladder made nearly singular: the magnetic vertex of W = 0 is rescaled so
    # that gamma chi~ of one q has an eigenvalue 1 - 1e-9 (cond(D) ~ 1e9 there).  Its
    # FP32 factorisation cannot deliver, the error control hands it to the FP64 LU,
    # and the mixed kernel then matches the FP64 path on every plane
    w = I.workload("paper_u20", nk=4, n_w=n_w, m_max=0)
    st, _ = oracle_first_pass(w)
    gd, gm = O.channel_vertices(w.gamma_uu, w.gamma_ud)
    q = 5
    ev = np.linalg.eigvals(gm[0] * st.chi[0, :, q][None, :])
    lead = ev[np.argmax(np.abs(ev))]
    gm = gm * ((1.0 - 1e-9) / lead)
    D = np.eye(n_w) - gm[0] * st.chi[0, :, q][None, :]
    assert np.linalg.cond(D) > 1e8
    kw = dict(dim=w.dim, nk=w.nk, t=w.t, tp=w.tp, beta=w.beta, mu=w.mu, n_w=w.n_w, m_max=w.m_max, g=w.g,
              delta=w.delta, gamma_d=gd, gamma_m=gm)
    with df.DualFermion(**kw) as d64:
        d64.bubble()
        d64.bse(3)
        k64 = d64.get_kernel()
    with df.DualFermion(precision=df.DF_FP32_IR, **kw) as d:
        d.bubble()
        d.bse(3)
        worst, back = d.ladder_stats()
        kmix = d.get_kernel()
    assert back >= 1 and worst > 1e-9
    # the handed-back ladder is the FP64 path's, bit for bit
    assert np.array_equal(kmix[1, 0, :, q], k64[1, 0, :, q])
    for c in range(2):
        assert nrel(kmix[c, 0], k64[c, 0]) < TOL_KERNEL, c


def test_mixed_cubic16_full_size_against_the_oracle(df):
    # the 3D workload at its stated size (16^3, n_w = 96, 21 bosonic frequencies,
    # 172,032 ladders of order 96): one mixed pass, the whole Sigma~ and every
    # ladder-kernel plane against the oracle (its ladders over a spawned pool)
    import oracle_pool
    w = I.workload("cubic16_crit")
    sig_ref, kref = oracle_pool.first_pass(w)
    with df.DualFermion.from_workload(w, precision=df.DF_FP32_IR) as d:
        d.bubble()
        d.bse(3)
        kern = d.get_kernel()
        worst_rho2, back = d.ladder_stats()
        d.sigma()
        sig = d.get_sigma()
    worst = max(nrel(kern[c, a], kref[c, a]) for c in range(2) for a in range(w.n_bos))
    err = nrel(sig, sig_ref)
    print(f"cubic16_crit mixed: worst kernel plane {worst:.2e}, Sigma~ {err:.2e} (elementwise "
          f"{erel(sig, sig_ref):.2e}), handed back {back}, worst rho^2 {worst_rho2:.1e}")
    assert worst < TOL_KERNEL
    assert err < TOL_SIGMA and erel(sig, sig_ref) < TOL_SIGMA


def test_tensor_core_sweep_matches_the_cuda_core_sweep(df):
    # the two FP32 Gauss-Jordan inversions of the large-order kernel (tcgen05 panel
    # updates with three-piece BF16 operands vs FP32 FMAs) give the same corrected
    # ladders within the mixed bound, and both within it of the FP64 path
    w = I.workload("cubic16_crit", nk=4, n_w=96, m_max=2)
    out = {}
    for sweep in (0, 1):
        with df.DualFermion.from_workload(w, precision=df.DF_FP32_IR, mixed_sweep=sweep) as d:
            d.bubble()
            d.bse(3)
            out[sweep] = d.get_kernel()
    with df.DualFermion.from_workload(w) as d:
        d.bubble()
        d.bse(3)
        k64 = d.get_kernel()
    for c in range(2):
        for a in range(w.n_bos):
            assert nrel(out[0][c, a], out[1][c, a]) < TOL_KERNEL
            assert nrel(out[0][c, a], k64[c, a]) < TOL_KERNEL


@pytest.mark.parametrize("n_w", [34, 40, 42, 48, 50, 58, 62, 64])
@pytest.mark.parametrize("wide", [False, True])
def test_mixed_two_ladder_blocks(df, n_w, wide):
    """Orders 33-64 where the kernel's tiles end (8-column panels, 16-row digit blocks, odd ladder
    counts: three orbits per plane), complex vertices without symmetry, each channel alone and both
    together; with `wide` the vertex's columns span twelve orders of magnitude and one is zero (the
    digits are relative to a power of two per column).  Bound: the stated one of the mixed path
    (each ladder's predicted error <= 1e-9 of its diag Gamma, or the FP64 solve)."""
    w = I.random_nonsymmetric(n_w, 1, 1, 4, seed=n_w, scale=0.5)
    if wide:
        s = 10.0 ** np.random.default_rng(n_w).uniform(-9.0, 3.0, n_w)
        s[n_w // 3] = 0.0
        w.gamma_uu = w.gamma_uu * s
        w.gamma_ud = w.gamma_ud * s
    _, kref = oracle_first_pass(w)
    with df.DualFermion.from_workload(w, precision=df.DF_FP32_IR, symmetry=1, eig_mode=0) as d:
        d.bubble()
        for mask, chans in ((1, (0,)), (2, (1,)), (3, (0, 1))):
            d.bse(mask)
            kern = d.get_kernel()
            for c in chans:
                for a in range(w.n_bos):
                    assert nrel(kern[c, a], kref[c, a]) < TOL_KERNEL, (mask, c, a)
        # the digit product carries T = S gamma to ~2^-47 of max|S_i| max|gamma_j|: what is left is the
        # FP32 sweep's error squared, far below the bound on these well-conditioned ladders
        assert nrel(kern, kref) < 1e-11


@pytest.mark.parametrize("n_w", [66, 72, 80, 94, 96, 98, 112, 126, 128])
@pytest.mark.parametrize("wide", [False, True])
def test_mixed_streamed_digits(df, n_w, wide):
    """Orders 65-128 where the kernel's tiles end (8-column panels, 16-row blocks, 64-column tiles,
    pieces of 32 K of the streamed digits), the same inputs and bound as for the orders below."""
    test_mixed_two_ladder_blocks(df, n_w, wide)


def test_mixed_orders_share_a_batch_class(df):
    """A batch's large-order class runs every order on the largest one's shared-memory layout."""
    ws = [I.half_filled_atom(f"b{n}", 1, 8, U=3.0 + 0.01 * n, beta=2.0, n_w=n, m_max=1) for n in (128, 66, 96, 80)]
    with df.DualFermionBatch(ws, precision=df.DF_FP32_IR) as b:
        b.iterate(1)
        for i, w in enumerate(ws):
            st, _ = oracle_first_pass(w)
            assert nrel(b.get_sigma(i), st.sigma) < TOL_SIGMA, w.n_w


@pytest.mark.parametrize("n_w", [2, 6, 8, 10, 14, 16, 18, 24, 26, 30, 32])
@pytest.mark.parametrize("wide", [False, True])
def test_mixed_ladder_per_warp(df, n_w, wide):
    """Orders up to 32 where the kernel's tiles end (padded orders 16 and 32, 8-column and 16-row
    product tiles, one or two lanes per row), the same inputs and bound as for the orders above."""
    test_mixed_two_ladder_blocks(df, n_w, wide)


def test_mixed_small_orders_share_a_batch_class(df):
    """Orders of one padded order in one queue; the points end inside a block's take, and a plane has
    more ladders than a block has warps."""
    ws = [I.half_filled_atom(f"b{n}", 1, 32, U=3.0 + 0.01 * n, beta=2.0, n_w=n, m_max=1)
          for n in (2, 32, 16, 18, 10, 30, 24)]
    with df.DualFermionBatch(ws, precision=df.DF_FP32_IR) as b:
        b.iterate(1)
        for i, w in enumerate(ws):
            st, _ = oracle_first_pass(w)
            assert nrel(b.get_sigma(i), st.sigma) < TOL_SIGMA, w.n_w


@pytest.mark.parametrize("n_w", [12, 40, 48, 80, 96, 98, 128])
def test_single_hand_back_is_split(df, n_w):
    """One nearly singular ladder (as above): a list this short is split into ranges of 16 right-hand sides
    (remainders at 40, 48 and 98), in shared memory up to order 96.  In a batch and on a handle the
    result is the FP64 path's for that ladder, so Sigma~ is within the mixed path's bound of it although the
    ladder's FP32 factorisation has no digit left."""
    w = I.workload("paper_u20", nk=4, n_w=n_w, m_max=0)
    st, _ = oracle_first_pass(w)
    gd, gm = O.channel_vertices(w.gamma_uu, w.gamma_ud)
    ev = np.linalg.eigvals(gm[0] * st.chi[0, :, 5][None, :])
    gm = gm * ((1.0 - 1e-9) / ev[np.argmax(np.abs(ev))])
    w.gamma_uu, w.gamma_ud = (gd + gm) / 2, (gd - gm) / 2
    with df.DualFermion.from_workload(w) as d64, df.DualFermion.from_workload(w, precision=df.DF_FP32_IR) as d:
        for h in (d64, d):
            h.bubble()
            h.bse(3)
        assert d.ladder_stats()[1] >= 1
        assert np.array_equal(d.get_kernel()[1, 0, :, 5], d64.get_kernel()[1, 0, :, 5])
    with df.DualFermionBatch([w]) as b64, df.DualFermionBatch([w], precision=df.DF_FP32_IR) as b:
        b64.iterate(1)
        b.iterate(1)
        assert nrel(b.get_sigma(0), b64.get_sigma(0)) < TOL_SIGMA


def rounds_to_singular(n, m_max=0):
    """Ladders that are exactly singular once D is rounded to FP32 and regular in FP64: g = Delta = 1,
    t = 0, N_k = 2, beta = 4 give chi~ = -1/16 exactly, and D = 1 + gamma / 16 is the identity but for
    [[2, 1], [2, 1 + 2^-30]] in its first and last rows and columns; every step of its LU is exact."""
    gam = np.zeros((1, n, n), complex)
    gam[0, 0, 0], gam[0, 0, n - 1], gam[0, n - 1, 0], gam[0, n - 1, n - 1] = 16.0, 16.0, 32.0, 16.0 * 2.0 ** -30
    g = np.ones(n, complex)
    return I.Workload("singular32", 1, 2, 0.0, 0.0, 1.0, 4.0, 0.0, n, 0, g, g, gam, np.zeros_like(gam))


@pytest.mark.parametrize("n_w,sweep", [(2, 0), (16, 0), (18, 0), (32, 0), (34, 0), (64, 0), (66, 0), (128, 0), (96, 1)])
def test_zero_fp32_pivot_is_left_to_the_fp64_solve(df, n_w, sweep):
    w = rounds_to_singular(n_w)
    with df.DualFermion.from_workload(w, eig_mode=0) as d:
        assert d.iterate(1)[2] == df.DF_OK
        ref, kref = d.get_sigma(), d.get_kernel()
    with df.DualFermion.from_workload(w, precision=df.DF_FP32_IR, eig_mode=0, mixed_sweep=sweep) as d:
        assert d.iterate(1)[2] == df.DF_OK
        assert d.ladder_stats()[1] == 4                     # 2 channels x 1 plane x 2 momenta
        assert nrel(d.get_kernel(), kref) < 1e-12 and nrel(d.get_sigma(), ref) < 1e-12
    # without the second solve it is reported
    with df.DualFermion.from_workload(w, precision=df.DF_FP32_IR, eig_mode=0, mixed_sweep=sweep, ladder_fallback=0) as d:
        with pytest.raises(df.DFError) as e:
            d.iterate(1)
        assert e.value.status == df.DF_ERR_SINGULAR


def test_zero_fp32_pivot_in_a_batch(df):
    ws = [rounds_to_singular(n) for n in (2, 18, 34, 66)]
    with df.DualFermionBatch(ws, precision=df.DF_FP32_IR) as b:
        b.iterate(1)
        for i, w in enumerate(ws):
            with df.DualFermion.from_workload(w, eig_mode=0) as d:
                d.iterate(1)
                assert nrel(b.get_sigma(i), d.get_sigma()) < 1e-12, w.n_w


@pytest.mark.parametrize("n_w,m_max", [(24, 3), (32, 3), (40, 4), (42, 4), (48, 4), (64, 3), (66, 2), (96, 2), (98, 2)])
def test_long_hand_back_list(df, n_w, m_max):
    """Lists longer than the blocks that run at once with their factors in shared memory (order 24: chunk lists only),
    and one just as long as a plane: every ladder is the FP64 path's, bit for bit, on a handle, and the batch's
    Sigma~ is within the FP64 parity bound."""
    w = I.random_nonsymmetric(n_w, m_max, 1, 64, seed=n_w, scale=0.5)
    with df.DualFermion.from_workload(w, eig_mode=0) as d64, \
            df.DualFermion.from_workload(w, precision=df.DF_FP32_IR, eig_mode=0, ladder_tol=1e-300) as d:
        d64.iterate(1)
        d.bubble()
        for mask, count in ((1, w.n_bos * w.N), (3, 2 * w.n_bos * w.N)):
            d.bse(mask)
            assert d.ladder_stats()[1] == count
            k, k64 = d.get_kernel(), d64.get_kernel()
            assert np.array_equal(k if mask == 3 else k[:1], k64 if mask == 3 else k64[:1])
        d.sigma()
        assert np.array_equal(d.get_sigma(), d64.get_sigma())


def test_long_hand_back_list_in_a_batch(df):
    # ladders near the edge of FP32 (square32_tp's critical planes at every momentum): hundreds are handed back, of
    # several orders at once, some of them beyond the shared-memory order
    ws = [I.workload("square32_tp", nk=16, n_w=n, m_max=1) for n in (24, 48, 64, 80, 98)]
    for w in ws:                                            # W = 0 scaled to |lambda| ~ 1e7: the list takes the plane
        w.gamma_uu[1] *= 1e4
        w.gamma_ud[1] *= 1e4
    with df.DualFermionBatch(ws) as b64, df.DualFermionBatch(ws, precision=df.DF_FP32_IR) as b:
        b64.iterate(1)
        b.iterate(1)
        for i in range(len(ws)):
            assert nrel(b.get_sigma(i), b64.get_sigma(i)) < TOL_SIGMA, ws[i].n_w


def test_long_hand_back_list_takes_the_fp64_path_s_time(df):
    # order 96, 3,200 ladders, all handed back: the second solve takes the FP64 path's time (22 ms; shared-memory
    # factors, one block per SM, took 1.45 times as long), beside the mixed kernel's own 3.4 ms
    w = I.random_nonsymmetric(96, 12, 1, 64, seed=1, scale=0.5)
    t = []
    for kw in (dict(), dict(precision=df.DF_FP32_IR), dict(precision=df.DF_FP32_IR, ladder_tol=1e-300)):
        with df.DualFermion.from_workload(w, eig_mode=0, **kw) as d:
            d.bubble()
            d.bse(3)
            best = 1e30
            for _ in range(3):
                d.set_timing(True)
                d.bse(3)
                best = min(best, d.get_timing()["bse"][0])
            t.append(best)
    assert t[2] - t[1] < 1.2 * t[0], t


def test_small_orders_error_on_the_paper_s_inputs(df):
    # the mean error of a (channel, W) plane against the FP64 path over orders 8-32 and 12 inputs each of the paper's
    # Example I: 1.6e-14 with the kernel that swept [D | gamma] (which rounds the pivot row once); 10% above that
    errs = []
    for n_w in (8, 16, 24, 32):
        for seed in range(1, 13):
            rng = np.random.default_rng(seed)
            w = I.half_filled_atom("p", 2, 8, U=float(rng.uniform(16.0, 24.0)), beta=float(rng.uniform(0.8, 1.2)),
                                   n_w=n_w, m_max=1)
            k = []
            for prec in (df.DF_FP64, df.DF_FP32_IR):
                with df.DualFermion.from_workload(w, precision=prec, eig_mode=0) as d:
                    d.bubble()
                    d.bse(3)
                    k.append(d.get_kernel())
            errs += [np.linalg.norm(k[1][c, a] - k[0][c, a]) / np.linalg.norm(k[0][c, a])
                     for c in range(2) for a in range(w.n_bos)]
    assert np.exp(np.mean(np.log(errs))) < 1.8e-14
