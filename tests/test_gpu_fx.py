"""The fixed-point FP64 operators (csrc/mdagm_fx.cu) at the edges of their shapes: the
smallest lattice, the largest block of each strip height, strips cut to two rows
(L mod 4 = 2 above 50), one slice per CTA and longer ranges; the scales of the exponent
range; and non-finite data, which must reach exactly the sites FP64 arithmetic takes it to.

Tolerance: 1e-12 of the largest element, as for the FP64 kernels (a slice is held to
2^-57 of its largest component or better, and the result rounded once).
"""
import numpy as np
import pytest
import torch

import oracle
from paper_2508_16298_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def hq():
    from paper_2508_16298_gb300 import build
    build.build()
    from paper_2508_16298_gb300 import hqmc
    return hqmc


def cuda(a):
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


def rel(a, b):
    return float(np.max(np.abs(a - b)) / np.max(np.abs(b)))


@pytest.mark.parametrize("L,N", [(18, 2), (18, 3), (20, 7), (34, 160), (50, 3), (52, 2), (54, 3), (58, 3), (62, 2), (64, 2),
                                 (66, 155), (68, 3)])
def test_shapes(hq, L, N):
    lat = oracle.Lattice(L, N)
    th = inputs.theta_hot(L, N, seed=10 + L)
    x = inputs.complex_gaussian(L, N, seed=20 + L)
    with hq.Config(L, N) as cfg:
        assert cfg.launch_shape(hq.FP64)["variant"] >= 200
        assert rel(hq.apply_MdagM(cfg, cuda(th), cuda(x)).cpu().numpy(), oracle.apply_MdagM(lat, th, x)) < 1e-12
        for dagger in (False, True):
            y = hq.apply_M(cfg, cuda(th), cuda(x), dagger=dagger).cpu().numpy()
            assert rel(y, oracle.apply_M(lat, th, x, dagger=dagger)) < 1e-12


@pytest.mark.parametrize("dtau,t,fixed", [(0.3, 1.0, True), (0.32, 1.0, False), (0.1, -2.0, True), (1.0, 1.0, False)])
def test_range_of_the_hopping(hq, dtau, t, fixed):
    """tanh(dtau |t|) up to 0.3 is in fixed point, beyond it in the FP64 kernels."""
    L, N = 18, 9
    lat = oracle.Lattice(L, N, dtau=dtau, t=t)
    th, x = inputs.theta_hot(L, N, seed=31), inputs.complex_gaussian(L, N, seed=32)
    with hq.Config(L, N, dtau=dtau, t=t) as cfg:
        assert (cfg.launch_shape(hq.FP64)["variant"] >= 200) == fixed
        assert rel(hq.apply_MdagM(cfg, cuda(th), cuda(x)).cpu().numpy(), oracle.apply_MdagM(lat, th, x)) < 1e-12


def test_scales(hq):
    """Every slice at its own scale: zero and graded slices, a point source, and the ends
    of the exponent range."""
    L, N = 18, 12
    lat = oracle.Lattice(L, N)
    th, base = inputs.theta_hot(L, N, seed=41), inputs.complex_gaussian(L, N, seed=42)
    one, point, graded = np.zeros_like(base), np.zeros_like(base), base.copy()
    one[3] = base[3]
    point[5, 2, 3] = 1 + 2j
    for k in range(N):
        graded[k] *= 10.0 ** (-6 * k)
    with hq.Config(L, N) as cfg:
        for x in (one, point, graded, base * 1e-290, base * 1e290):
            y, yo = hq.apply_MdagM(cfg, cuda(th), cuda(x)).cpu().numpy(), oracle.apply_MdagM(lat, th, x)
            for a, b in zip(y, yo):  # row by row: a graded vector's small rows count too
                m = np.max(np.abs(b))
                assert np.max(np.abs(a - b)) <= 1e-12 * m
        assert not hq.apply_MdagM(cfg, cuda(th), cuda(base * 0)).abs().max().item()


@pytest.mark.parametrize("bad", [np.nan, np.inf, -np.inf])
def test_non_finite_data_stays_local(hq, bad):
    L, N = 18, 12
    lat = oracle.Lattice(L, N)
    th, base = inputs.theta_hot(L, N, seed=51), inputs.complex_gaussian(L, N, seed=52)
    x, th2 = base.copy(), th.copy()
    x[4, 1, 2] = complex(bad, 0.0)
    th2[6, 3, 1, 0] = bad
    nan = lambda v: np.isnan(v.real) | np.isnan(v.imag) | np.isinf(v.real) | np.isinf(v.imag)  # noqa: E731
    with hq.Config(L, N) as cfg, np.errstate(all="ignore"):
        for t, v in ((th, x), (th2, base)):
            for y, yo in ((hq.apply_MdagM(cfg, cuda(t), cuda(v)), oracle.apply_MdagM(lat, t, v)),
                          (hq.apply_M(cfg, cuda(t), cuda(v)), oracle.apply_M(lat, t, v))):
                y = y.cpu().numpy()
                assert np.array_equal(nan(y), nan(yo))
                ok = ~nan(yo)
                assert np.max(np.abs(y[ok] - yo[ok])) < 1e-12 * np.max(np.abs(yo[ok]))


def test_large_angles(hq):
    """Angles beyond the integer reduction's range (2^28) take the library's functions."""
    L, N = 18, 5
    th = inputs.theta_hot(L, N, seed=61)
    x = inputs.complex_gaussian(L, N, seed=62)
    lat = oracle.Lattice(L, N)
    with hq.Config(L, N) as cfg:
        for s in (1e3, 1e8, 1e12):
            assert rel(hq.apply_MdagM(cfg, cuda(th * s), cuda(x)).cpu().numpy(), oracle.apply_MdagM(lat, th * s, x)) < 1e-12


MIXED = [(8, 16), (20, 24), (24, 18), (54, 8)]  # FP64 kernel; one shape of each strip height


@pytest.mark.parametrize("solver", ["cg64", "pcg64"])
@pytest.mark.parametrize("autotune", [False, True])
def test_batch_of_both_kernels_equals_single_chains(hq, solver, autotune):
    """Chains of the fixed-point and the FP64 kernels in one batch: bit for bit the
    single-chain runs, whatever the slice ranges."""
    th0 = [inputs.theta_ordered(L, N, 70 + i, tau_walk=0.0) for i, (L, N) in enumerate(MIXED)]
    phis = [cuda(inputs.complex_gaussian(L, N, 80 + i)) for i, (L, N) in enumerate(MIXED)]
    seeds, dts = [5, 6, 7, 8], [0.01, 0.01, 0.005, 0.005]
    with hq.Batch(MIXED, autotune=autotune) as b:
        b.set_solver(solver)
        xs, infos = b.cg_solve([cuda(t) for t in th0], phis, tol=1e-10)
        ths = [cuda(t) for t in th0]
        tinf = b.trajectory(ths, seeds, traj_counter=2, nsteps=2, dts=dts, tol=1e-9)
    for i, (L, N) in enumerate(MIXED):
        with hq.Config(L, N, variant=1) as cfg:
            x1, info1 = hq.cg_solve(cfg, cuda(th0[i]), phis[i], tol=1e-10, solver=solver)
            t1 = cuda(th0[i])
            ti = hq.trajectory(cfg, t1, seed=seeds[i], traj_counter=2, nsteps=2, dt=dts[i], tol=1e-9, solver=solver)
        assert infos[i]["status"] == 0 and infos[i]["iterations"] == info1["iterations"]
        assert torch.equal(xs[i], x1) and infos[i]["true_residual"] == info1["true_residual"]
        assert torch.equal(ths[i], t1) and tinf[i]["dH"] == ti["dH"] and tinf[i]["cg_iterations"] == ti["cg_iterations"]


@pytest.mark.parametrize("L,N", [(18, 2), (18, 9), (34, 16), (50, 3), (54, 3), (62, 2), (66, 9), (68, 3)])
@pytest.mark.parametrize("noncompact", [False, True])
def test_force_shapes(hq, L, N, noncompact):
    """The fixed-point force at both strip heights, cut strips and slice counts around the
    bosonic part's chunk of 8."""
    lat = oracle.Lattice(L, N, noncompact=noncompact)
    th, X = inputs.theta_hot(L, N, seed=91 + L), inputs.complex_gaussian(L, N, seed=92 + L)
    with hq.Config(L, N, noncompact=noncompact) as cfg:
        d = torch.empty((N, L, L, 2), dtype=torch.float64, device="cuda")
        F = hq.force(cfg, cuda(th), cuda(X), dSf=d).cpu().numpy()
        SB = hq.action_terms(cfg, cuda(th))[0]
    do = oracle.fermion_dS(lat, th, X)
    assert rel(d.cpu().numpy(), do) < 1e-12
    assert rel(F, -do - oracle.bosonic_dS(lat, th)) < 1e-12
    assert abs(SB - oracle.bosonic_action(lat, th)) < 1e-12 * abs(SB)


def test_force_scales_and_non_finite(hq):
    L, N = 18, 10
    lat = oracle.Lattice(L, N)
    th, base = inputs.theta_hot(L, N, seed=95), inputs.complex_gaussian(L, N, seed=96)
    small = th * 0  # angles and differences below the sine's series limit
    small[1::2] = 1e-4 * th[1::2]
    one, graded, bad = np.zeros_like(base), base.copy(), base.copy()
    one[3] = base[3]
    for k in range(N):
        graded[k] *= 10.0 ** (-5 * k)
    bad[4, 1, 2] = complex(np.nan, 0.0)
    with hq.Config(L, N) as cfg, np.errstate(all="ignore"):
        for t, x in ((th, one), (th, graded), (th, base * 1e-140), (th, base * 1e140), (small, base), (th, bad)):
            d = torch.empty((N, L, L, 2), dtype=torch.float64, device="cuda")
            F = hq.force(cfg, cuda(t), cuda(x), dSf=d).cpu().numpy()
            d, do = d.cpu().numpy(), oracle.fermion_dS(lat, t, x)
            assert np.array_equal(np.isnan(d), np.isnan(do))
            ok = ~np.isnan(do)
            assert np.max(np.abs(d[ok] - do[ok])) <= 1e-12 * np.max(np.abs(do[ok]))
            Fo = -do - oracle.bosonic_dS(lat, t)
            assert np.max(np.abs(F[ok] - Fo[ok])) <= 1e-12 * np.max(np.abs(Fo[ok]))


@pytest.mark.parametrize("L,N,dtau", [(4, 2, 0.1), (4, 17, 0.1), (6, 64, 0.1), (8, 65, 0.1), (10, 97, 0.05), (18, 240, 0.2),
                                      (24, 131, 0.1), (44, 450, 0.1), (8, 40, 0.5)])
def test_line_preconditioner(hq, L, N, dtau):
    """csrc/precond64.cu: lines shorter than the window, tiles and pieces cut by the end of
    the line, sites past a multiple of 32, windows from a few slices to 68 (FP64
    where rho < 0.6).  Tolerance: 1e-12 as above."""
    from oracle import precond as opc
    x = inputs.complex_gaussian(L, N, seed=50 + L)
    with hq.Config(L, N, dtau=dtau) as cfg:
        c = opc.coefficients(oracle.Lattice(L, N, dtau=dtau))
        want = opc.apply(c, x)
        for s in (1.0, 2.0**-1000, 2.0**900):
            z = hq.apply_precond(cfg, cuda(x * s)).cpu().numpy()
            assert rel(z / s, want) < 1e-12
        assert not np.any(hq.apply_precond(cfg, cuda(0 * x)).cpu().numpy())
        x[N // 2, 1, 1] = np.nan
        z = hq.apply_precond(cfg, cuda(x)).cpu().numpy()
        line = np.zeros(x.shape, bool)
        line[:, 1, 1] = True
        assert np.isnan(z[N // 2, 1, 1]) and rel(z[~line], want[~line]) < 1e-12


@pytest.mark.parametrize("L,N", [(4, 2), (4, 3), (4, 16), (4, 17), (6, 31), (6, 300), (8, 192), (10, 100)])
def test_cluster_solver(hq, L, N):
    """csrc/cg_cluster.cu: one slice a CTA and several, a last CTA with fewer, blocks that end
    inside a warp, up to the most threads.  The solution meets its tolerance by the oracle's
    operator; a solution as start; an iteration limit inside a body, where the recurrence is
    that of the two-kernel loop (variant 1) to rounding; and that loop's status for a zero
    and a non-finite source."""
    lat, theta = oracle.Lattice(L, N), inputs.theta_ordered(L, N, 61)
    th, phi = cuda(theta), inputs.complex_gaussian(L, N, 62)
    with hq.Config(L, N) as a, hq.Config(L, N, variant=1) as b:
        x, i = hq.cg_solve(a, th, cuda(phi), tol=1e-10)
        res = phi - oracle.apply_MdagM(lat, theta, x.cpu().numpy())
        assert i["status"] == 0 and np.linalg.norm(res) <= 1.01e-10 * np.linalg.norm(phi)
        _, k = hq.cg_solve(a, th, cuda(phi), x=x.clone(), tol=1e-10)
        assert k["status"] == 0 and k["iterations"] == 0
        m = min(7, i["iterations"] - 1)
        (x, i), (y, j) = (hq.cg_solve(c, th, cuda(phi), tol=1e-10, maxit=m, raise_on_fail=False) for c in (a, b))
        assert i["status"] == j["status"] != 0 and i["iterations"] == j["iterations"] == m
        assert rel(x.cpu().numpy(), y.cpu().numpy()) < 1e-9
        x, i = hq.cg_solve(a, th, cuda(0 * phi), tol=1e-10)
        assert i["status"] == 0 and not np.any(x.cpu().numpy())
        phi[N // 2, 1, 1] = np.nan
        i, j = (hq.cg_solve(c, th, cuda(phi), tol=1e-10, raise_on_fail=False)[1] for c in (a, b))
        assert i["status"] == j["status"] != 0


@pytest.mark.parametrize("solver", ["mixed", "pmixed"])
@pytest.mark.parametrize("maxit", [1, 6, 7, 8, 9])
def test_multi_correction_where_a_solve_ends(hq, solver, maxit):
    """The systems' FP32 corrections move by two steps every second iteration: ended after an
    odd and an even count, within a body (reliable interval 8) and at its end, a solution has
    all its steps.  Against one system alone; 9 FP32 iterations keep 1e-4 (rounding 6e-8, a
    few hundred operations an entry and iteration), a lost step is 1e-2 and more."""
    L, N, nsys = 8, 40, 3
    th = cuda(inputs.theta_ordered(L, N, 71))
    phi = np.stack([inputs.complex_gaussian(L, N, 72 + k) for k in range(nsys)])
    with hq.Config(L, N, reliable_interval=8) as cfg:
        hq.set_multi_rhs(cfg, nsys)
        X, infos = hq.cg_solve_multi(cfg, th, cuda(phi), tol=1e-10, maxit=maxit, solver=solver, raise_on_fail=False)
        for k in range(nsys):
            x, i = hq.cg_solve(cfg, th, cuda(phi[k]), tol=1e-10, maxit=maxit, solver=solver, raise_on_fail=False)
            assert i["iterations"] == infos[k]["iterations"] == maxit and i["status"] == infos[k]["status"]
            assert rel(X[k].cpu().numpy(), x.cpu().numpy()) < 1e-4


@pytest.mark.parametrize("L,N", [(8, 3), (10, 40), (18, 7), (34, 20), (44, 30), (66, 4)])
def test_apply_from_the_field_itself(hq, L, N):
    """FP32 M^dagger M with the angles wrapped in the kernel against the float table (which an
    event-timed apply uses): the same angles and arithmetic, so the same bits; angles far
    outside one turn, and a field with an infinity, among them."""
    th = inputs.theta_hot(L, N, 81)
    th[0, 1] *= 1000
    x = cuda(inputs.complex_gaussian(L, N, 82).astype(np.complex64))
    with hq.Config(L, N) as cfg:
        for bad in (False, True):
            if bad:
                th[N // 2, 2, 3, 0] = np.inf
            y = hq.apply_MdagM(cfg, cuda(th), x).cpu().numpy()
            hq.set_timing(cfg, True)
            z = hq.apply_MdagM(cfg, cuda(th), x).cpu().numpy()
            hq.set_timing(cfg, False)
            assert np.array_equal(y, z, equal_nan=True) and bool(np.isnan(y).any()) == bad


@pytest.mark.parametrize("L,N", [(12, 2), (12, 35), (14, 3), (16, 160)])
def test_batch_kernels_of_smaller_lattices(hq, L, N):
    """Variant 1 (a batch's kernels) is in fixed point from L = 12: blocks of 36, 49 and 64
    threads.  Tolerance as in test_shapes; a solve by the oracle's operator."""
    lat = oracle.Lattice(L, N)
    th, x = inputs.theta_ordered(L, N, 91), inputs.complex_gaussian(L, N, 92)
    with hq.Config(L, N) as cfg:
        assert cfg.launch_shape(hq.FP64)["variant"] < 200
    with hq.Config(L, N, variant=1) as cfg:
        assert cfg.launch_shape(hq.FP64)["variant"] >= 200
        assert rel(hq.apply_MdagM(cfg, cuda(th), cuda(x)).cpu().numpy(), oracle.apply_MdagM(lat, th, x)) < 1e-12
        for dagger in (False, True):
            assert rel(hq.apply_M(cfg, cuda(th), cuda(x), dagger=dagger).cpu().numpy(),
                       oracle.apply_M(lat, th, x, dagger=dagger)) < 1e-12
        for solver in ("cg64", "pcg64"):
            X, i = hq.cg_solve(cfg, cuda(th), cuda(x), tol=1e-9, solver=solver)
            res = x - oracle.apply_MdagM(lat, th, X.cpu().numpy())
            assert i["status"] == 0 and np.linalg.norm(res) <= 1.01e-9 * np.linalg.norm(x)


@pytest.mark.parametrize("L", [18, 54])
def test_force_at_the_ends_of_the_exponent_range(hq, L):
    """dS_f is bilinear in X: below 1e-162 its terms underflow and above 1e154 they overflow, as
    in FP64, also where a product of two slices' exponents is far outside a double's.  Mixed
    slices: a tiny slice beside a huge one, whose products are of order one."""
    N = 6
    lat = oracle.Lattice(L, N)
    th, base = inputs.theta_hot(L, N, seed=97), inputs.complex_gaussian(L, N, seed=98)
    mixed = base.copy()
    mixed[0::2] *= 1e-140
    mixed[1::2] *= 1e140
    with hq.Config(L, N) as cfg, np.errstate(all="ignore"):
        for x in (base * 1e-250, base * 1e-230, base * 1e-200, base * 1e-160, base * 1e150, base * 1e200, base * 1e250, mixed):
            d = torch.empty((N, L, L, 2), dtype=torch.float64, device="cuda")
            hq.force(cfg, cuda(th), cuda(x), dSf=d)
            d, do = d.cpu().numpy(), oracle.fermion_dS(lat, th, x)
            assert np.array_equal(np.isfinite(d), np.isfinite(do))
            ok = np.isfinite(do)
            if ok.any():  # 1e-12 of the largest, and a few subnormal units where FP64 underflows term by term
                assert np.max(np.abs(d[ok] - do[ok])) <= 1e-12 * np.max(np.abs(do[ok])) + 64 * 5e-324


@pytest.mark.parametrize("solver", ["cg64", "pcg64"])
@pytest.mark.parametrize("autotune", [False, True])
def test_batch_of_tall_strips_equals_single_chains(hq, solver, autotune):
    """4-row strips in one batch: both block sizes (up to 512 threads and 608), two lattices of each,
    whose blocks have idle rows (L mod 4 = 2) and surplus threads, several ranges a chain."""
    lats = [(54, 8), (62, 6), (66, 5), (68, 4)]
    th0 = [cuda(inputs.theta_ordered(L, N, 170 + i, tau_walk=0.0)) for i, (L, N) in enumerate(lats)]
    phis = [cuda(inputs.complex_gaussian(L, N, 180 + i)) for i, (L, N) in enumerate(lats)]
    with hq.Batch(lats, autotune=autotune) as b:
        b.set_solver(solver)
        xs, infos = b.cg_solve(th0, phis, tol=1e-10)
        ths = [t.clone() for t in th0]
        tinf = b.trajectory(ths, [5, 6, 7, 8], traj_counter=2, nsteps=2, dts=[0.005] * 4, tol=1e-9)
    for i, (L, N) in enumerate(lats):
        with hq.Config(L, N, variant=1) as cfg:
            x1, info1 = hq.cg_solve(cfg, th0[i], phis[i], tol=1e-10, solver=solver)
            t1 = th0[i].clone()
            ti = hq.trajectory(cfg, t1, seed=5 + i, traj_counter=2, nsteps=2, dt=0.005, tol=1e-9, solver=solver)
        assert infos[i]["status"] == 0 and infos[i]["iterations"] == info1["iterations"]
        assert torch.equal(xs[i], x1) and infos[i]["true_residual"] == info1["true_residual"]
        assert torch.equal(ths[i], t1) and tinf[i]["dH"] == ti["dH"] and tinf[i]["cg_iterations"] == ti["cg_iterations"]


@pytest.mark.parametrize("L,N", [(20, 9), (54, 7), (66, 5)])
@pytest.mark.parametrize("solver", ["mixed", "pmixed"])
def test_multi_system_residuals_in_fixed_point(hq, L, N, solver):
    """Systems solved together from L = 18: the FP64 residuals of every system, each range with its
    own scratch, by the oracle's operator; solutions as starts are accepted as they are."""
    lat, theta, nsys = oracle.Lattice(L, N), inputs.theta_ordered(L, N, 191, tau_walk=0.0), 3
    phi = np.stack([inputs.complex_gaussian(L, N, 192 + k) * 10.0 ** (3 * k) for k in range(nsys)])
    th = cuda(theta)
    with hq.Config(L, N, reliable_interval=10) as cfg:
        hq.set_multi_rhs(cfg, nsys)
        X, infos = hq.cg_solve_multi(cfg, th, cuda(phi), tol=1e-9, solver=solver)
        for k in range(nsys):
            res = phi[k] - oracle.apply_MdagM(lat, theta, X[k].cpu().numpy())
            true = np.linalg.norm(res) / np.linalg.norm(phi[k])
            # the reported residual is that of x to the rounding of O x, a few 1e-16 |O| |x| / |phi|
            assert infos[k]["status"] == 0 and abs(true - infos[k]["true_residual"]) < 1e-11 and true <= 1.01e-9
        _, again = hq.cg_solve_multi(cfg, th, cuda(phi), x=X.clone(), tol=1e-9, solver=solver)
        assert all(i["status"] == 0 and i["iterations"] == 0 for i in again)
