"""The grouped expansion on Fock matrices with a chosen spectrum: plans of a
context whose workspace holds few expansion buffers (Clenshaw's recurrence,
down to a single giant), and the refusal of a spectrum outside the interval.

F = L F~ L^T with S = L L^T and F~ = W diag(x) W^T for an orthogonal W, so the
eigenvalues of S^-1 F are x, and the expansion of order N_C is evaluated at
them exactly: P = L^-T W diag(p(x)) W^T L^-1."""
import numpy as np
import pytest
import scipy.fft

import workloads as w
from workloads.si_clusters import diamond_sphere, jitter, make_system

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no GPU", allow_module_level=True)

import paper_2108_13478_gb300 as dft  # noqa: E402
from oracle import dm  # noqa: E402

FP64, FP16 = dft.DFT_PREC_FP64, dft.DFT_PREC_FP16X3


def coarse(atoms):
    xyz = diamond_sphere(25.0)
    xyz = jitter(xyz[np.argsort((xyz ** 2).sum(1), kind="stable")[:atoms]], 0.05, 1)
    return make_system(xyz, h=1.0, grid_n=np.array([60, 60, 60]), grid_origin=xyz.min(0) - 7.0)


def few_slots():
    """K = 3500 on a coarse grid: a mixed context has 30 expansion buffers."""
    return coarse(350)


def given_spectrum(ctx, x, W):
    """F and L^-T W for the eigenvalues x (device)."""
    S, _ = ctx.overlap_kinetic()
    L = torch.linalg.cholesky(S)
    A = L @ W
    return ((A * x) @ A.T).contiguous(), torch.linalg.solve_triangular(L.T, W, upper=True)


def orthogonal(K, localised=False):
    g = torch.Generator(device="cuda").manual_seed(11)
    if localised:   # every eigenvector close to one function
        v = torch.randn(K, 1, generator=g, device="cuda", dtype=torch.float64)
        return torch.eye(K, device="cuda", dtype=torch.float64) - 2.0 / float((v ** 2).sum()) * (v @ v.T)
    return torch.linalg.qr(torch.randn(K, K, generator=g, device="cuda", dtype=torch.float64))[0]


def coefficients(mu, beta, n_c):
    """a_l on [-1, 1] from 4 N_C nodes, as the library takes them."""
    m = 4 * n_c
    a = scipy.fft.dct(dm.fermi(np.cos(np.pi * (np.arange(m) + 0.5) / m), mu, beta), type=2)[:n_c] / m
    a[0] *= 0.5
    return a


@pytest.mark.parametrize("n_c", [26, 40, 46])
def test_clenshaw_plan_with_a_single_giant(n_c):
    """One giant, no room to keep it with its sums: its moments still come
    from its own Gram sums (mu, and with it the electron count, depend on
    them)."""
    s = few_slots()
    beta = n_c / 2.0
    ctx = dft.Context(s, precision=FP16, e_min=-1.0, e_max=1.0, cheb_order=n_c, kT=1.0 / beta, skip_correction=1)
    K = ctx.K
    x = np.sort(np.random.default_rng(2).uniform(-0.95, 0.95, K))
    F, LW = given_spectrum(ctx, torch.from_numpy(x).cuda(), orthogonal(K))
    mom = dm.moments_from_eigs(x, n_c)
    mu = dm.bisect(lambda m: 2.0 * float(coefficients(m, beta, n_c) @ mom), s.n_electrons, -1.0 - 40 / beta, 1.0 + 40 / beta)
    for _ in range(2):   # the second call finds the first one's weights where its sums go
        P, info = ctx.density_matrix(F)
    ctx.close()
    ref = (LW * torch.from_numpy(dm.cheb_eval(x, coefficients(mu, beta, n_c))).cuda()) @ LW.T
    err = float((P - ref).abs().max() / ref.abs().max())
    print(f"K {K} N_C {n_c}: dmu {info.mu - mu:.2e}, N_e {info.n_e_trace:.6f} of {s.n_electrons}, max|dP| / max|P| {err:.2e}")
    assert abs(info.mu - mu) < 1e-5
    assert abs(info.n_e_trace - s.n_electrons) < 1e-5 * s.n_electrons
    assert err < 1e-4


@pytest.mark.parametrize("n_c", [90, 700, 2900])
def test_units_of_two_k_blocks(n_c):
    """K = 2060, above the line where accumulators take two k-blocks at a time:
    nine blocks per side, a last one of 12 columns, 65 k-blocks (a last unit of
    one); plans that keep few and many giants, and Clenshaw's recurrence."""
    s = coarse(206)
    beta = n_c / 4.0
    ctx = dft.Context(s, precision=FP16, e_min=-1.0, e_max=1.0, cheb_order=n_c, kT=1.0 / beta, skip_correction=1)
    x = np.sort(np.random.default_rng(3).uniform(-0.95, 0.95, ctx.K))
    F, LW = given_spectrum(ctx, torch.from_numpy(x).cuda(), orthogonal(ctx.K))
    P, info = ctx.density_matrix(F)
    ctx.close()
    ref = (LW * torch.from_numpy(dm.cheb_eval(x, coefficients(info.mu, beta, n_c))).cuda()) @ LW.T
    err = float((P - ref).abs().max() / ref.abs().max())
    print(f"K 2060 N_C {n_c}: N_e {info.n_e_trace:.6f} of {s.n_electrons}, max|dP| / max|P| {err:.2e}")
    assert abs(info.n_e_trace - s.n_electrons) < 1e-5 * s.n_electrons
    assert err < 1e-4


def outside(n_c, weight, at_last):
    """The eigenvalue above 1 whose T_{n_c - 1} makes an element of `at_last`
    with an eigenvector of largest squared component `weight`."""
    return float(np.cosh(np.arccosh(at_last / weight) / (n_c - 1)))


# (atoms, precision, N_C): one giant, two, a few; many (kept); Clenshaw's recurrence
PLANS = [(8, FP64, 26), (8, FP64, 40), (8, FP64, 71), (8, FP64, 140), (8, FP64, 1400), (8, FP64, 7000),
         (8, FP16, 26), (8, FP16, 40), (8, FP16, 71), (8, FP16, 140), (8, FP16, 1400), (8, FP16, 2900)]


@pytest.mark.parametrize("atoms,prec,n_c", PLANS)
def test_spectrum_outside_the_interval_is_refused(atoms, prec, n_c):
    """An eigenvalue above the interval makes the last term's largest element
    12: refused (the limit is 4), also where that term is never formed.  One
    that makes it 1.5 stays accepted; one that drives the operands or rho out
    of an FP16 pair is the same refusal, not an internal error."""
    s = w.config_system(f"tiny{atoms}")
    for at_last, ok in ((12.0, False), (1.5, True), (300.0, False), (1e7, False)):
        ctx = dft.Context(s, precision=prec, e_min=-1.0, e_max=1.0, cheb_order=n_c, kT=4.0 / n_c)
        K = ctx.K
        W = orthogonal(K)
        x = np.sort(np.random.default_rng(2).uniform(-0.9, 0.9, K))
        x[-1] = outside(n_c, float((W[:, -1] ** 2).max()), at_last)
        F, _ = given_spectrum(ctx, torch.from_numpy(x).cuda(), W)
        if ok:
            _, info = ctx.density_matrix(F)
            assert info.spectrum_ok == 1
        else:
            with pytest.raises(dft.DftError) as e:
                ctx.density_matrix(F)
            print(f"N_C {n_c}, x_max - 1 = {x[-1] - 1:.2e}, T_last {at_last}: {e.value}")
            assert e.value.status == dft._binding.DFT_ESPECTRUM
        ctx.close()


def test_spectrum_outside_the_interval_is_refused_where_mu_is_reused():
    """A cycle that takes over mu forms no giants: only the check itself sees
    a spectrum that left the interval since the cycles before."""
    s = w.config_system("tiny8")
    ref = dft.Context(s, model=dft.DFT_MODEL_NEUTRAL)
    S, T = ref.overlap_kinetic()
    Li = torch.linalg.inv(torch.linalg.cholesky(S))

    def edges(n):
        e = torch.linalg.eigvalsh(Li @ (T + ref.potential_matrix(ref.hartree_xc(n)[0])) @ Li.T)
        return float(e[0]), float(e[-1])
    n0 = ref.initial_density()
    n1 = 0.9 * n0
    if edges(n1)[1] < edges(n0)[1]:
        n0, n1 = n1, n0
    (lo, top0), (_, top1) = edges(n0), edges(n1)
    ref.close()
    # top1 at cosh(12 / 2899) of the interval, top0 well inside
    n_c, lo = 2900, lo - 1.0
    hi = lo + 2.0 * (top1 - lo) / (1.0 + np.cosh(12.0 / (n_c - 1)))
    assert top0 < hi - 1e-3
    ctx = dft.Context(s, precision=FP16, model=dft.DFT_MODEL_NEUTRAL, e_min=lo, e_max=hi, cheb_order=n_c, mix_alpha=0.0,
                      reuse_mu=1)
    ctx.overlap_kinetic()
    n = n0.clone()
    assert [ctx.scf_step(n).mu_reused for _ in range(3)] == [0, 0, 1]
    with pytest.raises(dft.DftError) as e:
        ctx.scf_step(n1.clone())
    print(f"top eigenvalues {top0:.4f}, {top1:.6f}, E_max {hi:.6f}: refused, {e.value}")
    assert e.value.status == dft._binding.DFT_ESPECTRUM
    ctx.close()


def test_fock_matrix_beyond_the_pair_is_an_internal_error():
    """Elements of F beyond the FP16 pair's range: the split reports them,
    whatever the expansion then makes of the operands."""
    s = w.config_system("tiny8")
    ctx = dft.Context(s, precision=FP16, e_min=-1.0, e_max=1.0, cheb_order=100, kT=0.04)
    W = orthogonal(ctx.K)
    F, _ = given_spectrum(ctx, torch.linspace(-0.9, 0.9, ctx.K, device="cuda", dtype=torch.float64), W)
    F[3, 3] = 1e6
    with pytest.raises(dft.DftError) as e:
        ctx.density_matrix(F)
    assert e.value.status == dft._binding.DFT_EINTERNAL
    ctx.close()


def test_clenshaw_sums_of_a_high_order_stay_in_the_pair():
    """b_q of Clenshaw's recurrence in T_s grows with the number of giants
    where the Fermi angle is near a multiple of pi / s: at N_C = 65536 with s
    = 24 it reaches 100, with eigenvectors that are nearly single functions
    also in its elements."""
    s = few_slots()
    n_c = 65536
    beta = n_c / 3.0
    ctx = dft.Context(s, precision=FP16, e_min=-1.0, e_max=1.0, cheb_order=n_c, kT=1.0 / beta, n_electrons=3500.0,
                      skip_correction=1)
    K = ctx.K
    near = np.pi / n_c * np.array([0.5, 1.0, 2.0, 3.0, 4.0, 6.0])
    x = np.concatenate([np.linspace(0.05, 0.9, K // 2 - len(near)), near])
    x = np.concatenate([x, -x])   # symmetric: mu = 0
    F, LW = given_spectrum(ctx, torch.from_numpy(x).cuda(), orthogonal(K, localised=True))
    P, info = ctx.density_matrix(F)
    ctx.close()
    p = dm.cheb_eval(x, coefficients(0.0, beta, n_c))
    ref = (LW * torch.from_numpy(p).cuda()) @ LW.T
    err = float((P - ref).abs().max() / ref.abs().max())
    # a relative error 2^-22 of H_N's pair shifts an eigenvalue, and f changes by up to beta / 4 per unit
    bound = 8 * beta / 4 * 2.0 ** -22
    print(f"K {K} N_C {n_c}: mu {info.mu:.2e}, N_e {info.n_e_trace:.4f}, max|dP| / max|P| {err:.2e} (bound {bound:.1e})")
    assert err < bound


def test_expired_waits_of_the_products_return_timeout_and_leave_the_context_usable(monkeypatch):
    """With DFT_TEST_EXPIRE_WAITS one epilogue warp of every CTA keeps back the
    release of its first accumulator: the waits of all roles run out (1 s), the
    CTAs drain their copies and MMAs, free tensor memory and return, the later
    launches of the call return at once, and the call reports DFT_ETIMEOUT.
    The same context then gives the density matrix."""
    import time
    s = w.config_system("tiny37")
    n_c = 300
    beta = n_c / 4.0
    ctx = dft.Context(s, precision=FP16, e_min=-1.0, e_max=1.0, cheb_order=n_c, kT=1.0 / beta)
    x = np.linspace(-0.9, 0.9, ctx.K)
    F, LW = given_spectrum(ctx, torch.from_numpy(x).cuda(), orthogonal(ctx.K))
    monkeypatch.setenv("DFT_TEST_EXPIRE_WAITS", "1")
    t0 = time.time()
    with pytest.raises(dft.DftError) as e:
        ctx.density_matrix(F)
    took = time.time() - t0
    print(f"expired waits: {e.value} after {took:.1f} s")
    assert e.value.status == dft._binding.DFT_ETIMEOUT
    assert took < 20.0
    monkeypatch.delenv("DFT_TEST_EXPIRE_WAITS")
    P, info = ctx.density_matrix(F)
    ctx.close()
    ref = (LW * torch.from_numpy(dm.cheb_eval(x, coefficients(info.mu - info.mu_correction, beta, n_c))).cuda()) @ LW.T
    assert info.spectrum_ok == 1
    assert float((P - ref).abs().max() / ref.abs().max()) < 1e-4


@pytest.mark.parametrize("prec", [FP16, dft.DFT_PREC_BF16X3])
def test_grouped_expansion_is_no_further_off_than_the_recurrence(prec, monkeypatch):
    """The distance of P from the FP64 context's (2-norm, six geometries, the
    first Fock matrix of an SCF run), by the grouped expansion and by the
    three-term recurrence."""
    err = {"grouped": 0.0, "three-term": 0.0}
    for seed in range(6):
        s = w.config_system("tiny8", seed=seed)
        ctx = dft.Context(s, model=dft.DFT_MODEL_NEUTRAL, cheb_tail_tol=1e-10)
        _, T = ctx.overlap_kinetic()
        F = (T + ctx.potential_matrix(ctx.hartree_xc(ctx.initial_density())[0])).contiguous()
        ref, info = ctx.density_matrix(F)
        ctx.close()
        for form in err:
            if form == "three-term":
                monkeypatch.setenv("DFT_TC_SHAPE", "32,0,256")
            else:
                monkeypatch.delenv("DFT_TC_SHAPE", raising=False)
            ctx = dft.Context(s, precision=prec, e_min=info.e_min, e_max=info.e_max, cheb_tail_tol=1e-6, skip_correction=1)
            ctx.overlap_kinetic()
            P, _ = ctx.density_matrix(F)
            ctx.close()
            err[form] += float(((P - ref) ** 2).sum() / (ref ** 2).sum()) / 6
    print({k: f"{v ** 0.5:.2e}" for k, v in err.items()})
    assert err["grouped"] <= err["three-term"]
