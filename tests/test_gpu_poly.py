"""The grouped evaluation of the Chebyshev expansion (babies, giants and the
weighted products or Clenshaw's recurrence) against the oracle's polynomial of
the same order in the eigenbasis, at the orders where its grouping changes:
no giant, one giant, ragged last groups, plans that keep the giants and
orders so high that they do not fit (Clenshaw)."""
import numpy as np
import pytest
import scipy.fft

import workloads as w
from oracle import basis, dm

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no GPU", allow_module_level=True)

import paper_2108_13478_gb300 as dft  # noqa: E402


@pytest.fixture
def dct_coefficients(monkeypatch):
    """The oracle's Gauss-Chebyshev sums by SciPy's DCT-II: the direct cosine
    sums take minutes per order at N_C of thousands."""
    def coeffs(mu, beta, e_min, e_max, n_c, m_nodes=None):
        m = int(m_nodes) if m_nodes else 8 * int(n_c)
        th = np.pi * (np.arange(m) + 0.5) / m
        f = dm.fermi(0.5 * (e_max + e_min) + 0.5 * (e_max - e_min) * np.cos(th), mu, beta)
        a = scipy.fft.dct(f, type=2)[:n_c] / m
        a[0] *= 0.5
        return a
    args = (0.1, 20.0, -1.0, 3.0, 40, 160)
    assert np.max(np.abs(coeffs(*args) - dm.cheb_coeffs(*args))) < 1e-14
    monkeypatch.setattr(dm, "cheb_coeffs", coeffs)


def problem(name, seed=3):
    s = w.config_system(name)
    S, T = basis.overlap_kinetic_system(s)
    D = np.random.default_rng(seed).normal(size=S.shape) * 0.02
    F = T - 0.5 * S + (D + D.T) / 2
    eps = dm.geneig(F, S)[0]
    return s, F, S, eps[0] - 0.05, eps[-1] + 0.05


@pytest.mark.parametrize("name,orders", [("tiny8", (2, 3, 4, 5, 8, 33, 64, 1000, 2900, 14000)), ("tiny3", (2, 17, 700)),
                                         ("tiny37", (65, 1500))])
def test_fp64_expansion_matches_the_oracle_at_every_grouping(name, orders, dct_coefficients):
    s, F, S, lo, hi = problem(name)
    Fd = torch.from_numpy(F).cuda()
    for n_c in orders:
        beta = n_c / (2.0 * (hi - lo))
        ref = dm.dm_cheb(F, S, s.n_electrons, beta, lo, hi, n_c, m_nodes=4 * n_c)
        ctx = dft.Context(s, e_min=lo, e_max=hi, cheb_order=n_c, kT=1.0 / beta)
        ctx.overlap_kinetic()
        P, info = ctx.density_matrix(Fd)
        ctx.close()
        err = float(np.max(np.abs(P.cpu().numpy() - ref["P"])))
        print(f"{name} N_C {n_c}: max|dP| {err:.2e} of {np.max(np.abs(ref['P'])):.2f}, "
              f"N_e {info.n_e_trace:.10f}, dmu {info.mu - ref['mu']:.1e}")
        # the requirement of the FP64 path; rounding errors grow with the order
        assert err < 1e-9 * max(1.0, np.max(np.abs(ref["P"])))
        assert abs(info.n_e_trace - s.n_electrons) < 1e-8 * s.n_electrons


@pytest.mark.parametrize("name,orders", [("tiny8", (2, 3, 5, 40, 700, 6000)), ("tiny37", (2, 33, 1500, 7000)),
                                         ("cluster64", (1400,))])
def test_split_expansion_matches_the_oracle_at_every_grouping(name, orders, dct_coefficients):
    """One, two and three 256-blocks per side (operands read in place and
    transposed, folded block rows, ragged last blocks), direct and Clenshaw
    plans; the gate of the mixed path's density matrices, 1e-4 of max|P|."""
    s, F, S, lo, hi = problem(name)
    Fd = torch.from_numpy(F).cuda()
    for n_c in orders:
        beta = n_c / (2.0 * (hi - lo))
        ref = dm.dm_cheb(F, S, s.n_electrons, beta, lo, hi, n_c, m_nodes=4 * n_c)
        ctx = dft.Context(s, e_min=lo, e_max=hi, cheb_order=n_c, kT=1.0 / beta, precision=dft.DFT_PREC_FP16X3,
                          skip_correction=1)
        ctx.overlap_kinetic()
        P, info = ctx.density_matrix(Fd)
        ctx.close()
        err = float(np.max(np.abs(P.cpu().numpy() - ref["P"]))) / np.max(np.abs(ref["P"]))
        print(f"{name} split N_C {n_c}: max|dP| / max|P| {err:.2e}, N_e {info.n_e_trace:.6f}, dmu {info.mu - ref['mu']:.1e}")
        assert info.spectrum_ok == 1
        assert err < 1e-4
        assert abs(info.n_e_trace - s.n_electrons) < 1e-4 * s.n_electrons
