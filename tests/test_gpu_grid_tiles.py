"""Collocation and quadrature by chunk pairs: lists shorter than a chunk, of
one chunk and a remainder, and of several chunks (chunks of 64 functions in
FP32, 32 in FP64), ragged grid tiles, mostly empty boxes, and a P that is not
symmetric, against the oracle's plain sums.  Collocation has a kernel for
contexts whose longest list has at most 160 terms in FP32 (tiny19: 156, tiny20:
161) and 32 in FP64 (tiny3: 29)."""
import numpy as np
import pytest

import workloads as w
from oracle import grid_ops

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no GPU", allow_module_level=True)

import paper_2108_13478_gb300 as dft  # noqa: E402

U32 = 2.0 ** -24


@pytest.mark.parametrize("name,pad", [("tiny1", 5.0), ("tiny3", 5.0), ("tiny7", 5.0), ("tiny13", 5.0), ("tiny19", 5.0),
                                      ("tiny20", 5.0), ("dtiny4", None), ("tiny2", 24.0)])
@pytest.mark.parametrize("mixed", [False, True])
def test_chunk_pairs_match_the_oracle(name, pad, mixed):
    s = w.config_system(name, pad=pad) if pad else w.config_system(name)
    rng = np.random.default_rng(21)
    v = rng.normal(size=tuple(int(t) for t in s.grid_n[::-1]))
    K = s.n_basis
    P = 0.1 * rng.normal(size=(K, K))   # not symmetric: n takes the full double sum
    ctx = dft.Context(s, precision=dft.DFT_PREC_FP16X3 if mixed else dft.DFT_PREC_FP64)
    V = ctx.potential_matrix(torch.from_numpy(v).cuda()).cpu().numpy()
    n = ctx.density_on_grid(torch.from_numpy(P).cuda()).cpu().numpy()
    ctx.close()
    Vr, nr = grid_ops.potential_matrix(s, v), grid_ops.density_on_grid(s, P)
    # bounds from the sums of absolute terms; FP32: chains of 64 terms, products
    # of up to five factors, conversions and 16 partial sums stay below 100 roundings
    Va = grid_ops.potential_matrix(s, np.abs(v))
    u = 100 * U32 if mixed else 1e-13
    tol_v = u * np.sqrt(np.outer(np.diag(Va), np.diag(Va))) + 1e3 * 2.0 ** -49   # Cauchy-Schwarz on |phi_a| |v| |phi_b|
    assert np.all(V == V.T)
    assert np.all(np.abs(V - Vr) <= tol_v)
    # |phi|^T |P| |phi| <= lambda_max(sym |P|) |phi|^2 at every point
    lam = np.linalg.eigvalsh(0.5 * (np.abs(P) + np.abs(P).T))[-1]
    tol_n = u * lam * grid_ops.density_on_grid(s, np.eye(K)) + 1e-15
    print(f"{name} {'FP32' if mixed else 'FP64'}: V {np.max(np.abs(V - Vr) / tol_v):.3f}, n {np.max(np.abs(n - nr) / tol_n):.3f} of the bounds")
    assert np.all(np.abs(n - nr) <= tol_n)
