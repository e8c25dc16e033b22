"""The eigensolver's precision where its block products run on the tensor cores."""
import pytest

torch = pytest.importorskip("torch")

import paper_1105_0542_gb300 as su  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("g,t,L,n,nev", [(10.0, 0.05, 4.0, 1700, 2), (48.0, 0.02, 8.0, 2001, 10)])
def test_residuals_are_a_double_products(g, t, L, n, nev):
    """Pairs that have converged far below the tolerance: the residual norm is
    the product's rounding.  That of a product in double, sums of 2w + 1 terms
    of a unit vector's elements, is some sqrt(2w) 2^-54: 1.6e-15 at w = 430."""
    E, R, info = su.speedup_evolution_spectrum("aho", [1.0, g], 8, t, L, n, nev)
    assert n * info["half_width"] * info["block"] >= 3_000_000   # the tensor-core product's share of sizes
    assert max(R) <= 2.0 ** -49


@pytest.mark.parametrize("n,L,t,nev", [(1100, 2.0, 0.05, 10), (1025, 2.0, 0.05, 8), (1025, 2.0, 0.05, 10), (900, 1.5, 0.05, 10),
                                       (1201, 2.0, 0.1, 2), (257, 2.0, 0.05, 10), (3001, 2.0, 0.05, 20)])
def test_blocks_that_reach_the_flat_end_of_the_spectrum_keep_their_rank(n, L, t, nev):
    """In a short interval the block's last eigenvalues are far below the
    first: energies against numpy's eigensolver on the dense matrix (its own
    rounding, 1e-15 of the largest eigenvalue, over t and the eigenvalue)."""
    import numpy as np

    U = torch.empty(n * n, dtype=torch.float64, device="cuda")
    su.speedup_evolution_matrix("aho", [1.0, 10.0], 8, t, L, n, U)
    lam = np.linalg.eigvalsh(U.reshape(n, n).cpu().numpy())[::-1][:nev]
    E, R, info = su.speedup_evolution_spectrum("aho", [1.0, 10.0], 8, t, L, n, nev)
    assert info["converged"]
    assert np.all(np.abs(np.array(E) + np.log(lam) / t) <= 1e-10 + 1e-13 * lam[0] / (lam * t))
