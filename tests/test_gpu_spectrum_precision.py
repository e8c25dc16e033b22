"""The eigensolver's precision where its block products run on the tensor cores."""
import pytest

torch = pytest.importorskip("torch")

import paper_1105_0542_gb300 as su  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,L,t,nev", [(1100, 2.0, 0.05, 10), (1025, 2.0, 0.05, 8), (1025, 2.0, 0.05, 10), (900, 1.5, 0.05, 10),
                                       (1201, 2.0, 0.1, 2), (257, 2.0, 0.05, 10)])
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
