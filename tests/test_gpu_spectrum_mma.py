"""The eigensolver's tensor-core block product at the edges of its tiles (rows
not a multiple of 128, one tile and a bit, a band wider than the matrix's half,
blocks of 8, 16 and 32 columns): energies against numpy's eigensolver on the
dense matrix of the same operator (the tolerance of the other spectrum tests:
1e-10 of max(1, |E|)), and orthonormal eigenfunctions."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import paper_1105_0542_gb300 as su  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,L,t,nev", [(1700, 4.0, 0.05, 2), (1409, 5.0, 0.02, 10), (1025, 2.0, 0.05, 8), (1281, 5.0, 0.02, 20),
                                       (2111, 6.0, 0.02, 9)])
def test_block_product_energies(n, L, t, nev):
    params = [1.0, 10.0]
    U = torch.empty(n * n, dtype=torch.float64, device="cuda")
    su.speedup_evolution_matrix("aho", params, 8, t, L, n, U)
    lam = np.linalg.eigvalsh(U.reshape(n, n).cpu().numpy())[::-1][:nev]
    ref = -np.log(lam) / t
    vec = torch.empty(nev * n, dtype=torch.float64, device="cuda")
    E, R, info = su.speedup_evolution_spectrum("aho", params, 8, t, L, n, nev, vectors=vec)
    w, _ = su.su_evolution_band_size(t, L, n)
    assert n * w * info["block"] >= 3_000_000     # the tensor-core product's share of sizes
    assert np.all(np.abs(np.array(E) - ref) <= 1e-10 * np.maximum(1.0, np.abs(ref))), np.array(E) - ref
    G = (vec.reshape(nev, n) @ vec.reshape(nev, n).T).cpu().numpy() * (2 * L / (n - 1))
    assert np.abs(G - np.eye(nev)).max() <= 1e-10
