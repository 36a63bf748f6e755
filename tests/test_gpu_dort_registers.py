"""Tridiagonalisation of one matrix with its rows in registers (n <= 512):
sizes around one lane's columns (32), one row per SM (152), the last size in
registers and the first beyond, with eigenvalues (1e-12 of the largest), the
eigenvectors made from the stored reflectors (residual 1e-10, orthonormal to
1e-12) and matrices whose columns are reduced already.  The tolerances are
those of every time-reversal test."""
import numpy as np
import pytest

import oracle.msd_oracle as O_
from paper_1409_8186_gb300 import workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [3, 4, 5, 31, 32, 33, 64, 65, 151, 153, 305, 511, 512, 513])
def test_one_matrix(n):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1409_8186_gb300 import msd
    rng = np.random.default_rng(n)
    pb = msd.Problem(W.four_disks())
    G = rng.standard_normal((n, n)) + 1j * rng.standard_normal((n, n))
    T = O_.time_reversal_matrix(G)
    lam = O_.dort_eigenvalues(T)
    K = 3
    eig, vec = pb.dort_eigenvectors(torch.from_numpy(G[None].copy()).cuda(), K)
    e, U = eig.cpu().numpy()[0], vec.cpu().numpy()[0].T
    assert np.abs(e - lam).max() <= 1e-12 * lam[0]
    assert np.abs(U.conj().T @ U - np.eye(K)).max() <= 1e-12
    for i in range(K):
        assert np.linalg.norm(T @ U[:, i] - e[i] * U[:, i]) <= 1e-10 * lam[0]
    Q, _ = np.linalg.qr(G)  # T = 4 I: nothing left to reduce
    e = pb.dort_eigen(torch.from_numpy(2.0 * Q[None]).cuda())[0].cpu().numpy()[0]
    assert np.abs(e - 4.0).max() <= 4e-12
    pb.close()
