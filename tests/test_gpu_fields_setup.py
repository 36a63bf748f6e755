"""Far field and generator kernels at the edges of their tiles: angle tiles
of 32, column groups of 1, 4 and 8, warps of four disks, configurations of
different truncation; unordered generator pairs for odd and even M, near and
far pairs, one disk, a geometry update with both precisions stored.

Tolerances (derived before the first run).  Far field: sums of up to M n ~
700 terms, each within ~20 eps of its value (phase and mode recurrences):
1e-12 of the largest value leaves a factor of six over the worst case 700 x 20
x 1.1e-16 = 1.6e-12 added without cancellation of signs, which random signs
reduce by sqrt(700).  Generators: 5e-12 relative to |H| against SciPy, as
the parity tests; the reversed pair equals (-1)^l exactly."""
import numpy as np
import pytest

import oracle.msd_oracle as O_
from paper_1409_8186_gb300 import workloads as W

torch = pytest.importorskip("torch")
pytestmark = [pytest.mark.gpu, pytest.mark.filterwarnings("ignore::RuntimeWarning")]


@pytest.fixture(scope="module")
def msd():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1409_8186_gb300 import msd as m
    return m


def _cluster(M, N, seed=5, k=2.0):
    return W.random_cluster(seed=seed, M=M, half_side=4.0 * np.sqrt(M) + 1.0, rmin=0.6, rmax=1.0, gap=0.2, k=k, N=N,
                            neumann_fraction=0.3)


@pytest.mark.parametrize("M,N,R,T", [(1, 1, 1, 1), (3, 10, 2, 31), (4, 12, 4, 32), (5, 10, 5, 33), (33, 9, 8, 64),
                                     (17, 20, 9, 5), (2, 55, 8, 40), (33, 10, 1, 360)])
def test_farfield_edges(msd, M, N, R, T):
    cls = [_cluster(M, N), _cluster(M + 2, max(1, N - 1), seed=6)]
    pb = msd.Problem(cls)
    rng = np.random.default_rng(M * 100 + R)
    rho = rng.standard_normal((pb.ntot, R)) + 1j * rng.standard_normal((pb.ntot, R))
    th = W.angles(T) + 0.3
    F = pb.farfield(torch.from_numpy(rho).cuda(), th).cpu().numpy()
    at = 0
    for c, cl in enumerate(cls):
        ref = O_.farfield(cl.centres, cl.radii, cl.k, cl.N, rho[at:at + cl.ntot], th).reshape(T, R)
        at += cl.ntot
        assert np.abs(F[c] - ref).max() <= 1e-12 * np.abs(ref).max()
    pb.close()


@pytest.mark.parametrize("M,N,k", [(1, 3, 1.0), (2, 12, 1.0), (3, 10, 30.0), (32, 8, 2.0), (33, 16, 9.0), (40, 4, 3.0)])
def test_generators_of_every_pair(msd, M, N, k):
    from scipy.special import hankel1
    cl = _cluster(M, N, k=k)
    pb = msd.Problem([_cluster(3, 5, seed=9), cl])
    moved = cl.centres + 0.01
    moved[0] += 0.02
    x32 = torch.ones((pb.ntot, 1), dtype=torch.complex64, device="cuda")
    pb.generators(1)
    pb.matvec(x32, msd.MSD_FP32)  # complex64 copy built too
    pb.update_geometry(centres=np.concatenate([pb.clusters[0].centres, moved]))
    G = pb.generators(1).cpu().numpy()  # [q][p][l]
    lmax = 2 * N
    l = np.arange(-lmax, lmax + 1)
    d = moved[None, :, :] - moved[:, None, :]  # [q][p] = O_p - O_q
    b, al = np.hypot(d[..., 0], d[..., 1]), np.arctan2(d[..., 1], d[..., 0])
    off = ~np.eye(M, dtype=bool)
    assert np.all(G[~off] == 0)
    if M > 1:
        ref = hankel1(l, k * b[off][:, None]) * np.exp(1j * l * al[off][:, None])
        assert np.abs(G[off] / ref - 1).max() <= 5e-12
    assert np.array_equal(G, np.swapaxes(G, 0, 1) * ((-1.0) ** l))
    pb.close()
