"""The row-per-thread FP64 product of few disks (tile code KB = 1, RT = 1),
pinned, against the oracle's dense operator: rows around blocks of 128, one to
many disks and columns, several configurations, and an FP64 solve that drops
converged systems.  Tolerance 1e-11 as for every FP64 product."""
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


@pytest.mark.parametrize("Ms,N,R", [((1,), 1, 1), ((4,), 12, 1), ((5, 2), 12, 3), ((3,), 21, 2), ((33,), 6, 5),
                                    ((2,), 55, 1)])
def test_rows_product(msd, Ms, N, R):
    cls = [W.random_cluster(seed=30 + i, M=M, half_side=4.0 * np.sqrt(M) + 2.0, rmin=0.6, rmax=1.0, gap=0.2, k=2.0,
                            N=N, neumann_fraction=0.3) for i, M in enumerate(Ms)]
    pb = msd.Problem(cls)
    pb.set_tile(R, msd.MSD_FP64, 1, 1)
    assert pb.plan_info(R, msd.MSD_FP64)[0]["KB"] == 1
    rng = np.random.default_rng(N)
    x = rng.standard_normal((pb.ntot, R)) + 1j * rng.standard_normal((pb.ntot, R))
    y = pb.matvec(torch.from_numpy(x).cuda()).cpu().numpy()
    for c, cl in enumerate(cls):
        rows = slice(pb.row_offset(c), pb.row_offset(c + 1))
        ref = O_.preconditioned_dense(cl.centres, cl.radii, cl.bc, cl.k, cl.N) @ x[rows]
        assert np.abs(y[rows] - ref).max() <= 1e-11 * np.abs(ref).max()
    if R > 1 and N < 55:
        betas = W.angles(R)
        res = pb.solve(betas, tol=1e-12)
        for c, cl in enumerate(cls):
            ref, _ = O_.solve(cl.centres, cl.radii, cl.bc, cl.k, cl.N, betas, method="lu")
            rows = slice(pb.row_offset(c), pb.row_offset(c + 1))
            assert np.abs(res.rho.cpu().numpy()[rows] - ref).max() <= 1e-9 * np.abs(ref).max()
    pb.close()
