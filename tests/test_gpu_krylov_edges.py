"""Krylov projections and updates at the edges of their shapes: column counts
that divide, exceed or do not divide a warp, odd numbers of elements (no
16-byte pairs), configurations of one to many reduction chunks, bases from one
vector to several batches, few and many systems, restarts.  Solutions against
the oracle's LU to 1e-10 (FP64) and 1e-9 (mixed) times a condition number below
10 (well separated disks), from relres 1e-12."""
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


@pytest.mark.parametrize("Ms,N,R", [((3,), 4, 1), ((5, 3), 6, 2), ((7,), 5, 3), ((9, 1, 4), 5, 12), ((4,), 7, 33),
                                    ((30,), 6, 64), ((60,), 10, 1), ((31,), 6, 5), ((12, 20), 8, 16), ((3, 3, 3), 4, 7)])
@pytest.mark.parametrize("precision", ["fp64", "mixed"])
def test_solves(msd, Ms, N, R, precision):
    cls = [W.random_cluster(seed=20 + i, M=M, half_side=8.0 * np.sqrt(M) + 2.0, rmin=0.5, rmax=0.9, gap=1.0, k=0.9,
                            N=N) for i, M in enumerate(Ms)]
    pb = msd.Problem(cls)
    betas = W.angles(R) + 0.2
    prec = msd.MSD_FP64 if precision == "fp64" else msd.MSD_MIXED
    for restart in (200, 4):
        res = pb.solve(betas, tol=1e-12, restart=restart, maxit=3000, precision=prec)
        assert res.status == msd.MSD_OK, res.relres.max()
        rho = res.rho.cpu().numpy()
        for c, cl in enumerate(cls):
            ref, _ = O_.solve(cl.centres, cl.radii, cl.bc, cl.k, cl.N, betas, method="lu")
            err = np.abs(rho[pb.row_offset(c):pb.row_offset(c + 1)] - ref).max() / np.abs(ref).max()
            assert err <= 10 * (1e-10 if precision == "fp64" else 1e-9), err
    pb.close()
