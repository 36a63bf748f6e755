"""The error path of the bounded waits of the shift-GEMM product, in both of its
block forms (two blocks of <= 8 modes, one of <= 16) and with one to several
folds of the accumulators: an expired wait (test hook, no GPU fault) is
reported, and the next product is right (1e-5 relative, as for every FP32
product)."""
import numpy as np
import pytest

import oracle.msd_oracle as O_
from paper_1409_8186_gb300 import workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("KB", [0, 1])
@pytest.mark.parametrize("M,N,R", [(3, 4, 8), (40, 10, 16), (150, 7, 8)])
def test_expired_wait_is_reported(KB, M, N, R):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1409_8186_gb300 import msd
    cl = W.random_cluster(seed=M, M=M, half_side=4.0 * np.sqrt(M) + 2.0, rmin=0.6, rmax=1.0, gap=0.2, k=2.0, N=N)
    pb = msd.Problem(cl)
    pb.set_tile(R, msd.MSD_FP32, KB, 8)
    rng = np.random.default_rng(M + KB)
    x = (rng.standard_normal((cl.ntot, R)) + 1j * rng.standard_normal((cl.ntot, R))).astype(np.complex64)
    xd = torch.from_numpy(x).cuda()
    pb.matvec(xd, msd.MSD_FP32)
    try:
        msd.msd_test_expire_waits(True)
        with pytest.raises(msd.MsdError) as e:
            for _ in range(3):
                pb.matvec(xd, msd.MSD_FP32)
            msd.msd_matvec_timing(pb.handle, -1)  # reports what the products recorded
        assert e.value.status == msd.MSD_ERR_CUDA, e.value
    finally:
        msd.msd_test_expire_waits(False)
    y = pb.matvec(xd, msd.MSD_FP32).cpu().numpy()
    msd.msd_matvec_timing(pb.handle, -1)
    ref = O_.preconditioned_dense(cl.centres, cl.radii, cl.bc, cl.k, cl.N) @ x.astype(np.complex128)
    assert np.abs(y - ref).max() <= 1e-5 * np.abs(ref).max()
    pb.close()
