"""Waits of two product kernels that expire in one call (a mixed solve whose FP32
sweeps and FP64 residuals both run on tensor cores; test hook, no GPU fault)
are reported by that call, and the next one works."""
import numpy as np
import pytest

import oracle.msd_oracle as O_
from paper_1409_8186_gb300 import workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("KB32,RT32,KB64", [(0, 16, 0), (0, 8, 0), (1, 8, 0), (5, 1, 0), (0, 16, 5), (0, 8, 5)])
def test_two_kinds_of_waits(KB32, RT32, KB64):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1409_8186_gb300 import msd
    cl = W.random_cluster(seed=3, M=20, half_side=9.0, rmin=0.6, rmax=1.0, gap=0.2, k=2.0, N=10)
    betas = W.angles(16)
    pb = msd.Problem(cl)
    pb.set_tile(16, msd.MSD_FP32, KB32, RT32)
    pb.set_tile(16, msd.MSD_FP64, KB64, 1)
    assert pb.plan_info(16, msd.MSD_FP64)[0]["KB"] == KB64
    x = torch.from_numpy(np.ones((cl.ntot, 16), np.complex128)).cuda()
    pb.matvec(x)  # (the generators of either precision are made, and checked, before)
    pb.matvec(x.to(torch.complex64), msd.MSD_FP32)
    ref, _ = O_.solve(cl.centres, cl.radii, cl.bc, cl.k, cl.N, betas, method="lu")
    try:
        msd.msd_test_expire_waits(True)
        pb.matvec(x)  # a wait of either product, reported by the next call that looks
        pb.matvec(x.to(torch.complex64), msd.MSD_FP32)
        with pytest.raises(msd.MsdError) as e:
            pb.solve(betas, tol=1e-10, precision=msd.MSD_MIXED)
        assert e.value.status == msd.MSD_ERR_CUDA, e.value
    finally:
        msd.msd_test_expire_waits(False)
    res = pb.solve(betas, tol=1e-10, precision=msd.MSD_MIXED)
    assert res.status == msd.MSD_OK
    assert np.abs(res.rho.cpu().numpy() - ref).max() <= 1e-9 * np.abs(ref).max()
    pb.close()
