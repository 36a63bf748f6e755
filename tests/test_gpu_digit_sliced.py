"""The digit-sliced FP64 product (tile code KB = 0, RT = 1), pinned, against the
oracle's dense operator at the edges of its tiles: targets around 32, sources
around 8, columns around 64 and not dividing it, one to several mode tiles and
groups of radii, uneven batches, the adjoint and raw products (gradient), the
formulations, the transmission product; non-finite input; radii that refuse
it.  Tolerance 1e-11 relative, as for every FP64 product (SciPy's own value
errors; the sliced sums themselves are exact to 2^-55 of the largest terms)."""
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


def _cluster(M, N, rmin=0.8, rmax=1.0, seed=5, k=2.0, neumann=0.3):
    return W.random_cluster(seed=seed, M=M, half_side=4.0 * np.sqrt(M) + 1.0, rmin=rmin, rmax=rmax, gap=0.1, k=k, N=N,
                            neumann_fraction=neumann)


def _dense(cl):
    return O_.preconditioned_dense(cl.centres, cl.radii, cl.bc, cl.k, cl.N)


def _x(n, R, seed):
    rng = np.random.default_rng(seed)
    return rng.standard_normal((n, R)) + 1j * rng.standard_normal((n, R))


def _pin(msd, pb, R):
    pb.set_tile(R, msd.MSD_FP64, 0, 1)
    assert pb.plan_info(R, msd.MSD_FP64)[0]["KB"] == 0


def _close(y, ref):
    return np.abs(y - ref).max() <= 1e-11 * np.abs(ref).max()


@pytest.mark.parametrize("M,N,R", [(1, 3, 1), (2, 1, 1), (8, 12, 1), (9, 20, 1), (31, 10, 3), (32, 9, 5), (33, 10, 1),
                                   (70, 12, 16), (70, 5, 33), (20, 4, 64), (20, 6, 65), (65, 20, 2), (4, 55, 1),
                                   (150, 8, 1), (12, 35, 7)])
def test_product_edges(msd, M, N, R):
    cl = _cluster(M, N, rmin=0.8 if N <= 20 else 0.97)  # radii within 2^{4.5/N}
    pb = msd.Problem(cl)
    _pin(msd, pb, R)
    x = _x(cl.ntot, R, M + R)
    assert _close(pb.matvec(torch.from_numpy(x).cuda()).cpu().numpy(), _dense(cl) @ x)
    pb.close()


def test_uneven_batch_wide_radii_and_update(msd):
    cls = [_cluster(40, 8, 0.5, 1.5, 1), _cluster(3, 11, 0.9, 1.0, 2), _cluster(90, 6, 0.5, 1.0, 3)]
    pb = msd.Problem(cls)
    for R in (1, 6):
        _pin(msd, pb, R)
        x = _x(pb.ntot, R, R)
        y = pb.matvec(torch.from_numpy(x).cuda()).cpu().numpy()
        ref = np.concatenate([_dense(c) @ x[pb.row_offset(i):pb.row_offset(i + 1)] for i, c in enumerate(cls)])
        assert _close(y, ref)
    rng = np.random.default_rng(9)
    for step in (0.01, 0.3):  # the groups stay, then change
        new = [W.Cluster(c.centres, c.radii * (1 - step * rng.uniform(0, 1, c.M)), c.bc, c.k, c.N) for c in cls]
        pb.update_geometry(radii=torch.from_numpy(np.concatenate([c.radii for c in new])).cuda())
        y = pb.matvec(torch.from_numpy(x).cuda()).cpu().numpy()
        ref = np.concatenate([_dense(c) @ x[pb.row_offset(i):pb.row_offset(i + 1)] for i, c in enumerate(new)])
        assert _close(y, ref)
    pb.close()


def test_radii_out_of_range_take_the_general_kernel(msd):
    cl = W.Cluster(np.array([[0.0, 0.0], [8.0, 0.0], [0.0, 8.0]]), np.array([0.2, 1.0, 2.0]), np.zeros(3, np.int8),
                   1.0, 12)
    pb = msd.Problem(cl)
    pb.set_tile(1, msd.MSD_FP64, 0, 1)
    assert pb.plan_info(1, msd.MSD_FP64)[0]["KB"] != 0
    x = _x(cl.ntot, 1, 1)
    assert _close(pb.matvec(torch.from_numpy(x).cuda()).cpu().numpy(), _dense(cl) @ x)
    pb.close()


@pytest.mark.parametrize("bad", [np.nan, np.inf])
def test_non_finite_input_stays_visible(msd, bad):
    cl = _cluster(40, 6)
    pb = msd.Problem(cl)
    _pin(msd, pb, 2)
    x = _x(cl.ntot, 2, 3)
    x[17, 1] = bad
    y = pb.matvec(torch.from_numpy(x).cuda()).cpu().numpy()
    assert np.isfinite(y[:, 0]).all() and not np.isfinite(y[:, 1]).any()
    pb.close()


def test_formulation_transmission_and_gradient(msd):
    cl = _cluster(34, 8, k=2.3)
    pb = msd.Problem(cl)
    pb.set_formulation("cfie")
    pb.set_tile(2, msd.MSD_FP64, 0, 1)  # the formulation's product over twice the columns
    x = _x(cl.ntot, 1, 4)
    y = pb.matvec(torch.from_numpy(x).cuda()).cpu().numpy()
    pb.set_tile(2, msd.MSD_FP64, 5, 1)
    ref = pb.matvec(torch.from_numpy(x).cuda()).cpu().numpy()
    assert _close(y, ref) and not np.array_equal(y, ref)
    pb.set_formulation(None)
    pb.set_penetrable(3.1)
    xm = _x(cl.ntot, 1, 5)
    out = []
    for KB in (0, 5):
        pb.set_tile(1, msd.MSD_FP64, KB, 1)
        yp, ym = pb.penetrable_matvec(torch.from_numpy(x).cuda(), torch.from_numpy(xm).cuda())
        out.append(torch.cat([yp, ym]).cpu().numpy())
    assert _close(out[0], out[1])
    pb.set_penetrable(None)
    th, betas = W.angles(20), W.angles(3)
    Ft = _x(20, 3, 6).reshape(1, 20, 3)
    g = []
    for KB in (0, 5):
        pb.set_tile(3, msd.MSD_FP64, KB, 1)
        g.append(pb.grad_farfield_misfit(betas, th, Ft, tol=1e-13))
    for u, v in zip(*g):
        assert np.abs(u - v).max() <= 1e-9 * np.abs(v).max()
    pb.close()


def test_expired_wait_is_reported(msd):
    cl = _cluster(40, 6)
    pb = msd.Problem(cl)
    _pin(msd, pb, 1)
    betas = [0.3]
    try:
        msd.msd_test_expire_waits(True)
        with pytest.raises(msd.MsdError) as e:
            pb.solve(betas, tol=1e-10)
        assert e.value.status == msd.MSD_ERR_CUDA, e.value
    finally:
        msd.msd_test_expire_waits(False)
    res = pb.solve(betas, tol=1e-12)
    ref, _ = O_.solve(cl.centres, cl.radii, cl.bc, cl.k, cl.N, betas, method="lu")
    assert res.status == msd.MSD_OK
    assert np.abs(res.rho.cpu().numpy() - ref).max() <= 1e-9 * np.abs(ref).max()
    pb.close()
