"""Sums of the Krylov kernels on given vectors: the solution update x += V y of
a mixed solve (FP32 basis and coefficients, batches of eight vectors summed in
FP32 and the batches in FP64), in every kernel and split that the sizes reach.

Tolerances: a batch of eight complex products in two chains is off by at most
12 x 2^-24 of the sum of its absolute terms, the coefficients' own rounding
included; FP64 adds nothing that shows."""
import numpy as np
import pytest

from paper_1409_8186_gb300 import workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def msd():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1409_8186_gb300 import msd as m
    return m


def _problem(msd, Ms, N):
    cls = []
    for M in Ms:
        side = int(np.ceil(np.sqrt(M)))
        g = 4.0 * np.stack(np.meshgrid(np.arange(side), np.arange(side)), -1).reshape(-1, 2)[:M]
        cls.append(W.Cluster(g + 0.0, np.full(M, 1.0), np.zeros(M, np.int8), 1.3, N))
    return msd.Problem(cls)


SIZES = [((3,), 4, 1), ((5, 3), 4, 3), ((40, 30), 10, 1), ((400,), 20, 1), ((80, 60), 3, 12), ((50,), 3, 33),
         ((30, 31), 4, 64), ((401,), 20, 3)]


@pytest.mark.parametrize("Ms,N,R", SIZES)
@pytest.mark.parametrize("nv", [1, 7, 40, 700])
def test_solution_update(msd, Ms, N, R, nv):
    pb = _problem(msd, Ms, N)
    g = torch.Generator(device="cuda").manual_seed(nv + R)
    V = torch.randn(nv, pb.ntot, R, dtype=torch.complex64, device="cuda", generator=g)
    y = torch.randn(pb.C, R, nv, dtype=torch.complex128, device="cuda", generator=g)
    x0 = torch.randn(pb.ntot, R, dtype=torch.complex128, device="cuda", generator=g)
    x = x0.clone()
    msd.msd_test_krylov(pb.handle, msd.MSD_TEST_SOLUTION_UPDATE, R, nv, V, y, x)
    for c in range(pb.C):
        s = slice(pb.row_offset(c), pb.row_offset(c + 1))
        ref = x0[s] + torch.einsum("inr,ri->nr", V[:, s].to(torch.complex128), y[c])
        size = torch.einsum("inr,ri->nr", V[:, s].abs().double(), y[c].abs()) + x0[s].abs()
        assert ((x[s] - ref).abs() <= 12 * 2.0 ** -24 * size).all()
    pb.close()


@pytest.mark.parametrize("Ms,N,R", [((400,), 20, 1), ((30,), 10, 1), ((30, 31), 4, 64), ((50,), 3, 33), ((3,), 4, 3)])
def test_small_terms_after_a_large_one(msd, Ms, N, R):
    """2^24 followed by 3999 terms of 0.1: in FP32 every later batch is lost."""
    nv = 4000
    pb = _problem(msd, Ms, N)
    V = torch.ones(nv, pb.ntot, R, dtype=torch.complex64, device="cuda")
    y = torch.full((pb.C, R, nv), 0.1, dtype=torch.complex128, device="cuda")
    y[..., 0] = 2.0 ** 24
    x = torch.zeros(pb.ntot, R, dtype=torch.complex128, device="cuda")
    msd.msd_test_krylov(pb.handle, msd.MSD_TEST_SOLUTION_UPDATE, R, nv, V, y, x)
    ref = 2.0 ** 24 + (nv - 1) * float(np.float32(0.1))
    # the first batch: eight additions next to 2^24, whose FP32 spacing is 2
    assert (x - ref).abs().max().item() <= 8.0 + 12 * 2.0 ** -24 * (nv - 1) * 0.1
    pb.close()


@pytest.mark.parametrize("Ms,N,R", [((40, 30), 4, 16), ((12,) * 9, 3, 1), ((50,), 3, 33)])
@pytest.mark.parametrize("eps", [1e-3, 1e-6, 1e-9])
def test_norm_after_a_second_projection_of_a_batch(msd, Ms, N, R, eps):
    """w = V c + t with |c| = 1 and a remainder |t| = eps across V, for more than
    eight systems: the norm that the step goes on with is that of what is left,
    t and the rounding of the projection (64 x 2^-53 and of V's orthonormality,
    which is formed in FP64), and not what a difference of squares near 1 leaves
    (1e-16, so that eps below 1e-8 would be lost)."""
    nv = 5
    pb = _problem(msd, Ms, N)
    assert pb.C * R > 8
    g = torch.Generator(device="cuda").manual_seed(7)
    B = torch.randn(nv + 1, pb.ntot, R, dtype=torch.complex128, device="cuda", generator=g)
    c = torch.randn(nv, pb.C, R, dtype=torch.complex128, device="cuda", generator=g)
    c = c / c.abs().square().sum(0).sqrt()
    w = torch.empty(pb.ntot, R, dtype=torch.complex128, device="cuda")
    for k in range(pb.C):
        s = slice(pb.row_offset(k), pb.row_offset(k + 1))
        Q = torch.linalg.qr(B[:, s].permute(2, 1, 0))[0].permute(2, 1, 0)  # [nv + 1, rows, R]
        B[:, s] = Q
        w[s] = torch.einsum("inr,ir->nr", Q[:nv], c[:, k]) + eps * Q[nv]
    norm2 = np.zeros(pb.C * R)
    msd.msd_test_krylov(pb.handle, msd.MSD_TEST_SECOND_PROJECTION, R, nv, B[:nv].contiguous(), None, w, norm2)
    left = torch.stack([w[pb.row_offset(k):pb.row_offset(k + 1)].abs().square().sum(0) for k in range(pb.C)])
    assert np.abs(norm2 - left.cpu().numpy().reshape(-1)).max() <= 1e-13 * eps ** 2
    assert np.abs(np.sqrt(norm2) - eps).max() <= 64 * 2.0 ** -53
    pb.close()


@pytest.mark.parametrize("M,R,pairs", [(4, 1, 1), (5, 1, 0), (87468, 1, 1), (87467, 1, 0), (5, 2, 1), (5, 3, 0),
                                       (87468, 2, 1), (40000, 1, 1)])
def test_single_columns_keep_their_pairs(msd, M, R, pairs):
    """16-byte loads wherever the vectors start on even elements: also where a
    256th of a single column is an odd number of rows (262404 / 256 = 1025)."""
    pb = _problem(msd, (M,), 1)
    assert msd.msd_test_pairs(pb.handle, R) == pairs
    pb.close()


def test_long_single_column(msd):
    """262404 rows in chunks of 1026, the last one shorter."""
    pb = _problem(msd, (87468,), 1)
    g = torch.Generator(device="cuda").manual_seed(3)
    V = torch.randn(9, pb.ntot, 1, dtype=torch.complex64, device="cuda", generator=g)
    y = torch.randn(1, 1, 9, dtype=torch.complex128, device="cuda", generator=g)
    x = torch.zeros(pb.ntot, 1, dtype=torch.complex128, device="cuda")
    msd.msd_test_krylov(pb.handle, msd.MSD_TEST_SOLUTION_UPDATE, 1, 9, V, y, x)
    ref = torch.einsum("inr,i->nr", V.to(torch.complex128), y[0, 0])
    size = torch.einsum("inr,i->nr", V.abs().double(), y[0, 0].abs())
    assert ((x - ref).abs() <= 12 * 2.0 ** -24 * size).all()
    pb.close()
