"""The digit-sliced FP64 product against its error bound, on source values whose
digits are the worst of the form (leading digit just above half its range,
every lower one -128) and on columns of very different size per disk.  The
reference multiplies the library's own generators and factors in extended
precision; the bound is the one of tests/test_digit_mirror.py per real product
of a (target, shift) maximum and a (mode) maximum, four products per complex
one, 2^-52 of it per folded sum, and one FP64 rounding per addition."""
import numpy as np
import pytest

from paper_1409_8186_gb300 import workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

PRODUCT = 1.01 * (2.0 ** -51.4 + 2.0 ** -53)
WORST = float(sum(d * 256.0 ** -(i + 1) * 2 for i, d in enumerate([65] + [-128] * 6)))


@pytest.mark.parametrize("M,N", [(60, 8), (33, 14)])
@pytest.mark.parametrize("kind", ["worst", "worst signs", "sizes"])
def test_error_bound(M, N, kind):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1409_8186_gb300 import msd
    n, rng = 2 * N + 1, np.random.default_rng(M)
    side = int(np.ceil(np.sqrt(M)))
    g = 3.0 * np.stack(np.meshgrid(np.arange(side), np.arange(side)), -1).reshape(-1, 2)[:M]
    cl = W.Cluster(g + 0.2 * rng.uniform(-1, 1, g.shape), np.full(M, 1.0), np.zeros(M, np.int8), 1.7, N)
    pb = msd.Problem(cl)
    pb.set_tile(1, msd.MSD_FP64, 0, 1)
    assert pb.plan_info(1, msd.MSD_FP64)[0]["KB"] == 0
    D = pb.diagonals().cpu().numpy().reshape(4, M, n)
    r, H = D[0].real, D[2]  # radius 1: column factor J_m, row factor 1 / H_m
    if kind == "sizes":
        x = (rng.standard_normal((M, n)) + 1j * rng.standard_normal((M, n))) * 10.0 ** rng.uniform(-6, 0, M)[:, None]
    else:
        sign = rng.choice([-1.0, 1.0], (2, M, n)) if kind == "worst signs" else np.ones((2, M, n))
        x = (sign[0] + 1j * sign[1]) * WORST / r  # scaled by r again: the worst digits, or the nearest to them
    G = pb.generators().cpu().numpy()  # [q][p][l]
    y = pb.matvec(torch.from_numpy(x.reshape(-1, 1)).cuda()).cpu().numpy().reshape(M, n)
    pb.close()
    xs = (r * x.real) + 1j * (r * x.imag)  # rounded as the library does
    part = np.maximum(np.abs(xs.real), np.abs(xs.imag)).max(0)            # [j]
    gmax = np.maximum(np.abs(G.real), np.abs(G.imag)).max(0)              # [p][l]
    ext = np.clongdouble
    s = np.zeros((M, n), ext)
    size, err = np.zeros((M, n)), np.zeros((M, n))
    for m in range(n):
        for j in range(n):
            col = G[:, :, j - m + 2 * N]
            s[:, m] += col.T.astype(ext) @ xs[:, j].astype(ext)
            size[:, m] += np.abs(col).T @ np.abs(xs[:, j])
            err[:, m] += (4 * M * PRODUCT + 16 * 2.0 ** -52) * gmax[:, j - m + 2 * N] * part[j]
    l = 1 / H.astype(ext)
    ref = x.astype(ext) + l * s
    # additions: the window's (n shifts, at most 16 folds and slots of it), the finalize kernel's
    err = np.abs(l) * (err + (16 * n + 32) * 2.0 ** -53 * size) + 16 * 2.0 ** -53 * np.abs(x)
    assert (np.abs((y - ref).astype(complex)) <= err).all()
