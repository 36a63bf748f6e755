"""Near field at the sizes where its kernel changes course: disks staged in
blocks of 64, columns in groups of one, four and eight, CTAs of 128 points,
pairs around the far limit k r = 20, points on a circle (field 0) and just
outside it.  Tolerance 1e-5 of the largest value, as for every near field (far
pairs are FP32 after an FP64 phase)."""
import numpy as np
import pytest

import oracle.msd_oracle as O_
from paper_1409_8186_gb300 import workloads as W

torch = pytest.importorskip("torch")
pytestmark = [pytest.mark.gpu, pytest.mark.filterwarnings("ignore::RuntimeWarning")]


@pytest.mark.parametrize("M,N,R,P", [(1, 1, 1, 1), (2, 4, 3, 127), (63, 3, 4, 128), (64, 9, 5, 129), (65, 9, 1, 300),
                                     (129, 2, 9, 257)])
def test_nearfield_edges(M, N, R, P):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1409_8186_gb300 import msd
    k, a = 2.0, 0.75
    side = int(np.ceil(np.sqrt(M)))
    g = np.arange(side * side)
    centres = 3.0 * np.stack([g % side, g // side], axis=1)[:M]
    cl = W.Cluster(centres, np.full(M, a), np.zeros(M, np.int8), k, N)
    rng = np.random.default_rng(M)
    pts = rng.uniform(-14.0, 3.0 * side + 14.0, (P, 2))
    special = [[a, 0.0], [0.0, a * (1 + 1e-12)], [10.0 * (1 + 1e-9), 0.0], [0.0, -10.0], [0.0, -10.0 * (1 - 1e-7)]]
    pts[:5] = np.array(special)[:min(P, 5)]
    rho = rng.standard_normal((cl.ntot, R)) + 1j * rng.standard_normal((cl.ntot, R))
    pb = msd.Problem(cl)
    u = pb.nearfield(torch.from_numpy(rho).cuda(), pts).cpu().numpy()
    pb.close()
    d = np.hypot(pts[:, None, 0] - centres[None, :, 0], pts[:, None, 1] - centres[None, :, 1])
    ins = (d <= a).any(axis=1)
    assert ins[0] and (u[ins] == 0).all()
    if (~ins).any():
        ref = O_.single_layer_potential(cl.centres, cl.radii, k, N, rho, pts[~ins])
        assert np.abs(u[~ins] - ref).max() <= 1e-5 * np.abs(ref).max()
