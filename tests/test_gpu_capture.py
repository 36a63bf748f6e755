"""FP64 products captured into a CUDA graph: a replay after a geometry update
multiplies by the new operator, and a capture leaves nothing behind that a
later product would take for made.  Against the oracle's dense operator,
1e-11 relative as for every FP64 product (formulation: against a problem made
with the new geometry)."""
import numpy as np
import pytest

import oracle.msd_oracle as O_
from paper_1409_8186_gb300 import workloads as W

torch = pytest.importorskip("torch")
pytestmark = [pytest.mark.gpu, pytest.mark.filterwarnings("ignore::RuntimeWarning")]


@pytest.mark.parametrize("pinned", [True, False])
@pytest.mark.parametrize("M,N,R,form", [(70, 10, 1, None), (100, 12, 6, None), (9, 5, 1, None), (40, 8, 2, "cfie")])
def test_replay_after_update(M, N, R, form, pinned):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1409_8186_gb300 import msd
    cl = W.random_cluster(seed=M, M=M, half_side=4.0 * np.sqrt(M) + 2.0, rmin=0.8, rmax=1.0, gap=0.2, k=2.5, N=N)
    rng = np.random.default_rng(M)
    moved = W.Cluster(cl.centres + 0.05 * rng.uniform(-1, 1, cl.centres.shape), cl.radii, cl.bc, cl.k, cl.N)
    resized = W.Cluster(moved.centres, cl.radii * rng.uniform(0.6, 1.0, M), cl.bc, cl.k, cl.N)  # other source groups

    def ref(c, x):
        if form is None:
            return O_.preconditioned_dense(c.centres, c.radii, c.bc, c.k, c.N) @ x.cpu().numpy()
        p = msd.Problem(c)
        p.set_formulation(form)
        p.set_tile(2 * R, msd.MSD_FP64, 5, 1)
        out = p.matvec(x).cpu().numpy()
        p.close()
        return out

    def close(y, r):
        return np.abs(y.cpu().numpy() - r).max() <= 1e-11 * np.abs(r).max()

    s = torch.cuda.Stream()
    with torch.cuda.stream(s):
        pb = msd.Problem(cl)
        if form:
            pb.set_formulation(form)
        if pinned:
            pb.set_tile(R if form is None else 2 * R, msd.MSD_FP64, 0, 1)
        x = torch.from_numpy(rng.standard_normal((cl.ntot, R)) + 1j * rng.standard_normal((cl.ntot, R))).cuda()
        y = torch.empty_like(x)
        assert close(pb.matvec(x), ref(cl, x))
        s.synchronize()
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph, stream=s):
            msd.msd_matvec(pb.handle, R, msd.MSD_FP64, x, y)
        graph.replay()
        assert close(y, ref(cl, x))
        for new in (moved, resized):
            pb.update_geometry(new.centres, new.radii)
            graph.replay()  # before any other product of the new geometry
            assert close(y, ref(new, x))
            assert close(pb.matvec(x), ref(new, x))
            y.zero_()
            graph.replay()  # nothing that it uses was moved by a product of other groups
            assert close(y, ref(new, x))
        pb.update_geometry(cl.centres, cl.radii)
        unused = torch.cuda.CUDAGraph()
        with torch.cuda.graph(unused, stream=s):
            msd.msd_matvec(pb.handle, R, msd.MSD_FP64, x, y)
        assert close(pb.matvec(x), ref(cl, x))
        s.synchronize()
        pb.close()
