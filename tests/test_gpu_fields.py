"""Far and near fields against the FP64 oracle where the kernels' splits can go
wrong: one direction or point, counts around the tiles of 16 and 32 directions and
of 8 to 128 points, more coefficients than one pass of a tile holds, one particle,
shapes of a few particles each, several solutions, directions that are not unit
vectors, points almost on a particle and far away.

Bar 1e-12: the oracle's sums over some 1e4 terms in another order."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from oracle import pmchwt as opm
from paper_2407_21724_gb300 import smr, workloads

from .test_gpu_parity import crandn, rel


@pytest.mark.parametrize("nx,ny,kinds,modes,R,nd,npt", [
    (1, 1, 1, (2, 1), 1, 1, 1), (5, 4, 3, (3, 3), 2, 16, 8), (7, 5, 9, (3, 2), 1, 33, 9),
    (4, 4, 1, (20, 15), 1, 17, 129), (6, 6, 2, (4, 4), 3, 100, 40)])
def test_fields(nx, ny, kinds, modes, R, nd, npt):
    rng = np.random.default_rng(nd)
    P = workloads.lattice(nx, ny)
    shapes = [(0.1 + 0.005 * k, *modes) for k in range(kinds)]
    sid = rng.integers(0, kinds, len(P)).astype(np.int32)
    ctx = smr.smr_create(pitch=workloads.PITCH)
    try:
        smr.add_shapes(ctx, shapes)
        smr.smr_set_scene(ctx, P, sid, 4.0)
        sc = opm.Scene(P, sid, shapes, eps_in=4.0)
        n = smr.smr_info(ctx)["n_unknowns"]
        X = np.stack([crandn(n, 5 + r) for r in range(R)])
        xd = torch.from_numpy(np.ascontiguousarray(X.T)).cuda()
        u = rng.standard_normal((nd, 3))
        u /= np.linalg.norm(u, axis=1)[:, None]
        u[0] = [0, 0, 1]
        u[nd // 2] *= 1.3
        pts = rng.uniform(-2, 2, (npt, 3))
        pts[:, 2] = rng.uniform(0.4, 3, npt)
        pts[0] = P[0] + [0, 0, shapes[sid[0]][0] + 1e-3]
        pts[-1] = [200.0, -100.0, 300.0] if npt > 1 else pts[-1]
        F = torch.empty(nd * 3 * R, dtype=torch.complex128, device="cuda")
        EH = torch.empty(npt * 6 * R, dtype=torch.complex128, device="cuda")
        smr.smr_far_field(ctx, xd, u, F, R=R)
        smr.smr_near_field(ctx, xd, pts, EH, R=R)
        torch.cuda.synchronize()
        F, EH = F.cpu().numpy().reshape(nd, 3, R), EH.cpu().numpy().reshape(npt, 6, R)
        for r in range(R):
            assert rel(F[:, :, r], opm.far_field(sc, X[r], u)) < 1e-12
            E0, H0 = opm.near_field(sc, X[r], pts)
            for i in range(npt):
                assert rel(EH[i, :3, r], E0[i]) < 1e-12
                assert rel(EH[i, 3:, r], H0[i]) < 1e-12
    finally:
        smr.smr_destroy(ctx)
