"""Solves whose Gram-Schmidt passes split the basis over CTAs and hold one row a
lane, at vector lengths around the segments of 64, 256 and 512 rows, with restarts
(few basis vectors) and several right-hand sides: the true FP64 residual meets the
tolerance, and the mixed solve's solution is the FP64 one's within a hundred times
its tolerance (the operator's condition on these arrays is below that)."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_2407_21724_gb300 import smr, workloads

from .test_gpu_parity import rel


@pytest.mark.parametrize("nx,ny,modes,R,restart", [(1, 1, (2, 1), 1, 0), (8, 8, (2, 2), 1, 0), (9, 7, (3, 2), 1, 5),
                                                   (13, 11, (8, 8), 1, 0), (6, 5, (4, 4), 3, 0)])
def test_solves(nx, ny, modes, R, restart):
    P = workloads.lattice(nx, ny)
    ctx = smr.smr_create(pitch=workloads.PITCH)
    try:
        smr.add_shapes(ctx, [(0.14, *modes)])
        smr.smr_set_scene(ctx, P, np.zeros(len(P), dtype=np.int32), 4.0)
        n = smr.smr_info(ctx)["n_unknowns"]
        kh = np.tile([0.0, 0.0, 1.0], (R, 1))
        pol = np.array([[1, 0, 0], [0, 1, 0], [1, 1j, 0]], dtype=complex)[:R]
        b = torch.empty(n * R, dtype=torch.complex128, device="cuda")
        smr.smr_rhs_plane_waves(ctx, kh, pol, b)
        x, y = torch.empty_like(b), torch.empty_like(b)
        out = []
        for prec, tol in ((smr.SMR_PREC_FP64, 1e-9), (smr.SMR_PREC_FP32, 1e-6)):
            rc, st = smr.smr_solve(ctx, b, x, R=R, tol=tol, precision=prec, maxit=400, max_outer=20, restart=restart)
            smr.smr_matvec(ctx, x, y, smr.SMR_PREC_FP64, R=R)
            torch.cuda.synchronize()
            Y, B = y.cpu().numpy().reshape(n, R), b.cpu().numpy().reshape(n, R)
            for r in range(R):
                assert rel(Y[:, r], B[:, r]) < 1.01 * tol
            out.append(x.cpu().numpy().copy())
        assert rel(out[1], out[0]) < 1e-4
    finally:
        smr.smr_destroy(ctx)
