"""The product on two circular fields against the FP64 oracle on four: level
spectra and products with an odd number of modes (CUDA-core aggregation and
receive), with more modes than one pass takes, one particle, several right-hand
sides, displaced particles and another background impedance, direct and captured,
and spectra read after other products.

Bars of the other parity tests: FP64 spectra 1e-12, product 1e-10; FP32 spectra
1e-5, product 2e-5."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from oracle import mlfma as oml
from oracle import pmchwt as opm
from paper_2407_21724_gb300 import smr, workloads

from .test_gpu_parity import crandn, rel


@pytest.mark.parametrize("nx,ny,kinds,modes,jitter,R,L0", [
    (1, 1, 1, (2, 1), 0.0, 1, 10), (9, 7, 3, (3, 2), 0.0, 3, 10), (10, 6, 2, (4, 4), 0.02, 2, 10),
    (8, 8, 1, (20, 15), 0.0, 1, 7), (17, 5, 8, (8, 8), 0.0, 1, 12)])
@pytest.mark.parametrize("prec", [smr.SMR_PREC_FP64, smr.SMR_PREC_FP32])
def test_levels_and_product(nx, ny, kinds, modes, jitter, R, L0, prec):
    rng = np.random.default_rng(nx)
    P = workloads.lattice(nx, ny)
    P = P + rng.uniform(-jitter, jitter, P.shape) * [1, 1, 0]
    shapes = [(0.11 + 0.005 * k, *modes) for k in range(kinds)]
    sid = rng.integers(0, kinds, len(P)).astype(np.int32)
    ctx = smr.smr_create(pitch=workloads.PITCH, L0=L0)
    try:
        smr.add_shapes(ctx, shapes)
        smr.smr_set_scene(ctx, P, sid, 4.0)
        M = oml.MLFMA(opm.Scene(P, sid, shapes, eps_in=4.0), workloads.PITCH, L0=L0)
        n = smr.smr_info(ctx)["n_unknowns"]
        X = np.stack([crandn(n, 3 + r) for r in range(R)])
        x = torch.from_numpy(np.ascontiguousarray(X.T)).cuda()
        y, yg = torch.empty_like(x), torch.empty_like(x)
        smr.smr_matvec(ctx, x, y, prec, R=R)
        smr.smr_matvec_graph(ctx, x, yg, prec, R=R)
        smr.smr_sync(ctx)
        cols = 1 if prec == smr.SMR_PREC_FP32 and R > 1 else R          # a split product leaves one column
        bar_l, bar_y = (1e-12, 1e-10) if prec == smr.SMR_PREC_FP64 else (1e-5, 2e-5)
        nlev = M.tree.n_levels
        got = [[smr.smr_copy_level(ctx, s, k, R=cols) for s in range(nlev)] for k in (0, 1)]
        again = smr.smr_copy_level(ctx, 0, 0, R=cols)
        assert np.array_equal(again, got[0][0])                         # reading changes nothing
        if cols < R:
            lanes = smr.smr_info(ctx)["column_lanes"]
            nl = 1 if jitter else max(1, min(R, lanes))
            which = [max(r for r in range(R) if r % nl == 0)]
        else:
            which = range(R)
        for q, r in enumerate(which):
            outs = [M.aggregate(X[r])]
            for s in range(nlev - 1):
                outs.append(M.upward(s, outs[s]))
            ins = [M.translate(s, outs[s]) for s in range(nlev)]
            for s in range(nlev - 2, -1, -1):
                ins[s] = ins[s] + M.downward(s, ins[s + 1])
            for s in range(nlev):
                assert rel(got[0][s][..., q], outs[s]) < bar_l
                if np.linalg.norm(ins[s]) > 0:
                    assert rel(got[1][s][..., q], ins[s]) < bar_l
                else:
                    assert np.all(got[1][s][..., q] == 0)
        for r in range(R):
            ref = M.matvec(X[r])
            assert rel(y.cpu().numpy()[:, r], ref) < bar_y
            assert rel(yg.cpu().numpy()[:, r], ref) < bar_y
    finally:
        smr.smr_destroy(ctx)
