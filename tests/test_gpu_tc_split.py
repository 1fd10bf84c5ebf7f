"""Tensor-core receive with its K chunks split over CTAs, and aggregation split
over M-tile pairs, where the splits can go wrong: a single particle, counts on
both sides of a 96-particle tile, several shapes with a nearly empty tile each,
enough tiles that nothing is split, odd chunk counts (L0), several right-hand
sides on concurrent lanes, direct and captured products.

Bars: the 3-term split against the CUDA cores' FP32 product 5e-6, against the
FP64 product 2e-5, the bars of the other tensor-core tests."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_2407_21724_gb300 import smr, workloads

from .test_gpu_parity import crandn, rel


@pytest.mark.parametrize("nx,ny,kinds,L0,R", [(1, 1, 1, 10, 1), (19, 5, 1, 10, 1), (12, 8, 1, 7, 2), (97, 1, 1, 12, 1),
                                              (11, 10, 5, 10, 5), (30, 30, 13, 8, 3), (121, 121, 1, 10, 1)])
def test_split_products(nx, ny, kinds, L0, R):
    P = workloads.lattice(nx, ny)
    ctx = smr.smr_create(pitch=workloads.PITCH, L0=L0)
    try:
        smr.add_shapes(ctx, [(0.12 + 0.01 * k, 3, 3) for k in range(kinds)])
        sid = np.minimum(np.arange(len(P)) // 7, kinds - 1).astype(np.int32)     # a few of each, the rest of the last
        smr.smr_set_scene(ctx, P, sid, 4.0)
        n = smr.smr_info(ctx)["n_unknowns"]
        x = torch.from_numpy(np.stack([crandn(n, 5 + r) for r in range(R)])).cuda()
        y64, y32, yg, yc = (torch.empty_like(x) for _ in range(4))
        smr.smr_matvec(ctx, x, y64, smr.SMR_PREC_FP64)
        smr.smr_matvec(ctx, x, y32, smr.SMR_PREC_FP32)
        smr.smr_matvec_graph(ctx, x, yg, smr.SMR_PREC_FP32)
        smr.smr_sync(ctx)
        smr.smr_set_tensor_cores(ctx, False)
        smr.smr_matvec(ctx, x, yc, smr.SMR_PREC_FP32)
        smr.smr_sync(ctx)
        y64, y32, yg, yc = (t.cpu().numpy() for t in (y64, y32, yg, yc))
        for r in range(R):
            for y in (y32, yg):
                assert rel(y[r], yc[r]) < 5e-6
                assert rel(y[r], y64[r]) < 2e-5
    finally:
        smr.smr_destroy(ctx)
