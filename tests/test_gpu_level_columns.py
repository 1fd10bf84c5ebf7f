"""Anterpolation and the products around it in FP32, and for several columns at once,
against the oracle: the marching and the gather kernel forced in turn where the grids
give both (stencils of more than 8 taps), FP32 products of one column
(smr_matvec), near and far parts of several (smr_matvec_parts, whose FP32 kernels run
all columns together).  The grids: 3-row and 4-row children, wide stencils, a parent
coarser than its child, missing children, narrow stencils.

Bars: FP64 spectra 1e-12, products 1e-10; FP32 spectra 1e-5, products 2e-5.  Above
the argument k r of the closest translation, 4 pi pitch, the factors grow with the
order like the Hankel function and cancel in the receive, which loses their digits:
orders of more than 4 pi pitch + 5 are left out of the FP32 products, and a pitch of
0.08 wavelengths at order 10 (factors of 1e9) out of the FP64 far parts too."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from oracle import mlfma as oml
from oracle import pmchwt as opm
from paper_2407_21724_gb300 import smr, workloads

from .test_gpu_march import CASES
from .test_gpu_parity import crandn, rel

F64, F32 = smr.SMR_PREC_FP64, smr.SMR_PREC_FP32


@pytest.mark.parametrize("n,keep,pitch,L0,modes", sorted({c[:5] for c in CASES} | {(12, 1.0, 2.0, 4, 2)}))
def test_anterpolation_and_parts(n, keep, pitch, L0, modes):
    rng = np.random.default_rng(n)
    C = workloads.lattice(n, n, pitch)
    on = rng.random(len(C)) < keep
    on[[0, -1]] = True
    C = C[on]
    ids = rng.integers(0, 2, len(C)).astype(np.int32)
    size = min(pitch, 1.0)
    shapes = [(0.2 * size, modes, modes), (0.3 * size, modes, modes)]
    ctx = smr.smr_create(pitch=pitch, L0=L0)
    try:
        smr.add_shapes(ctx, shapes)
        smr.smr_set_scene(ctx, C, ids, 4.0)
        well = L0 <= 4 * np.pi * pitch + 5
        N = smr.smr_info(ctx)["n_unknowns"]
        M = oml.MLFMA(opm.Scene(C, ids, shapes, eps_in=4.0), pitch, L0=L0)
        nl = M.tree.n_levels
        X = np.stack([crandn(N, 17 + r) for r in range(3)], axis=1)
        want = []
        for r in range(3):
            outs = [M.aggregate(X[:, r])]
            for s in range(nl - 1):
                outs.append(M.upward(s, outs[s]))
            ins = [M.translate(s, outs[s]) for s in range(nl)]
            for s in range(nl - 2, -1, -1):
                ins[s] = ins[s] + M.downward(s, ins[s + 1])
            want.append((outs, ins, M.near(X[:, r]), M.receive(ins[0])))

        def spectra(R, bar, what):
            for s in range(nl):
                for k in (0, 1):
                    g = smr.smr_copy_level(ctx, s, k, R)
                    for r in range(R):
                        assert rel(g[..., r], want[r][k][s]) < bar, (what, s, k, r)

        x = torch.from_numpy(X).cuda()
        x1 = x[:, 0].contiguous()
        for variant in (0, 1, 2, 4):
            for prec in (F64, F32):
                smr.smr_set_variant(ctx, smr.SMR_STEP_ANTERPOLATE, -1, prec, variant)
            y1, near, far = torch.empty_like(x1), torch.empty_like(x), torch.empty_like(x)
            smr.smr_matvec(ctx, x1, y1, F32)
            smr.smr_sync(ctx)
            spectra(1, 1e-5, ("fp32", variant))
            if well:
                assert rel(y1.cpu().numpy(), want[0][2] + want[0][3]) < 2e-5, variant
            for prec, bar_l, bar_y in ((F64, 1e-12, 1e-10), (F32, 1e-5, 2e-5)):
                smr.smr_matvec_parts(ctx, x, near, far, prec, R=3)
                smr.smr_sync(ctx)
                spectra(3, bar_l, (prec, "columns", variant))
                for r in range(3):
                    assert rel(near[:, r].cpu().numpy(), want[r][2]) < bar_y, (prec, variant, r)
                    if well or (prec == F64 and pitch > 0.1):
                        assert rel(far[:, r].cpu().numpy(), want[r][3]) < bar_y, (prec, variant, r)
    finally:
        smr.smr_destroy(ctx)
