"""The marching interpolation and anterpolation against the oracle's, level by
level, where their tiling can go wrong: 3-row grids whose windows reach both
poles, stencils wider than the compiled ones, parent grids coarser than their
children's, missing children, several right-hand sides, long rows in chunks.

Bars: FP64 spectra 1e-12 (the operations are the oracle's in another order,
sums of at most 16 x 16 terms); FP32 outgoing spectra 1e-5 (some 100 roundings
of 6e-8 per level on sums without cancellation)."""
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

# (sites per side, kept fraction, pitch, L0, modes per kind, columns)
CASES = [
    (7, 1.0, 0.5, 2, 3, 1),       # 3-row child grid, six-fold wider parent stencil
    (9, 0.8, 0.5, 3, 3, 2),       # 4-row child grid: one window position
    (8, 1.0, 1.5, 10, 3, 1),      # parent grid 3.5 times finer (14 transposed taps)
    (9, 0.9, 0.08, 10, 3, 1),     # parent grid coarser than the child's
    (11, 0.6, 0.5, 10, 3, 3),     # missing children, three columns
    (17, 0.15, 0.5, 16, 2, 5),    # sparse, five columns, narrow stencils
    (34, 0.03, 0.5, 10, 2, 1),    # rows in several column chunks
]


@pytest.mark.parametrize("n,keep,pitch,L0,modes,R", CASES)
def test_level_spectra_on_odd_grids(n, keep, pitch, L0, modes, R):
    rng = np.random.default_rng(n)
    C = workloads.lattice(n, n, pitch)
    on = rng.random(len(C)) < keep
    on[[0, -1]] = True
    C = C[on]
    ids = rng.integers(0, 2, len(C)).astype(np.int32)
    shapes = [(0.2 * pitch, modes, modes), (0.3 * pitch, modes, modes)]
    ctx = smr.smr_create(pitch=pitch, L0=L0)
    try:
        smr.add_shapes(ctx, shapes)
        smr.smr_set_scene(ctx, C, ids, 4.0)
        N = smr.smr_info(ctx)["n_unknowns"]
        M = oml.MLFMA(opm.Scene(C, ids, shapes, eps_in=4.0), pitch, L0=L0)
        nl = M.tree.n_levels
        x = np.stack([crandn(N, 7 + r) for r in range(R)], axis=1)
        xd = torch.from_numpy(x).cuda()
        yd = torch.empty_like(xd)
        want = []
        for r in range(R):
            outs = [M.aggregate(x[:, r])]
            for s in range(nl - 1):
                outs.append(M.upward(s, outs[s]))
            ins = [M.translate(s, outs[s]) for s in range(nl)]
            for s in range(nl - 2, -1, -1):
                ins[s] = ins[s] + M.downward(s, ins[s + 1])
            want.append((outs, ins))
        # the built-in rule, and the marching kernels at every level
        for variant in (0, 3):
            smr.smr_set_variant(ctx, smr.SMR_STEP_INTERPOLATE, -1, smr.SMR_PREC_FP64, variant)
            smr.smr_set_variant(ctx, smr.SMR_STEP_ANTERPOLATE, -1, smr.SMR_PREC_FP64, 4 if variant else 0)
            smr.smr_matvec(ctx, xd, yd, smr.SMR_PREC_FP64, R=R)
            torch.cuda.synchronize()
            for s in range(nl):
                go, gi = smr.smr_copy_level(ctx, s, 0, R), smr.smr_copy_level(ctx, s, 1, R)
                for r in range(R):
                    assert rel(go[..., r], want[r][0][s]) < 1e-12, ("out", s, r, variant)
                    assert rel(gi[..., r], want[r][1][s]) < 1e-12, ("in", s, r, variant)
        x1 = xd[:, 0].contiguous()
        y1 = torch.empty_like(x1)
        smr.smr_matvec(ctx, x1, y1, smr.SMR_PREC_FP32)
        smr.smr_sync(ctx)
        for s in range(nl):
            assert rel(smr.smr_copy_level(ctx, s, 0)[..., 0], want[0][0][s]) < 1e-5, ("out fp32", s)
    finally:
        smr.smr_destroy(ctx)
