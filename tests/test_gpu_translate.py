"""The FP32 translation's 4x4 target tiles against the FP64 one, level by level,
where the tiling can go wrong: levels that start off a tile's corner, partial
tiles, windows with missing rows and boxes, single boxes, direction counts that
leave part of a chunk, several arrays with empty tiles between them.

Bar: incoming spectra before anterpolation are sums of at most 27 products; the
received product after all levels stays within the FP32 bar of 2e-5, and the
top level's incoming spectrum (translation alone) within 2e-6 (some 30 roundings
of 6e-8 on random signs)."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_2407_21724_gb300 import smr, workloads

from .test_gpu_parity import crandn, rel


@pytest.mark.parametrize("nx,ny,keep,L0", [(3, 3, 1.0, 10), (4, 1, 1.0, 10), (1, 9, 1.0, 7), (9, 6, 0.5, 10),
                                           (17, 13, 0.9, 10), (23, 5, 0.25, 12), (33, 33, 0.04, 10)])
def test_tiles_against_fp64(nx, ny, keep, L0):
    rng = np.random.default_rng(nx * ny)
    C = workloads.lattice(nx, ny)
    on = rng.random(len(C)) < keep
    on[[0, -1]] = True
    ctx = smr.smr_create(pitch=workloads.PITCH, L0=L0)
    try:
        smr.add_shapes(ctx, [(0.15, 3, 3)])
        # two copies: the second array starts elsewhere on the common lattice
        P = np.concatenate([C[on], C[on][: max(2, on.sum() // 2)]])
        A = np.concatenate([np.zeros(on.sum(), dtype=np.int32), np.ones(len(P) - on.sum(), dtype=np.int32)])
        smr.smr_set_scene_arrays(ctx, P, np.zeros(len(P), dtype=np.int32), A, 4.0)
        info = smr.smr_info(ctx)
        x = torch.from_numpy(crandn(info["n_unknowns"], 3)).cuda()
        y64, y32 = torch.empty_like(x), torch.empty_like(x)
        top = info["n_levels"] - 1
        smr.smr_matvec(ctx, x, y64, smr.SMR_PREC_FP64)
        torch.cuda.synchronize()
        t64 = smr.smr_copy_level(ctx, top, 1)
        smr.smr_matvec(ctx, x, y32, smr.SMR_PREC_FP32)
        smr.smr_sync(ctx)
        t32 = smr.smr_copy_level(ctx, top, 1)
        if np.linalg.norm(t64) > 0:
            assert rel(t32, t64) < 2e-6
        else:
            assert np.all(t32 == 0)
        assert rel(y32.cpu().numpy(), y64.cpu().numpy()) < 2e-5
    finally:
        smr.smr_destroy(ctx)
