"""Products of arrays with sites tens of wavelengths apart: the parent grid is
hundreds of times finer than the child's, so a child column's transposed stencil
has some 800 taps (marching anterpolation in chunks of one column; in FP64 the taps
take two launches).  The marching kernel in FP64, alone and for two columns, and in
FP32 against the FP64 gather kernel, which the oracle tests check.

Bars: FP64 spectra 1e-12, product 1e-10.  FP32 spectra 1e-5: a sum of n terms of
random phase is rounded to about 6e-8 sqrt(n / 2) of itself, here twice with n
near 1000, 3e-6; product 2e-5."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_2407_21724_gb300 import smr, workloads

from .test_gpu_parity import crandn, rel


def test_eight_hundred_tap_stencils():
    pitch = 33.0
    C = workloads.lattice(7, 2, pitch)
    ctx = smr.smr_create(pitch=pitch, L0=2)
    try:
        smr.add_shapes(ctx, [(0.2, 2, 2)])
        smr.smr_set_scene(ctx, C, np.zeros(len(C), dtype=np.int32), 4.0)
        info = smr.smr_info(ctx)
        assert info["n_levels"] == 2 and info["L"][1] > 614
        X = np.stack([crandn(info["n_unknowns"], 11 + r) for r in range(2)], axis=1)

        def product(cols, prec, anterp):
            smr.smr_set_variant(ctx, smr.SMR_STEP_ANTERPOLATE, -1, prec, anterp)
            x = torch.from_numpy(np.ascontiguousarray(X[:, cols])).cuda()
            y = torch.empty_like(x)
            smr.smr_matvec(ctx, x, y, prec, R=len(cols))
            smr.smr_sync(ctx)
            return smr.smr_copy_level(ctx, 0, 1, len(cols)), y.cpu().numpy()

        want = [product([r], smr.SMR_PREC_FP64, 1) for r in range(2)]
        for cols, prec, bar_l, bar_y in (([0], smr.SMR_PREC_FP64, 1e-12, 1e-10), ([0, 1], smr.SMR_PREC_FP64, 1e-12, 1e-10),
                                         ([1], smr.SMR_PREC_FP32, 1e-5, 2e-5)):
            ins, y = product(cols, prec, 4)
            for q, r in enumerate(cols):
                assert rel(ins[..., q], want[r][0][..., 0]) < bar_l, (cols, prec)
                assert rel(y[:, q], want[r][1][:, 0]) < bar_y, (cols, prec)
    finally:
        smr.smr_destroy(ctx)
