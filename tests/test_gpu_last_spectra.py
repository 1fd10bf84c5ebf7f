"""smr_copy_level returns the spectra of the last product, whatever ran it."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_2407_21724_gb300 import smr, workloads

from .test_gpu_parity import crandn, rel


@pytest.fixture(scope="module")
def scene():
    ctx = smr.scene_from_workload(workloads.make("random", n=7, modes=6))
    yield ctx, smr.smr_info(ctx)["n_unknowns"]
    smr.smr_destroy(ctx)


def test_replayed_product_is_the_last_one(scene):
    """FP32 captured, FP64, FP32 replayed: the fields read are the FP32 product's,
    the very bits read after its capture (the kernels sum in a fixed order)."""
    ctx, n = scene
    x, u = (torch.from_numpy(crandn(n, s)).cuda() for s in (1, 2))
    y, v = torch.empty_like(x), torch.empty_like(x)
    smr.smr_matvec_graph(ctx, x, y, smr.SMR_PREC_FP32)
    smr.smr_sync(ctx)
    want = [smr.smr_copy_level(ctx, 0, k) for k in (0, 1)]
    smr.smr_matvec(ctx, u, v, smr.SMR_PREC_FP64)
    other = smr.smr_copy_level(ctx, 0, 0)
    smr.smr_matvec_graph(ctx, x, y, smr.SMR_PREC_FP32)
    smr.smr_sync(ctx)
    got = [smr.smr_copy_level(ctx, 0, k) for k in (0, 1)]
    assert rel(got[0], other) > 0.1
    assert all(np.array_equal(a, b) for a, b in zip(got, want))


@pytest.mark.parametrize("prec", [smr.SMR_PREC_FP64, smr.SMR_PREC_FP32])
def test_fields_combine_to_the_stored_spectra(scene, prec):
    """The fields read give the two combinations that the product stored, also when
    the launches it would now run have changed (tensor cores off: other FP32
    sums): equal to FP64 rounding of the few sums between, 1e-14, where another
    FP32 product's are 1e-8 to 1e-6 off."""
    ctx, n = scene
    nlev = smr.smr_info(ctx)["n_levels"]
    x = torch.from_numpy(crandn(n, 5)).cuda()
    y = torch.empty_like(x)

    def stored():
        out = []
        for s in range(nlev):
            for k in (0, 1):
                B = smr.smr_copy_level(ctx, s, k)[..., 0]
                out.append(np.stack([B[:, :, 0] + B[:, :, 3], B[:, :, 2] - B[:, :, 1]]))
        return out

    try:
        smr.smr_matvec_graph(ctx, x, y, prec)
        smr.smr_sync(ctx)
        want = stored()
        smr.smr_set_tensor_cores(ctx, 0)
        got = stored()
        assert all(rel(a, b) < 1e-14 if np.any(b) else not np.any(a) for a, b in zip(got, want))
        if prec == smr.SMR_PREC_FP32:
            smr.smr_matvec(ctx, x, y, prec)
            smr.smr_sync(ctx)
            assert rel(stored()[0], want[0]) > 1e-9       # the change of launches does show
    finally:
        smr.smr_set_tensor_cores(ctx, 1)


@pytest.mark.parametrize("prec,R,columns", [(smr.SMR_PREC_FP64, 1, 1), (smr.SMR_PREC_FP64, 3, 3),
                                            (smr.SMR_PREC_FP32, 1, 1), (smr.SMR_PREC_FP32, 3, 1)])
def test_profile_lists_the_copy_of_the_coefficients(scene, prec, R, columns):
    ctx, n = scene
    x = torch.from_numpy(np.stack([crandn(n, r) for r in range(R)], axis=1)).cuda()
    recs = [r for r in smr.smr_profile_matvec(ctx, x, torch.empty_like(x), prec, R=R) if r["name"] == "keep"]
    assert [(r["level"], r["bytes"]) for r in recs] == [(-1, 2.0 * 16 * n * columns)] and recs[0]["ms"] > 0
