"""Captured products of several columns outlive larger products of the same
context: an FP32 product with more columns takes new column buffers, and a graph
captured on the old ones must not be replayed on them.

Bar: the FP32 product's 2e-5 against FP64; a replay on released buffers is off by
order one."""
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_2407_21724_gb300 import smr, workloads


@pytest.mark.parametrize("cols", [(2, 5, 2), (3, 2, 9, 3, 2, 9), (1, 4, 6, 1, 4)])
def test_replays_after_larger_products(cols):
    ctx = smr.scene_from_workload(workloads.make("random", n=6, modes=4))
    try:
        n = smr.smr_info(ctx)["n_unknowns"]
        pairs = {}
        for R in sorted(set(cols)):
            g = torch.Generator(device="cuda").manual_seed(R)
            x = torch.randn((n, R), dtype=torch.complex128, device="cuda", generator=g)
            want = torch.empty_like(x)
            smr.smr_matvec(ctx, x, want, smr.SMR_PREC_FP64, R=R)
            pairs[R] = (x, torch.empty_like(x), want)
        for R in cols:
            x, y, want = pairs[R]
            y.fill_(float("nan"))
            smr.smr_matvec_graph(ctx, x, y, smr.SMR_PREC_FP32, R=R)
            smr.smr_sync(ctx)
            err = (y - want).norm(dim=0) / want.norm(dim=0)
            assert err.max().item() < 2e-5, (R, err)
    finally:
        smr.smr_destroy(ctx)
