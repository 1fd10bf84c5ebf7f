"""Far fields of scenes of many shapes over few directions, around the radiation
vectors' tiles of 4 and 16 directions and of 32 modes, against the FP64 oracle.

Bar 1e-12, as for the other field tests: sums of some 1e4 terms in another order."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from oracle import pmchwt as opm
from paper_2407_21724_gb300 import smr, workloads

from .test_gpu_parity import crandn, rel


@pytest.mark.parametrize("kinds,modes", [(12, (2, 1)), (40, (17, 16))])
def test_few_directions(kinds, modes):
    rng = np.random.default_rng(kinds)
    P = workloads.lattice(7, 6)
    shapes = [(0.1 + 0.002 * k, *modes) for k in range(kinds)]
    sid = rng.integers(0, kinds, len(P)).astype(np.int32)
    ctx = smr.smr_create(pitch=workloads.PITCH)
    try:
        smr.add_shapes(ctx, shapes)
        smr.smr_set_scene(ctx, P, sid, 4.0)
        sc = opm.Scene(P, sid, shapes, eps_in=4.0)
        x = crandn(smr.smr_info(ctx)["n_unknowns"], 3)
        xd = torch.from_numpy(x).cuda()
        u = rng.standard_normal((36, 3))
        u /= np.linalg.norm(u, axis=1)[:, None]
        u[0] = [0, 0, 1]
        want = opm.far_field(sc, x, u)
        for nd in (1, 2, 3, 4, 5, 12, 13, 16, 17, 28, 29, 36):
            F = torch.empty(nd * 3, dtype=torch.complex128, device="cuda")
            smr.smr_far_field(ctx, xd, u[:nd], F, R=1)
            assert rel(F.cpu().numpy().reshape(nd, 3), want[:nd]) < 1e-12, nd
    finally:
        smr.smr_destroy(ctx)
