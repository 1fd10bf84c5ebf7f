"""Arrays in a background of another impedance than 1, against the FP64 oracle: near
blocks, the cluster preconditioner, level spectra and products in FP64 (one and
several columns, direct and captured) and in FP32 (tensor cores and CUDA cores, one
column and the parts of several), fields.  A zeta for a 1 / zeta, or one left out,
shows in every factor of the circular components.

Bars of the other parity tests: blocks, spectra and fields 1e-12, products 1e-10 (each
current's rows by themselves), cluster solves 1e-10; FP32 spectra 1e-5, products 2e-5."""
import types

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from oracle import mlfma as oml
from oracle import pmchwt as opm
from paper_2407_21724_gb300 import smr, workloads

from .test_gpu_parity import _oracle_cluster_apply, crandn, rel

F64, F32 = smr.SMR_PREC_FP64, smr.SMR_PREC_FP32


# zeta 2 and 0.4 at the vacuum's wavenumber; zeta 1 / 1.2 in a denser one, displaced
@pytest.mark.parametrize("eps_out,mu_out,jitter", [(0.5, 2.0, 0.0), (2.5, 0.4, 0.0), (1.44, 1.0, 0.02)])
def test_background_impedance(eps_out, mu_out, jitter):
    rng = np.random.default_rng(8)
    P = workloads.lattice(9, 8)
    P = P + rng.uniform(-jitter, jitter, P.shape) * [1, 1, 0]
    shapes = [(0.12, 4, 4), (0.18, 4, 4)]
    sid = rng.integers(0, 2, len(P)).astype(np.int32)
    ctx = smr.smr_create(pitch=workloads.PITCH)
    try:
        smr.add_shapes(ctx, shapes)
        smr.smr_set_scene(ctx, P, sid, 4.0, eps_out, 1.0, mu_out)
        sc = opm.Scene(P, sid, shapes, eps_in=4.0, eps_out=eps_out, mu_out=mu_out)
        M = oml.MLFMA(sc, workloads.PITCH)
        assert abs(sc.outer.zeta - np.sqrt(mu_out / eps_out)) < 1e-12
        n, nl, R = smr.smr_info(ctx)["n_unknowns"], M.tree.n_levels, 2
        X = np.stack([crandn(n, 3 + r) for r in range(R)], axis=1)
        x = torch.from_numpy(X).cuda()
        cur = np.arange(n) // (n // len(P) // 2) % 2

        for mu, nu in [(0, 0), (0, 1), (1, 0), (10, 20), (20, 10), (30, 29)]:
            ref = M.near_block(mu, nu)
            B = smr.smr_copy_pair_block(ctx, mu, nu)
            h = ref.shape[0] // 2
            for i in (0, 1):
                for j in (0, 1):
                    q = np.s_[i * h:(i + 1) * h, j * h:(j + 1) * h]
                    assert rel(B[q], ref[q]) < 1e-12, (mu, nu, i, j)
        if not jitter:
            z = torch.empty_like(x[:, 0])
            smr.smr_precond_cluster(ctx, x[:, 0].contiguous(), z, F64)
            c = types.SimpleNamespace(w=dict(centres=P, pitch=workloads.PITCH), sc=sc)
            assert rel(z.cpu().numpy(), _oracle_cluster_apply(c, X[:, 0])) < 1e-10

        want = []
        for r in range(R):
            outs = [M.aggregate(X[:, r])]
            for s in range(nl - 1):
                outs.append(M.upward(s, outs[s]))
            ins = [M.translate(s, outs[s]) for s in range(nl)]
            for s in range(nl - 2, -1, -1):
                ins[s] = ins[s] + M.downward(s, ins[s + 1])
            want.append((outs, ins, M.near(X[:, r]), M.receive(ins[0])))

        def spectra(cols, bar, what):
            for s in range(nl):
                for k in (0, 1):
                    g = smr.smr_copy_level(ctx, s, k, len(cols))
                    for q, r in enumerate(cols):
                        assert rel(g[..., q], want[r][k][s]) < bar, (what, s, k, r)

        for f in (smr.smr_matvec, smr.smr_matvec_graph):
            y = torch.empty_like(x)
            f(ctx, x, y, F64, R=R)
            torch.cuda.synchronize()
            spectra(range(R), 1e-12, f.__name__)
            for r in range(R):
                for i in (0, 1):
                    ref = (want[r][2] + want[r][3])[cur == i]
                    assert rel(y[:, r].cpu().numpy()[cur == i], ref) < 1e-10, (f.__name__, r, i)
        x1 = x[:, 1].contiguous()
        for tc in (1, 0):
            smr.smr_set_tensor_cores(ctx, tc)
            y = torch.empty_like(x1)
            smr.smr_matvec(ctx, x1, y, F32)
            smr.smr_sync(ctx)
            spectra([1], 1e-5, ("fp32", tc))
            assert rel(y.cpu().numpy(), want[1][2] + want[1][3]) < 2e-5, tc
        near, far = torch.empty_like(x), torch.empty_like(x)
        smr.smr_matvec_parts(ctx, x, near, far, F32, R=R)
        torch.cuda.synchronize()
        for r in range(R):
            assert rel(near[:, r].cpu().numpy(), want[r][2]) < 2e-5
            assert rel(far[:, r].cpu().numpy(), want[r][3]) < 2e-5

        u = rng.standard_normal((5, 3))
        u /= np.linalg.norm(u, axis=1)[:, None]
        pts = rng.uniform(-2, 2, (5, 3)) + [0, 0, 3]
        F = torch.empty((5, 3, R), dtype=torch.complex128, device="cuda")
        EH = torch.empty((5, 6, R), dtype=torch.complex128, device="cuda")
        smr.smr_far_field(ctx, x, u, F, R=R)
        smr.smr_near_field(ctx, x, pts, EH, R=R)
        for r in range(R):
            assert rel(F[:, :, r].cpu().numpy(), opm.far_field(sc, X[:, r], u)) < 1e-12
            E, H = opm.near_field(sc, X[:, r], pts)
            assert rel(EH[:, :3, r].cpu().numpy(), E) < 1e-12 and rel(EH[:, 3:, r].cpu().numpy(), H) < 1e-12
    finally:
        smr.smr_destroy(ctx)
