"""The register-resident cluster kernel (float32, nx = 14): one reduction per
iteration, any CTAs per instance, clusters that split into groups."""
import numpy as np
import pytest
import scipy.sparse.linalg as spla

import oracle
from gpu_util import TOL_F32, TOL_KNOT_F32, knot_err, run_gpu, solver
from workload import gen

pytestmark = pytest.mark.gpu


# knots per CTA: 1 (a CTA faces both neighbours), 2, an empty last CTA, 32, and one CTA alone
@pytest.mark.parametrize("N,C", [(5, 5), (16, 16), (3, 2), (17, 16), (33, 16), (32, 1), (33, 2), (100, 7), (512, 16)])
def test_capped_iterate_at_every_packing(N, C):
    """After m iterations lambda is Algorithm 1's iterate, as in the general
    test of that name (same bar); m stays below the iterations that a tiny
    horizon takes to converge."""
    from paper_2309_08079_gb300.solver import make_opts
    m = 5
    lq = gen.kuka_lq(14, 7, N, 950 + N).astype(np.float32)
    Sd, So, g = oracle.schur_blocks(lq.astype(np.float64))
    lam0 = gen.warm_start(oracle.kkt_solve(lq.astype(np.float64))[0], 950, 0, rel=0.3).astype(np.float32)
    lo, it, _ = oracle.pcg(Sd, So, *oracle.precon_blocks(Sd, So), -g, lam0=lam0, tol=1e-30, max_iter=m)
    lam, _, _, st, _ = run_gpu(lq, lam0=lam0, opts=make_opts(mode=1, cluster=C, tol=1e-30, max_iter=m))
    assert it == m and st["status"][0] == 1 and st["iters"][0] == m, st
    assert oracle.relerr(lam, lo.reshape(lam.shape)) < 1e-3


def test_direct_sum_when_the_identity_cancels():
    """With a badly scaled preconditioner p^T S p falls below 1/16 of
    r~^T S r~, where the kernel sums p^T S p itself; its iterates are still
    Algorithm 1's."""
    import torch
    from paper_2309_08079_gb300.solver import LQTensors, make_opts, read_stats
    N, m = 48, 15
    lq = gen.kuka_lq(14, 7, N, 7).astype(np.float32)
    Sd, So, g = oracle.schur_blocks(lq.astype(np.float64))
    w = 1000.0 ** ((np.arange(N) * 7 % 5) / 4.0)
    Pd, Po = np.linalg.inv(Sd) * w[:, None, None], np.zeros_like(So)
    S, Phi = oracle.block_tridiag_sparse(Sd, So), oracle.block_tridiag_sparse(Pd, Po)
    r = -g.ravel()
    z = Phi @ r
    p, eta, ratio = z.copy(), r @ z, []
    for _ in range(m):
        Sp = S @ p
        ratio.append((p @ Sp) / (z @ (S @ z)))
        r = r - eta / (p @ Sp) * Sp
        z = Phi @ r
        eta, p = r @ z, z + (r @ z) / eta * p
    assert min(ratio) < 1 / 16 < max(ratio), ratio
    lo, _, _ = oracle.pcg(Sd, So, Pd, Po, -g, tol=1e-30, max_iter=m)
    s = solver()
    lt = LQTensors.from_numpy(lq)
    sch = s.alloc_schur(lt)
    s.form(lt, sch)
    sch.Pd.copy_(torch.as_tensor(Pd))
    sch.Po.zero_()
    lam = torch.zeros(N, 14, device="cuda")
    st = read_stats(s.pcg_solve(lt, sch, lam, make_opts(mode=1, tol=1e-30, max_iter=m)))
    assert st["status"][0] == 1 and st["iters"][0] == m, st
    assert oracle.relerr(lam.cpu().double().numpy().ravel(), lo) < 1e-3


@pytest.mark.parametrize("B,N_lo,N_hi", [(60, 1, 512), (200, 30, 70), (90, 120, 130), (20, 33, 512)])
def test_more_instances_than_clusters(B, N_lo, N_hi):
    """A queue of instances longer than the co-resident clusters: every group
    size down to one CTA, instances at the ends of a class, with one CTA per
    SM (20 instances) and two.  Against the
    exact solution of the S+ that was formed: its rounding alone takes the KKT
    solution of a long horizon to the bar."""
    import torch
    from paper_2309_08079_gb300.solver import LQTensors, make_opts, read_stats
    s = solver()
    Ns = gen.batch_horizons(B, N_lo, N_hi, 11)
    ends = [n for n in (1, 2, 32, 33, 64, 65, 128, 129, 256, 257, 512) if N_lo <= n <= N_hi]
    Ns[:len(ends)] = ends
    batch = gen.kuka_batch(14, 7, Ns, 3300).astype(np.float32)
    lt = LQTensors.from_batch(batch)
    sch = s.alloc_schur(lt)
    s.form(lt, sch)
    sh = s.pcg_shape(lt, sch, make_opts(mode=1))
    assert sh["clusters"] < B, sh
    lam = torch.zeros(lt.total, 14, device="cuda")
    st = read_stats(s.pcg_solve(lt, sch, lam, make_opts(mode=1)))
    assert (st["status"] == 0).all(), st
    lam, Sd, So, g = (t.cpu().double().numpy() for t in (lam, sch.Sd, sch.So, sch.gamma))
    for b, n in enumerate(Ns):
        k0, k1 = batch.knot_off[b], batch.knot_off[b + 1]
        S = oracle.block_tridiag_sparse(Sd[k0:k1], So[k0 - b:k1 - b - 1]).tocsc()
        ref = spla.spsolve(S, -g[k0:k1].ravel()).reshape(n, 14)
        assert oracle.relerr(lam[k0:k1], ref) < TOL_F32 and knot_err(lam[k0:k1], ref) < TOL_KNOT_F32, (b, n)
