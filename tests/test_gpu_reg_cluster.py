"""The cluster kernels with one reduction per iteration: float32 nx = 14 (any CTAs
per instance, clusters that split into groups), float32 nx = 36 and float64 nx
= 14 (a lane per row)."""
import numpy as np
import pytest
import scipy.sparse.linalg as spla

import oracle
from gpu_util import TOL_F32, TOL_KNOT_F32, knot_err, run_gpu, solver
from workload import gen

pytestmark = pytest.mark.gpu


# knots per CTA: 1 (a CTA faces both neighbours), 2, an empty last CTA, the
# largest of each variant, and one CTA alone
@pytest.mark.parametrize("nx,nu,dtype,N,C", [
    (14, 7, "float32", 5, 5), (14, 7, "float32", 16, 16), (14, 7, "float32", 3, 2), (14, 7, "float32", 17, 16),
    (14, 7, "float32", 33, 16), (14, 7, "float32", 32, 1), (14, 7, "float32", 33, 2), (14, 7, "float32", 100, 7),
    (14, 7, "float32", 512, 16), (36, 12, "float32", 16, 16), (36, 12, "float32", 17, 16), (36, 12, "float32", 6, 1),
    (36, 12, "float32", 8, 1), (36, 12, "float32", 24, 4), (36, 12, "float32", 27, 4), (36, 12, "float32", 128, 16),
    (14, 7, "float64", 7, 7), (14, 7, "float64", 16, 1), (14, 7, "float64", 33, 16), (14, 7, "float64", 250, 16)])
def test_capped_iterate_at_every_packing(nx, nu, dtype, N, C):
    """After m iterations lambda is Algorithm 1's iterate, as in the general
    test of that name (same bars); m stays below the iterations that a tiny
    horizon takes to converge."""
    from paper_2309_08079_gb300.solver import make_opts
    m = 5
    lq = gen.kuka_lq(nx, nu, N, 950 + N).astype(dtype)
    Sd, So, g = oracle.schur_blocks(lq.astype(np.float64))
    lam0 = gen.warm_start(oracle.kkt_solve(lq.astype(np.float64))[0], 950, 0, rel=0.3).astype(dtype)
    lo, it, _ = oracle.pcg(Sd, So, *oracle.precon_blocks(Sd, So), -g, lam0=lam0, tol=1e-30, max_iter=m)
    lam, _, _, st, _ = run_gpu(lq, dtype, lam0=lam0, opts=make_opts(mode=1, cluster=C, tol=1e-30, max_iter=m))
    assert it == m and st["status"][0] == 1 and st["iters"][0] == m, st
    assert oracle.relerr(lam, lo.reshape(lam.shape)) < (1e-3 if dtype == "float32" else 1e-9)


@pytest.mark.parametrize("N,C", [(2, 1), (3, 2), (4, 1), (20, 16), (31, 16), (64, 16), (65, 16), (8, 1), (9, 1), (115, 16), (128, 16)])
def test_capped_iterate_with_lanes_per_row(N, C):
    """float64: four lanes a row up to 2 knots per CTA, two up to 8."""
    test_capped_iterate_at_every_packing(14, 7, "float64", N, C)


@pytest.mark.parametrize("nx,nu,dtype", [(14, 7, "float32"), (36, 12, "float32"), (14, 7, "float64")])
@pytest.mark.parametrize("N", [16, 48])
def test_direct_sum_when_the_identity_cancels(nx, nu, dtype, N):
    """With a badly scaled preconditioner p^T S p falls below 1/16 of
    r~^T S r~, where the kernel sums p^T S p itself; its iterates are still
    Algorithm 1's.  N = 16: one knot per CTA."""
    import torch
    from paper_2309_08079_gb300.solver import LQTensors, make_opts, read_stats
    t = getattr(torch, dtype)
    lq = gen.kuka_lq(nx, nu, N, 7).astype(dtype)
    Sd, So, g = oracle.schur_blocks(lq.astype(np.float64))
    w = 1000.0 ** ((np.arange(N) * 7 % 5) / 4.0)
    Pd, Po = np.linalg.inv(Sd) * w[:, None, None], np.zeros_like(So)
    S, Phi = oracle.block_tridiag_sparse(Sd, So), oracle.block_tridiag_sparse(Pd, Po)
    r = -g.ravel()
    z = Phi @ r
    p, eta, ratio = z.copy(), r @ z, []
    while not ratio or min(ratio) >= 1 / 16:  # run past the first such iteration
        Sp = S @ p
        ratio.append((p @ Sp) / (z @ (S @ z)))
        r = r - eta / (p @ Sp) * Sp
        z = Phi @ r
        eta, p = r @ z, z + (r @ z) / eta * p
        assert len(ratio) < 40
    m = len(ratio) + 1
    lo, _, _ = oracle.pcg(Sd, So, Pd, Po, -g, tol=1e-30, max_iter=m)
    s = solver()
    lt = LQTensors.from_numpy(lq, dtype=t)
    sch = s.alloc_schur(lt)
    s.form(lt, sch)
    sch.Pd.copy_(torch.as_tensor(Pd))
    sch.Po.zero_()
    lam = torch.zeros(N, nx, dtype=t, device="cuda")
    st = read_stats(s.pcg_solve(lt, sch, lam, make_opts(mode=1, cluster=16, tol=1e-30, max_iter=m)))
    assert st["status"][0] == 1 and st["iters"][0] == m, st
    assert oracle.relerr(lam.cpu().double().numpy().ravel(), lo) < (1e-3 if dtype == "float32" else 1e-9)


@pytest.mark.parametrize("nx,nu,dtype,C", [(36, 12, "float32", 4), (14, 7, "float64", 2)])
def test_lane_per_row_queue(nx, nu, dtype, C):
    """More instances than co-resident clusters, one of them flagged."""
    import torch
    from paper_2309_08079_gb300.solver import LQTensors, make_opts, read_stats
    s = solver()
    Ns = [(i * 5) % 23 + 2 for i in range(200)]
    items = [gen.kuka_lq(nx, nu, n, 3400 + i) for i, n in enumerate(Ns)]
    items[5].Qd[0, 0] = 0.0
    batch = gen.concat_batch(items).astype(dtype)
    lt = LQTensors.from_batch(batch, dtype=getattr(torch, dtype))
    sch = s.alloc_schur(lt)
    s.form(lt, sch)
    o = make_opts(mode=1, cluster=C, tol=1e-6 if dtype == "float32" else 1e-13)
    assert s.pcg_shape(lt, sch, o)["clusters"] < len(Ns)
    lam = torch.full((lt.total, nx), 0.25, dtype=lt.dtype, device="cuda")
    st = read_stats(s.pcg_solve(lt, sch, lam, o))
    lam, Sd, So, g = (x.cpu().double().numpy() for x in (lam, sch.Sd, sch.So, sch.gamma))
    for b, n in enumerate(Ns):
        k0, k1 = batch.knot_off[b], batch.knot_off[b + 1]
        if b == 5:
            assert st["status"][b] == 4 and np.all(lam[k0:k1] == 0.25)
            continue
        ref = spla.spsolve(oracle.block_tridiag_sparse(Sd[k0:k1], So[k0 - b:k1 - b - 1]).tocsc(), -g[k0:k1].ravel())
        assert st["status"][b] == 0 and oracle.relerr(lam[k0:k1].ravel(), ref) < (TOL_F32 if dtype == "float32" else 1e-9), b


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


@pytest.mark.parametrize("B,top,C", [(60, 512, 16), (20, 512, 16), (60, 384, 12), (20, 257, 12), (70, 256, 8), (20, 256, 8),
                                     (60, 192, 6), (90, 128, 4), (40, 128, 4), (90, 96, 3), (300, 96, 3), (100, 64, 1), (200, 33, 1)])
def test_stages_of_a_ragged_batch(B, top, C):
    """Horizons at the ends of every stage's range, from batches that the
    device leaves to the form in registers (40 of 128, 20 of 512) to those of
    many waves; one instance flagged, one
    longer than a cluster of the launch holds; the launches of a captured graph give
    the same lambda, bit for bit."""
    import torch
    from paper_2309_08079_gb300.solver import LQTensors, make_opts, read_stats
    s = solver()
    edges = [n for n in (top, 385, 384, 257, 256, 193, 192, 129, 128, 97, 96, 65, 64, 48, 33, 32, 1) if n <= top]
    Ns = edges + gen.batch_horizons(B - 1 - len(edges), 2, min(top, 130), 12).tolist() + [(32 if C > 1 else 64) * C + 1]
    items = [gen.kuka_lq(14, 7, int(n), 3500 + i) for i, n in enumerate(Ns)]
    items[2].Qd[0, 0] = 0.0
    batch = gen.concat_batch(items).astype(np.float32)
    lt = LQTensors.from_batch(batch)
    sch, stats, ws = s.alloc_schur(lt), s.alloc_stats(lt.nb), s.alloc_workspace(lt)
    s.form(lt, sch)
    o = make_opts()
    assert s.pcg_shape(lt, sch, o, N=top)["C"] == C
    lam = torch.full((lt.total, 14), 0.25, device="cuda")
    s.pcg_solve(lt, sch, lam, o, stats, ws, N=top)
    torch.cuda.synchronize()
    st = read_stats(stats)
    again = torch.empty_like(lam)
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        again.fill_(0.25)
        s.pcg_solve(lt, sch, again, o, stats, ws, N=top)
        after = again + 0.0  # ordered behind every stage
    for _ in range(3):
        g.replay()
        torch.cuda.synchronize()
        assert torch.equal(again, lam) and torch.equal(after, lam)
    lam, Sd, So, gam = (t.cpu().double().numpy() for t in (lam, sch.Sd, sch.So, sch.gamma))
    for b, n in enumerate(Ns):
        k0, k1 = batch.knot_off[b], batch.knot_off[b + 1]
        if b in (2, B - 1):
            assert st["status"][b] == 4 and np.all(lam[k0:k1] == 0.25), (b, n)
            continue
        S = oracle.block_tridiag_sparse(Sd[k0:k1], So[k0 - b:k1 - b - 1]).tocsc()
        ref = spla.spsolve(S, -gam[k0:k1].ravel()).reshape(n, 14)
        assert st["status"][b] == 0 and oracle.relerr(lam[k0:k1], ref) < TOL_F32, (b, n)


@pytest.mark.parametrize("nx,nu,N,seed,scale,shift,precon", [
    (14, 7, 6, 9, 2.0, 0.42199, 2), (14, 7, 40, 0, 3.0, 0.42199, 2), (36, 12, 6, 19, 3.0, 0.39835, 2),
    (14, 7, 16, 2, 1.0, 0.05, 0), (36, 12, 16, 0, 1.0, 0.05, 0)])
@pytest.mark.parametrize("dtype", ["float32", "float64"])
def test_breakdown_after_the_first_iteration(nx, nu, N, seed, scale, shift, precon, dtype):
    """S+ made indefinite so that p^T S p turns negative in a later iteration, by
    a small share of |r~^T S r~| where the preconditioner is not symmetric:
    MPCG_BREAKDOWN in the iteration of Algorithm 1.  (Smallest |p^T S p| over
    the sum of the identity's terms: 8e-3, against 1e-6 of rounding.)"""
    import torch
    from paper_2309_08079_gb300.solver import LQTensors, make_opts, read_stats
    t = getattr(torch, dtype)
    lq = gen.kuka_lq(nx, nu, N, seed)
    Sd, So, g = oracle.schur_blocks(lq)
    Pd, Po = oracle.precon_blocks(Sd, So)
    Po = scale * Po
    rng = np.random.default_rng(seed)
    for k in range(N):
        if rng.random() < 0.5:
            Sd[k] -= shift * np.trace(Sd[k]) / nx * np.eye(nx)
    S, P = oracle.block_tridiag_sparse(Sd, So), oracle.block_tridiag_sparse(Pd, Po).toarray()
    if precon == 2:  # even block rows keep their diagonal block alone
        for k in range(0, N, 2):
            rows = slice(k * nx, (k + 1) * nx)
            P[rows, :k * nx] = 0.0
            P[rows, (k + 1) * nx:] = 0.0
    r = -g.ravel()
    z = P @ r
    p, eta = z.copy(), r @ z
    for it in range(1, 10):
        Sp = S @ p
        if not p @ Sp > 0:
            break
        r = r - eta / (p @ Sp) * Sp
        z = P @ r
        eta, p = r @ z, z + (r @ z) / eta * p
    assert p @ Sp < 0 and it >= 2
    s = solver()
    lt = LQTensors.from_numpy(lq, dtype=t)
    sch = s.alloc_schur(lt)
    s.form(lt, sch)
    for dst, src in ((sch.Sd, Sd), (sch.So, So), (sch.Pd, Pd), (sch.Po, Po), (sch.gamma, g)):
        dst.copy_(torch.as_tensor(src))
    for C in (1 if N <= 8 else 4, 16):
        lam = torch.zeros(N, nx, dtype=t, device="cuda")
        st = read_stats(s.pcg_solve(lt, sch, lam, make_opts(mode=1, cluster=C, precon=precon)))
        assert st["status"][0] == 2 and st["iters"][0] == it, (C, it, st)
        assert torch.isfinite(lam).all()


@pytest.mark.parametrize("nx,nu,dtype,scale,small", [(14, 7, "float32", 85, 20), (36, 12, "float32", 85, 20),
                                                     (14, 7, "float64", 900, 60)])
def test_small_scale(nx, nu, dtype, scale, small):
    """S+ times 2^scale, Phi^-1 as much smaller, gamma 2^-small: r^T r~ and p^T S p
    leave the normal range before the solve ends (no vector does), and 1 / (r^T
    r~) overflows.  As the unscaled problem does, it converges, and the
    residual meets the tolerance to a tenth."""
    import torch
    from paper_2309_08079_gb300.solver import LQTensors, make_opts, read_stats
    t = getattr(torch, dtype)
    N, tol = 64, 1e-3 if dtype == "float32" else 1e-6
    s = solver()
    lt = LQTensors.from_numpy(gen.kuka_lq(nx, nu, N, 31).astype(dtype), dtype=t)
    sch = s.alloc_schur(lt)
    s.form(lt, sch)
    Sd, So, g = (x.cpu().double().numpy() for x in (sch.Sd, sch.So, sch.gamma))
    for x, e in ((sch.Sd, scale), (sch.So, scale), (sch.Pd, -scale), (sch.Po, -scale), (sch.gamma, -small)):
        x.mul_(2.0 ** e)
    for C in (2 if nx == 14 else 8, 16):
        lam = torch.zeros(N, nx, dtype=t, device="cuda")
        st = read_stats(s.pcg_solve(lt, sch, lam, make_opts(mode=1, cluster=C, tol=tol)))
        assert st["status"][0] == 0 and 0 < st["eta"][0] < (2.0 ** -128 if dtype == "float32" else 2.0 ** -1024), st
        y = np.ldexp(lam.cpu().double().numpy().ravel(), scale + small)
        res = oracle.block_tridiag_sparse(Sd, So) @ y + g.ravel()
        assert np.linalg.norm(res) < 1.1 * tol * np.linalg.norm(g)


@pytest.mark.parametrize("nx,nu,N,dtype,dot", [(14, 7, 64, "float32", 0), (14, 7, 64, "float32", 1), (14, 7, 256, "float32", 0),
                                               (36, 12, 64, "float32", 0), (14, 7, 64, "float64", 0)])
def test_steps_are_as_exact_as_with_a_direct_sum(nx, nu, N, dtype, dot):
    """alpha takes the residual to zero along p: the share of v^T r that step v
    leaves, (v^T r_{m+1}) / (v^T r_m), is the relative error of alpha.  Its rms
    over 48 steps of three problems whose solution is white noise (errors of a
    carried p^T S p would show) stays within twice that of the tiled
    kernel, which sums p^T S p itself.  Emulated in float32: both 3e-7 to
    6e-7 per problem; carried in float32 1e-6 to 3e-6."""
    import torch
    from paper_2309_08079_gb300.solver import LQTensors, make_opts
    t = getattr(torch, dtype)
    wide = np.longdouble if dtype == "float64" else np.float64
    s, M, rms = solver(), 48, {1: 0.0, 3: 0.0}
    for seed in range(3):
        lt = LQTensors.from_numpy(gen.kuka_lq(nx, nu, N, seed).astype(dtype), dtype=t)
        sch = s.alloc_schur(lt)
        s.form(lt, sch)
        D, O = (x.cpu().numpy().astype(wide) for x in (sch.Sd, sch.So))

        def mul(v):
            y = (D * v[:, None, :]).sum(2)
            y[1:] += (O * v[:-1, None, :]).sum(2)
            y[:-1] += (O * v[1:, :, None]).sum(1)
            return y
        b = mul(np.random.default_rng(seed).standard_normal((N, nx)).astype(wide)).astype(dtype)
        sch.gamma.copy_(torch.as_tensor(-b))
        for mode in rms:
            lams = [np.zeros((N, nx), wide)]
            for m in range(1, M + 1):
                lam = torch.zeros(N, nx, dtype=t, device="cuda")
                s.pcg_solve(lt, sch, lam, make_opts(mode=mode, tol=1e-30, max_iter=m, dot=dot))
                lams.append(lam.cpu().numpy().astype(wide))
            r = [b - mul(x) for x in lams]
            for m in range(M):
                v = lams[m + 1] - lams[m]
                rms[mode] += float(((v * r[m + 1]).sum() / (v * r[m]).sum()) ** 2) / (3 * M)
    assert np.sqrt(rms[1]) < 2.0 * np.sqrt(rms[3]), {k: np.sqrt(v) for k, v in rms.items()}
    print({k: np.sqrt(v) for k, v in rms.items()})


@pytest.mark.parametrize("nx,nu,dtype,N,C,at_once", [(14, 7, "float64", 32, 4, True), (14, 7, "float64", 32, 16, True),
                                                     (36, 12, "float32", 16, 8, False), (14, 7, "float64", 32, 2, True)])
def test_fixed_cluster_batches_run_at_once_where_that_is_faster(nx, nu, dtype, N, C, at_once):
    """40 instances with a given number of CTAs: in float64 the general kernel,
    which holds them all at once, unless the lane-per-row kernel does; at nx =
    36 the latter in several waves.  The solutions are those of the formed S+."""
    import torch
    from paper_2309_08079_gb300.solver import LQTensors, make_opts, read_stats
    s = solver()
    Ns = [N] * 39 + [N - 3]
    batch = gen.kuka_batch(nx, nu, Ns, 3900).astype(dtype)
    lt = LQTensors.from_batch(batch, dtype=getattr(torch, dtype))
    sch = s.alloc_schur(lt)
    s.form(lt, sch)
    o = make_opts(cluster=C, tol=1e-6 if dtype == "float32" else 1e-13)
    sh = s.pcg_shape(lt, sch, o)
    assert sh["C"] == C and (sh["clusters"] == 40) == at_once, sh
    lam = torch.zeros(lt.total, nx, dtype=lt.dtype, device="cuda")
    st = read_stats(s.pcg_solve(lt, sch, lam, o))
    lam, Sd, So, g = (x.cpu().double().numpy() for x in (lam, sch.Sd, sch.So, sch.gamma))
    for b in (0, 17, 39):
        k0, k1 = batch.knot_off[b], batch.knot_off[b + 1]
        ref = spla.spsolve(oracle.block_tridiag_sparse(Sd[k0:k1], So[k0 - b:k1 - b - 1]).tocsc(), -g[k0:k1].ravel())
        assert st["status"][b] == 0 and oracle.relerr(lam[k0:k1].ravel(), ref) < (TOL_F32 if dtype == "float32" else 1e-9), b


@pytest.mark.parametrize("N,C", [(16, 8), (16, 4), (5, 2)])
def test_fixed_cluster_batch_without_a_workspace(N, C):
    """nx = 36, 40 (80) instances with a given number of CTAs: the general kernel
    holds them all at once and needs no workspace, so the lane-per-row kernel,
    which takes them in turn, needs none either; the same bits as with one."""
    import ctypes

    import torch
    from paper_2309_08079_gb300.solver import LQTensors, make_opts, read_stats
    s = solver()
    B = 80 if N == 5 else 40
    lt = LQTensors.from_batch(gen.kuka_batch(36, 12, [N] * B, 3950).astype(np.float32))
    sch = s.alloc_schur(lt)
    s.form(lt, sch)
    o, ss = make_opts(cluster=C), sch.struct()
    assert s.pcg_shape(lt, sch, o)["clusters"] < B
    out = []
    for ws in (s.alloc_workspace(lt), None):
        lam, st = torch.zeros(lt.total, 36, device="cuda"), s.alloc_stats(B)
        assert s.lib.mpcg_pcg_solve_batched(s.h, lt.dims(), lt.nb, lt.knot_off.data_ptr(), ctypes.byref(ss), lam.data_ptr(),
                                            ctypes.byref(o), st.data_ptr(), None if ws is None else ws.data_ptr(),
                                            torch.cuda.current_stream().cuda_stream) == 0
        assert (read_stats(st)["status"] == 0).all()
        out.append(lam)
    assert torch.equal(*out)
