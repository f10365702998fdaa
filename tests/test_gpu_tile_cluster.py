"""The tiled PCG kernel with a cluster of CTAs per instance (float32, nx = 36),
against the exact solution of the S+ that was formed and against the same
kernel with one CTA per instance.

Bars: TOL_F32 / TOL_KNOT_F32 for the solutions, as everywhere; a capped iterate
against Algorithm 1 in float64 at 1e-3, as in test_gpu_reg_cluster.py."""
import ctypes

import numpy as np
import pytest
import scipy.sparse.linalg as spla

import oracle
from gpu_util import TOL_F32, TOL_KNOT_F32, knot_err, run_gpu, solver
from workload import gen

pytestmark = pytest.mark.gpu


def _formed(Ns, seed, flagged=None):
    from paper_2309_08079_gb300.solver import LQTensors
    items = [gen.kuka_lq(36, 12, n, seed + i) for i, n in enumerate(Ns)]
    if flagged is not None:
        items[flagged].Qd[0, 0] = 0.0
    batch = gen.concat_batch(items).astype(np.float32)
    s = solver()
    lt = LQTensors.from_batch(batch)
    sch = s.alloc_schur(lt)
    s.form(lt, sch)
    return s, batch, lt, sch


# every cluster size; horizons below the cluster's CTAs (some have no knots),
# of one knot each, and with unequal shares; more instances than clusters
# (without a workspace too), and fewer
@pytest.mark.parametrize("Ns,C", [
    ([70, 9, 1, 2, 13, 69, 15] * 20, 2), ([33, 1, 3, 4, 5, 17, 40] * 6, 4),
    ([67, 7, 8, 9, 1, 70, 31, 33] * 3, 8), ([130, 15, 16, 17, 5, 1, 131, 150, 2, 33], 16), ([257], 16)])
@pytest.mark.parametrize("queue", [True, False])
def test_solutions_at_every_cluster_size(Ns, C, queue):
    import torch
    from paper_2309_08079_gb300.solver import make_opts, read_stats
    flagged = 3 if len(Ns) > 1 else None
    s, batch, lt, sch = _formed(Ns, 5100, flagged)
    o = make_opts(tol=1e-6, refine_tol=1e-3)
    sh = s.pcg_shape(lt, sch, o)
    assert sh["form"] == "cta_tma" and sh["C"] == C, sh
    ws = s.alloc_workspace(lt)
    stats = s.alloc_stats(lt.nb)
    lam = torch.full((lt.total, 36), 0.25, device="cuda")
    if queue:
        s.pcg_solve(lt, sch, lam, o, stats, ws)
    else:
        ss = sch.struct()
        assert s.lib.mpcg_pcg_solve_batched(s.h, lt.dims(), lt.nb, lt.knot_off.data_ptr(), ctypes.byref(ss), lam.data_ptr(),
                                            ctypes.byref(o), stats.data_ptr(), None, torch.cuda.current_stream().cuda_stream) == 0
    st = read_stats(stats)
    s.refine_step(lt, sch, lam, o, s.alloc_stats(lt.nb), ws)
    lam, Sd, So, g = (x.cpu().double().numpy() for x in (lam, sch.Sd, sch.So, sch.gamma))
    for b, n in enumerate(Ns):
        k0, k1 = batch.knot_off[b], batch.knot_off[b + 1]
        if b == flagged:
            assert st["status"][b] == 4 and np.all(lam[k0:k1] == 0.25)
            continue
        S = oracle.block_tridiag_sparse(Sd[k0:k1], So[k0 - b:k1 - b - 1]).tocsc()
        ref = spla.spsolve(S, -g[k0:k1].ravel()).reshape(n, 36)
        assert st["status"][b] == 0, (b, st[b])
        assert oracle.relerr(lam[k0:k1], ref) < TOL_F32 and knot_err(lam[k0:k1], ref) < TOL_KNOT_F32, (b, n)


@pytest.mark.parametrize("precon", [0, 1, 2])
@pytest.mark.parametrize("N", [129, 200, 255])
def test_capped_iterate(N, precon):
    """After m iterations lambda is Algorithm 1's iterate, and one CTA per
    instance (mode 3) leaves the same to rounding."""
    from paper_2309_08079_gb300.solver import make_opts
    m = 5
    lq = gen.kuka_lq(36, 12, N, 5200 + N).astype(np.float32)
    Sd, So, g = oracle.schur_blocks(lq.astype(np.float64))
    lam0 = gen.warm_start(oracle.kkt_solve(lq.astype(np.float64))[0], 5200, 0, rel=0.3).astype(np.float32)
    got = [run_gpu(lq, lam0=lam0, opts=make_opts(mode=mode, tol=1e-30, max_iter=m, precon=precon)) for mode in (0, 3)]
    for lam, _, _, st, _ in got:
        assert st["status"][0] == 1 and st["iters"][0] == m, st
    assert oracle.relerr(got[0][0], got[1][0]) < 1e-4
    if precon == 0:
        lo, it, _ = oracle.pcg(Sd, So, *oracle.precon_blocks(Sd, So), -g, lam0=lam0, tol=1e-30, max_iter=m)
        assert it == m and oracle.relerr(got[0][0], lo.reshape(N, 36)) < 1e-3


def _capped(s, lt, sch, mode, m=4, lam0=0.25):
    import torch
    from paper_2309_08079_gb300.solver import make_opts
    lam = torch.full((lt.total, 36), lam0, device="cuda")
    s.pcg_solve(lt, sch, lam, make_opts(mode=mode, tol=1e-30, max_iter=m), s.alloc_stats(lt.nb), s.alloc_workspace(lt))
    return lam


def _median_ms(f):
    import torch
    f()
    t = []
    for _ in range(9):
        a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        a.record()
        f()
        b.record()
        b.synchronize()
        t.append(a.elapsed_time(b))
    return sorted(t)[4]


@pytest.mark.parametrize("Ns,one", [([200] * 152, True), ([72] * 100, True), ([100] * 120, True), ([256, 64, 80, 90] * 40, False),
                                    ([160] * 60, False)])
def test_batch_takes_the_form_that_its_horizons_favour(Ns, one):
    """Equal horizons that fill the GPU run with a CTA per instance: the bits of
    mode 3 (which has no other form), eagerly, from a captured graph and with a
    padded list, and within 1.1 of its time (clusters took 1.3).  Ragged ones,
    and few, run with clusters: other bits (another order of sums), less time."""
    import torch
    from paper_2309_08079_gb300.solver import make_opts
    s, batch, lt, sch = _formed(Ns, 5300)
    assert s.pcg_shape(lt, sch, make_opts())["C"] > 1
    want, got = _capped(s, lt, sch, 3), _capped(s, lt, sch, 0)
    assert torch.equal(got, want) == one
    assert oracle.relerr(got.cpu().double().numpy(), want.cpu().double().numpy()) < 1e-4
    g = torch.cuda.CUDAGraph()
    stats, ws, lam = s.alloc_stats(lt.nb), s.alloc_workspace(lt), torch.empty_like(got)
    o = make_opts(tol=1e-30, max_iter=4)
    with torch.cuda.graph(g):
        lam.fill_(0.25)
        s.pcg_solve(lt, sch, lam, o, stats, ws)
    for _ in range(2):
        g.replay()
    assert torch.equal(lam, got)
    t0, t3 = (_median_ms(lambda: _capped(s, lt, sch, mode, 40)) for mode in (0, 3))
    assert t0 < (1.1 if one else 0.95) * t3, (t0, t3)
