"""The tiled formation and the flat recovery (float32, the two measured
shapes) against the kernels that serve every shape."""
import numpy as np
import pytest

from gpu_util import solver
from workload import gen

pytestmark = pytest.mark.gpu


def _rel(a, b):
    a, b = a.double(), b.double()
    return ((a - b).norm() / b.norm()).item() if b.numel() else 0.0


# knots per CTA: 15 (nx = 14) and 11 (nx = 36) once a batch is large; horizons
# that end on, before and after a CTA's last knot, and single knots
@pytest.mark.parametrize("nx,nu,Ns", [(14, 7, [1]), (14, 7, [5]), (14, 7, [512]), (14, 7, [1, 15, 16, 14, 2, 31] * 40),
                                      (36, 12, [1]), (36, 12, [3]), (36, 12, [130]), (36, 12, [1, 11, 12, 10, 2, 23] * 40)])
@pytest.mark.parametrize("shift", [0, 1])
def test_form_equals_the_separate_calls(nx, nu, Ns, shift):
    """form (one launch) gives what form_schur and form_precon give, to the
    rounding of differently contracted multiply-adds (1 ulp an entry, times
    the condition of a diagonal block in Phi^-1); shift = 1 misaligns A, which
    takes the general kernel."""
    import torch
    from paper_2309_08079_gb300.solver import LQTensors
    s = solver()
    b = gen.kuka_batch(nx, nu, Ns, 7000).astype(np.float32)
    lt = LQTensors.from_batch(b) if len(Ns) > 1 else LQTensors.from_numpy(b.items[0])
    if shift:
        a = torch.empty(lt.A.numel() + 1, device="cuda")[1:].view(lt.A.shape)
        a.copy_(lt.A)
        lt.A = a
    one, two = s.alloc_schur(lt), s.alloc_schur(lt)
    for x in (one, two):
        for t in (x.Sd, x.So, x.Pd, x.Po, x.gamma):
            t.fill_(float("nan"))
    s.form(lt, one)
    s.form_schur(lt, two)
    s.form_precon(lt, two)
    K, J = lt.total, lt.total - lt.nb
    for f, n, bar in (("Sd", K, 1e-6), ("So", J, 1e-6), ("gamma", K, 1e-6), ("Pd", K, 1e-5), ("Po", J, 1e-5)):
        x, y = getattr(one, f)[:n], getattr(two, f)[:n]
        assert torch.isfinite(x).all() and _rel(x, y) < bar, (f, _rel(x, y))
    for d in (one.Sd, one.Pd):
        assert torch.equal(d, d.mT)
    assert one.info.sum().item() == 0
    if one.Sdp is not None:
        i, j = np.triu_indices(nx)
        at = torch.as_tensor(j * (j + 1) // 2 + i)
        for p, d in ((one.Sdp, one.Sd), (one.Pdp, one.Pd)):
            assert torch.equal(p[:, at], d[:, i, j]) and (p[:, nx * (nx + 1) // 2:] == 0).all()


@pytest.mark.parametrize("nx,nu", [(14, 7), (36, 12)])
def test_bad_weight_marks_its_own_instance(nx, nu):
    """A bad weight at a knot that two CTAs read marks its instance only."""
    from paper_2309_08079_gb300.solver import LQTensors
    s = solver()
    items = [gen.kuka_lq(nx, nu, n, 40 + n) for n in (7, 1, 30, 16)]
    items[1].Qd[0, 3] = -1.0
    items[2].Rd[10, 0] = np.inf
    lt = LQTensors.from_batch(gen.concat_batch(items).astype(np.float32))
    sch = s.form(lt, s.alloc_schur(lt))
    assert sch.info.tolist() == [0, 1, 1, 0]


@pytest.mark.parametrize("dtype", ["float32", "float64"])
@pytest.mark.parametrize("nx,nu,Ns", [(14, 7, [1, 12, 13, 11, 40]), (36, 12, [1, 5, 6, 4, 17])])
def test_flat_recovery(nx, nu, Ns, dtype):
    """dz of the flat kernel is the float64 recovery, rounded: the sums carry
    44 bits or more, so an entry is off by its own rounding and 2^-40 of the
    terms it cancels."""
    import torch
    from paper_2309_08079_gb300.solver import LQTensors
    s = solver()
    t = getattr(torch, dtype)
    b = gen.kuka_batch(nx, nu, Ns, 7100).astype(np.float32)
    lt = LQTensors.from_batch(b, dtype=t)
    lam = torch.as_tensor(np.cumsum(np.random.default_rng(5).normal(size=(lt.total, nx)), 0), dtype=t, device="cuda")
    dx, du = (x.cpu().double().numpy() for x in s.recover_step(lt, lam))
    L = lam.cpu().double().numpy()
    eps = 2.0 ** -23 if dtype == "float32" else 2.0 ** -50
    for i, it in enumerate(b.items):
        it = it.astype(np.float64)
        k0, j0 = b.knot_off[i], b.knot_off[i] - i
        x, u = L[k0:k0 + it.N] - it.q, -it.r
        x[:-1] -= np.einsum("kij,ki->kj", it.A, L[k0 + 1:k0 + it.N])
        u = u - np.einsum("kij,ki->kj", it.B, L[k0 + 1:k0 + it.N])
        big = np.abs(L[k0:k0 + it.N]).max() * nx
        for got, ref in ((dx[k0:k0 + it.N], x / it.Qd), (du[j0:j0 + it.N - 1], u / it.Rd)):
            assert np.all(np.abs(got - ref) <= eps * np.abs(ref) + 2.0 ** -40 * big / 0.01)


@pytest.mark.parametrize("Ns", [[1], [6], [300], [1, 15, 16, 14, 2, 31] * 10])
def test_dense_costs_equal_the_separate_calls(Ns):
    """Dense SPD cost blocks at nx = 14: the tiled formation against the two
    general launches, and the recovery against float64 (bars as above; the
    inverse cost blocks add their condition to S+'s rounding)."""
    import torch
    from paper_2309_08079_gb300.solver import LQTensors
    s = solver()
    b = gen.kuka_batch(14, 7, Ns, 7200, dense=True).astype(np.float32)
    lt = LQTensors.from_batch(b) if len(Ns) > 1 else LQTensors.from_numpy(b.items[0])
    one, two = s.alloc_schur(lt), s.alloc_schur(lt)
    s.form(lt, one)
    s.form_schur(lt, two)
    s.form_precon(lt, two)
    K, J = lt.total, lt.total - lt.nb
    for f, n in (("Sd", K), ("So", J), ("gamma", K), ("Pd", K), ("Po", J)):
        x, y = getattr(one, f)[:n], getattr(two, f)[:n]
        assert torch.isfinite(x).all() and _rel(x, y) < 1e-5, (f, _rel(x, y))
    lam = torch.as_tensor(np.cumsum(np.random.default_rng(5).normal(size=(K, 14)), 0), dtype=torch.float32, device="cuda")
    dx, du = (x.cpu().double().numpy() for x in s.recover_step(lt, lam))
    L = lam.cpu().double().numpy()
    for i, it in enumerate(b.items):
        it = it.astype(np.float64)
        k0, j0 = b.knot_off[i], b.knot_off[i] - i
        x, u = L[k0:k0 + it.N] - it.q, -it.r
        x[:-1] -= np.einsum("kij,ki->kj", it.A, L[k0 + 1:k0 + it.N])
        u = u - np.einsum("kij,ki->kj", it.B, L[k0 + 1:k0 + it.N])
        for got, M, rhs in ((dx[k0:k0 + it.N], it.Q, x), (du[j0:j0 + it.N - 1], it.R, u)):
            ref = np.linalg.solve(M, rhs[..., None])[..., 0]
            assert np.linalg.norm(got - ref) <= 1e-5 * np.linalg.norm(ref)


def test_dense_block_that_is_not_spd_is_flagged():
    from paper_2309_08079_gb300.solver import LQTensors
    s = solver()
    items = [gen.kuka_lq(14, 7, n, 50 + n, dense=True) for n in (5, 20, 9)]
    items[1].R[7] = -items[1].R[7]
    items[2].Q[8] = np.nan
    lt = LQTensors.from_batch(gen.concat_batch(items).astype(np.float32))
    assert s.form(lt, s.alloc_schur(lt)).info.tolist() == [0, 1, 1]


def test_misaligned_arrays_keep_a_specialised_kernel():
    """A misaligned A (4 bytes off) takes the formation away from the tiled
    kernel, to the one with a warp per knot, whose sizes are fixed at compile
    time: half the time of the two separate calls (the general sizes: 1.03 of
    it)."""
    import torch
    from paper_2309_08079_gb300.solver import LQTensors
    s = solver()
    lt = LQTensors.from_batch(gen.kuka_batch(14, 7, [32] * 256 + [300] * 128, 5).astype(np.float32))
    a = torch.empty(lt.A.numel() + 1, device="cuda")[1:].view(lt.A.shape)
    a.copy_(lt.A)
    lt.A = a
    sch = s.alloc_schur(lt)

    def two():
        s.form_schur(lt, sch)
        s.form_precon(lt, sch)

    def median(f):
        f()
        torch.cuda.synchronize()
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g):
            f()
        t = []
        for _ in range(21):
            a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            a.record()
            g.replay()
            b.record()
            b.synchronize()
            t.append(a.elapsed_time(b))
        return sorted(t)[10]
    assert median(lambda: s.form(lt, sch)) < 0.75 * median(two)
