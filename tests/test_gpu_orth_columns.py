"""The cooperative Gram-Schmidt kernel at every number of basis vectors it has
a form for: one Newton correction from m GMRES iterations, m = 1 .. 31, in the
graph and in the host-driven loop, against GMRES with modified Gram-Schmidt
applied twice on the host over the library's own operators (frozen Jv and FP64
preconditioner), on one, two and three levels.  The preconditioner is weakened
(one damped sweep), so that no cycle converges and the basis stays well
conditioned; one pass of classical Gram-Schmidt then loses a few digits at
most, and a column left out or taken twice changes the correction by its
Hessenberg entry, a thousandth or more.  Bound 1e-7 of the largest entry."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu

from paper_1302_6303_gb300 import workloads as W  # noqa: E402


@pytest.fixture(scope="module")
def nrd():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__ as g
    g.build()
    from paper_1302_6303_gb300 import nrd as m
    return m


HIERS = {
    "one": lambda: W.uniform((12, 11, 9)),
    "two": lambda: W.config_amr2(16, seed=3, band=4, ncubes=4)[0],
    "three": lambda: W.tiny_amr(8, True),
}
A0, DT = 1.0, 5e-2
WEAK = dict(nmg=1, nu1=1, nu2=0, coarse_sweeps=1, omega=0.02, pc_precision=0, max_newton=1,
            eta0=1e-13, rtol=1e-14)


def context(nrd, h, z, **kw):
    ctx = nrd.Context(smoother=nrd.SMOOTH_JACOBI, **WEAK, **kw)
    ctx.set_hierarchy_from(h)
    ctx.set_material(z)
    return ctx


@pytest.mark.parametrize("name", list(HIERS))
def test_columns(nrd, name):
    h = HIERS[name]()
    N = h.ncells
    z = torch.from_numpy(W.material_from_cubes(h, [((2, 2, 2), 3, 10.0)])).cuda()
    u = torch.from_numpy(W.front_state(h, seed=2, noise=0.0)).cuda()
    b = u * (1 + 1e-3 * torch.sin(torch.arange(2 * N, device="cuda", dtype=torch.float64)))
    leaf = torch.from_numpy(~h.covered_mask()).cuda().repeat(2)
    L = h.cell_ijk()[0]
    vol = np.array([1.0 / np.prod(h.level_n(l)) for l in range(h.nlevels)])[L]
    wt = torch.from_numpy(np.concatenate([vol] * 2)).cuda() * leaf
    ref = context(nrd, h, z)
    F = ref.linearise(u, b, A0, DT)
    dot = lambda x, y: float((wt * x * y).sum())  # noqa: E731
    V, Z, H = [-F / dot(F, F) ** 0.5], [], np.zeros((32, 31))
    for j in range(31):
        Z.append(ref.precond_apply(V[j]))
        w = ref.jv(u, Z[j], A0, DT, mode=nrd.JV_FROZEN)
        for _ in range(2):
            for i in range(j + 1):
                c = dot(w, V[i])
                H[i, j] += c
                w = w - c * V[i]
        H[j + 1, j] = dot(w, w) ** 0.5
        V.append(w / H[j + 1, j])
    for graph in (1, 0):
        for m in range(1, 32):
            e1 = np.zeros(m + 1)
            e1[0] = dot(F, F) ** 0.5
            y, res = np.linalg.lstsq(H[:m + 1, :m], e1, rcond=None)[:2]
            assert res[0] ** 0.5 > 1e-6 * e1[0]          # not converged: every column counts
            dx = sum(float(q) * zq for q, zq in zip(y, Z))
            ctx = context(nrd, h, z, restart=m, max_krylov=m, graph=graph)
            got = u.clone()
            st = ctx.newton(got, b, A0, DT, check=False)
            dx = dx * st["min_lambda"]                   # the update's positivity damping
            assert st["krylov_its"] == m and st["min_lambda"] > 0.0
            err = ((got - u - dx) * leaf).abs().max()
            assert float(err) <= 1e-7 * float((dx * leaf).abs().max()), (graph, m)
            ctx.close()


@pytest.mark.parametrize("name", list(HIERS))
def test_two_passes(nrd, name):
    """The adjoint solve (always two passes) stopped after m = 1 .. 31
    iterations: its true residual is the smallest over the space, so it is
    orthogonal to its difference from the one before, which lies in it."""
    h = HIERS[name]()
    z = torch.from_numpy(W.material_from_cubes(h, [((2, 2, 2), 3, 10.0)])).cuda()
    u = torch.from_numpy(W.front_state(h, seed=2, noise=0.0)).cuda()
    leaf = torch.from_numpy(~h.covered_mask()).cuda().repeat(2)
    g = torch.from_numpy(W.random_direction(h, 7)).cuda() * leaf
    last = g
    for m in range(1, 32):
        ctx = context(nrd, h, z, restart=m, max_krylov=m)
        ctx.linearise(u, u, A0, DT)
        lam, st = ctx.adjoint_solve(g, A0, DT, rtol=1e-13, check=False)
        assert st["krylov_its"] == m
        r = g - ctx.vjp(lam, A0, DT, want_dz=False)[0]
        d = last - r
        nr, nd = ctx.dot(r, r) ** 0.5, ctx.dot(d, d) ** 0.5
        assert abs(ctx.dot(r, d)) <= 1e-7 * nr * ctx.dot(g, g) ** 0.5, m
        assert nd > 1e-6 * nr, m                         # the column did change it
        last = r
        ctx.close()
