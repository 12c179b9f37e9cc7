"""The frozen Jv has forms for hierarchies of few tiles (up to 304 and 1,216 of
them), the residual one (up to 1,216); each against the oracle on either side of
the lines, on whole and ragged boxes and on patches, with and without Robin
faces.  Tolerance 1e-12 of each cell's term scale, as in the parity tests."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu

from oracle.oracle import Oracle  # noqa: E402
from paper_1302_6303_gb300 import workloads as W  # noqa: E402


@pytest.fixture(scope="module")
def nrd():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__ as g
    g.build()
    from paper_1302_6303_gb300 import nrd as m
    return m


def dev(a):
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


# (tiles are launched in two halves on hierarchies as small as these)
CASES = {
    "box304": (lambda: W.uniform((32, 32, 76)), (32, 4, 4)),
    "ragged305": (lambda: W.uniform((31, 18, 121)), (32, 4, 4)),
    "box320": (lambda: W.uniform((32, 32, 80)), (32, 4, 4)),
    "box1216": (lambda: W.uniform((32, 80, 152)), (32, 4, 4)),
    "ragged1236": (lambda: W.uniform((31, 77, 154)), (32, 4, 4)),
    "neumann304": (lambda: W.all_neumann(W.uniform((31, 29, 75))), (32, 4, 4)),
    "amr_few": (lambda: W.config_amr2(16, seed=3, band=4, ncubes=4)[0], (8, 8, 4)),
    "amr_many": (lambda: W.config_batching(24, seed=0)[0], (8, 8, 8)),
}


@pytest.mark.parametrize("name", list(CASES))
def test_frozen_jv(nrd, name):
    mk, tile = CASES[name]
    h = mk()
    z = W.material_from_cubes(h, [((2, 2, 2), 3, 10.0)])
    u = W.front_state(h, seed=2, noise=0.1)
    v = W.random_direction(h, 7)
    ctx = nrd.Context(nmg=1, tile_x=tile[0], tile_y=tile[1], tile_z=tile[2])
    ctx.set_hierarchy_from(h)
    ctx.set_material(dev(z))
    a0, dt = 1.5, 3e-3
    ctx.linearise(dev(u), dev(u), a0, dt)
    J = ctx.jv(dev(u), dev(v), a0, dt, mode=nrd.JV_FROZEN).cpu().numpy()
    o = Oracle(h, z)
    S = o.jv_scale(u, v, a0, dt)
    assert np.all(np.abs(J - o.jv_analytic(u, v, a0, dt)) <= 1e-12 * S + 1e-300)


@pytest.mark.parametrize("name", list(CASES))
def test_residual(nrd, name):
    mk, tile = CASES[name]
    h = mk()
    z = W.material_from_cubes(h, [((2, 2, 2), 3, 10.0)])
    u = W.front_state(h, seed=2, noise=0.1)
    b = u * (1 + 0.05 * np.random.default_rng(4).uniform(-1, 1, u.size))
    ctx = nrd.Context(nmg=1, tile_x=tile[0], tile_y=tile[1], tile_z=tile[2])
    ctx.set_hierarchy_from(h)
    ctx.set_material(dev(z))
    a0, dt = 1.5, 3e-3
    F = ctx.residual(dev(u), dev(b), a0, dt)
    o = Oracle(h, z)
    S = o.residual_scale(u, b, a0, dt)
    assert np.all(np.abs(F.cpu().numpy() - o.residual(u, b, a0, dt)) <= 1e-12 * S + 1e-300)
    # the linearisation's residual has the same bits
    assert torch.equal(ctx.linearise(dev(u), dev(b), a0, dt), F)
