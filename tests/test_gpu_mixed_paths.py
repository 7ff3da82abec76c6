"""Mixed-precision shared-operator kernels, which advance two elements per thread, at the sizes where their pairs,
tiles and halos are partial: element counts around half a tile and a tile in 1D, every remainder of the tile in
2D, both signs of the velocity, periodic and inflow faces; and the general kernels' face feet, taken in pairs up to
13 nodes and from a list above and on nonconforming meshes.  Bound: 1e-6 relative L2 against the oracle, the mixed
path's bound after one step; global mass on a periodic mesh to 1e-12 relative over 20 steps."""
import numpy as np
import pytest

from oracle import sl_oracle as O

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

TOL = 1e-6


@pytest.fixture(scope="module")
def sl():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1910_06476_gb300 import build as B
    B.build()
    import paper_1910_06476_gb300 as pkg
    return pkg


def rel(a, b):
    return float(np.sqrt(np.sum((a - b) ** 2) / np.sum(b ** 2)))


@pytest.mark.parametrize("K", [1, 2, 3, 127, 128, 129, 255, 256, 257, 513])
@pytest.mark.parametrize("case", [(9, 1.0, 0, 7, 0), (8, -0.7, 1, 3, 0), (5, 0.6, 1, 7, 0), (4, -1.0, 0, 1, 0),
                                  (6, -0.8, 0, 3, 1), (17, 0.9, 1, 3, 0), (2, 0.5, 0, 1, 0)])
def test_1d_pairs_and_tiles(sl, K, case):
    n, a, bc, cons, fit = case
    box = (0.0, 1.0, 0.0, 0.0)
    ctx = sl.Context(1, K, 1, box, n, 0, sl.MIXED, (bc,) * 4, 0.4)
    setup = O.Setup(1, K, 1, box, n, 0, (bc,) * 4, 0.4)
    x, _ = ctx.node_coords()
    phi = 1.0 + 0.5 * np.sin(2 * np.pi * x) + 0.2 * np.cos(4 * np.pi * x)
    gv = sl.velocity(0, a)
    dt = ctx.max_dt(gv, sl.RULE_PAPER)
    src = ctx.pack(torch.tensor(phi.ravel(), device="cuda"))
    dst = ctx.new_state()
    ctx.step(src, dst, gv, 0.0, dt, sl.options(cons, 4, fit))
    assert ctx.sync() & ~sl.ST_PICARD_NOCONV == 0
    got = ctx.unpack(dst).cpu().numpy().reshape(K, n)
    ref, infos = O.step_1d(setup, phi, O.StepOpts(O.Vel(0, (a, 0, 0, 0, 0, 0)), 0.0, dt, cons, 4, fit,
                                                  energy_skip_rtol=1e-9))
    good = np.array([infos[k]["converged"] for k in range(K)])
    if good.any():
        assert rel(got[good], ref[good]) <= TOL


@pytest.mark.parametrize("size", [(1, 1), (2, 3), (3, 2), (7, 5), (8, 4), (9, 4), (8, 5), (17, 9)])
@pytest.mark.parametrize("case", [(9, 1.0, 0.5, 0, 3), (8, -0.7, 0.6, 1, 3), (5, -0.5, -0.9, 1, 2), (4, 0.8, -0.6, 0, 1),
                                  (10, -0.8, -0.4, 0, 3), (13, 0.6, 0.9, 1, 3), (2, 0.6, 0.9, 0, 3), (3, -0.6, 0.9, 1, 3)])
def test_2d_pairs_and_tiles(sl, size, case):
    kx, ky = size
    n, a, b, bc, cons = case
    box = (0.0, 1.0, 0.0, 1.0)
    ctx = sl.Context(2, kx, ky, box, n, 0, sl.MIXED, (bc,) * 4, 0.4)
    setup = O.Setup(2, kx, ky, box, n, 0, (bc,) * 4, 0.4)
    x, y = ctx.node_coords()
    phi = 1.0 + 0.5 * np.sin(2 * np.pi * x) * np.cos(2 * np.pi * y) + 0.1 * np.cos(4 * np.pi * y)
    gv = sl.velocity(0, a, b)
    dt = ctx.max_dt(gv, sl.RULE_PAPER)
    src = ctx.pack(torch.tensor(phi.ravel(), device="cuda"))
    dst = ctx.new_state()
    ctx.step(src, dst, gv, 0.0, dt, sl.options(cons, 4))
    assert ctx.sync() == 0
    got = ctx.unpack(dst).cpu().numpy().reshape(phi.shape)
    ref, _ = O.step_2d(setup, phi, O.StepOpts(O.Vel(0, (a, b, 0, 0, 0, 0)), 0.0, dt, cons, 4))
    assert rel(got, ref) <= TOL


@pytest.mark.parametrize("dim", [1, 2])
def test_mass_over_partial_tiles(sl, dim):
    kx, ky, n = (777, 1, 7) if dim == 1 else (21, 11, 7)
    ctx = sl.Context(dim, kx, ky, (0.0, 1.0, 0.0, 1.0 if dim == 2 else 0.0), n, 0, sl.MIXED, (0,) * 4, 0.0)
    x, y = ctx.node_coords()
    phi = 1.0 + 0.5 * np.sin(2 * np.pi * x) * (np.cos(2 * np.pi * y) if dim == 2 else 1.0)
    gv = sl.velocity(0, -0.9, 0.7)
    dt = ctx.max_dt(gv, sl.RULE_PAPER)
    a = ctx.pack(torch.tensor(phi.ravel(), device="cuda"))
    m0 = ctx.mass(a)
    out = ctx.run(a, ctx.new_state(), gv, 0.0, dt, 20, sl.options(3, 4))
    assert ctx.sync() == 0
    assert abs(ctx.mass(out) / m0 - 1.0) <= 1e-12


@pytest.mark.parametrize("rk", [1, 2, 3, 4])
@pytest.mark.parametrize("n", [3, 4, 8, 9, 13, 14])
@pytest.mark.parametrize("when", [0.3, "reversal"])
def test_2d_face_feet_of_the_swirl(sl, n, rk, when):
    """Every RK order's distinct stage times, and a step over which the flow reverses, so that a face point flows
    out at some of them only; the mass row carries the face fluxes into the result."""
    kx, ky, box = 5, 4, (0.0, 1.0, 0.0, 1.0)
    ctx = sl.Context(2, kx, ky, box, n, 0, sl.MIXED, (1,) * 4, 0.3)
    setup = O.Setup(2, kx, ky, box, n, 0, (1,) * 4, 0.3)
    x, y = ctx.node_coords()
    phi = 1.0 + 0.5 * np.sin(2 * np.pi * x) * np.cos(2 * np.pi * y) + 0.1 * np.cos(4 * np.pi * y)
    gv = sl.velocity(sl.VEL_SWIRL, 5.0)
    dt = ctx.max_dt(gv)
    t = 2.5 - 0.3 * dt if when == "reversal" else when
    src = ctx.pack(torch.tensor(phi.ravel(), device="cuda"))
    dst = ctx.new_state()
    ctx.step(src, dst, gv, t, dt, sl.options(sl.C_BOUNDARY | sl.C_MASS, rk))
    assert ctx.sync() == 0
    got = ctx.unpack(dst).cpu().numpy().reshape(phi.shape)
    ref, _ = O.step_2d(setup, phi, O.StepOpts(O.Vel(sl.VEL_SWIRL, (5.0, 0, 0, 0, 0, 0)), t, dt, 3, rk))
    assert rel(got, ref) <= TOL
