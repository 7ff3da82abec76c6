"""FP64 2D kernels at the sizes where their layout changes: several elements per CTA with a partial last
CTA, the constant-velocity operators against the per-element solve, and each form of the swirl's small-angle
evaluation.  Tolerance: 1e-12 relative L2 per step against the oracle, the FP64 path's bound; two paths that
each meet it differ by at most twice that."""
import numpy as np
import pytest

import sl_inputs
from oracle import sl_oracle as O

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

TOL = 1e-12
BOX = (0.0, 1.0, 0.0, 1.0)


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


def advance(sl, kx, ky, n, kind, p, bc, cons, rk, factor=1.0, orders=None, ghost=0.2, fit=0, basis=0):
    ctx = sl.Context(2, kx, ky, BOX, n, basis, sl.FP64, (bc,) * 4, ghost, orders=orders)
    gv = sl.velocity(kind, *p)
    x, y = sl.Context(2, kx, ky, BOX, n, basis, sl.FP64, (bc,) * 4, ghost).node_coords()
    phi = 1.0 + 0.5 * np.sin(2 * np.pi * x) * np.cos(2 * np.pi * y) + 0.02 * sl_inputs.random_state(x.shape, kx + n)
    dt = factor * ctx.max_dt(gv, sl.RULE_PAPER)
    a = torch.tensor(phi.ravel(), device="cuda")
    b = torch.empty_like(a)
    ctx.step(a, b, gv, 0.3, dt, sl.options(cons, rk, fit))
    return phi, dt, b.cpu().numpy().reshape(phi.shape), ctx.sync()


PACKED = [
    # kx, ky, n, kind, params, bc, cons, rk: element counts that fill several slots per CTA and leave the
    # last CTA partial
    (61, 53, 5, 2, (5.0,), 1, 3, 4),
    (41, 31, 8, 2, (5.0,), 1, 7, 4),
    (41, 31, 8, 1, (2 * np.pi, 0.5, 0.5), 1, 3, 3),
    (47, 41, 7, 1, (2 * np.pi, 0.5, 0.5), 1, 3, 2),
    (35, 27, 9, 2, (5.0,), 0, 3, 4),
    (31, 23, 11, 1, (2 * np.pi, 0.5, 0.5), 1, 3, 4),
    (83, 61, 3, 2, (5.0,), 1, 3, 4),
    (83, 61, 2, 1, (2 * np.pi, 0.5, 0.5), 1, 3, 1),
    (131, 73, 9, 0, (1.0, 0.5), 0, 3, 4),
    (131, 73, 9, 0, (-0.4, 0.9), 1, 7, 4),
    (97, 101, 4, 0, (0.7, -0.6), 1, 3, 3),
    (41, 31, 13, 0, (-0.7, -0.6), 0, 3, 2),
]


@pytest.mark.parametrize("case", PACKED, ids=[f"{c[0]}x{c[1]}n{c[2]}v{c[3]}c{c[6]}rk{c[7]}" for c in PACKED])
def test_packed_elements(sl, case):
    kx, ky, n, kind, p, bc, cons, rk = case
    phi, dt, got, bits = advance(sl, *case)
    assert bits & ~sl.ST_PICARD_NOCONV == 0
    setup = O.Setup(2, kx, ky, BOX, n, 0, (bc,) * 4, 0.2)
    pick = sl_inputs.sample_elements(24, kx * ky, 5)
    pick = np.unique(np.concatenate([pick, [0, kx - 1, kx * ky - 2, kx * ky - 1]]))
    els = [(int(e % kx), int(e // kx)) for e in pick]
    ref, infos = O.step_2d(setup, phi, O.StepOpts(O.Vel(kind, tuple(p) + (0,) * (6 - len(p))), 0.3, dt, cons, rk),
                           elements=els)
    good = [e for e in els if infos[e]["converged"]]
    assert len(good) > len(els) // 2
    g = np.array([got[ey, ex] for ex, ey in good])
    r = np.array([ref[ey, ex] for ex, ey in good])
    assert rel(g, r) <= TOL


SHIFT = [
    # kx, ky, n, params, bc, cons, rk, fit, basis: constant velocity, shared operators against the per-element
    # solve (reached through an element map whose node counts are all equal)
    (6, 5, 9, (1.0, 0.5), 0, 3, 4, 0, 0),
    (5, 4, 2, (-1.0, 0.5), 1, 3, 4, 0, 0),       # (n = 2: the faces fix every value, no energy row)
    (5, 4, 5, (0.6, -0.9), 1, 7, 3, 0, 1),
    (5, 4, 6, (0.6, -0.9), 1, 2, 2, 0, 0),
    (5, 4, 6, (-0.6, -0.9), 1, 4, 1, 0, 0),
    (5, 4, 7, (0.8, 0.0), 1, 3, 4, 0, 0),
    (4, 5, 7, (0.0, -0.8), 0, 7, 4, 0, 0),
    (4, 5, 6, (0.7, 0.8), 0, 3, 4, 1, 0),
    (4, 5, 6, (0.7, 0.8), 0, 0, 4, 0, 0),
    (1, 1, 8, (0.7, 0.8), 0, 3, 4, 0, 0),
    (3, 2, 17, (0.7, -0.8), 1, 3, 4, 0, 0),
    (37, 29, 10, (0.7, -0.8), 1, 3, 4, 0, 0),
]


@pytest.mark.parametrize("case", SHIFT, ids=[f"{c[0]}x{c[1]}n{c[2]}a{c[3][0]}b{c[3][1]}bc{c[4]}c{c[5]}rk{c[6]}f{c[7]}"
                                             for c in SHIFT])
@pytest.mark.parametrize("factor", [0.3, 1.0, 3.0])
def test_shared_operators_match_per_element_solve(sl, case, factor):
    kx, ky, n, p, bc, cons, rk, fit, basis = case
    kw = dict(fit=fit, basis=basis, factor=factor)
    _, _, a, ba = advance(sl, kx, ky, n, 0, p, bc, cons, rk, **kw)
    _, _, b, bb = advance(sl, kx, ky, n, 0, p, bc, cons, rk, orders=np.full((ky, kx), n), **kw)
    assert ba == bb
    assert rel(a, b) <= 2 * TOL


@pytest.mark.parametrize("case", [(4, 3, 4, 1.0), (4, 4, 8, 1.0), (5, 5, 8, 0.05), (3, 3, 6, 2.0), (9, 7, 5, 0.2)])
@pytest.mark.parametrize("rk", [1, 2, 3, 4])
def test_swirl_small_angle_forms(sl, case, rk):
    """Steps whose largest stage angle falls in the short series, the long series and the direct form."""
    kx, ky, n, factor = case
    phi, dt, got, bits = advance(sl, kx, ky, n, 2, (5.0,), 1, 3, rk, factor=factor)
    assert bits == 0
    setup = O.Setup(2, kx, ky, BOX, n, 0, (1,) * 4, 0.2)
    ref, _ = O.step_2d(setup, phi, O.StepOpts(O.Vel(2, (5.0, 0, 0, 0, 0, 0)), 0.3, dt, 3, rk))
    assert rel(got, ref) <= TOL
