"""FP64 1D kernels at the sizes where their launch shape changes (one, several and partial CTAs of each block
size), the constant-velocity operators against the per-element form, and each form of the small-angle
evaluation of u = -sin x.  Tolerance: 1e-12 relative L2 per step against the oracle, the FP64 path's bound;
two paths that each meet it differ by at most twice that."""
import numpy as np
import pytest

import sl_inputs
from oracle import sl_oracle as O

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

TOL = 1e-12


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


def smooth(x, box, seed):
    z = 2 * np.pi * (x - box[0]) / (box[1] - box[0])
    return 1.0 + 0.5 * np.sin(z) + 0.2 * np.cos(3 * z) + 1e-3 * sl_inputs.random_state(x.shape, seed)


SIZES = [1, 2, 29, 30, 31, 61, 62, 63, 126, 127, 1000, 300007]


@pytest.mark.parametrize("K", SIZES)
@pytest.mark.parametrize("case", [(4, 0, 1.0, 3, 4, 0), (5, 0, -0.7, 3, 3, 1), (4, 3, 0.0, 3, 4, 0), (6, 3, 0.0, 3, 2, 0)])
def test_mesh_sizes(sl, K, case):
    n, kind, a, cons, rk, bc = case
    box = (0.0, 2.0 * np.pi, 0.0, 0.0) if kind == 3 else (0.0, 1.0, 0.0, 0.0)
    ctx = sl.Context(1, K, 1, box, n, 0, sl.FP64, (bc,) * 4, 0.3)
    setup = O.Setup(1, K, 1, box, n, 0, (bc,) * 4, 0.3)
    gv = sl.velocity(kind, a) if kind == 0 else sl.velocity(kind)
    ov = O.Vel(kind, (a, 0, 0, 0, 0, 0))
    x, _ = ctx.node_coords()
    phi = smooth(x, box, K)
    dt = ctx.max_dt(gv, sl.RULE_PAPER)
    src = torch.tensor(phi, device="cuda")
    dst = torch.empty_like(src)
    ctx.step(src, dst, gv, 0.1, dt, sl.options(cons, rk))
    assert ctx.sync() == 0
    pick = np.arange(K) if K <= 1000 else np.unique(np.concatenate([sl_inputs.sample_elements(60, K, 3), [0, 1, K - 2, K - 1]]))
    got = dst.cpu().numpy().reshape(K, n)
    op = O.StepOpts(ov, 0.1, dt, cons, rk)
    ref = np.array([O.element_step_1d(setup, phi, int(k), op)[0] for k in pick])
    assert rel(got[pick], ref) <= TOL


@pytest.mark.parametrize("case", [(9, 1.0, 0, 7, 4, 0, 0), (5, -0.6, 1, 3, 3, 0, 1), (7, 0.8, 1, 7, 2, 0, 0),
                                  (4, -1.0, 0, 2, 1, 0, 0), (6, 0.5, 0, 3, 4, 1, 0), (17, 0.9, 1, 3, 4, 0, 0),
                                  (2, 0.9, 1, 1, 4, 0, 0), (6, 0.0, 0, 3, 4, 0, 0), (5, 0.4, 0, 0, 4, 0, 0)])
@pytest.mark.parametrize("factor", [0.3, 1.0, 3.0])
def test_shared_operators_match_per_element_form(sl, case, factor):
    """The same constant velocity given at the nodes takes the per-element kernel."""
    n, a, bc, cons, rk, fit, basis = case
    K, box = 37, (0.0, 1.0, 0.0, 0.0)
    ctx = sl.Context(1, K, 1, box, n, basis, sl.FP64, (bc,) * 4, 0.3)
    gv = sl.velocity(0, a)
    x, _ = ctx.node_coords()
    phi = torch.tensor(smooth(x, box, 5), device="cuda")
    dt = factor * ctx.max_dt(sl.velocity(0, a or 1.0), sl.RULE_PAPER)
    field = torch.full((2, 1, phi.numel()), a, dtype=torch.float64, device="cuda")
    one, two = torch.empty_like(phi), torch.empty_like(phi)
    opts = sl.options(cons, rk, fit)
    ctx.step(phi, one, gv, 0.0, dt, opts)
    b1 = ctx.sync()
    ctx.step(phi, two, sl.nodal_velocity(field, abs(a)), 0.0, dt, opts)
    assert ctx.sync() == b1
    assert rel(one.cpu().numpy(), two.cpu().numpy()) <= 2 * TOL


@pytest.mark.parametrize("K,n", [(3, 4), (12, 6), (40, 6), (400, 7)])
@pytest.mark.parametrize("rk", [1, 2, 3, 4])
@pytest.mark.parametrize("bvalue", [0, 1])
def test_sinx_small_angle_forms(sl, K, n, rk, bvalue):
    """Meshes whose step takes the direct form (coarse), the long and the short series (fine)."""
    box = (0.0, 2.0 * np.pi, 0.0, 0.0)
    ctx = sl.Context(1, K, 1, box, n, 1, sl.FP64, (0,) * 4, 0.0)
    setup = O.Setup(1, K, 1, box, n, 1, (0,) * 4, 0.0)
    gv = sl.velocity(3)
    x, _ = ctx.node_coords()
    phi = smooth(x, box, n)
    dt = ctx.max_dt(gv, sl.RULE_PAPER)
    src = torch.tensor(phi, device="cuda")
    dst = torch.empty_like(src)
    ctx.step(src, dst, gv, 0.0, dt, sl.options(3, rk, 0, bvalue))
    assert ctx.sync() == 0
    ref, _ = O.step_1d(setup, phi, O.StepOpts(O.Vel(3, (0.0,) * 6), 0.0, dt, 3, rk, 0, bvalue))
    assert rel(dst.cpu().numpy(), ref) <= TOL
