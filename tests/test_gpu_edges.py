"""The kernels at the sizes where their tiles, chunks and rings end: axes of
three to five nodes, one past a warp, a tile or a span, elongated grids --
against the CPU oracle and the numpy V-cycle, with the bounds of the tests
those references come from."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu

from oracle import nn as N  # noqa: E402
from oracle import pyoracle as O  # noqa: E402
from paper_1901_08269_gb300 import cfp  # noqa: E402
from paper_1901_08269_gb300 import workloads as W  # noqa: E402
from test_gpu_multigrid import build_levels, vcycle  # noqa: E402
from test_gpu_nn import act_in, bf16, close, npad, rnd, unpad  # noqa: E402
from test_gpu_parity import Pair, dev  # noqa: E402


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    torch.cuda.set_device(0)


def grid(nx, ny, nz, body=None):
    axes = W.tanh_grid(-1, 1, nx, 0.9), W.tanh_grid(-1, 1, ny, 0.5), W.uniform_grid(-1, 1, nz)
    return W.Workload("edge", *axes, [body] if body else [], W._c2_u, W._c2_f)


BALL = W.sphere((0.04, -0.02, 0.03), 0.4)
GRIDS = {
    "3-3-3": lambda: grid(3, 3, 3),                    # a single unknown
    "3-40-5": lambda: grid(3, 40, 5),                  # one column
    "34-12-3": lambda: grid(34, 12, 3),                # a full warp of columns, one plane
    "35-4-70": lambda: grid(35, 4, 70),                # one column past a warp, past 64 planes
    "130-19-4": lambda: grid(130, 19, 4),              # rows past a CTA of 4 warps x 4
    "17-18-33": lambda: grid(17, 18, 33, BALL),
    "258-15-12": lambda: grid(258, 15, 12, BALL),      # the widest row of the 256-column ring
    "259-14-37": lambda: grid(259, 14, 37, BALL),      # the narrowest of the 512-column one
    "515-13-12": lambda: grid(515, 13, 12, BALL),      # copied row by row, one column in the last tile
}
SHAPES = [(cfp.APPLY_STREAM, 2, 16), (cfp.APPLY_STREAM, 4, 64), (cfp.APPLY_RING, 2, 32), (cfp.APPLY_RING, 2, 64)]


@pytest.mark.parametrize("name", list(GRIDS))
def test_classify_apply_rhs(name):
    """Types and IBI points equal the oracle's; the FP64 operator and
    right-hand side within 1e-12 and the FP32 operator within 64 * 2^-24
    (regular rows; irregular rows 2^29 * 1e-12) of the sum of absolute terms;
    every FP32 kernel and shape the same bits."""
    p = Pair(GRIDS[name]())
    np.testing.assert_array_equal(p.type.cpu().numpy(), p.otype)
    np.testing.assert_array_equal(p.xyz.cpu().numpy().reshape(-1), np.asarray(p.oxyz).reshape(-1))
    x = p.rand_field(3, zero_off=False).astype(np.float32).astype(np.float64)
    want, scale = p.P.apply_B(x), p.P.apply_B(x, absval=True)
    unk = np.zeros(p.w.N, bool)
    unk[p.unk] = True
    y = torch.full((p.w.N,), float("nan"), dtype=torch.float64, device="cuda")
    p.ctx.apply(dev(x), y)
    got = y.cpu().numpy()
    assert np.all(np.abs(got - want) <= 1e-12 * scale + 1e-300) and np.all(got[~unk] == 0.0)
    xd = torch.as_tensor(x, dtype=torch.float32, device="cuda")
    outs = []
    for shape in [None] + SHAPES:
        if shape:
            p.ctx.tune_apply(cfp.PREC_MIXED, shape[1], shape[2], kernel=shape[0])
        o = torch.full((p.w.N,), float("nan"), dtype=torch.float32, device="cuda")
        p.ctx.apply_f32(xd, o)
        outs.append(o)
        assert torch.equal(o, outs[0]), shape
    err = np.abs(outs[0].double().cpu().numpy() - want)
    bound = np.where(p.otype == O.IRREGULAR, 2.0 ** 29 * 1e-12, 64 * 2.0 ** -24) * scale + 1e-30
    assert np.all(err <= bound)
    f, g = p.w.fields()
    gi = p.w.g_at(p.oxyz)
    rhs = torch.full((p.w.N,), float("nan"), dtype=torch.float64, device="cuda")
    p.ctx.assemble_rhs(dev(f), dev(g), dev(gi), rhs)
    ro = p.P.rhs(f, g, gi)
    X, Y, Z = p.w.mesh()
    u = p.w.u(X, Y, Z, np).reshape(-1)
    u[p.otype == O.SOLID] = 0.0
    scale = p.P.apply_B(u, absval=True) + np.abs(ro) + 1.0
    assert np.all(np.abs(rhs.cpu().numpy() - ro) <= 1e-12 * scale)
    p.ctx.close()


# the coarse levels of one launch: distributed and whole levels, long in each axis in turn
@pytest.mark.parametrize("nu,post", [(2, 2), (1, 2)])
@pytest.mark.parametrize("n", [(17, 17, 17), (18, 40, 71), (70, 17, 33), (131, 18, 17), (33, 98, 20)])
def test_vcycle_sizes(n, nu, post):
    """FP64 within 1e-12 and FP32 within 1e-5 of the V-cycle's definition, as
    for the ordinary sizes."""
    w = grid(*n, BALL)
    P = O.Problem(w.x, w.y, w.z, w.bodies, w.fluid_inside)
    otype = P.classify()
    P.ibi()
    P.assemble()
    levels = build_levels(w.x, w.y, w.z, otype, P.export(O.MAT_K))
    u = levels[0]["unk"]
    rho = np.where(u, np.random.default_rng(2).standard_normal(w.N), 0.0)
    want = vcycle(levels, rho, nu, post=post)
    ctx = cfp.Context(w.x, w.y, w.z, w.bodies, w.fluid_inside)
    ctx.classify_points()
    for precision, tol in ((cfp.PREC_FP64, 1e-12), (cfp.PREC_MIXED, 1e-5)):
        phi = torch.full((w.N,), 7.0, dtype=torch.float64, device="cuda")
        ctx.precondition_ex(dev(rho), phi, precond=cfp.PRECOND_MG, mg_smooth=nu, mg_post=post, precision=precision)
        got = phi.cpu().numpy()
        assert np.all(got[~u] == 0.0)
        err = np.max(np.abs(got[u] - want[u])) / np.max(np.abs(want[u]))
        assert err <= tol, (precision, err)
    ctx.close()


# fewer rows than a tile of 128, a remainder past one and several tiles, planes
# marched one by one (40 x 7 x 11) and in chunks (the last one short)
@pytest.mark.parametrize("d,cin,cout", [((5, 3, 3), 16, 16), ((5, 3, 3), 128, 128), ((17, 9, 3), 64, 32),
                                        ((40, 7, 11), 16, 16), ((40, 7, 11), 32, 64), ((40, 7, 11), 128, 128),
                                        ((126, 30, 21), 16, 16), ((126, 30, 21), 16, 32), ((62, 61, 21), 32, 32)])
def test_layer_sizes(d, cin, cout):
    axis = np.linspace(-1.0, 1.0, 9)
    ctx = cfp.Context(axis, axis, axis)
    x_d, x = act_in(d, cin, 1, relu=True)
    g_d, g = act_in(d, cout, 2)
    w_d, w = bf16(rnd((cout, 27, cin), 3, 0.3))
    b = rnd(cout, 4, 0.5).astype(np.float32).astype(np.float64)
    out = torch.empty(npad(d) * cout, dtype=torch.float32, device="cuda")
    ctx.nn_conv3d(d, cin, cout, x_d, w_d, out, bias=torch.as_tensor(b, dtype=torch.float32).cuda(), flags=cfp.NN_OUT_F32)
    close(unpad(out.double().cpu().numpy(), d, cout)[1], N.conv3d(x, w, b, d),
          N.conv3d(np.abs(x), np.abs(w), np.abs(b), d), False, "forward")
    gin = torch.empty(npad(d) * cin, dtype=torch.bfloat16, device="cuda")
    ctx.nn_conv3d(d, cout, cin, g_d, w_d, gin, act=x_d, flags=cfp.NN_DGRAD | cfp.NN_MASK)
    close(unpad(gin.double().cpu().numpy(), d, cin)[1], N.conv3d_dgrad(g, w, d) * (x > 0),
          N.conv3d_dgrad(np.abs(g), np.abs(w), d), True, "input gradient")
    dw = torch.zeros(cout * 27 * cin, dtype=torch.float32, device="cuda")
    db = torch.zeros(cout, dtype=torch.float32, device="cuda")
    ctx.nn_wgrad(d, cin, cout, x_d, g_d, dw, db)
    want, wantb = N.conv3d_wgrad(x, g, d)
    scale, scaleb = N.conv3d_wgrad(np.abs(x), np.abs(g), d)
    close(dw.double().cpu().numpy().reshape(cout, 27, cin), want, scale, False, "weight gradient")
    close(db.double().cpu().numpy(), wantb, scaleb, False, "bias gradient")
    ctx.close()
