"""The apply's shape handed from one context to another of the same grid size
(cfp_apply_shape -> cfp_tune_apply): the second reports, and so launches, what
the first does, whether the tuner chose the shape, the grid's size did, or the
shape was set."""
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu

from paper_1901_08269_gb300 import cfp  # noqa: E402
from paper_1901_08269_gb300 import workloads as W  # noqa: E402

BALL = W.sphere((0.04, -0.02, 0.03), 0.4)


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    torch.cuda.set_device(0)


def context(n, bodies=()):
    ctx = cfp.Context(*[W.tanh_grid(-1, 1, q, 0.7) for q in n], list(bodies))
    ctx.classify_points()
    return ctx


GRIDS = [(33, 33, 33), (97, 65, 82), (129, 129, 129), (257, 257, 257), (321, 129, 65)]


@pytest.mark.parametrize("prec", [cfp.PREC_FP64, cfp.PREC_MIXED])
@pytest.mark.parametrize("n", GRIDS)
@pytest.mark.parametrize("how", ["size", "tuned", "set"])
def test_shape_goes_to_another_context(n, prec, how):
    a, b = context(n, [BALL]), context(n, [BALL])
    a.time_kernel(cfp.KERNEL_APPLY, prec, 1)  # sets up the ring where it applies
    if how == "tuned":
        a.tune_apply(prec)
    elif how == "set":
        a.tune_apply(prec, 2, 32)
    kernel, rows, planes = a.apply_shape(prec)
    b.tune_apply(prec, rows, planes, kernel=kernel)
    assert b.apply_shape(prec) == (kernel, rows, planes)
    if how == "set":
        assert (kernel, rows, planes) == (cfp.APPLY_STREAM, 2, 32)
    # the dot products are summed per CTA: the same shape, the same bits
    x = torch.randn(a.N, dtype=torch.float64, device="cuda", generator=torch.Generator("cuda").manual_seed(1))
    gi = torch.zeros(a.n_ibi, dtype=torch.float64, device="cuda")
    us = []
    for ctx in (a, b):
        u = torch.zeros(a.N, dtype=torch.float64, device="cuda")
        ctx.solve(x, x, gi, u, tol=1e-3, maxit=2, check=False, precision=prec)
        us.append(u)
    assert torch.equal(us[0], us[1])
    a.close()
    b.close()


def test_by_size_shapes_differ_from_the_listed_ones():
    """33^3 in FP64 runs smaller tiles than any shape of the tuner's list."""
    a = context((33, 33, 33))
    kernel, rows, planes = a.apply_shape(cfp.PREC_FP64)
    assert kernel == cfp.APPLY_STREAM and rows in (1, 2, 4) and planes < 16
    a.close()


@pytest.mark.parametrize("prec", [cfp.PREC_FP64, cfp.PREC_MIXED])
def test_other_shapes_stay_refused(prec):
    a = context((129, 129, 129))
    own = a.apply_shape(prec)
    for s in [(1, 3, 64), (1, 4, 7), (1, 4, 128), (1, 8, 16), (2, 2, 16), (2, 2, 33), (2, 4, 64), (3, 2, 64), (1, 0, 64),
              (1, 2, 0)]:
        assert s != own
        with pytest.raises(cfp.CfpError) as e:
            a.tune_apply(prec, s[1], s[2], kernel=s[0])
        assert e.value.status == cfp.EINVAL
        assert a.apply_shape(prec) == own
    a.close()


def test_ring_planes_of_a_body_free_grid_and_unaligned_fields():
    """A ring of more planes than the streaming kernel stages: with fields that
    are not 16-byte aligned that kernel takes its place, with the same bits."""
    n = (259, 402, 402)
    tiles = (n[1] - 2 + 1) // 2 * (n[2] - 2)
    planes = min(128, tiles // 1024)
    assert planes > 64
    a = context(n, [BALL])
    x = torch.randn(a.N + 4, dtype=torch.float32, device="cuda", generator=torch.Generator("cuda").manual_seed(2))
    outs = []
    for kernel, rows, q in [(cfp.APPLY_STREAM, 4, 64), (cfp.APPLY_RING, 2, planes)]:
        a.tune_apply(cfp.PREC_MIXED, rows, q, kernel=kernel)
        assert a.apply_shape() == (kernel, rows, q)
        for off in (0, 1):
            v = torch.empty(a.N + 4, dtype=torch.float32, device="cuda")[off:off + a.N]
            v.copy_(x[:a.N])
            y = torch.full((a.N,), float("nan"), dtype=torch.float32, device="cuda")
            a.apply_f32(v, y)
            outs.append(y)
    assert all(torch.equal(o, outs[0]) for o in outs)
    a.close()
