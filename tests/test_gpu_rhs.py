"""The right-hand side where there is no fluid at all (the inside of no body):
zero at every node, whatever f and g hold there, like the row-by-row form of
cfp_assemble_rhs_noalloc; and where it shares memory with an input."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu

from oracle import pyoracle as O  # noqa: E402
from paper_1901_08269_gb300 import cfp  # noqa: E402
from paper_1901_08269_gb300 import workloads as W  # noqa: E402


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    torch.cuda.set_device(0)


@pytest.mark.parametrize("n", [(3, 4, 5), (17, 9, 12), (41, 35, 38)])
def test_interior_of_no_body(n):
    axes = [W.tanh_grid(-1, 1, q, 0.7) for q in n]
    ctx = cfp.Context(*axes, [], fluid_inside=True)
    types = torch.empty(ctx.N, dtype=torch.uint8, device="cuda")
    ctx.classify_points(types)
    P = O.Problem(*axes, [], True)
    np.testing.assert_array_equal(types.cpu().numpy(), P.classify())
    solid = types == O.SOLID
    assert int(solid.sum()) == np.prod([q - 2 for q in n])
    f = torch.randn(ctx.N, dtype=torch.float64, device="cuda", generator=torch.Generator("cuda").manual_seed(1))
    g = torch.randn(ctx.N, dtype=torch.float64, device="cuda", generator=torch.Generator("cuda").manual_seed(2))
    f[solid] = float("nan")  # the values at solid nodes are not read
    for entry in (ctx.assemble_rhs, ctx.assemble_rhs_noalloc):
        rhs = torch.full((ctx.N,), float("nan"), dtype=torch.float64, device="cuda")
        entry(f, g, None, rhs)
        assert torch.equal(rhs, torch.zeros_like(rhs)), entry
    ctx.close()


BALL = W.sphere((0.05, -0.03, 0.02), 0.3)


@pytest.mark.parametrize("which", ["f", "g", "g_ibi", "shifted"])
def test_rhs_may_share_memory_with_an_input(which):
    """The same bits as with memory of its own: rhs in the place of f, of g,
    over g_ibi, and beginning in the middle of f."""
    n = (41, 35, 38)
    axes = [W.tanh_grid(-1, 1, q, 0.7) for q in n]
    ctx = cfp.Context(*axes, [BALL])
    ctx.classify_points()
    gen = torch.Generator("cuda").manual_seed(3)

    def field(m):
        return torch.randn(m, dtype=torch.float64, device="cuda", generator=gen)

    f, g, gi = field(ctx.N), field(ctx.N), field(ctx.n_ibi)
    want = torch.empty(ctx.N, dtype=torch.float64, device="cuda")
    ctx.assemble_rhs(f, g, gi, want)
    room = torch.zeros(2 * ctx.N, dtype=torch.float64, device="cuda")
    start = 0 if which != "shifted" else ctx.N // 2 + 1
    src = {"f": f, "g": g, "g_ibi": gi, "shifted": f}[which]
    inp, rhs = room[:src.numel()], room[start:start + ctx.N]
    inp.copy_(src)
    a = {"f": f, "g": g, "g_ibi": gi}
    a["f" if which == "shifted" else which] = inp
    ctx.assemble_rhs(a["f"], a["g"], a["g_ibi"], rhs)
    assert torch.equal(rhs, want)
    ctx.close()
