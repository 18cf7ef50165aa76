"""Grids whose z axis is longer than 65535 block rows of one launch cover."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu

from paper_1901_08269_gb300 import cfp  # noqa: E402
from paper_1901_08269_gb300 import workloads as W  # noqa: E402


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    torch.cuda.set_device(0)


@pytest.mark.parametrize("precision,nz,unit", [(cfp.PREC_FP64, 131075, 2.0 ** -53), (cfp.PREC_FP64, 263001, 2.0 ** -53),
                                               (cfp.PREC_MIXED, 197001, 2.0 ** -24)])
def test_red_black_sweeps_along_a_long_axis(precision, nz, unit):
    """The same sweeps with the long axis as z and as x: a node's colour, its
    neighbours and coefficients are the same and only the order of its six
    products and three diagonal terms differs.  A half-sweep commits some 17
    roundings of at most twice the largest value and carries earlier errors
    with weights that sum to at most one: 8 x 34 = 272 units, bounded by 512."""
    long, short = W.uniform_grid(-1, 1, nz), [W.tanh_grid(-1, 1, q, 0.7) for q in (11, 9)]
    rho = np.random.default_rng(5).standard_normal((nz, 9, 11))
    out = {}
    for name, axes, r in (("z", (short[0], short[1], long), rho),
                          ("x", (long, short[1], short[0]), np.ascontiguousarray(rho.transpose(2, 1, 0)))):
        ctx = cfp.Context(*axes)
        ctx.classify_points()
        phi = torch.full((ctx.N,), float("nan"), dtype=torch.float64, device="cuda")
        ctx.precondition_ex(torch.as_tensor(r.reshape(-1), device="cuda"), phi, precond=cfp.PRECOND_RBGS, sweeps=4,
                            precision=precision, mg_tma=0)
        got = phi.cpu().numpy().reshape(r.shape)
        out[name] = got if name == "z" else got.transpose(2, 1, 0)
        ctx.close()
    assert np.max(np.abs(out["z"])) > 0 and np.all(np.isfinite(out["z"]))
    assert np.max(np.abs(out["z"] - out["x"])) <= 512 * unit * np.max(np.abs(out["x"]))


def test_multigrid_on_too_long_a_grid_is_refused():
    """The V-cycle's transfers take one block row per coarse plane: 70001 of
    them are refused, by the solve (whose loop is captured) as by the
    preconditioner, every time, and the context goes on."""
    axes = [W.uniform_grid(-1, 1, n) for n in (17, 17, 140001)]
    ctx = cfp.Context(*axes)
    ctx.classify_points()
    f = torch.ones(ctx.N, dtype=torch.float64, device="cuda")
    g = torch.zeros_like(f)
    for _ in range(2):
        u = torch.zeros_like(f)
        with pytest.raises(cfp.CfpError) as e:
            ctx.solve(f, g, None, u, tol=1e-10, precond=cfp.PRECOND_MG, maxit=2)
        assert e.value.status == cfp.ECUDA
        with pytest.raises(cfp.CfpError) as e:
            ctx.precondition_ex(f, u, precond=cfp.PRECOND_MG)
        assert e.value.status == cfp.ECUDA
    ctx.precondition(f, u, sweeps=1)
    assert float(u.abs().max()) > 0.0
    ctx.close()
