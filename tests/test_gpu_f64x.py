"""FP64 apply on the tensor pipe (levels of more than 304 elements): every side
degree and mortar size against the oracle, and the properties that the exact
digit arithmetic has to keep."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from gpu_util import oracle_mesh, single  # noqa: E402
from oracle import sipg  # noqa: E402
from paper_1907_01572_gb300 import dgell, inputs  # noqa: E402

pytestmark = pytest.mark.gpu

# one launch for all degrees: n = 2..9 with every mortar size, hanging faces; turned blocks
# a launch per degree: one degree (each end of the FP64 / integer volume passes, n = 5 | 6, n = 9) and many
MESHES = {
    "hp_fused": lambda: inputs.sweep_mesh(level=3, seed=5, pmin=1, pmax=8),
    "blocks_fused": lambda: inputs.block_pair_mesh(rot=5, level=3, refine_block=0, seed=2, pmin=1, pmax=8, refine_count=9),
    "p1": lambda: single(1, level=3, warp=(0.02, (1, 2, 1))),
    "p4": lambda: single(4, level=3, warp=(0.02, (1, 2, 1))),
    "p5": lambda: single(5, level=3, warp=(0.02, (1, 2, 1))),
    "p8": lambda: single(8, level=3, warp=(0.02, (1, 2, 1))),
    "hp_buckets": lambda: inputs.sweep_mesh(level=4, seed=3, pmin=1, pmax=8),
}


def _apply(ctx, x):
    return ctx.apply(x, torch.empty_like(x))


@pytest.mark.parametrize("name", list(MESHES))
def test_against_the_oracle(name):
    desc = MESHES[name]()
    m = oracle_mesh(desc)
    assert m.n_elems > 304
    ctx = dgell.Context(desc)
    x = inputs.random_vector(m.n_dofs, seed=7)
    y = _apply(ctx, torch.tensor(x, device="cuda")).cpu().numpy()
    rng = np.random.default_rng(1)
    sample = sorted(set(rng.choice(m.n_elems, 16, replace=False).tolist()))
    ref = sipg.apply_local(m, x, 10.0, elems=sample)
    num = sum(np.sum((y[m.dof_off[e]:m.dof_off[e + 1]] - ref[e]) ** 2) for e in sample)
    den = sum(np.sum(ref[e] ** 2) for e in sample)
    assert np.sqrt(num / den) < 1e-12   # the parity bound of every FP64 apply


@pytest.mark.parametrize("name", ["hp_fused", "p8", "p4"])
def test_scaling_zeros_and_additivity(name):
    ctx = dgell.Context(MESHES[name]())
    n = ctx.level_info()["n_dofs"]
    g = torch.Generator(device="cuda").manual_seed(3)
    x = torch.randn(n, dtype=torch.float64, device="cuda", generator=g)
    y = _apply(ctx, x)
    for e in (-400, 1, 400):   # a power of two changes exponents only
        assert torch.equal(_apply(ctx, x * 2.0 ** e), y * 2.0 ** e)
    for e in (-900, 900):      # outside the integers' range: the FP64 code, rounded differently
        z = _apply(ctx, x * 2.0 ** e) * 2.0 ** -e
        assert float((z - y).norm()) <= 1e-13 * float(y.norm())
    assert not _apply(ctx, torch.zeros_like(x)).any()
    # integers add without rounding, so the sum's apply differs by the arithmetic's rounding alone
    a = torch.randint(-2 ** 20, 2 ** 20, (n,), device="cuda", generator=g).double()
    b = torch.randint(-2 ** 20, 2 ** 20, (n,), device="cuda", generator=g).double()
    s = _apply(ctx, a + b)
    assert float((_apply(ctx, a) + _apply(ctx, b) - s).norm()) <= 1e-15 * float(s.norm())


@pytest.mark.parametrize("value", [float("nan"), float("inf")])
def test_non_finite_values_stay_where_they_belong(value):
    """The element and its face neighbours, and no others."""
    desc = single(3, level=3)
    ctx = dgell.Context(desc)
    off = ctx.level_leaves()[2]
    leaves = np.asarray(desc["leaves"])
    e0 = int(np.nonzero((leaves[:, 1:] == 3).all(1))[0][0])
    x = torch.ones(ctx.level_info()["n_dofs"], dtype=torch.float64, device="cuda")
    x[int(off[e0]) + 21] = value   # an interior node
    y = _apply(ctx, x).cpu().numpy()
    near = np.abs(leaves[:, 1:] - 3).sum(1) <= 1
    for e in range(len(leaves)):
        fin = np.isfinite(y[off[e]:off[e + 1]])
        assert fin.all() if not near[e] else not fin.all()
    assert not np.isfinite(y[off[e0]:off[e0 + 1]]).any()


@pytest.mark.parametrize("name", ["hp_fused", "p8"])
def test_zeroth_order_term(name):
    """(L + M_c - L) 1 = int c psi, the right-hand side of g = c."""
    ctx = dgell.Context(MESHES[name]())
    i = ctx.level_info()
    c = 1.0 + torch.rand(i["n_vol_qp"], dtype=torch.float64, device="cuda") * 1e3
    one = torch.ones(i["n_dofs"], dtype=torch.float64, device="cuda")
    y0 = _apply(ctx, one)
    ctx.set_zeroth_order(c)
    y1 = _apply(ctx, one)
    F = ctx.rhs(c, None, torch.empty_like(one))
    assert float((y1 - y0 - F).norm()) <= 1e-12 * float(y1.norm())
