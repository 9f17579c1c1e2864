"""FP64 apply on the tensor pipe (levels of more than 304 elements): every side
degree and mortar size against the oracle, and the properties that the exact
digit arithmetic has to keep."""
import os
import subprocess
import sys

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


def _native(name, x, tmp_path, plan=2):
    """The same apply by the FP64 kernels (a process of its own: the plan is fixed at the first apply)."""
    here = os.path.dirname(os.path.abspath(__file__))
    np.save(tmp_path / "x.npy", x)
    code = ("import sys, numpy as np, torch, test_gpu_f64x as t\n"
            "ctx = t.dgell.Context(t.MESHES[sys.argv[1]]())\n"
            "y = [t._apply(ctx, torch.tensor(v, device='cuda')).cpu().numpy() for v in np.load(sys.argv[2])]\n"
            "np.save(sys.argv[3], np.array(y))\n")
    path = os.pathsep.join([here, os.path.dirname(here), os.environ.get("PYTHONPATH", "")])
    subprocess.run([sys.executable, "-c", code, name, str(tmp_path / "x.npy"), str(tmp_path / "y.npy")], check=True,
                   env=dict(os.environ, DGELL_APPLY_PLAN=str(plan), PYTHONPATH=path), cwd=os.path.dirname(here))
    return np.load(tmp_path / "y.npy")


MESHES["p7"] = lambda: single(7, level=3)
MESHES["p8_affine"] = lambda: single(8, level=3)
MESHES["shell_1e9"] = lambda: inputs.cubed_sphere_mesh(level=2, a=1.0, r=3.0, r_out=1e9, pmin=3, pmax=8)


@pytest.mark.parametrize("name", ["p7", "p8_affine"])
def test_concentrated_values_keep_the_accuracy_of_fp64_arithmetic(name, tmp_path):
    """Unit vectors at a corner node and values that fall off from a corner by
    many orders of magnitude, in every third element per axis: each entry of such
    an element follows its own size.  An entry is a chain of twelve contractions
    of n terms, each rounded to n 2^-53 of it in either arithmetic where nothing
    cancels: the bound is put to the median entry."""
    desc = MESHES[name]()
    ctx = dgell.Context(desc)
    off, leaves, n = ctx.level_leaves()[2], np.asarray(desc["leaves"])[:, 1:], int(desc["p"][0]) + 1
    mid = np.nonzero((leaves % 3 == 1).all(1))[0]
    t = np.linspace(-1.0, 1.0, n)
    r = np.sqrt(sum((v + 1.0) ** 2 for v in np.meshgrid(t, t, t, indexing="ij")))
    shapes = [(r == 0).astype(float), np.exp(-30.0 * r)]
    x = np.zeros((len(shapes), int(off[-1])))
    for v, s in zip(x, shapes):
        for e in mid:
            v[off[e]:off[e + 1]] = s.ravel()
    native = _native(name, x, tmp_path)
    for v, want in zip(x, native):
        y = _apply(ctx, torch.tensor(v, device="cuda")).cpu().numpy()
        assert (y != want).any()   # not the same kernels
        own = np.concatenate([np.arange(off[e], off[e + 1]) for e in mid])
        own = own[want[own] != 0]
        assert np.median(np.abs(y[own] - want[own]) / np.abs(want[own])) <= 12 * n * 2.0 ** -53


@pytest.mark.parametrize("name", ["hp_fused", "hp_buckets", "shell_1e9"])
def test_graded_values_element_by_element(name, tmp_path):
    """Magnitudes over eight orders inside every element, and the elements of the
    shell to r = 1e9: each element agrees with the FP64 kernels to 1e-13 by itself."""
    ctx = dgell.Context(MESHES[name]())
    off = ctx.level_leaves()[2]
    assert len(off) - 1 > 304
    rng = np.random.default_rng(2)
    x = rng.standard_normal((2, int(off[-1])))
    x[1] *= 10.0 ** rng.uniform(-8, 0, x.shape[1])
    native = _native(name, x, tmp_path)
    for v, want in zip(x, native):
        y = _apply(ctx, torch.tensor(v, device="cuda")).cpu().numpy()
        d2, w2 = np.add.reduceat((y - want) ** 2, off[:-1]), np.add.reduceat(want ** 2, off[:-1])
        assert (y != want).any()
        assert np.sqrt((d2 / w2).max()) <= 1e-13


@pytest.mark.parametrize("value", [float("nan"), float("inf")])
@pytest.mark.parametrize("p", [5, 8])
def test_non_finite_values_in_the_volume_terms(p, value):
    """As above where the volume terms run on digits too, in the vector and in the zeroth-order coefficient."""
    desc = single(p, level=3)
    ctx = dgell.Context(desc)
    off, n = ctx.level_leaves()[2], p + 1
    leaves = np.asarray(desc["leaves"])
    e0 = int(np.nonzero((leaves[:, 1:] == 3).all(1))[0][0])
    inner = 1 + n + n * n
    x = torch.ones(ctx.level_info()["n_dofs"], dtype=torch.float64, device="cuda")
    c = torch.ones(ctx.level_info()["n_vol_qp"], dtype=torch.float64, device="cuda")
    c[e0 * n ** 3 + inner] = value
    ctx.set_zeroth_order(c)
    y = _apply(ctx, x).cpu().numpy()
    for e in range(len(leaves)):   # the coefficient is the element's own
        assert np.isfinite(y[off[e]:off[e + 1]]).all() == (e != e0)
    ctx.set_zeroth_order(None)
    x[int(off[e0]) + inner] = value
    y = _apply(ctx, x).cpu().numpy()
    near = np.abs(leaves[:, 1:] - 3).sum(1) <= 1
    for e in range(len(leaves)):
        fin = np.isfinite(y[off[e]:off[e + 1]])
        assert fin.all() if not near[e] else not fin.all()
    assert not np.isfinite(y[off[e0]:off[e0 + 1]]).any()


MESHES_LOW = {"p1_4096": lambda: single(1, level=4), "p1to2": lambda: inputs.sweep_mesh(level=3, pmin=1, pmax=2)}
MESHES.update(MESHES_LOW)


@pytest.mark.parametrize("name", list(MESHES_LOW))
def test_low_degrees_stay_on_the_native_kernels(name, tmp_path):
    """Bit for bit one of the native plans (which one is timed)."""
    ctx = dgell.Context(MESHES[name]())
    x = torch.randn(ctx.level_info()["n_dofs"], dtype=torch.float64, device="cuda")
    y = _apply(ctx, x).cpu().numpy()
    assert any(np.array_equal(y, _native(name, x.cpu().numpy()[None], tmp_path, plan)[0]) for plan in range(3))
