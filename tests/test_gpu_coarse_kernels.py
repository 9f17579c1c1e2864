"""Kernels that carry the small levels: the CG step of the smoother's eigenvalue
estimate (one cluster, or three launches on longer vectors) and the product
with the Galerkin blocks of the zeroth-order term."""
import math

import pytest

torch = pytest.importorskip("torch")

from paper_1907_01572_gb300 import dgell, inputs  # noqa: E402
from tests.gpu_util import single  # noqa: E402

pytestmark = pytest.mark.gpu


def _smooth_reference(apply, b, x, ne, nc, Lam=20.0):
    """Algs. 4-5 in FP64 vector operations around the given operator."""
    x = x.clone()
    r = b - apply(x)
    p, rr, lam, prev = r.clone(), float(r @ r), 0.0, None
    for _ in range(ne):
        Ap = apply(p)
        a = rr / float(p @ Ap)
        x += a * p
        r = r - a * Ap
        new = float(r @ r)
        beta = new / rr
        row = 1 / a + math.sqrt(beta) / a + ((prev[1] + math.sqrt(prev[1])) / prev[0] if prev else 0.0)
        lam, prev, rr = max(lam, row), (a, beta), new
        p = r + beta * p
    lo = lam / Lam
    c, d = 0.5 * (lam - lo), 0.5 * (lam + lo)
    p, a = torch.zeros_like(x), 0.0
    for k in range(nc):
        a = 1 / d if k == 0 else (2 * d / (2 * d * d - c * c) if k == 1 else 1 / (d - a * c * c / 4))
        p = a * (b - apply(x)) + (a * d - 1) * p
        x = x + p
    return x, lam


# 8 DOFs; the last vector of one value a thread (4,096) and longer ones up to the cluster's 16,384; beyond it
@pytest.mark.parametrize("desc", [single(1), single(1, level=3), single(4, level=2), inputs.sweep_mesh(level=2, seed=4, pmax=4),
                                  single(5, level=2), single(6, level=2)],
                         ids=["8", "4096", "8000", "hp", "13824", "21952"])
def test_cg_step_and_estimate(desc):
    ctx = dgell.Context(desc)
    n = ctx.level_info()["n_dofs"]
    g = torch.Generator(device="cuda").manual_seed(n)
    b = torch.randn(n, dtype=torch.float64, device="cuda", generator=g)
    x = torch.randn(n, dtype=torch.float64, device="cuda", generator=g)
    ne = min(6, max(1, n // 4))
    want, lam = _smooth_reference(lambda v: ctx.apply(v, torch.empty_like(v)), b, x, ne, 5)
    got_lam = ctx.smooth(b, x, n_eigs=ne, n_cheb=5)
    # six CG steps amplify the rounding of the dot products (n eps) by at most a few hundred
    assert abs(got_lam - lam) <= 1e-11 * lam
    assert float((x - want).norm()) <= 1e-11 * float(want.norm())


def _curved(p):
    return single(p, level=1, warp=(0.03, (1, 2, 1)))


# every remainder of the 32 rows a block takes; elements carried over between levels and mixed degrees on
# three levels; turned blocks
@pytest.mark.parametrize("desc", [_curved(1), _curved(2), _curved(3), _curved(6), _curved(8),
                                  inputs.sweep_mesh(level=1, seed=3, pmin=1, pmax=8),
                                  inputs.block_pair_mesh(rot=5, level=2, seed=1)],
                         ids=["p1", "p2", "p3", "p6", "p8", "hp", "blocks"])
def test_galerkin_blocks_on_the_coarse_levels(desc):
    """O^H x = (I^T O^h I) x, with O^h from the finest level's quadrature."""
    ctx = dgell.Context(desc)
    Lt = ctx.n_levels - 1
    assert Lt >= 1
    n = [ctx.level_info(l)["n_dofs"] for l in range(Lt + 1)]
    g = torch.Generator(device="cuda").manual_seed(n[0])
    coef = 1.0 + torch.rand(ctx.level_info()["n_vol_qp"], dtype=torch.float64, device="cuda", generator=g)
    for low in range(Lt):
        x = torch.randn(n[low], dtype=torch.float64, device="cuda", generator=g)
        xf = x
        for l in range(low, Lt):
            up = torch.zeros(n[l + 1], dtype=torch.float64, device="cuda")
            xf = ctx.transfer(l, 0, xf, up)

        def both(z):
            ctx.set_zeroth_order(coef if z else None)
            lowp = ctx.apply(x.float(), torch.empty(n[low], device="cuda"), level=low)
            return [ctx.apply(x, torch.empty_like(x), level=low), ctx.apply(xf, torch.empty_like(xf)), lowp.double()]

        (c1, f1, s1), (c0, f0, s0) = both(True), both(False)
        want = f1 - f0
        for l in range(Lt - 1, low - 1, -1):
            want = ctx.transfer(l, 1, want, torch.empty(n[l], dtype=torch.float64, device="cuda"))
        # both sides are differences of applies: their rounding is that of the applies
        size = float(c1.norm()) + float(f1.norm())
        assert float((c1 - c0 - want).norm()) <= 1e-13 * size
        assert float((s1 - s0 - want).norm()) <= 1e-6 * size


@pytest.mark.parametrize("dtype", [torch.float64, torch.float32])
@pytest.mark.parametrize("desc", [inputs.sweep_mesh(level=5, seed=2, pmin=1, pmax=2), single(1, level=5)], ids=["hp", "p1"])
def test_restriction_of_large_levels_is_the_transposed_prolongation(desc, dtype):
    """f_H . v = r . (P v), with more coarse elements than run their children side by side (2,048),
    carried-over ones among them; each product is rounded a few dozen times."""
    ctx = dgell.Context(desc)
    low = ctx.n_levels - 2
    n_c, n_f = ctx.level_info(low)["n_dofs"], ctx.level_info(low + 1)["n_dofs"]
    assert ctx.level_info(low)["n_elems"] > 2048
    g = torch.Generator(device="cuda").manual_seed(1)
    r = torch.randn(n_f, dtype=dtype, device="cuda", generator=g)
    v = torch.randn(n_c, dtype=dtype, device="cuda", generator=g)
    f = ctx.transfer(low, 1, r, torch.full_like(v, float("nan")))
    up = ctx.transfer(low, 0, v, torch.zeros_like(r))
    want = r.double() * up.double()
    assert abs(float((f.double() * v.double()).sum() - want.sum())) <= 32 * torch.finfo(dtype).eps * float(want.abs().sum())
