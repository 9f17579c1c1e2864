"""FP32 apply in one launch (small levels): against the oracle over side
degrees, hanging faces, turned blocks and coarse levels.  Which plan a level
takes is timed, except under stream capture, where a level of up to 304
elements takes the one-launch form, or with DGELL_APPLY_PLAN=4, read at a
process's first apply: so the tests capture the apply or run it in a child."""
import os
import subprocess
import sys

import pytest

torch = pytest.importorskip("torch")

from gpu_util import CASES, oracle_mesh, rel_l2  # noqa: E402
from oracle import sipg  # noqa: E402
from paper_1907_01572_gb300 import dgell, inputs  # noqa: E402

pytestmark = pytest.mark.gpu

MESHES = dict({k: CASES[k] for k in ("config1_affine_p3", "mixed_curved_2to1_l1", "single_element_p1", "single_element_p8_curved",
                                     "uniform_p8_2x2x2", "blocks_turned_fine_side", "blocks_turned_coarse_side",
                                     "cubed_sphere_shell_2to1")},
              hp_1to8=lambda: inputs.sweep_mesh(level=1, seed=11, pmin=1, pmax=8))


@pytest.mark.parametrize("dtype", [torch.float32, torch.bfloat16], ids=["f32", "bf16"])
@pytest.mark.parametrize("name", list(MESHES))
def test_captured_apply_against_the_oracle(name, dtype):
    desc = MESHES[name]()
    st = torch.cuda.Stream()
    ctx = dgell.Context(desc, stream=st.cuda_stream)
    m = oracle_mesh(desc)
    x = torch.tensor(inputs.random_vector(m.n_dofs, seed=5), device="cuda").to(dtype)
    y = torch.full((m.n_dofs,), float("nan"), device="cuda")
    torch.cuda.synchronize()
    launches = ctx.launch_count()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, stream=st):
        ctx.apply(x, y)
    assert ctx.launch_count() == launches + 1   # one kernel
    g.replay()
    torch.cuda.synchronize()
    want = sipg.assemble(m) @ x.double().cpu().numpy()
    assert rel_l2(y.double().cpu().numpy(), want) < 1e-5   # the FP32 parity bound, on the rounded input


def test_captured_apply_on_coarse_levels_with_the_zeroth_order_term():
    """The one-launch form adds to the Galerkin blocks' product like the others:
    FP32 against the FP64 apply of the same level."""
    st = torch.cuda.Stream()
    ctx = dgell.Context(inputs.sweep_mesh(level=2, seed=4, pmin=1, pmax=8), stream=st.cuda_stream)
    c = 1.0 + torch.rand(ctx.level_info()["n_vol_qp"], dtype=torch.float64, device="cuda")
    torch.cuda.synchronize()
    ctx.set_zeroth_order(c)
    for level in range(ctx.n_levels):
        n = ctx.level_info(level)["n_dofs"]
        x = torch.tensor(inputs.random_vector(n, seed=level), device="cuda").float()
        y, y64 = torch.empty_like(x), torch.empty(n, dtype=torch.float64, device="cuda")
        torch.cuda.synchronize()
        ctx.apply(x.double(), y64, level=level)
        st.synchronize()
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g, stream=st):
            ctx.apply(x, y, level=level)
        g.replay()
        torch.cuda.synchronize()
        assert rel_l2(y.double().cpu().numpy(), y64.cpu().numpy()) < 1e-5


def _plan4(code):
    here = os.path.dirname(os.path.abspath(__file__))
    path = os.pathsep.join([here, os.path.dirname(here), os.environ.get("PYTHONPATH", "")])
    code = ("import torch\nfrom gpu_util import CASES, single, rel_l2\nfrom paper_1907_01572_gb300 import dgell, inputs\n"
            "def randn(n):\n    return torch.tensor(inputs.random_vector(n, seed=3), device='cuda')\n" + code)
    return subprocess.run([sys.executable, "-c", code], check=True, capture_output=True, text=True,
                          env=dict(os.environ, DGELL_APPLY_PLAN="4", PYTHONPATH=path), cwd=os.path.dirname(here)).stdout.split()


def test_levels_of_up_to_608_elements():
    """512 elements of one degree and of mixed degrees, against the FP64 apply."""
    out = _plan4("""
for d in (single(5, level=3, warp=(0.02, (1, 2, 1))), inputs.sweep_mesh(level=3, seed=5, pmin=1, pmax=8, refine_octant=False)):
    ctx = dgell.Context(d)
    n = ctx.level_info()["n_dofs"]
    assert 304 < ctx.level_info()["n_elems"] <= 608
    for dt in (torch.float32, torch.bfloat16):
        x = randn(n).to(dt)
        y, want = torch.empty(n, device="cuda"), torch.empty(n, dtype=torch.float64, device="cuda")
        ctx.apply(x.double(), want)
        k = ctx.launch_count()
        ctx.apply(x, y)
        print(ctx.launch_count() - k, rel_l2(y.double().cpu().numpy(), want.cpu().numpy()))
""")
    assert out[::2] == ["1"] * 4
    assert all(float(v) < 1e-5 for v in out[1::2])   # the FP32 parity bound


def test_element_diagonal_blocks():
    """The smoother with element subdomains (the neighbour's traces taken as 0): FP32 against FP64 V-cycle,
    with a fixed number of local CG steps.  FP32 rounding, amplified by the local problems' condition
    (a few hundred), stays below 1e-3; a neighbour's trace left in would change a fifth of the values' size."""
    out = _plan4("""
for name in ("config1_affine_p3", "mixed_curved_2to1_l1"):
    ctx = dgell.Context(CASES[name]())
    f = randn(ctx.level_info()["n_dofs"])
    v = [torch.empty_like(f, dtype=t) for t in (torch.float64, torch.float32)]
    for w in v:
        ctx.vcycle(f.to(w.dtype), w, smoother=1, local_iters=6, local_tol=1e-12)
    print(rel_l2(v[1].double().cpu().numpy(), v[0].cpu().numpy()))
""")
    assert all(float(v) < 1e-3 for v in out) and len(out) == 2
