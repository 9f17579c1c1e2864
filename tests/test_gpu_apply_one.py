"""FP32 apply in one launch (small levels): against the oracle over side
degrees, hanging faces, turned blocks and coarse levels.  Which plan a level
takes is timed, except under stream capture, where a level of up to 304
elements takes the one-launch form: so the tests capture the apply."""
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
