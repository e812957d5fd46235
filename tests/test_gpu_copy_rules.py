"""When a march reads gather copies, seen in the kernels that a call launches
(the copy is one more; the diagonal from copies also expands its packed sums):
copies where they pay, none where the gathers they save cost less."""
import numpy as np
import pytest

from gpu_common import empty

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("call,dtype,G,cams,W,H,launches", [
    ("render", "f32", 128, 10, 800, 800, 2),
    ("render", "f32", 64, 5, 800, 800, 1),        # the L1s nearly hold the grid
    ("render", "f32", 93, 7, 165, 165, 1),
    ("residual", "bf16", 256, 4, 800, 800, 2),
    ("residual", "bf16", 128, 4, 800, 800, 1),
    ("vjp", "f32", 128, 1, 800, 800, 2),
    ("vjp", "bf16", 121, 1, 65, 676, 1),          # 0.2 samples a voxel
    ("diag", "f32", 128, 1, 800, 800, 3),
    ("diag", "f32", 62, 2, 69, 519, 1),           # most rays miss the grid
    ("apply", "f32", 128, 1, 800, 800, 2),
    ("apply", "bf16", 152, 1, 190, 796, 1),
    ("jvp", "f32", 128, 2, 800, 800, 2),
    ("jvp", "f32", 129, 1, 690, 112, 1),
])
def test_marches_copy_where_it_pays(call, dtype, G, cams, W, H, launches):
    import torch
    from paper_2112_05598_gb300 import PERF_BF16, PERF_F32, Context
    from paper_2112_05598_gb300._binding import launch_count
    from scenegen import make_cameras
    c2w, focal = make_cameras(np.random.default_rng(2), cams, W, 4.0, "hemisphere", 40.0)
    bf = dtype == "bf16"
    ctx = Context(G, (), 0, 0, c2w, focal, W, H, dtype=PERF_BF16 if bf else PERF_F32)
    x = torch.full((4 * G ** 3,), 0.1, dtype=torch.bfloat16 if bf else torch.float32, device="cuda")
    rays, n = ctx.n_rays, x.numel()
    t = torch.zeros(3 * rays, dtype=x.dtype, device="cuda")
    out = empty(max(3 * rays, n))
    p = torch.ones(n, device="cuda")
    calls = {"render": lambda: ctx.render(x, out),
             "residual": lambda: ctx.residual(x, t, torch.empty_like(t), empty(1, torch.float64)),
             "vjp": lambda: ctx.vjp(x, torch.ones(3 * rays, device="cuda"), out),
             "diag": lambda: ctx.diag_jtj(x, out), "apply": lambda: ctx.apply_normal(x, p, out),
             "jvp": lambda: ctx.jvp(x, p, out)}
    before = launch_count()
    calls[call]()
    assert launch_count() - before == launches
    torch.cuda.synchronize()
