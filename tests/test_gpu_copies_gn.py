"""Gauss-Newton steps, the diagonal's block couplings, Adam and per-call PCG on
launches large enough for gather copies, the spread lane order and the packed
diagonal, against the FP64 oracle: full, partial and no coefficient store, the
auxiliary term, brick order, BF16 scenes, and the step that is redone with
Jacobi after the line search's trial points have taken the copy's place."""
import dataclasses

import numpy as np
import pytest

from conftest import rel_l2
from gpu_common import TOL_FP32, TOL_GN, cuda_tensor, empty, host

pytestmark = pytest.mark.gpu
LAM = 0.1


def _scene(G, cams, W, H):
    """A small-workload scene at other sizes, a state halfway to its ground
    truth, and the FP64 oracle."""
    from oracle import Oracle
    from scenegen import CONFIGS, make_scene
    sc = make_scene(dataclasses.replace(CONFIGS["small32"], G=G, n_cams=cams, width=W, height=H,
                                        env_h=16, env_w=32, max_samples=2 * G))
    tiles = -(-W // 8) * -(-H // 4) * cams
    assert tiles > 1824, "small launches gather from the grid itself"
    orc = Oracle.from_scene(sc)
    target = orc.render(sc.x_gt)[0].astype(np.float32).ravel()
    return sc, orc, target, (0.5 * sc.x0 + 0.5 * sc.x_gt).astype(np.float32)


@pytest.fixture(scope="module")
def mid():
    return _scene(24, 7, 150, 135)


def _launches(call):
    from paper_2112_05598_gb300._binding import launch_count
    before = launch_count()
    call()
    return launch_count() - before


def _same_step(orc, st, x, ref):
    """What a step determines well: its objective and the image it renders
    (barely observed parameters magnify the rounding of their rows)."""
    assert abs(st["F_after"] - ref.F_after) <= TOL_GN * ref.F_after
    assert rel_l2(orc.render(x)[0], orc.render(ref.x)[0]) < TOL_GN


@pytest.mark.parametrize("brick", [1, 4])
@pytest.mark.parametrize("budget", ["full", "half", "none"])
@pytest.mark.parametrize("aux", [0, 1])
def test_gn_step_from_copies_against_oracle(mid, aux, budget, brick):
    """One step of 3 PCG iterations: F before within 1e-5, F after and the image
    within the Gauss-Newton tolerance.  The plain operators of the same context launch
    the copy beside their march, so the step's do too."""
    from oracle import Oracle, gn_step
    from paper_2112_05598_gb300 import Context
    sc, _, target, x = mid
    orc = Oracle.from_scene(sc, aux=bool(aux), aux_lambda=LAM)
    ctx = Context.from_scene(sc, pcg_iters=3, pcg_fixed=1, aux=aux, aux_lambda=LAM)
    d = empty(x.size)
    ctx.diag_jtj(cuda_tensor(x), d)
    assert _launches(lambda: ctx.diag_jtj(cuda_tensor(x), d)) == 3   # copy, march, expansion
    ctx.set_brick(brick)
    td = cuda_tensor(target)
    if budget == "half":
        ctx.gn_solve(cuda_tensor(x), td, 1)
        ctx.set_coef_budget(ctx.coef_info()["bytes"] // 2)
    elif budget == "none":
        ctx.set_coef_budget(0)
    xd = cuda_tensor(x)
    st = ctx.gn_solve(xd, td, 1)[0]
    cov = ctx.coef_info()
    assert cov["used"] == (budget != "none")
    if budget == "half":
        assert 0.2 < cov["coverage"] < 0.8
    ref = gn_step(orc, x.astype(np.float64), target.astype(np.float64), 3)
    assert st["accepted"] and abs(st["gamma"] - ref.gamma) < 1e-9
    assert abs(st["F_before"] - ref.F_before) <= TOL_FP32 * ref.F_before
    _same_step(orc, st, host(xd), ref)


def test_bf16_gn_step_at_the_size_of_copies_against_oracle(mid):
    """A BF16 scene's step keeps the plain scatters at this size: the objective
    before and after the step against the oracle on the BF16-rounded state
    (p and the trial point are rounded to BF16 on the way, 2^-9 a value, so F
    after the step is held to 1%)."""
    import torch
    from oracle import gn_step
    from paper_2112_05598_gb300 import PERF_BF16, Context
    sc, orc, target, x = mid
    ctx = Context.from_scene(sc, pcg_iters=3, pcg_fixed=1, dtype=PERF_BF16)
    td = cuda_tensor(target, torch.bfloat16)
    x16 = host(cuda_tensor(x, torch.bfloat16).float())
    t16 = host(td.float())
    xd = cuda_tensor(x16.astype(np.float32))
    st = ctx.gn_solve(xd, td, 1)[0]
    ref = gn_step(orc, x16, t16, 3)
    assert st["accepted"] and abs(st["gamma"] - ref.gamma) < 1e-9
    assert abs(st["F_before"] - ref.F_before) <= 1e-3 * ref.F_before
    assert abs(st["F_after"] - ref.F_after) <= 1e-2 * ref.F_before


def test_step_redone_with_jacobi_reads_the_right_copy():
    """Blocks that are indefinite in the opacities give a step that raises F; it
    is redone with Jacobi, on a half store, so the recomputing A p reads x's
    copy, whose place the trial point had taken.  100^3: the forward marches
    read copies too."""
    from oracle import gn_step
    from paper_2112_05598_gb300 import PERF_JUDGE_OBJECTIVE, PERF_PRECOND_BLOCK4, Context
    sc, orc, target, x = _scene(100, 3, 520, 512)
    xd, td, n = cuda_tensor(x), cuda_tensor(target), x.size
    ctx = Context.from_scene(sc, pcg_iters=4, pcg_fixed=1, ls_max=0, precond=PERF_PRECOND_BLOCK4,
                             precond_judge=PERF_JUDGE_OBJECTIVE)
    rgb = empty(3 * ctx.n_rays)
    ctx.render(xd, rgb)
    assert _launches(lambda: ctx.render(xd, rgb)) == 2
    diag = empty(n)
    ctx.diag_jtj(xd, diag)
    host_diag = host(diag)[:4 * 100 ** 3].reshape(-1, 4)
    P = np.zeros((100 ** 3, 4, 4), np.float32)
    for c in range(4):
        seen = host_diag[:, c] > 1e-30
        P[seen, c, c] = (-1.0 if c == 3 else 1.0) / host_diag[seen, c]
    blocks = cuda_tensor(P.reshape(-1))
    ctx.set_blocks(blocks, 100 ** 3)
    ctx.gn_solve(xd.clone(), td, 1)
    ctx.set_coef_budget(ctx.coef_info()["bytes"] // 2)
    got = xd.clone()
    st = ctx.gn_solve(got, td, 1)[0]
    assert 0.2 < ctx.coef_info()["coverage"] < 0.8
    ref = gn_step(orc, x.astype(np.float64), target.astype(np.float64), 4, ls_max=0)
    assert ref.accepted and st["accepted"] and st["precond_fallback"] and st["ls_evals"] == 2
    _same_step(orc, st, host(got), ref)


def test_block_couplings_from_copies(mid):
    from paper_2112_05598_gb300 import Context
    sc, orc, _, x = mid
    ctx = Context.from_scene(sc)
    d, cr = empty(x.size), empty(4 * sc.G ** 3)
    ctx.diag_cross(cuda_tensor(x), d, cr)
    assert _launches(lambda: ctx.diag_cross(cuda_tensor(x), d, cr)) == 3
    dref, cref = orc.block_cross(x.astype(np.float64))
    assert rel_l2(host(d), dref) < TOL_FP32
    assert rel_l2(host(cr).reshape(-1, 4)[:, :3], np.asarray(cref).reshape(-1, 4)[:, :3]) < TOL_FP32


def test_adam_step_from_copies(mid):
    import torch
    from oracle import adam_step
    from paper_2112_05598_gb300 import Context
    sc, orc, target, x = mid
    ctx = Context.from_scene(sc)
    xd, m, v = cuda_tensor(x), empty(x.size), empty(x.size)
    F = empty(1, torch.float64)
    ctx.adam_step(xd, cuda_tensor(target), m, v, 1, F_out=F)
    _, mr, vr, Fr = adam_step(orc, x.astype(np.float64), target.astype(np.float64),
                              np.zeros(x.size), np.zeros(x.size), 1)
    assert abs(F.item() - Fr) <= TOL_FP32 * Fr
    # m = (1 - beta1) J^T r: the gradient itself (x's step is its sign at t = 1)
    assert rel_l2(host(m), mr) < TOL_FP32
    assert rel_l2(host(v), vr) < 2 * TOL_FP32


def test_per_call_pcg_from_copies(mid):
    """pcg_begin and three pcg_step on the grad and diagonal of the context: the
    direction of the oracle's CG."""
    from oracle import jacobi_apply, pcg
    from paper_2112_05598_gb300 import Context
    sc, orc, target, x = mid
    ctx = Context.from_scene(sc, pcg_iters=3, pcg_fixed=1)
    x64 = x.astype(np.float64)
    r, _ = orc.residual(x64, target.astype(np.float64))
    diag, grad = orc.diag_grad(x64, r)
    xd, dd, gd = cuda_tensor(x), cuda_tensor(diag.astype(np.float32)), cuda_tensor(grad.astype(np.float32))
    ctx.pcg_begin(gd, dd)
    for _ in range(3):
        ctx.pcg_step(xd)
    delta = empty(x.size)
    ctx.pcg_result(delta)
    ref = pcg(lambda p: orc.apply_A(x64, p), -grad, lambda q: jacobi_apply(diag, q), 3, fixed=True)
    assert rel_l2(host(delta), ref.x) < TOL_GN
