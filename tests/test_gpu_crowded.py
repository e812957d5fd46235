"""Scenes whose parameters are each seen by very many rays: a parameter is then
a long chain of binary32 additions, and the scatters keep the plain lane order."""
import importlib.util
import os

import numpy as np
import pytest

from conftest import ROOT, rel_l2
from gpu_common import TOL_FP32, assert_elementwise, cuda_tensor, empty, host

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("cube", [False, True])
@pytest.mark.parametrize("G", [2, 4])
def test_operators_on_a_tiny_grid_against_oracle(G, cube):
    """92 k rays into 8 and 64 voxels: J p, J^T v, A p and the gradient within the
    library's bars (the diagonal, whose terms are all positive, rounds to 1.5e-5
    to 3e-5 there in every order of its additions)."""
    from gpu_common import make_pair
    from test_gpu_copies import _problem
    rng, a, x = _problem(G, 421, 219, 1, cube)
    ctx, orc = make_pair(*a, env_kind=int(cube))
    p, v = rng.normal(size=x.size).astype(np.float32), rng.normal(size=3 * 421 * 219).astype(np.float32)
    xd, pd, vd = cuda_tensor(x), cuda_tensor(p), cuda_tensor(v)
    jp, jtv, ap, dg, gr = empty(v.size), empty(x.size), empty(x.size), empty(x.size), empty(x.size)
    ctx.jvp(xd, pd, jp)
    ctx.vjp(xd, vd, jtv)
    ctx.apply_normal(xd, pd, ap)
    ctx.diag_jtj(xd, dg, vd, gr)
    x64, p64, v64 = (q.astype(np.float64) for q in (x, p, v))
    ref, mag = orc.jvp(x64, p64, mag=True)
    assert rel_l2(host(jp), ref) < TOL_FP32
    ref, mag = orc.vjp(x64, v64, mag=True)
    assert rel_l2(host(jtv), ref) < TOL_FP32
    assert_elementwise(host(jtv), ref, mag, what=f"J^T v {G}")
    assert rel_l2(host(ap), orc.apply_A(x64, p64)) < TOL_FP32
    assert rel_l2(host(gr), orc.diag_grad(x64, v64)[1]) < TOL_FP32


def test_gauss_newton_step_of_a_crowded_scene_against_oracle():
    """2.2 M rays on a 26^3 grid and shells of 11 x 22 texels, 6 PCG iterations:
    the objective after the step within 2e-5 of the FP64 step's, which is 2^-24
    times the sqrt(1e5) additions of its fullest parameters."""
    from oracle import Oracle, gn_step
    spec = importlib.util.spec_from_file_location("perf_cases", os.path.join(ROOT, "perf", "cases.py"))
    cases = importlib.util.module_from_spec(spec)
    spec.loader.exec_module(cases)
    case = dict(op="gn", G=26, S=4, He=11, W=674, H=69, cams=47, layout="ring", cube=False, bf16=False,
                late=False, jitter=False, aux=False, pcg=6, block=False)
    st = cases.prepare(case, 235)
    x0, target = host(st["x0"]), host(st["target"])
    got = cases.run(st)
    _, c2w, focal, He, We = cases._geometry(case, 235)
    orc = Oracle(26, cases.RADII, He, We, c2w, focal, 674, 69, max_samples=512)
    ref = gn_step(orc, x0, target, 6)
    assert ref.accepted
    print(f"[crowded] F_after {got['F_after']:.9g}, FP64 {ref.F_after:.9g}, "
          f"rel {got['F_after'] / ref.F_after - 1:.2e}")
    assert abs(got["F_before"] - ref.F_before) <= 1e-6 * ref.F_before
    assert abs(got["F_after"] - ref.F_after) <= 2e-5 * ref.F_after
