"""The gather-copy workspace of a context between calls: a call waits for the
last one that used it, on whichever stream and from whichever thread."""
import threading

import numpy as np
import pytest

from gpu_common import cuda_tensor, empty

pytestmark = pytest.mark.gpu


def _context(G=64, W=400, cams=12):
    """A context whose renders read copies and take long enough to overlap the
    next call's copy."""
    from paper_2112_05598_gb300 import Context
    from scenegen import make_cameras, random_params
    rng = np.random.default_rng(12)
    c2w, focal = make_cameras(rng, cams, W, 3.2, "sphere", 40.0)
    x = random_params(rng, G, 0, 0, 0, 0.01, 0.2)
    ctx = Context(G, (), 0, 0, c2w, focal, W, W)
    return ctx, [cuda_tensor(x), cuda_tensor((0.5 * x).astype(np.float32))]


def _reference(ctx, xs):
    import torch
    want = []
    for x in xs:
        out = empty(3 * ctx.n_rays)
        ctx.render(x, out)
        torch.cuda.synchronize()
        want.append(out)
    return want


def test_a_solve_of_no_steps_does_not_forget_a_render_in_flight():
    import torch
    ctx, xs = _context()
    want = _reference(ctx, xs)
    a, b = torch.cuda.Stream(), torch.cuda.Stream()
    got = [empty(3 * ctx.n_rays) for _ in xs]
    x, target = xs[1].clone(), empty(3 * ctx.n_rays)
    torch.cuda.synchronize()
    for _ in range(8):
        ctx.render(xs[0], got[0], stream=b)
        ctx.gn_solve(x, target, 0, stream=a)
        ctx.render(xs[1], got[1], stream=a)
        torch.cuda.synchronize()
        assert torch.equal(got[0], want[0]) and torch.equal(got[1], want[1])


def test_two_threads_in_turn_on_their_default_streams():
    """cudaStreamPerThread (handle 2) is another stream in each host thread."""
    import torch
    ctx, xs = _context()
    want = _reference(ctx, xs)
    got = [empty(3 * ctx.n_rays) for _ in xs]
    torch.cuda.synchronize()
    mine = torch.cuda.ExternalStream(2)
    turns, fault = [threading.Semaphore(1), threading.Semaphore(0)], []

    def work(i):
        try:
            for _ in range(8):
                turns[i].acquire()
                ctx.render(xs[i], got[i], stream=mine)
                turns[1 - i].release()
        except Exception as e:   # the other thread must not wait for ever
            fault.append(e)
            turns[1 - i].release()

    threads = [threading.Thread(target=work, args=(i,)) for i in range(2)]
    for t in threads:
        t.start()
    for t in threads:
        t.join(60)
    torch.cuda.synchronize()
    assert not fault and not any(t.is_alive() for t in threads)
    assert torch.equal(got[0], want[0]) and torch.equal(got[1], want[1])


def test_a_call_after_a_failed_solve_waits_for_its_marches():
    """A solve that ends in an error (a non-finite objective) leaves the
    workspace to the next call on another stream."""
    import torch
    from paper_2112_05598_gb300 import PerfError
    ctx, xs = _context(G=32, W=300, cams=4)
    want = _reference(ctx, xs)
    bad = torch.full((3 * ctx.n_rays,), float("nan"), device="cuda")
    a, b = torch.cuda.Stream(), torch.cuda.Stream()
    out = empty(3 * ctx.n_rays)
    torch.cuda.synchronize()
    for _ in range(3):
        with pytest.raises(PerfError):
            ctx.gn_solve(xs[0].clone(), bad, 1, stream=a)
        ctx.render(xs[1], out, stream=b)
        torch.cuda.synchronize()
        assert torch.equal(out, want[1])


def test_first_calls_leave_a_capture_on_another_stream_alone():
    """Calls on a stream that is not under capture may allocate their workspace
    while another stream of the thread is: the capture goes on."""
    import torch
    from paper_2112_05598_gb300 import Batch
    from scenegen import make_cameras, random_params
    ctx, xs = _context(G=32, W=300, cams=4)
    want = _reference(*_context(G=32, W=300, cams=4))[0]
    rng = np.random.default_rng(3)
    c2w, focal = make_cameras(rng, 4, 200, 3.2, "sphere", 40.0)
    batch = Batch([dict(G=24, radii=(), env_h=0, env_w=0, c2w=c2w, focal=focal, width=200, height=200)] * 2)
    xb = cuda_tensor(np.concatenate([random_params(rng, 24, 0, 0, 0, 0.01, 0.2)] * 2))
    out, diag, rgb, y = empty(3 * ctx.n_rays), empty(xs[0].numel()), empty(3 * batch.n_rays), empty(4)
    other, graph = torch.cuda.Stream(), torch.cuda.CUDAGraph()
    torch.cuda.synchronize()
    with torch.cuda.graph(graph):
        y.add_(1.0)
        ctx.render(xs[0], out, stream=other)
        ctx.diag_jtj(xs[0], diag, stream=other)
        batch.render(xb, rgb, stream=other)
        y.add_(1.0)
    torch.cuda.synchronize()
    assert torch.equal(out, want) and float(diag.sum()) > 0 and float(rgb.sum()) > 0
    graph.replay()
    torch.cuda.synchronize()
    assert y.tolist() == [2.0] * 4


def test_growing_the_workspace_does_not_wait_for_marches_in_flight():
    """The diagonal needs more of the workspace than the renders before it; the
    call returns while they run (calls are asynchronous)."""
    import torch
    ctx, xs = _context()
    out, diag = empty(3 * ctx.n_rays), empty(xs[0].numel())
    _context()[0].diag_jtj(xs[0], diag)   # its kernels loaded: a first launch may wait for that
    torch.cuda.synchronize()
    ctx.render(xs[0], out)
    torch.cuda.synchronize()
    for _ in range(300):
        ctx.render(xs[0], out)
    done = torch.cuda.Event()
    done.record()
    ctx.diag_jtj(xs[0], diag)
    early = not done.query()
    torch.cuda.synchronize()
    assert early
    again = empty(xs[0].numel())
    ctx.diag_jtj(xs[0], again)
    ap, jp = empty(xs[0].numel()), empty(3 * ctx.n_rays)
    ctx.apply_normal(xs[0], xs[0], ap)
    ctx.jvp(xs[0], xs[0], jp)
    torch.cuda.synchronize()
    # the same sums in another order of their binary32 additions
    assert float((again - diag).norm() / diag.norm()) < 1e-5
    dot = float((xs[0].double() * ap.double()).sum())
    assert abs(dot - float(jp.double().square().sum())) < 1e-5 * dot
