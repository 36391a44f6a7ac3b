"""The streams an evaluation branches to: shared by the plans of one stream, closed with the last of them, and
safe where several host threads evaluate, on one stream or on their own."""
import ctypes
import threading

import pytest

pytestmark = pytest.mark.gpu


def _count():
    from paper_2402_08725_gb300 import _native
    return ctypes.CDLL(_native.load()._name)._ZN2sr19branch_stream_countEv()


def _problem(k, stream=None):
    from paper_2402_08725_gb300 import synthetic as syn
    from paper_2402_08725_gb300.binding import Problem
    fd = syn.small_deconv(seed=900 + k, E=4, N=32, f=2, K=21, M=2, J=4, lam=1.0)
    p = Problem.from_field(fd, conv_mode="fft" if k % 2 else "direct", stream=stream)
    p.set_lambda_pts(0.5)
    return p, fd


def test_plans_of_one_stream_share_their_branches():
    import gc
    import torch
    gc.collect()
    before = _count()
    one, two = torch.cuda.Stream(), torch.cuda.Stream()
    probs = []
    for k in range(6):
        p, fd = _problem(k, one)
        with torch.cuda.stream(one):
            p.loss_and_grad(torch.from_numpy(fd.params).cuda())
        probs.append(p)
        if k == 3:
            first = _count() - before
            assert 2 <= first <= 8  # two for each kind of branch of either form
    assert _count() - before == first
    p, fd = _problem(1, two)
    with torch.cuda.stream(two):
        p.loss_and_grad(torch.from_numpy(fd.params).cuda())
    assert first < _count() - before < 2 * first  # a first evaluation opens one of each
    for q in probs + [p]:
        q.close()
    assert _count() == before


@pytest.mark.parametrize("shared", [True, False])
def test_threads_on_one_stream_and_on_their_own(shared):
    import torch
    common = torch.cuda.Stream()
    got, want = {}, {}
    for k in range(4):
        p, fd = _problem(k)
        loss, grad = p.loss_and_grad(torch.from_numpy(fd.params).cuda())
        want[k] = (loss, grad.clone())
        p.close()
    torch.cuda.synchronize()

    def work(k):
        stream = common if shared else torch.cuda.Stream()
        p, fd = _problem(k, stream)
        with torch.cuda.stream(stream):
            P = torch.from_numpy(fd.params).cuda()
            for _ in range(20):
                loss, grad = p.loss_and_grad(P)
            stream.synchronize()
            got[k] = (loss, grad.clone())
            stream.synchronize()
        p.close()

    threads = [threading.Thread(target=work, args=(k,)) for k in range(4)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    for k in range(4):
        assert got[k][0] == want[k][0] and torch.equal(got[k][1], want[k][1])


def test_a_callers_capture_takes_the_branches_along():
    """An evaluation recorded in the caller's own graph, with another plan of the stream alive, replays to the
    same bits on new parameters."""
    import torch
    stream = torch.cuda.Stream()
    other, fo = _problem(0, stream)
    p, fd = _problem(1, stream)
    with torch.cuda.stream(stream):
        other.loss_and_grad(torch.from_numpy(fo.params).cuda())
        P = torch.from_numpy(fd.params).cuda()
        grad = torch.empty_like(P)
        p.loss_and_grad(P, grad, sync=False)  # the plan is built before the capture
        stream.synchronize()
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph, stream=stream):
            loss, _ = p.loss_and_grad(P, grad, sync=False)
        for scale in (1.0, 1.25):
            P.mul_(scale)
            graph.replay()
            stream.synchronize()
            got = (float(loss), grad.clone())
            want = p.loss_and_grad(P, torch.empty_like(P))
            assert got[0] == float(want[0]) and torch.equal(got[1], want[1])
            other.loss_and_grad(torch.from_numpy(fo.params).cuda())
    p.close()
    other.close()
