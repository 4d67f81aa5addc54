"""Folded launches of one to four waves of tiles, whose sums pass through a scratch of the context:
overlapping calls on two streams and from two threads do not disturb one another, and a captured
call replays after later, larger calls have replaced that scratch."""
import threading

import pytest

import workloads
from oracle.events import make_event, make_proposal
from gpu_common import m, torch, gpu_context, set_metric  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def wide(m, torch):  # noqa: F811
    w = workloads.scaled(workloads.bns_population(n_events=1), f_hi=148.0)  # 16,385 bins: three parts
    ev, th, _ = make_event(w, w.events[0])
    prop = make_proposal(ev, w, th)
    ctx = gpu_context(m, ev, w, w.events[0], th, m.MIXED)
    set_metric(m, ctx, prop)
    wave = torch.cuda.get_device_properties(0).multi_processor_count * 7 * 128

    def draw(seed, n):
        theta = torch.empty((len(prop["ids"]), n), dtype=torch.float64, device="cuda")
        m.mbis_draw(ctx, seed, 0, n, theta)
        # pieces of less than a wave, one after another
        want = torch.empty(n, dtype=torch.float64, device="cuda")
        for i in range(0, n, 100_000):
            part = torch.empty(min(100_000, n - i), dtype=torch.float64, device="cuda")
            m.mbis_loglike(ctx, len(part), theta[:, i:i + len(part)].contiguous(), part)
            want[i:i + len(part)] = part
        torch.cuda.synchronize()
        return n, theta, want, torch.empty_like(want)

    yield ctx, draw, wave
    m.mbis_destroy(ctx)


def test_two_streams(m, torch, wide):  # noqa: F811
    ctx, draw, wave = wide
    calls = [draw(1, wave + 1), draw(2, 2 * wave - 5), draw(3, wave + 77), draw(4, 3 * wave)]
    streams = [torch.cuda.Stream(), torch.cuda.Stream()]
    for rep in range(3):  # the second call grows the scratch under the first
        for i, (n, theta, _, out) in enumerate(calls):
            m.mbis_loglike(ctx, n, theta, out, streams[i % 2])
        torch.cuda.synchronize()
        for n, _, want, out in calls:
            assert torch.equal(out, want), (rep, n)
            out.zero_()
        torch.cuda.synchronize()


def test_two_threads(m, torch, wide):  # noqa: F811
    ctx, draw, wave = wide
    calls = [draw(5, wave + 300), draw(6, 2 * wave + 1)]
    streams = [torch.cuda.Stream(), torch.cuda.Stream()]

    def work(i):
        n, theta, _, out = calls[i]
        for _ in range(5):
            m.mbis_loglike(ctx, n, theta, out, streams[i])

    threads = [threading.Thread(target=work, args=(i,)) for i in range(2)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    torch.cuda.synchronize()
    for n, _, want, out in calls:
        assert torch.equal(out, want), n


def test_captured_call_outlives_the_scratch(m, torch, wide):  # noqa: F811
    ctx, draw, wave = wide
    n, theta, want, out = draw(7, wave + 9)
    m.mbis_loglike(ctx, n, theta, out)  # the scratch holds such a call
    torch.cuda.synchronize()
    graph, side = torch.cuda.CUDAGraph(), torch.cuda.Stream()
    with torch.cuda.graph(graph, stream=side):
        m.mbis_loglike(ctx, n, theta, out, side)
    n2, theta2, want2, out2 = draw(8, 3 * wave + 1000)
    m.mbis_loglike(ctx, n2, theta2, out2)
    out.zero_()
    graph.replay()
    torch.cuda.synchronize()
    assert torch.equal(out, want) and torch.equal(out2, want2)
