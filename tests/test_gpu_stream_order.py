"""Layer calls are ordered on the caller's stream like any other work: inputs refilled on the stream
right after a call and outputs copied on the stream right behind it, with no synchronisation anywhere,
eagerly and as a captured graph.  One input buffer serves all layers, so a kernel that starts before
its inputs are there, or still reads when they are overwritten, shows in the results."""
import pytest
import torch

from paper_2609_07306_b200 import workload as W
from paper_2609_07306_b200.ledger import BucketSet, RouteLedger, config_from_workload, device_tensor

pytestmark = pytest.mark.gpu

NAMES = ("routes", "sentinels", "ages", "kth_score", "margin", "flags", "refresh_count")
CASES = {
    "bf16": (W.sweep(512, 0.15).replace(heads=8, chunk_tokens=16), {}),
    "bf16_wide": (W.sweep(512, 0.15).replace(heads=8, k=48, m=24), {}),
    "bf16_streaming": (W.sweep(256, 0.15).replace(heads=8), dict(streaming=True)),
    "bf16_two_pass": (W.sweep(256, 0.15).replace(heads=4), dict(two_pass=True)),
    "fp32": (W.tiny().replace(heads=12, n_q=300, n_k=256, rho=0.15), {}),
}
LAYERS = 7
ANCHORS = [l in (0, 1, 4) for l in range(LAYERS)]        # an anchor after an anchor, after relays, at the start


def _inputs(w):
    q, k = W.generate(w, layers=LAYERS)
    return [(device_tensor(q[l]), device_tensor(k[l])) for l in range(LAYERS)]


def _snapshot(ledgers):
    return [{n: getattr(led, n).clone() for n in NAMES} for led in ledgers]


def _run(call, ledgers, inputs, buf):
    """All layers through one pair of buffers; what each layer left behind."""
    out = []
    for l, (q, k) in enumerate(inputs):
        if buf is None:
            call(q, k, l, ANCHORS[l])
            torch.cuda.synchronize()
        else:
            buf[0].copy_(q); buf[1].copy_(k)
            call(buf[0], buf[1], l, ANCHORS[l])
        out.append(_snapshot(ledgers))
        if buf is not None:
            buf[0].fill_(float("nan")); buf[1].fill_(float("nan"))
    return out


def _check(make, inputs):
    call, ledgers, reset, close = make()
    want = _run(call, ledgers, inputs, None)
    buf = tuple(torch.empty_like(x) for x in inputs[0])
    stream = torch.cuda.Stream()
    for _ in range(3):                                   # (a race need not show at once)
        with torch.cuda.stream(stream):
            reset()
            got = _run(call, ledgers, inputs, buf)
        torch.cuda.synchronize()
        _equal(got, want)
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.stream(stream):
        reset()
        with torch.cuda.graph(graph, stream=stream):
            got = _run(call, ledgers, inputs, buf)
    torch.cuda.synchronize()
    for _ in range(2):
        with torch.cuda.stream(stream):
            reset()
            graph.replay()
        torch.cuda.synchronize()
        _equal(got, want)
    assert all(led.status() == 0 for led in ledgers)
    del graph
    close()


def _equal(got, want):
    for l, (a, b) in enumerate(zip(got, want)):
        for x, y in zip(a, b):
            for n in NAMES:
                assert torch.equal(x[n], y[n]), (l, n)


@pytest.mark.parametrize("case", sorted(CASES))
def test_ledger_calls_on_a_stream(case):
    w, kw = CASES[case]

    def make():
        led = RouteLedger(config_from_workload(w, **kw))
        return (lambda q, k, l, a: (led.route_anchor if a else led.route_relay)(q, k, l)), [led], led.reset, led.close
    _check(make, _inputs(w))


def test_bucket_calls_on_a_stream():
    w = W.sweep(512, 0.15).replace(heads=9)

    def make():
        bs = BucketSet(config_from_workload(w), [(8, 16, 32)[p % 3] for p in range(9)])
        return bs.route_layer, bs.buckets, bs.reset, bs.close
    _check(make, _inputs(w))
