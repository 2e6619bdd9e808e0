"""Calls on streams: a change of streams is ordered on the device, and calls can be captured on another stream than they ran on."""
import time

import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from gen import problems  # noqa: E402


def _outputs(hap, hp):
    out = hap.hap_pipeline_dp(hp, 0, hp.n_cand, partition=True)
    return {**out, "best": hap.hap_argmin(hp, out["cost"])}


@pytest.mark.parametrize("first,second", [("default", "side"), ("side", "default"), ("side", "other")])
def test_a_change_of_streams_waits_on_the_device_only(first, second):
    import paper_2609_39350_b200 as hap
    streams = {"default": torch.cuda.default_stream(), "side": torch.cuda.Stream(), "other": torch.cuda.Stream()}
    hp = hap.hap_problem_create(problems.small())
    hap.hap_enumerate(hp)
    want = _outputs(hap, hp)
    torch.cuda.synchronize()
    with torch.cuda.stream(streams[second]):
        scratch = torch.zeros(1, device="cuda")           # (the stream's first use, before the clock runs)
    with torch.cuda.stream(streams[first]):
        _outputs(hap, hp)
        torch.cuda.synchronize()
        torch.cuda._sleep(400_000_000)                    # 0.2 s
        done = torch.cuda.Event()
        a = _outputs(hap, hp)
        done.record()
    t0 = time.perf_counter()
    with torch.cuda.stream(streams[second]):
        b = _outputs(hap, hp)
    waited = time.perf_counter() - t0
    assert not done.query() and waited < 0.1, waited      # the host went on while the first stream was still asleep
    torch.cuda.synchronize()
    for k, v in want.items():
        assert torch.equal(a[k], v) and torch.equal(b[k], v), k
    del scratch
    hap.hap_problem_destroy(hp)


@pytest.mark.parametrize("warm", ["default", "side"])
def test_capture_on_another_stream_than_the_warm_up(warm):
    """Asynchronous calls only before the capture: nothing has waited for the upload or the calls on the host yet."""
    import paper_2609_39350_b200 as hap
    pb = problems.small()
    ref = hap.hap_problem_create(pb)
    hap.hap_enumerate(ref)
    want = _outputs(hap, ref)
    torch.cuda.synchronize()
    hp = hap.hap_problem_create(pb)
    hap.hap_enumerate(hp)
    out = dict(cost=torch.empty_like(want["cost"]), bottleneck=torch.empty_like(want["bottleneck"]),
               partition=torch.empty_like(want["partition"]), recompute=torch.empty_like(want["recompute"]))
    side = torch.cuda.default_stream() if warm == "default" else torch.cuda.Stream()
    side.wait_stream(torch.cuda.current_stream())
    with torch.cuda.stream(side):
        hap.hap_pipeline_dp(hp, 0, hp.n_cand, out=out)
    graph = torch.cuda.CUDAGraph()
    stream = torch.cuda.Stream()
    with torch.cuda.graph(graph, stream=stream):
        hap.hap_pipeline_dp(hp, 0, hp.n_cand, out=out)
    torch.cuda.synchronize()
    for v in out.values():
        v.zero_()
    for _ in range(3):
        graph.replay()
    torch.cuda.synchronize()
    for k, v in out.items():
        assert torch.equal(v, want[k]), k
    again = _outputs(hap, hp)                             # a call outside of the graph, behind it
    torch.cuda.synchronize()
    assert torch.equal(again["best"], want["best"])
    hap.hap_problem_destroy(hp)
    hap.hap_problem_destroy(ref)
