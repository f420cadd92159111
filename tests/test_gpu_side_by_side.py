"""Calls on several streams at once share the SMs: a launch that leaves most of an SM idle must not keep the others out (needs a B200)."""
import pytest
import torch

from paper_2501_00692_b200 import binding as B
from paper_2501_00692_b200 import synth
from paper_2501_00692_b200.build import build_library

pytestmark = pytest.mark.gpu
DEV = "cuda:0"
CALLS, STREAMS = 16, 4


def test_small_forwards_side_by_side():
    """1,024 x 64 fp32: 128 CTAs of four warps a launch.  On four streams at once a call takes 0.32 of the time that it takes alone; 0.48
    where the scan kernels keep others off their SMs.  Graphs, so that the host's part does not count."""
    build_library()
    w = synth.custom_workload("beside", 67, 1, 1024, 64, io="f32")
    theta = synth.layer_params(w, 0, DEV)
    x, _ = synth.activations(w, DEV)
    sh = B.shape_of(x)
    kept = []
    for _ in range(STREAMS):
        ws, y, s, graph = B.alloc_workspace(B.as_workspace_bytes(sh, 1024)[0], DEV), torch.empty_like(x), torch.cuda.Stream(), torch.cuda.CUDAGraph()
        B.as_ssm_forward(sh, theta, x, y, ws)
        torch.cuda.synchronize()
        with torch.cuda.graph(graph, stream=s):
            for _ in range(CALLS):
                B.as_ssm_forward(sh, theta, x, y, ws, stream=s)
        kept.append((graph, s, ws, y))

    def us_a_call(n):
        times = []
        for _ in range(20):
            main, t0, t1 = torch.cuda.current_stream(), torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            torch.cuda._sleep(200000)   # the replays are enqueued before the first begins
            t0.record(main)
            for graph, s, _, _ in kept[:n]:
                s.wait_stream(main)
                with torch.cuda.stream(s):
                    graph.replay()
            for _, s, _, _ in kept[:n]:
                main.wait_stream(s)
            t1.record(main)
            torch.cuda.synchronize()
            times.append(t0.elapsed_time(t1) * 1e3 / (CALLS * n))
        return sorted(times)[len(times) // 2]

    us_a_call(STREAMS)
    alone, beside = us_a_call(1), us_a_call(STREAMS)
    assert all(torch.equal(y, kept[0][3]) for _, _, _, y in kept)
    assert beside < 0.4 * alone, (alone, beside)
