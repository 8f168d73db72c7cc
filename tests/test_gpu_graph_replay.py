"""Captured calls replayed between eager ones of other kernels and sizes on the same stream (GPU)."""
import pytest
import torch

from paper_2403_10444_b200 import workloads as wl

pytestmark = pytest.mark.gpu


# (entry point, B, gamma, V, kernel): the phase kernel and, with diagnostics, the flow kernel on one shape; a larger flow call; a
# few sequences; unaligned rows
CALLS = [("bv_verify", 128, 8, 65536, 5), ("bv_verify_ex", 320, 8, 65536, 1), ("bv_verify", 320, 8, 65536, 5), ("tv_verify", 320, 8, 65536, 1),
         ("bv_verify", 4, 4, 32768, 4), ("bv_verify", 200, 2, 5089, 5)]


@pytest.mark.parametrize("warm", [True, False])
def test_replays_between_eager_calls(warm):
    import paper_2403_10444_b200 as bv
    inputs = []
    for i, (fn, B, gamma, V, kernel) in enumerate(CALLS):
        inp = wl.make_inputs(wl.Workload("g", B, gamma, V, "bf16", 0.9, 40 + i, 2.0, 0.0, 0, 0.0, 0.5), "cuda:0")
        inputs.append([inp[k] for k in ("target_logits", "draft_logits", "draft_tokens", "uniforms")] + [inp["temperature"]])
    torch.cuda.synchronize()
    want = []
    for c, a in zip(CALLS, inputs):                       # (on torch's own stream: another workspace)
        want.append(getattr(bv, c[0])(*a)[:2])
        assert bv.bv_last_kernel() == c[4], c
    side = torch.cuda.Stream()
    side.wait_stream(torch.cuda.current_stream())
    with torch.cuda.stream(side):
        def eager(i):
            got = getattr(bv, CALLS[i][0])(*inputs[i])[:2]
            assert bv.bv_stream_status() == 0 and all(torch.equal(x, y) for x, y in zip(got, want[i])), CALLS[i]

        for i in range(len(CALLS)):
            if warm:
                eager(i)
            torch.cuda.synchronize()
            graph = torch.cuda.CUDAGraph()
            with torch.cuda.graph(graph, stream=side):
                out = getattr(bv, CALLS[i][0])(*inputs[i])[:2]
            assert bv.bv_last_kernel() == CALLS[i][4]
            for j in range(len(CALLS)):
                for _ in range(2):
                    for t in out:
                        t.fill_(-7)
                    graph.replay()
                    assert bv.bv_stream_status() == 0 and all(torch.equal(x, y) for x, y in zip(out, want[i])), (CALLS[i], CALLS[j])
                    eager(j)
            side.synchronize()
            del graph
