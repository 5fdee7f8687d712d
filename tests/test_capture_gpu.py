"""run_block under stream capture, for a small block (whose kernels are programmatic dependent launches)
and a larger one: two blocks captured as one graph give what the same two blocks give launched one by
one, also when the graph is replayed, and blocks enqueued back to back without waiting equal blocks
that are waited for."""

import numpy as np
import pytest

from synth import generate as G

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

N = 256


@pytest.mark.parametrize("S,F,B,M,prec", [(8, 1, 4, 64, "fp32"), (8, 1, 4, 255, "fp32"), (24, 4, 40, 128, "fp32"),
                                          (16, 1, 20, 64, "fp16tc"), (3, 1, 2, 16, "fp32")])
def test_captured_blocks_equal_launched_blocks(S, F, B, M, prec):
    from paper_1105_0661_gb300 import Plan, build_lib
    build_lib.build()
    dev = torch.device("cuda:0")
    rng = np.random.default_rng(S)
    wl = G.Workload("cap", G.lofar_positions(rng, S // 2, S - S // 2), G.subband_centres(F, 120e6),
                    G.hex_beam_grid(B, 0.05), (0.3, 0.4), M * N, 1, "I")
    xs = [torch.from_numpy(G.make_block(wl, seed=2, block_index=k)).to(dev) for k in range(4)]

    def outs(p):
        return [torch.zeros(p.shape("stokes"), dtype=torch.float32, device=dev) for _ in range(4)]

    p = Plan.from_workload(wl, precision=prec)
    want = outs(p)
    for x, o in zip(xs, want):
        p.run_block(x, o)
        torch.cuda.synchronize()
    p.reset_state()
    queued = outs(p)
    for x, o in zip(xs, queued):                     # no waiting in between
        p.run_block(x, o)
    torch.cuda.synchronize()
    for a, b in zip(want, queued):
        assert torch.equal(a, b)
    # one graph of two blocks (the history's two buffers alternate), replayed for blocks 2 and 3
    p.reset_state()
    bufs = [torch.zeros_like(xs[0]) for _ in range(2)]
    got = [torch.zeros_like(want[0]) for _ in range(2)]
    side = torch.cuda.Stream()
    side.wait_stream(torch.cuda.current_stream())
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.stream(side):
        graph.capture_begin()
        for x, o in zip(bufs, got):
            p.run_block(x, o, stream=side)
        graph.capture_end()
    for half in range(2):
        for b, x in zip(bufs, xs[2 * half:]):
            b.copy_(x)
        torch.cuda.synchronize()
        graph.replay()
        torch.cuda.synchronize()
        for a, b in zip(want[2 * half:], got):
            assert torch.equal(a, b), half
    assert p.device_status() == 0
    p.close()
