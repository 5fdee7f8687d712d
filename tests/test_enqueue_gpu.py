"""Enqueueing a block of one long stream takes the host about as long as one of many short streams: the
cut of the streams into filter-bank spans is made with the plan."""

import time

import numpy as np
import pytest

from synth import generate as G

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

N = 256


def _enqueue_us(S, F, M):
    from paper_1105_0661_gb300 import Plan, build_lib
    build_lib.build()
    dev = torch.device("cuda:0")
    rng = np.random.default_rng(S)
    wl = G.Workload("enq", G.lofar_positions(rng, S // 2, S - S // 2), G.subband_centres(F, 120e6),
                    G.hex_beam_grid(1, 0.05), (0.3, 0.4), M * N, 1, "I")
    p = Plan.from_workload(wl)
    x = torch.zeros(p.shape("in"), dtype=torch.int16, device=dev)
    o = torch.empty(p.shape("stokes"), dtype=torch.float32, device=dev)
    best = 1e9
    for _ in range(40):
        torch.cuda.synchronize()
        t = time.perf_counter()
        p.run_block(x, o)
        best = min(best, time.perf_counter() - t)
    torch.cuda.synchronize()
    p.close()
    return best * 1e6


def test_long_stream_costs_the_host_no_more():
    many, one = _enqueue_us(64, 10, 16), _enqueue_us(1, 1, 38912)   # 640 and 2432 tiles, three launches each
    print(f"enqueue: {many:.1f} us for 640 short streams, {one:.1f} us for one long")
    assert one <= many + 5.0
