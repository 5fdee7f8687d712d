"""Small blocks, whose filter bank and few-beam kernel start behind one another's tails: blocks queued
back to back, each into its own output, equal blocks that are waited for, for every output kind, also
with the input of each block written by a copy queued directly before it."""

import numpy as np
import pytest

from synth import generate as G

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

N = 256


@pytest.mark.parametrize("S,B,M,out,bits,inc", [(8, 4, 256, "IQUV", 16, False), (3, 1, 16, "V", 8, False),
                                                (8, 8, 64, "I", 16, True), (16, 3, 128, "IQUV", 8, True)])
def test_queued_blocks_equal_waited_blocks(S, B, M, out, bits, inc):
    from paper_1105_0661_gb300 import Plan, build_lib
    build_lib.build()
    dev = torch.device("cuda:0")
    rng = np.random.default_rng(S)
    wl = G.Workload("dep", G.lofar_positions(rng, S // 2, S - S // 2), G.subband_centres(1, 120e6),
                    G.hex_beam_grid(B, 0.05), (0.3, 0.4), M * N, 1 if out == "V" else 4, out, sample_bits=bits)
    n = 24
    xs = [torch.from_numpy(G.make_block(wl, seed=3, block_index=k)).to(dev) for k in range(n)]
    p = Plan.from_workload(wl, incoherent_beam=inc)
    which, dtype = ("vol", torch.complex64) if out == "V" else ("stokes", torch.float32)
    outs = [[torch.zeros(p.shape(which), dtype=dtype, device=dev) for _ in range(n)] for _ in range(3)]
    staged = torch.empty_like(xs[0])
    for mode in range(3):                             # waited for; queued; queued behind a copy each
        p.reset_state()
        for x, o in zip(xs, outs[mode]):
            if mode == 2:
                staged.copy_(x)
                x = staged
            p.run_block(x, o)
            if mode == 0:
                torch.cuda.synchronize()
        torch.cuda.synchronize()
    for a, b, c in zip(*outs):
        assert torch.equal(a, b) and torch.equal(a, c)
    assert p.device_status() == 0
    p.close()
