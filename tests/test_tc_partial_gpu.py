"""Tensor-core beam former with lane quadrants and whole M tiles without beams, which are not drained: a
plan of few beams gives bit for bit the first beams of a plan of 128, over several items per CTA, for
rows that can be stored 16 bytes wide and odd ones."""

import numpy as np
import pytest

from synth import generate as G

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

N = 256


@pytest.mark.parametrize("prec", ["fp16tc", "fp16tc2"])
@pytest.mark.parametrize("M,Q,out", [(68, 4, "I"), (68, 4, "IQUV"), (128, 4, "IQUV"), (66, 2, "I"), (66, 2, "IQUV"), (65, 1, "IQUV"),
                                     (64, 1, "I"), (72, 8, "IQUV"), (160, 32, "I"), (65, 1, "V"), (128, 1, "V")])
def test_few_beams_equal_the_first_of_many(M, Q, out, prec):
    from paper_1105_0661_gb300 import Plan, build_lib
    build_lib.build()
    dev = torch.device("cuda:0")
    S, F = 9, 2                                      # 512 items
    rng = np.random.default_rng(S)
    xyz = G.lofar_positions(rng, S // 2, S - S // 2)
    grid = G.hex_beam_grid(128, 0.05)
    which, dtype = ("vol", torch.complex64) if out == "V" else ("stokes", torch.float32)
    outs, x = {}, None
    for B in (128, 9, 16, 17, 33, 64, 65, 81):
        wl = G.Workload("part", xyz, G.subband_centres(F, 120e6), grid[:B], (0.3, 0.4), M * N, Q, out)
        if x is None:
            x = torch.from_numpy(G.make_block(wl, seed=8)).to(dev)
        p = Plan.from_workload(wl, precision=prec)
        assert p.dims.bf_kernel == 3
        o = outs[B] = torch.full(p.shape(which), float("nan"), dtype=dtype, device=dev)
        p.run_block(x, o)
        assert p.device_status() == 0
        p.close()
        assert torch.equal(o, outs[128][:B]), B
