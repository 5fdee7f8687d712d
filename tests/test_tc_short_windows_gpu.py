"""Tensor-core beam former with short integration windows (1, 2 and 4 spectra), whose rows go through
shared memory: partly filled beam blocks, spectra that end inside a tile and rows that are not 16-byte
aligned, against the oracle at the bars of the precision (three products: 1e-3 of I per element; two:
1e-3 of I's RMS per beam)."""

import numpy as np
import pytest

from oracle import lbf_oracle as O
from synth import generate as G

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

N = 256


@pytest.mark.parametrize("prec", ["fp16tc", "fp16tc2"])
@pytest.mark.parametrize("out", ["I", "IQUV"])
@pytest.mark.parametrize("Q", [1, 2, 4])
@pytest.mark.parametrize("S,B,M", [(24, 70, 96), (40, 133, 68), (9, 9, 140)])
def test_short_windows_match_the_oracle(S, B, M, Q, out, prec):
    from paper_1105_0661_gb300 import Plan, build_lib
    build_lib.build()
    dev = torch.device("cuda:0")
    rng = np.random.default_rng(S)
    wl = G.Workload("short", G.lofar_positions(rng, S // 2, S - S // 2), G.subband_centres(1, 120e6),
                    G.hex_beam_grid(B, 0.05), (0.3, 0.4), M * N, Q, out, sample_bits=8, sigma=8.0)
    if Q == 1:
        M -= 1                                   # odd rows
        wl.block_samples = M * N
    blk = G.make_block(wl, seed=3)
    p = Plan.from_workload(wl, precision=prec)
    assert p.dims.bf_kernel == 3
    o = torch.full(p.shape("stokes"), float("nan"), dtype=torch.float32, device=dev)
    p.run_block(torch.from_numpy(blk).to(dev), o)
    assert p.device_status() == 0
    got = o.cpu().numpy().astype(np.float64)
    ref = O.observation_from_workload(wl).run_block(blk)
    err = np.abs(got - ref)
    if prec == "fp16tc":
        # an element that the stations nearly cancel in is measured against its beam's mean
        bar = 1e-3 * np.maximum(ref[:, :1], ref[:, :1].mean(axis=(2, 3, 4), keepdims=True))
        assert np.all(err <= bar)
    else:
        rms = np.sqrt((err ** 2).mean(axis=(2, 3, 4)))
        assert np.all(rms <= 1e-3 * np.sqrt((ref[:, :1] ** 2).mean(axis=(2, 3, 4))))
    p.close()
