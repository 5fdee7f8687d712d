"""Batch tuning times each set of kernels once: plans that the split beam former serves under every
variant add no candidates, plans that another variant would move to it add one."""

import numpy as np
import pytest

from synth import generate as G

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

N = 256


@pytest.mark.parametrize("S,B,variant,candidates", [(24, 40, "auto", 4), (24, 130, "auto", 4), (16, 12, "auto", 7),
                                                    (24, 40, "many64", 10), (66, 40, "auto", 10), (66, 130, "auto", 7),
                                                    (24, 4, "auto", 4)])
def test_candidates(S, B, variant, candidates):
    from paper_1105_0661_gb300 import Batch, Plan, build_lib
    build_lib.build()
    dev = torch.device("cuda:0")
    rng = np.random.default_rng(S)
    wl = G.Workload("tune", G.lofar_positions(rng, S // 2, S - S // 2), G.subband_centres(1, 120e6),
                    G.hex_beam_grid(B, 0.05), (0.3, 0.4), 64 * N, 4, "I")
    plans = [Plan.from_workload(wl, bf_variant=variant) for _ in range(2)]
    x = [torch.zeros(p.shape("in"), dtype=torch.int16, device=dev) for p in plans]
    o = [torch.empty(p.shape("stokes"), dtype=torch.float32, device=dev) for p in plans]
    b = Batch(plans)
    info = b.tune(x, o, reps=1)
    assert len(info["candidates"]) == candidates
    b.close()
    for p in plans:
        p.close()
