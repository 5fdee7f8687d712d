"""The incoherent beam of a tensor-core Stokes I plan, summed inside the beam former: bit for bit the
separate kernel's (which a batch uses), and the oracle's to FP32 rounding of the hi+lo planes (2^-22
per component, twice that in power)."""

import numpy as np
import pytest

from oracle import lbf_oracle as O
from synth import generate as G

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

N = 256


@pytest.mark.parametrize("prec", ["fp16tc", "fp16tc2"])
@pytest.mark.parametrize("S,B,M,Q", [(20, 70, 65, 1), (48, 140, 96, 2), (9, 300, 64, 8), (64, 9, 160, 32), (33, 127, 200, 4)])
def test_incoherent_beam_in_the_beam_former(S, B, M, Q, prec):
    from paper_1105_0661_gb300 import Batch, Plan, build_lib
    build_lib.build()
    dev = torch.device("cuda:0")
    rng = np.random.default_rng(S)
    wl = G.Workload("inc", G.lofar_positions(rng, S // 2, S - S // 2), G.subband_centres(1, 120e6),
                    G.hex_beam_grid(B, 0.05), (0.3, 0.4), M * N, Q, "I", bandpass=G.bandpass_ripple(N))
    blk = G.make_block(wl, seed=6)
    x = torch.from_numpy(blk).to(dev)
    outs = []
    for batched in (False, True):
        p = Plan.from_workload(wl, precision=prec, incoherent_beam=True)
        o = torch.full(p.shape("stokes"), float("nan"), dtype=torch.float32, device=dev)
        if batched:
            b = Batch([p])
            b.run([x], [o])
        else:
            p.run_block(x, o)
        assert p.device_status() == 0
        outs.append(o)
        if batched:
            b.close()
        p.close()
    assert torch.equal(outs[0], outs[1])
    ob = O.observation_from_workload(wl, incoherent_beam=True)
    ref = ob.incoherent(ob.delay_correct(ob.ppf(blk)))
    got = outs[0][-1].cpu().numpy().astype(np.float64)
    assert np.all(np.abs(got - ref) <= 2e-6 * ref.max())
