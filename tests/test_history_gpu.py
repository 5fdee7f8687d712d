"""The history between blocks in both forms of its update (inside the filter bank for a few tiles per
SM, a kernel of its own for more) and for blocks shorter than the history: consecutive short blocks give
the spectra of one long block, bit for bit."""

import numpy as np
import pytest

from synth import generate as G

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

N = 256


@pytest.mark.parametrize("bits", [16, 8])
@pytest.mark.parametrize("S,F,M", [(3, 1, 1), (8, 2, 20), (12, 60, 3), (12, 60, 18)])
def test_short_blocks_equal_one_long_block(S, F, M, bits):
    from paper_1105_0661_gb300 import Plan, build_lib
    build_lib.build()
    dev = torch.device("cuda:0")
    rng = np.random.default_rng(S)

    def wl(blocks):
        return G.Workload("hist", G.lofar_positions(np.random.default_rng(S), S // 2, S - S // 2),
                          G.subband_centres(F, 120e6), G.hex_beam_grid(1, 0.05), (0.3, 0.4), blocks * M * N, 1, "I",
                          sample_bits=bits)

    n = 20 // M + 2                                  # past 15 frames + d_max of history
    big = torch.from_numpy(rng.integers(-100, 100, (S, F, n * M * N, 2, 2)).astype(np.int16 if bits == 16 else np.int8))
    long, short = Plan.from_workload(wl(n)), Plan.from_workload(wl(1))
    whole = torch.empty(long.shape("chan"), dtype=torch.complex64, device=dev)
    long.ppf(big.to(dev), whole)
    part = torch.empty(short.shape("chan"), dtype=torch.complex64, device=dev)
    for k in range(n):
        short.ppf(big[:, :, k * M * N:(k + 1) * M * N].contiguous().to(dev), part)
        assert torch.equal(part, whole[:, :, :, k * M:(k + 1) * M]), k
    long.close()
    short.close()
