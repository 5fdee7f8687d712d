"""The FP32 beam former on the tensor cores is no further from the 64-bit result than FP32 FMAs are,
for stations of equal and of very different level.

The bar is the few-beam FMA kernel itself on the same block and the same first eight beams (both take
their weights from the same 32-bit phases; what differs there is the rounding of the FP32 sine and
cosine, for which the ratio of the two RMS errors gets 5 %).  Of the slice products, leaving out any
one costs far more: W3 Y1, the smallest that matters for equal stations, quadruples the error."""

import numpy as np
import pytest

from oracle import lbf_oracle as O
from synth import generate as G

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

N = 256


def _rms(S, M, gain, scale=1.0, F=1):
    """RMS errors of the two kernels over 8 beams, relative to the RMS voltage."""
    from paper_1105_0661_gb300 import Plan, build_lib
    build_lib.build()
    dev = torch.device("cuda:0")
    rng = np.random.default_rng(S)
    xyz = G.lofar_positions(rng, S // 2, S - S // 2)
    shape = (F, N, S, 2, M)
    ct = ((rng.standard_normal(shape) + 1j * rng.standard_normal(shape)) * gain[None, None, :, None, None]).astype(np.complex64)
    ct *= np.float32(scale)
    x = torch.from_numpy(ct).to(dev)
    err = []
    for B in (40, 8):
        wl = G.Workload("prec", xyz, G.subband_centres(F, 120e6), G.hex_beam_grid(40, 0.05)[:B], (0.3, 0.4), M * N, 1, "V")
        p = Plan.from_workload(wl)
        o = torch.empty(p.shape("vol"), dtype=torch.complex64, device=dev)
        p.trace_begin()
        p.beamform(x, o)
        assert ("bf_split" if B == 40 else "bf_few") in p.trace_end()
        assert p.device_status() == 0
        got = o.cpu().numpy()[:8].astype(np.complex128)
        if B == 40:
            ref = O.observation_from_workload(wl).beamform(ct.astype(np.complex128))[:8]
        err.append(float(np.sqrt(np.mean(np.abs(got - ref) ** 2) / np.mean(np.abs(ref) ** 2))))
        p.close()
    return err


GAINS = {"equal": lambda S: np.ones(S), "first_30": lambda S: np.where(np.arange(S) == 0, 30.0, 1.0),
         "last_30": lambda S: np.where(np.arange(S) == S - 1, 30.0, 1.0),
         "last_1000": lambda S: np.where(np.arange(S) == S - 1, 1000.0, 1.0),
         "three_decades": lambda S: 10.0 ** (3.0 * np.random.default_rng(7).random(S))}


@pytest.mark.parametrize("gain", list(GAINS))
@pytest.mark.parametrize("S,M,F", [(9, 512, 4), (12, 512, 2), (16, 320, 1), (24, 255, 1), (48, 256, 1), (64, 258, 1)])
def test_no_further_from_64_bits_than_fp32_fmas(S, M, F, gain):
    split, fma = _rms(S, M, GAINS[gain](S), F=F)
    print(f"{S} stations, {gain}: split {split:.3e}, FMAs {fma:.3e}")
    assert split <= 1.05 * fma


@pytest.mark.parametrize("scale", [1e-36, 1e-39])
def test_small_and_denormal_columns(scale):
    """Samples down to denormal numbers, too small for the power of two that scales a column."""
    split, fma = _rms(24, 256, np.ones(24), scale)
    print(f"scale {scale}: split {split:.3e}, FMAs {fma:.3e}")
    assert split <= 1.05 * fma
