"""The FP32 beam former on the tensor cores (error-free slices) at the edges of its tiles.

Error bound, elementwise: a weight component is off by at most 2^-24 (its FP32 sincos) plus the phase
rounding (4e-9 cycle, 3e-8 rad); a sample component by 2^-24 of its column's peak (the second slice's
rounding) and, through the FP16-rounded weight of that slice, by 2^-12 x 2^-11 of the peak.  Summed
over the real and imaginary parts of S stations that is below 8e-7 x S x the column's largest |Y|
(worst case, all errors aligned), and the FP32 additions and the scaling add 2^-23 of the result.
"""

import numpy as np
import pytest

from oracle import lbf_oracle as O
from synth import generate as G

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

N = 256


@pytest.fixture(scope="module")
def dev():
    from paper_1105_0661_gb300 import build_lib
    build_lib.build()
    assert torch.cuda.is_available(), "GPU tests need CUDA"
    torch.cuda.set_device(0)
    return torch.device("cuda:0")


def _wl(S, B, M, Q, out, seed=0):
    rng = np.random.default_rng(seed)
    return G.Workload("split", G.lofar_positions(rng, S // 2, S - S // 2), G.subband_centres(1, 120e6),
                      G.hex_beam_grid(B, 0.05), (0.3, 0.4), M * N, Q, out)


def _ct(shape, seed, spread=0.0):
    """Complex normal samples, the stations' gains spread over `spread` decades."""
    rng = np.random.default_rng(seed)
    x = rng.standard_normal(shape) + 1j * rng.standard_normal(shape)
    gain = 10.0 ** (spread * rng.random(shape[2]))
    return (x * gain[None, None, :, None, None]).astype(np.complex64)


def _run(wl, ct, dev, **over):
    from paper_1105_0661_gb300 import Plan
    p = Plan.from_workload(wl, **over)
    d = torch.from_numpy(ct).to(dev)
    if wl.output == "V":
        o = torch.empty(p.shape("vol"), dtype=torch.complex64, device=dev)
        p.beamform(d, o)
    else:
        o = torch.empty(p.shape("stokes"), dtype=torch.float32, device=dev)
        p.beamform_stokes(d, o)
    assert p.device_status() == 0
    p.close()
    return o.cpu().numpy()


# stations at the edges of the 16-station steps and of Kpad; beams of one and several 64-beam items,
# partly filled lane quadrants; spectra around the 64-spectrum tile, odd (8-byte loads) and spans of
# several tiles
SHAPES = [(1, 40, 64), (8, 33, 1), (9, 64, 63), (24, 65, 65), (37, 127, 130), (48, 133, 255), (64, 50, 320)]


@pytest.mark.parametrize("S,B,M", SHAPES)
@pytest.mark.parametrize("spread", [0.0, 3.0])
def test_voltages_within_the_bound(dev, S, B, M, spread):
    wl = _wl(S, B, M, 1, "V")
    ct = _ct((1, N, S, 2, M), 1, spread)
    got = _run(wl, ct, dev, bf_variant="many").astype(np.complex128)
    ref = O.observation_from_workload(wl).beamform(ct.astype(np.complex128))
    peak = np.abs(ct.astype(np.complex128)).max(axis=2)[None]                  # [1][F][N][P][M]
    assert np.all(np.abs(got - ref) <= 8e-7 * S * peak + 2.0 ** -22 * np.abs(ref))


@pytest.mark.parametrize("out", ["I", "IQUV"])
@pytest.mark.parametrize("Q", [1, 2, 4, 8, 16, 32])
@pytest.mark.parametrize("S,B,M", [(24, 65, 32), (48, 37, 160), (16, 40, 352)])
def test_stokes_match_the_oracle(dev, S, B, M, Q, out):
    """Every integration length, spectra that end inside a tile and inside an output flush."""
    wl = _wl(S, B, M, Q, out)
    ct = _ct((1, N, S, 2, M), 2)
    got = _run(wl, ct, dev).astype(np.float64)
    ob = O.observation_from_workload(wl)
    ref = ob.stokes(ob.beamform(ct.astype(np.complex128)))
    # |dI| <= 2 |V| |dV| + |dV|^2 summed over pols and spectra, dV as above
    scale = (ref[:, :1] * Q) ** 0.5 * 2 * 2 * 8e-7 * S * np.abs(ct).max() + 4e-7 * ref[:, :1]
    assert np.all(np.abs(got - ref) <= scale)


@pytest.mark.parametrize("scale", [1e-30, 1e30])
def test_column_scales_cover_the_float_range(dev, scale):
    wl = _wl(24, 40, 64, 1, "V")
    ct = (_ct((1, N, 24, 2, 64), 3) * np.float32(scale)).astype(np.complex64)
    got = _run(wl, ct, dev).astype(np.complex128)
    ref = O.observation_from_workload(wl).beamform(ct.astype(np.complex128))
    assert np.all(np.abs(got - ref) <= 8e-7 * 24 * np.abs(ct).max() + 2.0 ** -22 * np.abs(ref))


@pytest.mark.parametrize("out,Q", [("V", 1), ("I", 1), ("IQUV", 16)])
def test_infinities_and_nans_stay_in_their_columns(dev, out, Q):
    """As the FP32 FMA kernel gives them: the same finite, infinite and NaN outputs."""
    S, M = 16, 96
    ct = _ct((1, N, S, 2, M), 4)
    ct[0, 3, 5, 0, 7] = np.inf
    ct[0, 9, 2, 1, 70] = complex(1.0, -np.inf)
    ct[0, 20, 0, 0, 33] = np.nan
    wl = _wl(S, 8, M, Q, out)
    few = _run(wl, ct, dev, bf_variant="few")
    many = _run(wl, ct, dev, bf_variant="many")
    for part in (np.real, np.imag):
        a, b = part(few), part(many)
        assert np.array_equal(np.isnan(a), np.isnan(b)) and np.array_equal(np.isinf(a), np.isinf(b))
        ok = np.isfinite(a)
        assert np.abs(a[ok] - b[ok]).max() <= 1e-4 * np.abs(a[ok]).max()


def test_incoherent_beam_beside_the_split_kernel(dev):
    wl = _wl(24, 40, 96, 8, "IQUV")
    ct = _ct((1, N, 24, 2, 96), 5)
    got = _run(wl, ct, dev, incoherent_beam=True).astype(np.float64)
    ob = O.observation_from_workload(wl, incoherent_beam=True)
    inc = ob.incoherent(ct.astype(np.complex128))
    assert np.all(np.abs(got[-1] - inc) <= 1e-5 * inc[:1])
    plain = _run(wl, ct, dev)
    assert np.array_equal(got[:-1].astype(np.float32), plain)
