"""The split beam former where its dispatch sends it at the edges of its tiles (the trace names it): the
single K step of few stations with mostly padded rows, blocks that end inside a tile, odd rows read 8
bytes at a time, one and several 64-beam items, every station count class of the converters, windows
of every length, infinities and NaN, and the incoherent beam beside it.

Bound for the voltages, with the samples held to 2^-33 of the column's peak and the FP32 weights to
2^-24 plus 4e-9 cycle of phase (9e-8 in all for each of the two components): 2e-7 x S x peak, and the
rounding of the result; Stokes follow from |dI| <= 2 |V| |dV| + |dV|^2 over pols and spectra."""

import numpy as np
import pytest

from oracle import lbf_oracle as O
from synth import generate as G

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

N = 256


def _wl(S, B, M, Q, out, F=1):
    rng = np.random.default_rng(S)
    return G.Workload("edges", G.lofar_positions(rng, S // 2, S - S // 2), G.subband_centres(F, 120e6),
                      G.hex_beam_grid(B, 0.05), (0.3, 0.4), M * N, Q, out)


def _ct(S, M, seed, F=1):
    rng = np.random.default_rng(seed)
    shape = (F, N, S, 2, M)
    return (rng.standard_normal(shape) + 1j * rng.standard_normal(shape)).astype(np.complex64)


def _run(wl, ct, kernel="bf_split", **over):
    from paper_1105_0661_gb300 import Plan, build_lib
    build_lib.build()
    dev = torch.device("cuda:0")
    p = Plan.from_workload(wl, **over)
    which, dtype = ("vol", torch.complex64) if wl.output == "V" else ("stokes", torch.float32)
    o = torch.full(p.shape(which), float("nan"), dtype=dtype, device=dev)
    p.trace_begin()
    (p.beamform if wl.output == "V" else p.beamform_stokes)(torch.from_numpy(ct).to(dev), o)
    assert kernel in p.trace_end()
    assert p.device_status() == 0
    p.close()
    return o.cpu().numpy()


@pytest.mark.parametrize("S,B,M,F", [(9, 60, 512, 4), (16, 40, 258, 2), (20, 40, 129, 4), (24, 129, 65, 2), (31, 40, 130, 1),
                                     (33, 40, 64, 1), (40, 33, 36, 1), (48, 133, 255, 1), (49, 40, 66, 1), (57, 40, 65, 1),
                                     (64, 50, 320, 1), (64, 64, 33, 1), (64, 64, 7, 4)])
def test_voltages(S, B, M, F):
    ct = _ct(S, M, 1, F)
    wl = _wl(S, B, M, 1, "V", F)
    ref = O.observation_from_workload(wl).beamform(ct.astype(np.complex128))
    peak = np.abs(ct).max(axis=2)[None].astype(np.float64)
    assert np.all(np.abs(_run(wl, ct) - ref) <= 2e-7 * S * peak + 2.0 ** -23 * np.abs(ref))


@pytest.mark.parametrize("S,B,M,Q,out,F", [
    (1, 40, 768, 32, "I", 4), (2, 64, 544, 16, "I", 4), (1, 40, 512, 2, "IQUV", 1), (3, 40, 514, 2, "IQUV", 2),
    (4, 32, 516, 4, "I", 4), (5, 40, 512, 32, "IQUV", 1), (5, 65, 512, 32, "I", 1), (7, 40, 520, 8, "IQUV", 1),
    (8, 32, 257, 1, "I", 2), (16, 40, 255, 1, "I", 1), (16, 24, 257, 1, "IQUV", 4), (48, 40, 66, 1, "IQUV", 4),
    (24, 129, 66, 2, "I", 2), (50, 40, 66, 2, "IQUV", 1), (56, 40, 68, 4, "IQUV", 1), (64, 40, 72, 8, "IQUV", 1),
    (64, 70, 160, 32, "I", 1), (64, 40, 63, 1, "IQUV", 1)])
def test_stokes(S, B, M, Q, out, F):
    ct = _ct(S, M, 2, F)
    wl = _wl(S, B, M, Q, out, F)
    ob = O.observation_from_workload(wl)
    ref = ob.stokes(ob.beamform(ct.astype(np.complex128)))
    dv = 2e-7 * S * np.abs(ct).max()
    assert np.all(np.abs(_run(wl, ct) - ref) <= 4 * dv * (ref[:, :1] * Q) ** 0.5 + 4e-7 * ref[:, :1])


@pytest.mark.parametrize("out,Q,M", [("V", 1, 96), ("I", 1, 96), ("IQUV", 16, 96), ("I", 4, 68)])
def test_infinities_and_nans_stay_in_their_columns(out, Q, M):
    """The same finite, infinite and NaN outputs as the FMA many-beam kernel's."""
    S = 24
    ct = _ct(S, M, 4)
    ct[0, 3, 5, 0, 7] = np.inf
    ct[0, 9, 2, 1, 66] = complex(1.0, -np.inf)
    ct[0, 20, 0, 0, 33] = np.nan
    wl = _wl(S, 40, M, Q, out)
    split, fma = _run(wl, ct), _run(wl, ct, kernel="bf_many64", bf_variant="many64")
    for part in (np.real, np.imag):
        a, b = part(fma), part(split)
        assert np.array_equal(np.isnan(a), np.isnan(b)) and np.array_equal(np.isinf(a), np.isinf(b))
        ok = np.isfinite(a)
        assert np.abs(a[ok] - b[ok]).max() <= 1e-5 * np.abs(a[ok]).max()


@pytest.mark.parametrize("out,Q", [("I", 1), ("I", 8), ("IQUV", 4)])
def test_incoherent_beam_beside_it(out, Q):
    ct = _ct(24, 128, 5)
    wl = _wl(24, 40, 128, Q, out)
    got = _run(wl, ct, incoherent_beam=True)
    inc = O.observation_from_workload(wl, incoherent_beam=True).incoherent(ct.astype(np.complex128))
    assert np.all(np.abs(got[-1] - inc) <= 1e-5 * inc[:1])
    assert np.array_equal(got[:-1], _run(wl, ct))
