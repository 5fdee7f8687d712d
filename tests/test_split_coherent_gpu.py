"""Stations that add up in phase with every component near the column's peak: the leading slice product
of the split beam former reaches its largest sum and must still be exact.

All stations stand on one spot, so that every weight of a beam and channel is the same w, which the
column with a single unit sample returns.  The others hold components of 0.9 to 1 throughout; the
reference is w times their sum in 64 bits.  Bound: half a unit in the last place for V, and for the
small products' accumulator (below 2^16, where V is at least 2^23) 40 truncations of 2^-7: together
below one unit.  An accumulator that passes 2^24 truncates by up to a unit in each of its last steps."""

import numpy as np
import pytest

from synth import generate as G

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

N = 256


@pytest.mark.parametrize("S", [46, 48, 64])
def test_coherent_sums_are_exact_to_the_last_place(S):
    from paper_1105_0661_gb300 import Plan, build_lib
    build_lib.build()
    dev = torch.device("cuda:0")
    M, B = 256, 40
    rng = np.random.default_rng(S)
    xyz = np.tile(np.array([[31e3, -17e3, 0.0]]), (S, 1))
    wl = G.Workload("coh", xyz, G.subband_centres(1, 120e6), G.hex_beam_grid(B, 0.05), (0.3, 0.4), M * N, 1, "V")
    y = np.zeros((1, N, S, 2, M), dtype=np.complex64)
    y[..., 1:] = (rng.uniform(0.9, 1.0, (1, N, S, 2, M - 1)) + 1j * rng.uniform(0.9, 1.0, (1, N, S, 2, M - 1)))
    y[..., 0] = 0
    y[:, :, 0, :, 0] = 1
    p = Plan.from_workload(wl)
    o = torch.empty(p.shape("vol"), dtype=torch.complex64, device=dev)
    p.trace_begin()
    p.beamform(torch.from_numpy(y).to(dev), o)
    assert "bf_split" in p.trace_end()
    assert p.device_status() == 0
    p.close()
    v = o.cpu().numpy()                              # [B][F][N][P][M]
    w = v[..., :1].astype(np.complex128)
    ref = w * y.astype(np.complex128).sum(axis=2)[None]
    checked = 0
    for part in (np.real, np.imag):
        got, want = part(v)[..., 1:].astype(np.float64), part(ref)[..., 1:]
        big = np.abs(want) > 1.1 * S                 # both components of w count
        ulp = np.spacing(np.abs(want[big]).astype(np.float32)).astype(np.float64)
        assert np.max(np.abs(got[big] - want[big]) / ulp) <= 1.0
        checked += int(big.sum())
    assert checked > 10 ** 5
