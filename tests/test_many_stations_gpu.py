"""More than 64 stations, where the FP32 FMA many-beam kernels are the only ones: every window length,
the incoherent beam they sum themselves, and their grouped form in a batch (both beam tiles), also for
plans of fewer stations that name them.

Bound: FP32 rounding of the weights and of 2 S accumulations, each at most 2^-24 of the sum of the
moduli, which stays below 8e-7 x S x peak as for the split kernel."""

import numpy as np
import pytest

from oracle import lbf_oracle as O
from synth import generate as G

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

N = 256


def _wl(S, B, M, Q, out, F=1):
    rng = np.random.default_rng(S)
    return G.Workload("stations", G.lofar_positions(rng, S // 2, S - S // 2), G.subband_centres(F, 120e6),
                      G.hex_beam_grid(B, 0.05), (0.3, 0.4), M * N, Q, out)


@pytest.mark.parametrize("S,B,M,Q,out,kernel", [(65, 70, 64, 2, "I", "bf_many"), (65, 127, 96, 4, "IQUV", "bf_many"),
                                                (113, 40, 64, 8, "I", "bf_many64"), (113, 127, 64, 16, "I", "bf_many"),
                                                (80, 40, 96, 32, "IQUV", "bf_many64"), (80, 127, 32, 32, "IQUV", "bf_many"),
                                                (72, 127, 41, 1, "I", "bf_many")])
@pytest.mark.parametrize("inc", [False, True])
def test_stokes_over_windows(S, B, M, Q, out, kernel, inc):
    from paper_1105_0661_gb300 import Plan, build_lib
    build_lib.build()
    dev = torch.device("cuda:0")
    wl = _wl(S, B, M, Q, out)
    rng = np.random.default_rng(1)
    shape = (1, N, S, 2, M)
    ct = (rng.standard_normal(shape) + 1j * rng.standard_normal(shape)).astype(np.complex64)
    p = Plan.from_workload(wl, incoherent_beam=inc)
    o = torch.full(p.shape("stokes"), float("nan"), dtype=torch.float32, device=dev)
    p.trace_begin()
    p.beamform_stokes(torch.from_numpy(ct).to(dev), o)
    assert kernel in p.trace_end()
    p.close()
    got = o.cpu().numpy().astype(np.float64)
    ob = O.observation_from_workload(wl, incoherent_beam=inc)
    ref = ob.stokes(ob.beamform(ct.astype(np.complex128)))[:B]
    dv = 8e-7 * S * np.abs(ct).max()
    assert np.all(np.abs(got[:B] - ref) <= 4 * dv * (ref[:, :1] * Q) ** 0.5 + 4e-7 * ref[:, :1])
    if inc:
        ri = ob.incoherent(ct.astype(np.complex128))
        assert np.all(np.abs(got[B] - ri) <= 1e-5 * ri[:1])


@pytest.mark.parametrize("out,inc", [("I", True), ("IQUV", False), ("V", False)])
def test_grouped_launches(out, inc):
    from paper_1105_0661_gb300 import Batch, Plan, build_lib
    build_lib.build()
    dev = torch.device("cuda:0")
    specs = [(66, 127, 48, "auto"), (70, 40, 32, "auto"), (20, 127, 64, "many"), (33, 70, 41 if out == "V" else 44, "many64")]
    wls = [_wl(S, B, M, 4 if out != "V" else 1, out) for S, B, M, _ in specs]
    solo = [Plan.from_workload(w, bf_variant=s[3], incoherent_beam=inc) for w, s in zip(wls, specs)]
    grouped = [Plan.from_workload(w, bf_variant=s[3], incoherent_beam=inc) for w, s in zip(wls, specs)]
    batch = Batch(grouped)
    so = [torch.zeros(p.dims.out_bytes // 4, dtype=torch.float32, device=dev) for p in solo]
    bo = [torch.ones_like(o) for o in so]
    for k in range(2):
        x = [torch.from_numpy(G.make_block(w, seed=i, block_index=k)).to(dev) for i, w in enumerate(wls)]
        for p, xi, o, kernel in zip(solo, x, so, ("bf_many", "bf_many64", "bf_many", "bf_many64")):
            p.trace_begin()
            p.run_block(xi, o)
            assert kernel in p.trace_end()
        batch.run(x, bo)
        torch.cuda.synchronize()
        for a, b in zip(so, bo):
            assert torch.equal(a, b)
    ref = O.observation_from_workload(wls[0], incoherent_beam=inc)
    if out == "I":                                   # the group's first observation against the oracle
        for k in range(2):
            r = ref.run_block(G.make_block(wls[0], seed=0, block_index=k))
        got = bo[0].cpu().numpy().astype(np.float64).reshape(r.shape)
        assert np.abs(got - r).max() <= 1e-5 * r.max()
    batch.close()
    for p in solo + grouped:
        p.close()
