"""Which FP32 beam former a plan runs, as its trace names it: the FMA kernel that bf_variant asks for,
and under AUTO the split tensor-core kernel except for few beams, more than 64 stations and small blocks
of few stations.  The same for the voltages call of a Stokes plan, and for tensor-core plans that
name the few-beam kernel."""

import numpy as np
import pytest

from synth import generate as G

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

N = 256


@pytest.mark.parametrize("variant,prec,S,B,M,out,stokes,volts", [
    ("few", "fp32", 24, 20, 64, "I", "bf_few", "bf_few"), ("many", "fp32", 24, 40, 64, "I", "bf_many", "bf_many"),
    ("many64", "fp32", 24, 40, 64, "IQUV", "bf_many64", "bf_many64"), ("few", "fp32", 48, 130, 64, "IQUV", "bf_few", "bf_few"),
    ("auto", "fp32", 24, 40, 64, "I", "bf_split", "bf_split"), ("auto", "fp32", 24, 8, 64, "I", "bf_few", "bf_few"),
    ("auto", "fp32", 32, 9, 64, "I", "bf_few", "bf_few"),
    ("auto", "fp32", 19, 40, 64, "I", "bf_split", "bf_many64"), ("auto", "fp32", 65, 40, 64, "I", "bf_many64", "bf_many64"),
    ("auto", "fp32", 65, 127, 64, "I", "bf_many", "bf_many"), ("few", "fp16tc", 24, 40, 64, "I", "bf_few", "bf_few")])
def test_kernel_that_runs(variant, prec, S, B, M, out, stokes, volts):
    from paper_1105_0661_gb300 import Plan, build_lib
    build_lib.build()
    dev = torch.device("cuda:0")
    rng = np.random.default_rng(S)
    wl = G.Workload("disp", G.lofar_positions(rng, S // 2, S - S // 2), G.subband_centres(1, 120e6),
                    G.hex_beam_grid(B, 0.05), (0.3, 0.4), M * N, 4, out)
    p = Plan.from_workload(wl, bf_variant=variant, precision=prec)
    ct = torch.zeros(p.shape("ct"), dtype=torch.complex64, device=dev)
    o = torch.empty(p.shape("stokes"), dtype=torch.float32, device=dev)
    v = torch.empty(p.shape("vol"), dtype=torch.complex64, device=dev)
    for call, dst, kernel in ((p.beamform_stokes, o, stokes), (p.beamform, v, volts)):
        p.trace_begin()
        call(ct, dst)
        assert [k for k in p.trace_end() if k.startswith("bf_")] == [kernel]
    p.trace_begin()
    p.run_block(torch.zeros(p.shape("in"), dtype=torch.int16, device=dev), o)
    assert stokes in p.trace_end()
    assert p.device_status() == 0
    p.close()


def test_empty_block_beside_others_in_a_batch():
    """A plan of no spectra takes no kernel (its cost is not asked for), alone or in a batch."""
    from paper_1105_0661_gb300 import Batch, Plan, build_lib
    build_lib.build()
    dev = torch.device("cuda:0")
    rng = np.random.default_rng(1)
    plans = [Plan.from_workload(G.Workload("empty", G.lofar_positions(rng, 12, 12), G.subband_centres(1, 120e6),
                                           G.hex_beam_grid(40, 0.05), (0.3, 0.4), M * N, 1, "I")) for M in (0, 64)]
    x = [torch.zeros(max(1, p.dims.in_bytes // 2), dtype=torch.int16, device=dev) for p in plans]
    o = [torch.ones(max(1, p.dims.out_bytes // 4), dtype=torch.float32, device=dev) for p in plans]
    b = Batch(plans)
    b.run(x, o)
    torch.cuda.synchronize()
    assert o[0].item() == 1.0 and torch.count_nonzero(o[1]).item() == 0
    plans[0].trace_begin()
    plans[0].run_block(x[0], o[0])
    assert [k for k in plans[0].trace_end() if not k.startswith("_")] == []
    b.close()
    for p in plans:
        p.close()
