"""Plans of different sizes launched from several host threads at once: the shared-memory limit of a
kernel is state of the whole process, so a launch must not depend on another thread's last setting.
The kernels are launched back to back by two threads each (the calls release the interpreter lock)."""

import threading

import numpy as np
import pytest

from synth import generate as G

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

N = 256


def _plan(S, B, variant, prec, M=64):
    from paper_1105_0661_gb300 import Plan
    rng = np.random.default_rng(S)
    wl = G.Workload("thr", G.lofar_positions(rng, S // 2, S - S // 2), G.subband_centres(1, 120e6),
                    G.hex_beam_grid(B, 0.05), (0.3, 0.4), M * N, 4, "I")
    return Plan.from_workload(wl, bf_variant=variant, precision=prec)


@pytest.mark.parametrize("variant,prec,B,sizes", [("auto", "fp32", 40, (16, 64)), ("few", "fp32", 4, (16, 800)),
                                                  ("many", "fp32", 5, (66, 110)), ("auto", "fp16tc", 40, (16, 64))])
def test_launches_of_two_sizes_from_two_threads(variant, prec, B, sizes):
    from paper_1105_0661_gb300 import build_lib
    build_lib.build()
    dev = torch.device("cuda:0")
    plans = [_plan(S, B, variant, prec) for S in sizes]
    ct = [torch.zeros(p.shape("ct"), dtype=torch.complex64, device=dev) for p in plans]
    out = [torch.empty(p.shape("stokes"), dtype=torch.float32, device=dev) for p in plans]
    streams = [torch.cuda.Stream() for _ in plans]
    torch.cuda.synchronize()
    errors = []
    start = threading.Barrier(len(plans))

    def work(i):
        try:
            torch.cuda.set_device(dev)
            start.wait()
            for _ in range(60):
                for _ in range(50):
                    plans[i].beamform_stokes(ct[i], out[i], stream=streams[i])
                streams[i].synchronize()
        except Exception as e:                       # reported by the main thread
            errors.append(e)

    threads = [threading.Thread(target=work, args=(i,)) for i in range(len(plans))]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    torch.cuda.synchronize()
    for p in plans:
        p.close()
    assert not errors, errors[0]
