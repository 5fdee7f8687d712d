"""The workloads this library's speed is measured on, each one pass through its public entry points.

A case is a plain dict; its "op" names the calls that a user's program makes:

  block         Plan.run_block: station samples to beams, the streaming call
  split         Plan.ppf, delay_correct, beamform, stokes: the same path step by step
  pulsar        Plan.run_block to beam voltages, dedisperse in place, stokes
  superstation  Plan.superstation on a corner-turned block, then beamform_stokes of the plan whose
                stations are the superstations
  batch         Batch.launch: a block of many small observations, replayed from its graph

The other keys are the observation: S stations, F subbands, B beams, M spectra per block (256
samples each), Q spectra per integration, sample width, output kind and precision.  Every plan
keeps its filter history between passes, as a stream does; the first pass starts from silence.
"""

from __future__ import annotations

import math

import numpy as np
import torch

from paper_1105_0661_gb300 import Batch, Plan

N, L = 256, 16                  # channels per subband, filter taps per channel
RATE = 195312.5                 # complex sample rate of a subband (Hz)
LIGHT = 299792458.0
CENTRE = (0.3, 0.4)             # direction cosines of the phase centre
K_DM = 4.148808e15              # dispersion constant, s Hz^2 per pc cm^-3
DM = 13.8


def listed():
    return [
        # One subband of a small station group, watched live: launches and latency are all there is.
        dict(name="tiny", op="block", S=8, F=1, B=4, M=256, Q=4, bits=16, output="I", precision="fp32", inc=False),
        # The survey observation: the whole station set and band, a tied-array beam per hexagon of a
        # six-ring grid, a second of data per block.  The largest case.
        dict(name="lofar", op="block", S=48, F=244, B=127, M=768, Q=16, bits=16, output="I", precision="fp32",
             inc=False),
        # A quarter of its band, as a streaming server's chunk plan holds it, on the tensor cores.
        dict(name="lofar_tc", op="block", S=48, F=61, B=127, M=768, Q=16, bits=16, output="I", precision="fp16tc",
             inc=False),
        # Full polarisation over a thousand beams from 8-bit stations: the contraction is everything.
        dict(name="beams1024_tc", op="block", S=48, F=30, B=1024, M=768, Q=16, bits=8, output="IQUV",
             precision="fp16tc", inc=False),
        # The cheaper two-product precision with a ragged beam count and short integrations.
        dict(name="beams300_tc2", op="block", S=40, F=24, B=300, M=384, Q=4, bits=8, output="IQUV",
             precision="fp16tc2", inc=False),
        # A handful of beams on known sources: the block streams through, little arithmetic per sample.
        dict(name="few_beams", op="block", S=48, F=61, B=8, M=768, Q=16, bits=16, output="I", precision="fp32",
             inc=False),
        # A ragged mid-size observation without integration: odd stations, beams and spectra.
        dict(name="ragged_iquv", op="block", S=37, F=29, B=29, M=255, Q=1, bits=8, output="IQUV", precision="fp32",
             inc=False),
        # A survey with the incoherent beam beside the tied-array ones.
        dict(name="incoherent_tc", op="block", S=48, F=30, B=127, M=768, Q=16, bits=16, output="I",
             precision="fp16tc", inc=True),
        # The pulsar mode: complex voltages at full rate, dedispersed, then detected.
        dict(name="pulsar", op="pulsar", S=48, F=16, B=127, M=768, Q=16, bits=16, precision="fp32", K=256),
        # The path step by step, for a program that keeps the intermediate products.
        dict(name="split", op="split", S=24, F=16, B=61, M=768, Q=4, bits=16, output="IQUV", precision="fp32"),
        # Core stations summed in pairs before a beam former with a modest grid.
        dict(name="superstation", op="superstation", S=48, G=24, F=24, B=37, M=768, Q=16, output="I",
             precision="fp32"),
        # Sixty-four small observations sharing the GPU, one graph launch per block.
        dict(name="batch_small", op="batch", n=64, M=64, layout=5),
    ]


def draw(rng):
    """A case of the same ranges, at most as costly as the survey observation."""
    def log_int(lo, hi):
        return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))

    op = rng.choice(["block", "block", "block", "block", "split", "pulsar", "superstation", "batch"])
    if op == "batch":
        return dict(op="batch", n=rng.randint(8, 64), M=rng.choice([16, 33, 64, 100, 128]),
                    layout=rng.randint(1, 10 ** 6))
    while True:
        S, F, B = rng.randint(8, 64), log_int(1, 244), log_int(1, 1024)
        Q = rng.choice([1, 2, 4, 4, 8, 16, 16, 32])
        M = Q * rng.randint(max(1, 48 // Q), 768 // Q)
        case = dict(op=op, S=S, F=F, B=B, M=M, Q=Q)
        if op == "superstation":
            case.update(G=max(1, S // rng.choice([2, 2, 3, 4])), output=rng.choice(["I", "IQUV"]), precision="fp32")
        elif op == "pulsar":
            K = rng.choice([256, 256, 64, 128])
            M = K * max(1, M // K)
            case.update(M=M, Q=min(Q, K), bits=rng.choice([8, 16]), precision=rng.choice(["fp32", "fp16tc"]), K=K)
        else:
            case.update(bits=rng.choice([8, 16]), output=rng.choice(["I", "IQUV"]),
                        precision="fp32" if op == "split" else rng.choice(["fp32", "fp32", "fp16tc", "fp16tc2"]))
            if op == "block":
                case.update(inc=rng.random() < 0.2)
        w = work(case)
        ct = S * F * M * N * 16
        if w["bytes"] <= 6e9 and w["flops"] <= 1.2e12 and ct <= 6e9:
            return case


# ------------------------------------------------------------------ geometry, filter and inputs
def _stations(S):
    """Half the stations in a 1 km core, the rest log-uniform out to 80 km."""
    r = np.random.default_rng(S)
    core = S // 2
    rad = np.concatenate([1000.0 * np.sqrt(r.random(core)), np.exp(r.uniform(np.log(1e3), np.log(8e4), S - core))])
    th = 2 * np.pi * r.random(S)
    return np.stack([rad * np.cos(th), rad * np.sin(th), np.zeros(S)], axis=1)


def _subbands(F, start=110e6):
    return start + (np.arange(F) + 0.5) * RATE


def _beams(B, pitch_deg=0.05):
    """The first B points of a hexagonal grid, centre first, ring by ring."""
    pts, k = [(0, 0)], 1
    while len(pts) < B:
        q, r = -k, k
        for dq, dr in ((1, 0), (1, -1), (0, -1), (-1, 0), (-1, 1), (0, 1)):
            for _ in range(k):
                pts.append((q, r))
                q, r = q + dq, r + dr
        k += 1
    p = np.radians(pitch_deg)
    return np.array([(p * (q + 0.5 * r), p * math.sqrt(3.0) / 2 * r) for q, r in pts[:B]])


def _taps():
    n = np.arange(L * N, dtype=np.float64)
    h = np.kaiser(L * N, 9.0) * np.sinc((n - (L * N - 1) / 2.0) / N)
    return (h / h.sum()).astype(np.float32)


def _bandpass():
    return (1.0 + 0.1 * np.cos(6 * np.pi * np.arange(N) / N)).astype(np.float32)


def _delays(xyz, l, m):
    return -(xyz[:, 0] * l + xyz[:, 1] * m + xyz[:, 2] * math.sqrt(1 - l * l - m * m)) / LIGHT


def _samples(xyz, f0, M, bits, seed):
    """Receiver noise plus a narrow tone from the first beam's direction, in the stations' integers:
    [S][F][T][2][2] on the GPU."""
    S, F, T = len(xyz), len(f0), M * N
    gen = torch.Generator(device="cuda")
    gen.manual_seed(int(seed))
    sigma, top = (32.0, 32767) if bits == 16 else (8.0, 127)
    out = torch.empty((S, F, T, 2, 2), dtype=torch.int16 if bits == 16 else torch.int8, device="cuda")
    offset = 32 * RATE / N
    t = torch.arange(T, device="cuda", dtype=torch.float64) * (2 * math.pi * offset / RATE)
    tone = math.sqrt(0.1 * 2) * sigma * torch.polar(torch.ones_like(t), t).to(torch.complex64)
    tau = _delays(xyz, *CENTRE)
    for s in range(S):
        x = torch.randn((F, T, 2, 2), generator=gen, device="cuda").mul_(sigma)
        ph = torch.tensor(np.exp(-2j * np.pi * ((f0 + offset) * tau[s])), dtype=torch.complex64, device="cuda")
        x += torch.view_as_real(ph[:, None] * tone[None, :])[:, :, None, :]
        out[s] = x.round_().clamp_(-top - 1, top)
    return out


def _groups(case):
    return np.arange(case["S"]) % case["G"]


def _small(case):
    """The observations of a batch: 8-16 stations, 2-8 subbands, 1-8 beams each."""
    r = np.random.default_rng(case["layout"])
    return [dict(S=int(r.integers(8, 17)), F=int(r.integers(2, 9)), B=int(r.integers(1, 9)), M=case["M"],
                 Q=4 if case["M"] % 4 == 0 else 1, bits=16, output="I", precision="fp32", inc=False, start=120e6 + 1e6 * i)
            for i in range(case["n"])]


def _plan(case, xyz=None, **over):
    kw = dict(station_xyz=_stations(case["S"]) if xyz is None else xyz,
              subband_hz=_subbands(case["F"], case.get("start", 110e6)), beam_dlm=_beams(case["B"]),
              phase_centre=CENTRE, taps=_taps(), bandpass=_bandpass(), block_samples=case["M"] * N,
              int_factor=case["Q"], output=case.get("output", "I"), sample_bits=case.get("bits", 16),
              precision=case["precision"], incoherent_beam=case.get("inc", False))
    kw.update(over)
    return Plan(**kw)


def _block(case, seed):
    return _samples(_stations(case["S"]), _subbands(case["F"], case.get("start", 110e6)), case["M"], case["bits"], seed)


def _corner_turned(case, seed):
    gen = torch.Generator(device="cuda")
    gen.manual_seed(int(seed))
    x = torch.randn((case["F"], N, case["S"], 2, case["M"], 2), generator=gen, device="cuda").mul_(2.0)
    return torch.view_as_complex(x)


def _empty(plan, which):
    return torch.empty(plan.shape(which), dtype=torch.float32 if which == "stokes" else torch.complex64, device="cuda")


# ------------------------------------------------------------------------------ one pass of a case
def prepare(case, seed):
    op = case["op"]
    if op == "batch":
        obs = _small(case)
        plans = [_plan(c) for c in obs]
        ins = [_block(c, seed * 1000 + i) for i, c in enumerate(obs)]
        outs = [_empty(p, "stokes") for p in plans]
        batch = Batch(plans)
        batch.capture(ins, outs)
        return dict(op=op, plans=plans, batch=batch, ins=ins, outs=outs)
    if op == "superstation":
        fine = _plan(case, precision="fp32", external_workspace=True)
        grp, xyz = _groups(case), _stations(case["S"])
        coarse = _plan(case, xyz=np.stack([xyz[grp == g].mean(axis=0) for g in range(case["G"])]))
        return dict(op=op, plan=fine, coarse=coarse, groups=grp, ct=_corner_turned(case, seed),
                    ss=torch.empty((case["F"], N, case["G"], 2, case["M"]), dtype=torch.complex64, device="cuda"),
                    out=_empty(coarse, "stokes"))
    state = dict(op=op, x=_block(case, seed))
    if op == "pulsar":
        state["plan"] = _plan(case, output="V", int_factor=1)
        state["detect"] = _plan(case, output="I", external_workspace=True)
        state.update(K=case["K"], vol=_empty(state["plan"], "vol"), out=_empty(state["detect"], "stokes"))
        return state
    plan = state["plan"] = _plan(case)
    if op == "split":
        state.update(chan=_empty(plan, "chan"), ct=_empty(plan, "ct"), vol=_empty(plan, "vol"))
    state["out"] = _empty(plan, "stokes")
    return state


def run(state):
    op = state["op"]
    if op == "batch":
        state["batch"].launch()
        return state["outs"]
    plan = state["plan"]
    if op == "block":
        plan.run_block(state["x"], state["out"])
        return state["out"]
    if op == "split":
        plan.ppf(state["x"], state["chan"])
        plan.delay_correct(state["chan"], state["ct"])
        plan.beamform(state["ct"], state["vol"])
        plan.stokes(state["vol"], state["out"])
        return {k: state[k] for k in ("chan", "ct", "vol", "out")}
    if op == "pulsar":
        plan.run_block(state["x"], state["vol"])
        plan.dedisperse(DM, state["K"], state["vol"], state["vol"])
        state["detect"].stokes(state["vol"], state["out"])
        return {"vol": state["vol"], "out": state["out"]}
    plan.superstation(state["groups"], state["ct"], state["ss"])
    state["coarse"].beamform_stokes(state["ss"], state["out"])
    return {"ss": state["ss"], "out": state["out"]}


def work(case):
    """Bytes: each input once, each returned output once.  Flops: 16 multiply-adds of a complex
    sample by a real tap and 5 log2 N per sample of the FFT, 8 per complex multiply-add of the beam
    former, and the detections."""
    op = case["op"]
    if op == "batch":
        parts = [work(dict(c, op="block")) for c in _small(case)]
        return {k: sum(p[k] for p in parts) for k in ("bytes", "flops")}
    S, F, B, T = case["S"], case["F"], case["B"], case["M"] * N
    samples = 2.0 * S * F * T              # complex samples, both polarisations
    beamed = 2.0 * B * F * T
    ns = 4 if case.get("output", "I") == "IQUV" else 1
    stokes = 4.0 * (B + case.get("inc", False)) * ns * F * T / case["Q"]
    word = case.get("bits", 16) / 4.0      # bytes of one complex sample of one polarisation
    flops = 8.0 * samples * B + 4.0 * beamed * ns
    if op == "superstation":
        summed = samples * case["G"] / S
        return {"bytes": 8 * (samples + summed) + stokes, "flops": 2 * samples + 8.0 * summed * B + 4.0 * beamed * ns}
    flops += samples * (4 * L + 5 * 8 + 8)
    total = samples * word + stokes
    if op == "split":
        total += 8 * (2 * samples + beamed)    # the channels, the corner-turned block, the voltages
    if op == "pulsar":
        total += 8 * beamed
        flops += beamed * (10 * math.log2(case["K"]) + 6)
    return {"bytes": total, "flops": flops}


# --------------------------------------------------------------- the same path in 64 bits, plainly
def _filtered(x, f, d):
    """Subband f of integer samples, first block of a stream: [S][P][M][N] channels in frequency order."""
    S, T = x.shape[0], x.shape[2]
    M = T // N
    h = torch.tensor(_taps(), dtype=torch.float64, device=x.device).reshape(L, N)
    out = torch.empty((S, 2, M, N), dtype=torch.complex128, device=x.device)
    for s in range(S):
        v = x[s, f].to(torch.float64)
        v = torch.complex(v[..., 0], v[..., 1]).T                        # [P][T]
        pad = torch.zeros((2, (L - 1) * N + int(d[s])), dtype=v.dtype, device=v.device)
        fr = torch.cat([pad, v], dim=1)[:, :(M + L - 1) * N].reshape(2, M + L - 1, N)
        acc = torch.zeros((2, M, N), dtype=v.dtype, device=v.device)
        for t in range(L):
            acc += h[t] * fr[:, t:t + M]
        out[s] = torch.fft.fftshift(torch.fft.fft(acc, dim=-1), dim=-1)
    return out


def _unit(cycles):
    a = 2 * math.pi * (cycles - torch.round(cycles))
    return torch.polar(torch.ones_like(a), a)


def _stokes_of(v, output, Q):
    """v [..., P, M] -> [nS][..., M/Q]."""
    X, Y = v[..., 0, :], v[..., 1, :]
    xx, yy = X.real ** 2 + X.imag ** 2, Y.real ** 2 + Y.imag ** 2
    p = [xx + yy]
    if output == "IQUV":
        xy = X * Y.conj()
        p += [xx - yy, 2 * xy.real, 2 * xy.imag]
    return torch.stack([q.reshape(q.shape[:-1] + (-1, Q)).sum(dim=-1) for q in p])


def _exact_path(case, xyz, f0s, x=None, ct_in=None, want=("stokes",)):
    """The path from samples `x` (or a corner-turned block) in 64 bits; the products in `want`."""
    dev = "cuda"
    S, F, B, M, Q = len(xyz), len(f0s), case["B"], case["M"], case["Q"]
    output = case.get("output", "I")
    ns = 4 if output == "IQUV" else 1
    tau = _delays(xyz, *CENTRE)
    n = np.sign(tau) * np.floor(np.abs(tau * RATE) + 0.5)
    d = n.max() - n
    resid = torch.tensor(tau - n / RATE, device=dev)
    dtau = torch.tensor(np.stack([_delays(xyz, CENTRE[0] + a, CENTRE[1] + b) - tau for a, b in _beams(B)]), device=dev)
    tau = torch.tensor(tau, device=dev)
    df = (torch.arange(N, dtype=torch.float64, device=dev) - N // 2) * (RATE / N)
    bp = torch.tensor(_bandpass(), dtype=torch.float64, device=dev)
    c128 = dict(dtype=torch.complex128, device=dev)
    got = {}
    if "chan" in want:
        got["chan"] = torch.empty((F, S, 2, M, N), **c128)
    if "ct" in want:
        got["ct"] = torch.empty((F, N, S, 2, M), **c128)
    if "vol" in want:
        got["vol"] = torch.empty((B, F, N, 2, M), **c128)
    got["stokes"] = torch.empty((B + int(case.get("inc", False)), ns, F, N, M // Q), dtype=torch.float64, device=dev)
    step = max(1, min(N, int(2e8) // (B * 2 * M)))
    for f in range(F):
        if ct_in is None:
            X = _filtered(x, f, d)
            if "chan" in got:
                got["chan"][f] = X
            y = X * (bp * _unit(float(f0s[f]) * tau[:, None] + df[None, :] * resid[:, None]))[:, None, None, :]
            y = y.permute(3, 0, 1, 2).contiguous()                        # [N][S][P][M]
            if "ct" in got:
                got["ct"][f] = y
        else:
            y = ct_in[f].to(torch.complex128)
        if case.get("inc"):
            got["stokes"][B, :, f] = _stokes_of(y, output, Q).sum(dim=2)
        for c in range(0, N, step):
            w = _unit((float(f0s[f]) + df[c:c + step, None, None]) * dtau[None])
            v = torch.matmul(w, y[c:c + step].reshape(-1, S, 2 * M)).reshape(-1, B, 2, M).transpose(0, 1)
            if "K" in case:
                K = case["K"]
                k = torch.arange(K, dtype=torch.float64, device=dev)
                nu = torch.where(k < K // 2, k, k - K) * (RATE / N / K)
                fc = (float(f0s[f]) + df[c:c + step])[:, None]
                chirp = _unit(-K_DM * DM * nu * nu / (fc * fc * (fc + nu)))
                v = torch.fft.ifft(torch.fft.fft(v.reshape(B, -1, 2, M // K, K), dim=-1) * chirp[None, :, None, None, :],
                                   dim=-1).reshape(B, -1, 2, M)
            if "vol" in got:
                got["vol"][:, f, c:c + step] = v
            got["stokes"][:B, :, f, c:c + step] = _stokes_of(v, output, Q).transpose(0, 1)
            del w, v
    return got


def exact(case, seed):
    op = case["op"]
    if op == "batch":
        return [exact(dict(c, op="block"), seed * 1000 + i) for i, c in enumerate(_small(case))]
    xyz, f0s = _stations(case["S"]), _subbands(case["F"], case.get("start", 110e6))
    if op == "superstation":
        grp, ct = _groups(case), _corner_turned(case, seed)
        ss = torch.zeros((case["F"], N, case["G"], 2, case["M"]), dtype=torch.complex128, device="cuda")
        for s in range(case["S"]):
            ss[:, :, int(grp[s])] += ct[:, :, s]
        sums = np.stack([xyz[grp == g].mean(axis=0) for g in range(case["G"])])
        return {"ss": ss, "out": _exact_path(case, sums, f0s, ct_in=ss)["stokes"]}
    x = _block(case, seed)
    if op == "block":
        return _exact_path(case, xyz, f0s, x)["stokes"]
    want = ("chan", "ct", "vol", "stokes") if op == "split" else ("vol", "stokes")
    got = _exact_path(case, xyz, f0s, x, want=want)
    return dict({k: got[k] for k in want[:-1]}, out=got["stokes"])
