"""The work that users have this library do: forward passes of integer LSTM stacks through its public entry points.

A case is one call of one entry point on one stack:

  call      "run"    QLSTM.run on device buffers (the state h, c is carried from call to call, as in streaming)
            "host"   QLSTM.run_host_raw: host buffers in and out, copies inside the call
            "bidir"  BiQLSTM.run: a forward and a backward stack over the same input
  layers    depth; every layer has n_cell cells, and n_output outputs where it has a projection (else n_cell)
  proj, peep, norm, cifg    the variants of Section 2 of the paper (arXiv 2101.05453)
  T, B      time steps of the call, batch rows

Weights, inputs and scales follow the distributions of workloads/configs.py: W ~ N(0, 1/sqrt(n_in)), x ~ N(0, 1), and
the ranges that calibration logs for such stacks (quoted in _ranges).
"""
import math

import numpy as np
import torch

import paper_2101_05453_b200 as qlstm


def _case(name, call, layers, n_input, n_cell, n_output, T, B, proj=False, peep=False, norm=False, cifg=False):
    return dict(name=name, call=call, layers=layers, n_input=n_input, n_cell=n_cell,
                n_output=n_output if proj else n_cell, proj=proj, peep=peep, norm=norm, cifg=cifg, T=T, B=B)


def listed():
    deep = dict(layers=8, n_input=640, n_cell=2048, n_output=640, proj=True, norm=True)
    return [
        # one user dictating into the production-shaped encoder, one frame per call: pure latency
        _case("step 8x2048 b1", "run", T=1, B=1, **deep),
        # a few streams served together in chunks of 16 frames
        _case("chunk 5x1024 b4", "run", 5, 640, 1024, 1024, T=16, B=4, cifg=True),
        # a small acoustic model on log-mel frames
        _case("basic 2x256 b8", "run", 2, 80, 256, 256, T=100, B=8),
        # one wide layer with every extra (layer norm, peephole, projection)
        _case("peephole 1x2048 b32", "run", 1, 512, 2048, 640, T=200, B=32, proj=True, peep=True, norm=True),
        # a coupled-gate stack over a batch of long utterances
        _case("cifg 5x1024 b64", "run", 5, 640, 1024, 1024, T=500, B=64, cifg=True),
        # the production-shaped encoder on whole utterances: one, a handful, a server's batch, offline transcription
        _case("deep 8x2048 b1", "run", T=300, B=1, **deep),
        _case("deep 8x2048 b8", "run", T=300, B=8, **deep),
        _case("deep 8x2048 b64", "run", T=300, B=64, **deep),
        _case("deep 8x2048 b256", "run", T=300, B=256, **deep),
        # sizes that no tile, vector or warp divides
        _case("odd 3x1000 b37", "run", 3, 40, 1000, 300, T=131, B=37, proj=True, norm=True, cifg=True),
        # a bidirectional encoder
        _case("bidirectional 2x512 b16", "bidir", 2, 80, 512, 512, T=150, B=16),
        # end to end from host memory, an odd number of rows and steps
        _case("host 4x1024 b100", "host", 4, 320, 1024, 512, T=123, B=100, proj=True, norm=True),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """Any stack of one to eight layers over the sizes of the listed ones, with any of the variants."""
    call = rng.choice(["run"] * 6 + ["host", "bidir"])
    layers = rng.choice([1, 2, 2, 3, 4, 5, 6, 8])
    proj, norm = rng.random() < 0.5, rng.random() < 0.5
    peep, cifg = rng.random() < 0.25, rng.random() < 0.35
    n_input, n_cell = _log(rng, 16, 640), _log(rng, 32, 2048)
    n_output = _log(rng, 16, min(n_cell, 640))
    odd = rng.random() < 0.2
    if not odd:
        n_input, n_cell, n_output = (max(16, (v + 8) // 16 * 16) for v in (n_input, n_cell, n_output))
    if call == "bidir":
        n_input = max(16, (n_input + 8) // 16 * 16)          # the reversed copy of the input is made in 16-byte pieces
    T, B = _log(rng, 1, 500), _log(rng, 1, 256)
    T = min(T, (300 if odd else 2400) // (layers * (2 if call == "bidir" else 1)))
    return {k: v for k, v in _case("", call, layers, n_input, n_cell, n_output, max(1, T), B, proj, peep, norm, cifg).items()
            if k != "name"}


class _Layer:
    """One layer description as QLSTM takes it (the fields of qlstm_layer_t)."""


def _scale(v):
    """real = multiplier 2^(shift - 31), multiplier in [2^30, 2^31)."""
    m, e = math.frexp(v)
    q = int(round(m * (1 << 31)))
    return (1 << 30, e + 1) if q == 1 << 31 else (q, e)


def _asym(lo, hi):
    s = (hi - lo) / 255.0
    return s, max(-128, min(127, int(round(-128.0 - lo / s))))


def _ranges(case, l):
    """What calibration logs for layer l of such a stack: |h|, |m|, |c| and, with layer norm, |gate sum| at most."""
    if case["norm"]:
        m, c, g = 0.97, (3.6 if l == 0 else 20.0), (5.0 if l == 0 else 2.5)
        return (1.1 if l == 0 else 1.6) if case["proj"] else m, m, c, g
    fade = max(0.3, 0.75 ** l)
    m, c = (0.7 * fade, 0.95 * fade) if case["cifg"] else (0.9 * fade, 2.8 * fade)
    return 1.1 * m if case["proj"] else m, m, c, 0.0


def _weights(gen, rows, cols):
    """int8 weights ~ N(0, 1 / sqrt(cols)) with a symmetric scale, and that scale."""
    w = torch.randn((rows, cols), generator=gen, device="cuda") / math.sqrt(cols)
    s = float(w.abs().max()) / 127.0
    return torch.round(w / s).to(torch.int8).cpu().numpy(), s


def _stack(case, gen, rng):
    layers, n_in = [], case["n_input"]
    s_x, zp_x = _asym(-4.6, 4.5)
    for l in range(case["layers"]):
        C, O = case["n_cell"], case["n_output"]
        h_max, m_max, c_max, g_max = _ranges(case, l)
        q = _Layer()
        q.n_input, q.n_cell, q.n_output = n_in, C, O
        q.flags = case["proj"] * 1 + case["peep"] * 2 + case["norm"] * 4 + case["cifg"] * 8
        q.cell_int_bits = max(0, math.ceil(math.log2(c_max)))
        s_h, q.zp_h = _asym(-1.02 * h_max, h_max)
        s_m, q.zp_m = _asym(-m_max, 1.02 * m_max) if case["proj"] else (s_h, q.zp_h)
        q.zp_x = zp_x
        q.W, q.R, q.P, q.b, q.L = ([None] * 4 for _ in range(5))
        q.eff_x, q.eff_h, q.eff_c, q.eff_ln = ([(0, 0)] * 4 for _ in range(4))
        for g in range(1 if case["cifg"] else 0, 4):
            q.W[g], s_w = _weights(gen, C, n_in)
            q.R[g], s_r = _weights(gen, C, O)
            s_gate, s_b = 2.0 ** -12, s_r * s_h
            if case["norm"]:
                s_gate, s_l = g_max / 32767.0, 1.4 / 32767.0
                q.L[g] = np.clip(np.rint(rng.normal(1.0, 0.1, C) / s_l), -32767, 32767).astype(np.int16)
                s_b = s_l * 2.0 ** -10
                q.eff_ln[g] = _scale(s_b * 4096.0)
            bias = rng.normal(0.0, 0.1, C) + (1.0 if g == 1 else 0.0)
            q.b[g] = np.rint(bias / s_b).astype(np.int32)
            q.eff_x[g], q.eff_h[g] = _scale(s_w * s_x / s_gate), _scale(s_r * s_h / s_gate)
            if case["peep"] and g != 2:
                s_p = 0.35 / 32767.0
                q.P[g] = np.clip(np.rint(rng.normal(0.0, 0.1, C) / s_p), -32767, 32767).astype(np.int16)
                q.eff_c[g] = _scale(s_p * 2.0 ** (q.cell_int_bits - 15) / s_gate)
        q.eff_m = _scale(2.0 ** -30 / s_m)
        q.W_proj = q.b_proj = None
        q.eff_proj = (0, 0)
        if case["proj"]:
            q.W_proj, s_wp = _weights(gen, O, C)
            q.b_proj = np.rint(rng.normal(0.0, 0.1, O) / (s_wp * s_m)).astype(np.int32)
            q.eff_proj = _scale(s_wp * s_m / s_h)
        layers.append(q)
        n_in, s_x, zp_x = O, s_h, q.zp_h
    return layers


def prepare(case, seed):
    gen, rng = torch.Generator(device="cuda"), np.random.default_rng(seed)
    gen.manual_seed(seed)
    T, B = case["T"], case["B"]
    stacks = [_stack(case, gen, rng) for _ in range(2 if case["call"] == "bidir" else 1)]
    where = "cpu" if case["call"] == "host" else "cuda"
    s_x, _ = _asym(-4.6, 4.5)
    x = torch.randn((T, B, case["n_input"]), generator=gen, device="cuda")
    x = torch.clamp(torch.round(x / s_x) + stacks[0][0].zp_x, -128, 127).to(torch.int8).to(where)
    # initial state: float zero, layer after layer
    h = [torch.cat([torch.full((B * q.n_output,), q.zp_h, dtype=torch.int8) for q in s]).to(where) for s in stacks]
    c = [torch.zeros(B * sum(q.n_cell for q in s), dtype=torch.int16, device=where) for s in stacks]
    y = torch.empty((T, B, len(stacks) * stacks[0][-1].n_output), dtype=torch.int8, device=where)
    if where == "cpu":
        x, h, c, y = x.pin_memory(), [v.pin_memory() for v in h], [v.pin_memory() for v in c], y.pin_memory()
    model = qlstm.BiQLSTM(*stacks, T, B) if len(stacks) == 2 else qlstm.QLSTM(stacks[0], T, B)
    return dict(call=case["call"], model=model, T=T, B=B, x=x, h=h, c=c, y=y)


def run(state):
    model, T, B, x, h, c, y = (state[k] for k in ("model", "T", "B", "x", "h", "c", "y"))
    if state["call"] == "host":
        model.run_host_raw(x.data_ptr(), T, B, h[0].data_ptr(), c[0].data_ptr(), y.data_ptr())
    elif state["call"] == "bidir":
        model.run(x, T, B, h[0], c[0], h[1], c[1], y, stream=torch.cuda.current_stream().cuda_stream)
    else:
        model.run(x, T, B, h[0], c[0], y, stream=torch.cuda.current_stream().cuda_stream)
    return [y] + h + c


def work(case):
    """Weights, input and state read once, output and state written once; two operations per multiply-add of the matrix
    products (the integer elementwise work between them comes on top)."""
    T, B, C, O = case["T"], case["B"], case["n_cell"], case["n_output"]
    gates, stacks = (3 if case["cifg"] else 4), (2 if case["call"] == "bidir" else 1)
    weights = state = 0
    n_in = case["n_input"]
    for _ in range(case["layers"]):
        weights += gates * C * (n_in + O) + (C * O if case["proj"] else 0)
        state += O + 2 * C
        n_in = O
    return {"bytes": T * B * (case["n_input"] + stacks * O) + stacks * (weights + 2 * B * state),
            "flops": 2 * T * B * stacks * weights}


def tolerance(case):
    return "exact"          # an integer method: every value has one correct result
