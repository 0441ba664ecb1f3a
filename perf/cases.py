"""Timed cases: whole training steps under a memory budget, through the public entry points.

One pass is one call of ``mebptt_lstm_train_step`` (or of its host-buffer or allocation-free
variant): every forward, recomputed forward and backward operation that the plan dictates over the
sequence, giving the loss and every gradient.  The plan, the weights, the workspace and the output
buffers are made beforehand, as a training loop keeps them from step to step.

The sizes are those of the five benchmark workloads and of the paper's own timing experiment, of the
tests' two-layer and GRU problems grown to a size that is trained in earnest, and of data that does
not come in multiples of eight (features of a spectrogram, a short last batch).
"""
import math

import torch

from paper_1606_03401_b200 import binding as B

#: storage types of (operands, everything else), tolerance of another correct implementation
_OPERAND = {"fp32": torch.float32, "tf32": torch.float32, "bf16": torch.bfloat16}
# fp32: 32-bit sums in another order, carried through a few hundred dependent steps.  tf32: products
# of 16-bit mantissas.  bf16: h, gates and staged gradients are rounded to 8 bits at every step.
_REL = {"fp32": 2e-5, "tf32": 1e-4, "bf16": 1e-2}


def _case(name, dtype, layers, input, hidden, readout, batch, t, mode, m, beta=0, cell="lstm", dx=False,
          entry="device"):
    c = {"name": name} if name else {}
    c.update(dtype=dtype, layers=layers, input=input, hidden=hidden, readout=readout, batch=batch, t=t, mode=mode, m=m,
             beta=beta, cell=cell, dx=dx, entry=entry)
    return c


def listed():
    return [
        # the smallest workload: a few hundred tiny operations in exact float32, all latency
        _case("fp32_h64_hsm8", "fp32", 1, 32, 64, 32, 4, 64, "hsm", 8),
        # an ordinary float32 layer with sizes as a dataset gives them, gradient handed to what lies below
        _case("fp32_2x200_msm40", "fp32", 2, 77, 200, 61, 13, 120, "msm", 40, beta=3, dx=True),
        # a mid-sized bf16 layer under hidden-state memorisation
        _case("bf16_h512_hsm64", "bf16", 1, 512, 512, 512, 64, 256, "hsm", 64),
        # the paper's timing experiment: a thousand steps of 256 units, a tenth of the states kept
        _case("bf16_h256_hsm100", "bf16", 1, 256, 256, 256, 64, 1000, "hsm", 100),
        # the headline workload: t = 1000, H = 1024 under mixed memorisation with m = 100
        _case("bf16_h1024_msm100", "bf16", 1, 1024, 1024, 1024, 64, 1000, "msm", 100),
        # the same under a tight budget: short runs, many recomputations
        _case("bf16_h1024_msm10", "bf16", 1, 1024, 1024, 1024, 64, 1000, "msm", 10),
        # full-memory BPTT as a layer inside a model has it: with the gradient of its input
        _case("bf16_h1024_full_dx", "bf16", 1, 1024, 1024, 1024, 64, 1000, "ism", 1000, dx=True),
        # the headline workload from and to pinned host memory
        _case("bf16_h1024_msm100_host", "bf16", 1, 1024, 1024, 1024, 64, 1000, "msm", 100, entry="host"),
        # a very long sequence in float32 storage on the tensor cores
        _case("tf32_h1024_t4000_ism50", "tf32", 1, 256, 1024, 256, 32, 4000, "ism", 50),
        # a deep, wide network with one GiB for its states
        _case("bf16_2x2048_msm341", "bf16", 2, 1024, 2048, 1024, 128, 1000, "msm", 341),
        # a two-layer GRU in bf16, its input gradient wanted
        _case("bf16_gru_2x256_msm48", "bf16", 2, 128, 256, 128, 32, 128, "msm", 48, beta=3, cell="gru", dx=True),
        # bf16 with nothing a multiple of eight: 161 spectrogram bins, 29 symbols, a short last batch
        _case("bf16_2x300_ragged_msm60", "bf16", 2, 161, 300, 29, 20, 160, "msm", 60, beta=3, dx=True),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _width(rng, lo, hi, whole):
    """A width; `whole`: a multiple of eight, as widths are usually chosen."""
    v = _log(rng, lo, hi)
    return max(8, v - v % 8) if whole else v


def _batch(rng, lo, hi):
    """A batch: half the time a multiple of 32 (where the range reaches one)."""
    v = _log(rng, lo, hi)
    return v if rng.random() < 0.5 or hi < 32 else max(32, v - v % 32)


def _gate_flops(c, width):
    """Flops of the contraction of `width` input columns with all gates of one layer at one step."""
    return 2.0 * c["batch"] * width * (3 if c["cell"] == "gru" else 4) * c["hidden"]


def _flops(c):
    """Flops of the step the plan dictates: its forward operations, one backward operation a time step
    (gradients of state and weights), the readout with its two gradients."""
    H, plan = c["hidden"], _plan(c)
    ins = [c["input"]] + [H] * (c["layers"] - 1)
    fwd = sum(_gate_flops(c, i + H) for i in ins)
    into = sum(_gate_flops(c, i) for k, i in enumerate(ins) if k or c["dx"])   # gradients handed down
    bwd = fwd + into + _gate_flops(c, H) * c["layers"]
    return plan.cost * fwd + c["t"] * (bwd + 6.0 * c["batch"] * H * c["readout"])


# family, cell: (types, layers, input, hidden, batch, t), the most flops and layer operations of a case.  The
# last two keep a drawn case below the largest listed one whatever kernels serve it.
_FAMILIES = {
    "small": (("fp32",), (1, 2), (16, 160), (32, 256), (2, 32), (32, 256), 6e11, 3000),
    "layer": (("bf16",), (1, 1), (64, 1024), (64, 1024), (8, 64), (64, 1000), 1e12, 6000),
    "deep": (("bf16",), (2, 3), (128, 1024), (256, 2048), (32, 128), (32, 500), 8e12, 4000),
    "long": (("tf32",), (1, 1), (64, 512), (64, 1024), (8, 64), (128, 4000), 1e12, 6000),
    "gru": (("fp32", "bf16", "bf16"), (1, 2), (32, 256), (64, 512), (4, 64), (32, 256), 6e11, 3000),
    "ragged": (("bf16",), (1, 2), (33, 320), (65, 512), (3, 64), (32, 256), 6e11, 3000),
}


def draw(rng):
    family = rng.choice(("small", "layer", "layer", "deep", "long", "gru", "ragged"))
    dtypes, layers, inputs, hiddens, batches, ts, most_flops, most_ops = _FAMILIES[family]
    c = _case(None, rng.choice(dtypes), rng.randint(*layers), 0, 0, 0, 0, _log(rng, *ts), rng.choice(("hsm", "ism", "msm")), 0,
              cell="gru" if family == "gru" else "lstm", dx=rng.random() < 0.4, entry="host" if rng.random() < 0.15 else "device")
    if family == "ragged":
        c.update(input=_log(rng, *inputs), hidden=_log(rng, *hiddens), readout=_log(rng, 10, 256), batch=_log(rng, *batches))
    else:
        whole = rng.random() < 0.8
        c.update(input=_width(rng, *inputs, whole), hidden=_width(rng, *hiddens, whole), readout=_width(rng, *inputs, whole),
                 batch=_batch(rng, *batches))
    # a budget between a handful of states and nearly everything; ISM counts states four times as large
    c["m"] = max(4, _log(rng, 8, c["t"]) // (2 if c["mode"] == "ism" else 1))
    c["beta"] = rng.choice((0, 3)) if c["mode"] == "msm" else 0
    while c["t"] > 16 and (_flops(c) > most_flops or (_plan(c).cost + c["t"]) * c["layers"] > most_ops):
        c["t"] = c["t"] * 4 // 5
        c["m"] = max(4, min(c["m"], c["t"]))
    return c


def _plan(c):
    return B.mebptt_plan_ex(c["t"], c["m"], B.MODES[c["mode"]], 4, c["beta"])


def prepare(case, seed):
    c = case
    dev = torch.device("cuda", torch.cuda.current_device())
    g = torch.Generator(device=dev).manual_seed(int(seed))
    L, I, H, O, N, t = (c[k] for k in ("layers", "input", "hidden", "readout", "batch", "t"))
    op, ng = _OPERAND[c["dtype"]], 3 if c["cell"] == "gru" else 4

    def normal(n, dtype, scale=1.0):
        return torch.randn(n, generator=g, device=dev).mul_(scale).to(dtype)

    def uniform(n, dtype, lim):
        return torch.rand(n, generator=g, device=dev).mul_(2 * lim).sub_(lim).to(dtype)

    nW = sum(ng * H * ((I if l == 0 else H) + H) for l in range(L))
    # weights as they are initialised, biases a little way into training, a carried-over initial state
    b = uniform(L * ng * H, torch.float32, 0.3).view(L, ng, H)
    if c["cell"] == "lstm":
        b[:, 1] += 1.0
    inputs = [uniform(nW, op, H ** -0.5), b.reshape(-1), uniform(O * H, op, H ** -0.5), uniform(O, torch.float32, 0.3),
              normal(t * N * I, op), normal(t * N * O, torch.float32), normal(L * N * H, op, 0.5),
              normal(L * N * H, torch.float32, 0.5)]
    sizes = {"loss": 1, "dW": nW, "db": L * ng * H, "dW_out": O * H, "db_out": O, "dx": t * N * I if c["dx"] else 0}
    host = c["entry"] == "host"
    where = dict(pin_memory=True) if host else dict(device=dev)
    out = {k: torch.zeros(n, dtype=torch.float32, **where) for k, n in sizes.items() if n}
    out["counters"] = torch.zeros(8, dtype=torch.int64, **where)
    if host:
        inputs = [x.cpu().pin_memory() for x in inputs]
    desc = B.make_desc(L, I, H, O, N, t, c["dtype"], want_dx=int(c["dx"]), flags=B.MEBPTT_FLAG_GRU if c["cell"] == "gru" else 0)
    plan = _plan(c)
    nbytes = (B.mebptt_lstm_host_workspace_bytes if host else B.mebptt_lstm_workspace_bytes)(desc, plan)
    return {"desc": desc, "plan": plan, "inputs": inputs, "out": out, "workspace": torch.empty(nbytes, dtype=torch.uint8, device=dev),
            "step": B.mebptt_lstm_train_step_host if host else B.mebptt_lstm_train_step}


def run(state):
    o = state["out"]
    state["step"](state["desc"], state["plan"], *state["inputs"], state["workspace"], torch.cuda.current_stream().cuda_stream,
                  o["loss"], o["dW"], o["db"], o["dW_out"], o["db_out"], o.get("dx"), o["counters"])
    return o


def work(case):
    c = case
    L, I, H, O, N, t = (c[k] for k in ("layers", "input", "hidden", "readout", "batch", "t"))
    e, ng = (2 if c["dtype"] == "bf16" else 4), 3 if c["cell"] == "gru" else 4
    nW = sum(ng * H * ((I if l == 0 else H) + H) for l in range(L)) + O * H
    nb = L * ng * H + O
    read = nW * e + nb * 4 + t * N * (I * e + O * 4) + L * N * H * (e + 4)
    written = 4 * (nW + nb + (t * N * I if c["dx"] else 0))
    return {"bytes": read + written, "flops": _flops(c)}


def tolerance(case):
    return {"rel": _REL[case["dtype"]]}
