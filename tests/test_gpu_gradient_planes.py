"""GPU: with bfloat16 storage, gradients keep their 24 bits through the tensor cores of the walking kernels.

Gradients are float32 there and go to the tensor cores as three bfloat16 planes that add up to them.  Against an
oracle that rounds nothing the rounding of h and of the gates hides that: a dropped plane is 2^-9 or 2^-17 of a
gradient, and the tolerance of the type is 2e-2.  So the problems here are such that the stored values are known
exactly -- gates and states that do not depend on a sum -- and what is left is 32-bit arithmetic on gradients.

The bounds: sums of at most some 40 terms and a dozen roundings of 2^-24 each, 1e-7 to 6e-7 together; without the
third plane an operand is off by up to 2^-18, some 2e-6 in the mean square, and each of the outputs below is linear
in such operands.
"""
import numpy as np
import pytest

from paper_1606_03401_b200 import synth
from tests.util import rel_l2

BOUND = 1.2e-6
CHUNK_BOUND = 4e-7                   # (elementwise derivatives and sums of at most three rows)
KEYS = ("layers", "input", "hidden", "readout", "batch", "t")
SIZES = [("pods", (1, 20, 31, 7, 5, 6)), ("pods", (2, 21, 130, 7, 9, 6)), ("teams", (2, 20, 515, 7, 3, 6)),
         ("teams", (3, 24, 400, 9, 20, 5))]
CHUNKS = [("pods", (1, 20, 31, 7, 2, 1)), ("pods", (2, 21, 130, 7, 2, 1)), ("teams", (2, 20, 515, 7, 3, 1)), ("teams", (3, 24, 515, 9, 2, 1))]
BIAS = (0.4, 1.1, -0.7, 0.9)         # i, f, g, o


def _sigmoid(a):
    return 1.0 / (1.0 + np.exp(-a))


def _stored(v):
    """v as bfloat16; v is far enough from a tie for float32 arithmetic to round it the same way."""
    r = synth.round_to_bf16(np.array([v, v * (1 + 1e-6), v * (1 - 1e-6)]))
    assert r[0] == r[1] == r[2]
    return r[0]


def _problem(size, bias):
    cfg = synth.with_overrides(synth.CONFIGS["c1"], dtype="bf16", **dict(zip(KEYS, size)))
    prob = synth.make_problem(cfg)
    rng = np.random.default_rng(11)
    prob["W"] = [np.zeros_like(w) for w in prob["W"]]
    prob["b"] = [synth.round_to_fp32(np.repeat(bias, cfg.hidden)) for _ in prob["b"]]
    prob["b_out"] = synth.round_to_fp32(rng.uniform(-0.3, 0.3, cfg.readout))
    return cfg, prob, rng


def _planes(n):
    """A gradient as n bfloat16 planes hold it (0: all of it)."""
    def op(v):
        if not n:
            return v
        total = np.zeros_like(v)
        for _ in range(n):
            total = total + synth.round_to_bf16(v - total)
        return total
    return op


def _run(cfg, prob, route):
    from paper_1606_03401_b200 import binding as B
    from paper_1606_03401_b200 import harness as H
    dp = H.DeviceProblem(cfg, prob, want_dx=True)
    plan = dp.plan("msm", 7)
    assert B.mebptt_test_route(dp.desc, plan)["route"] == route
    res = dp.run(plan)
    assert res["counters"][3] == 0
    return res, dp


def _carried_problem(size):
    """No inputs, no state, g = tanh(0): h and c stay zero and the gates i, f, o are constants, while the gradients
    of g run through W_hh, through W_ih into the layers below and into dx, from dy W_out."""
    cfg, prob, rng = _problem(size, (BIAS[0], BIAS[1], 0.0, BIAS[3]))
    lim = 1.0 / np.sqrt(cfg.hidden)
    units = rng.choice(cfg.hidden, 16, replace=False)         # the units whose gradients are handed on: short sums
    for w in prob["W"]:
        w[2 * cfg.hidden + units] = synth.round_to_bf16(rng.uniform(-lim, lim, (16, w.shape[1])) * 4)
    prob["x"][:], prob["h0"][:], prob["c0"][:] = 0, 0, 0
    return cfg, prob


def _carried_gradients(size, prob, op):
    L, I, H, O, N, t = size
    gi, gf, go = (_stored(_sigmoid(np.float64(np.float32(b)))) for b in (BIAS[0], BIAS[1], BIAS[3]))
    dz, carry = ([np.zeros((N, H)) for _ in range(L)] for _ in range(2))
    out = {"db %d" % l: np.zeros(4 * H) for l in range(L)}
    for k in range(t, 0, -1):
        above = op(2.0 * (prob["b_out"] - prob["targets"][k - 1]) / (N * O)) @ prob["W_out"]
        for l in range(L - 1, -1, -1):
            I_l = I if l == 0 else H
            w = prob["W"][l][2 * H:3 * H]
            dc = (above + op(dz[l]) @ w[:, I_l:]) * go + carry[l]
            carry[l], dz[l] = dc * gf, dc * gi
            out["db %d" % l][2 * H:3 * H] += dz[l].sum(0)
            above = op(dz[l]) @ w[:, :I_l]
        out["dx of step %d" % k] = above
    return out


def _chunk_problem(size):
    """No recurrent or input weights: gates and states are the same for all units and known, and the weight
    gradients are sums over rows of float32 gradients times bfloat16 values."""
    cfg, prob, rng = _problem(size, BIAS)
    prob["W_out"] = np.zeros_like(prob["W_out"])
    keep = rng.choice(cfg.hidden, 12, replace=False)          # y and dy W_out: short sums
    prob["W_out"][:, keep] = synth.round_to_bf16(rng.uniform(-1, 1, (cfg.readout, 12)))
    prob["h0"][:], prob["c0"][:] = 0.5, 0.25
    return cfg, prob


def _chunk_gradients(size, prob, op):
    L, I, H, O, N, t = size
    gates = [np.tanh(np.float64(np.float32(b))) if q == 2 else _sigmoid(np.float64(np.float32(b))) for q, b in enumerate(BIAS)]
    g = [_stored(v) for v in gates]
    c, h = [0.25], [0.5]
    for k in range(t):
        c.append(gates[1] * c[-1] + gates[0] * gates[2])
        h.append(_stored(gates[3] * np.tanh(c[-1])))
    I_l = I if L == 1 else H
    dW, db, dW_out, carry = np.zeros((4 * H, I_l + H)), np.zeros(4 * H), np.zeros((O, H)), np.zeros((N, H))
    for k in range(t, 0, -1):
        y = h[k] * prob["W_out"].sum(1) + prob["b_out"]
        dy = 2.0 * (y - prob["targets"][k - 1]) / (N * O)
        dh = op(dy) @ prob["W_out"]
        th = np.tanh(c[k])
        dc = dh * g[3] * (1 - th * th) + carry
        dz = np.concatenate([dc * g[2] * g[0] * (1 - g[0]), dc * c[k - 1] * g[1] * (1 - g[1]), dc * g[0] * (1 - g[2] * g[2]),
                             dh * th * g[3] * (1 - g[3])], 1)
        carry = dc * g[1]
        inp = prob["x"][k - 1] if L == 1 else np.full((N, H), h[k])
        dW += op(dz).T @ np.concatenate([inp, np.full((N, H), h[k - 1])], 1)
        db += dz.sum(0)
        dW_out += op(dy).T @ np.full((N, H), h[k])
    return {"dW": dW, "db": db, "dW_out": dW_out}


@pytest.mark.gpu
@pytest.mark.parametrize("route,size", SIZES)
def test_gradients_carried_through_time_and_layers(route, size):
    L, I, H, O, N, t = size
    cfg, prob = _carried_problem(size)
    res, _ = _run(cfg, prob, route)
    dx, db = res["dx"].reshape(t, N, I), res["db"].reshape(L, 4 * H)
    errs = {}
    for name, want in _carried_gradients(size, prob, _planes(0)).items():
        errs[name] = rel_l2(db[int(name[3:])] if name.startswith("db") else dx[int(name.split()[-1]) - 1], want)
    print(size, {k: "%.1e" % v for k, v in errs.items()})
    assert max(errs.values()) < BOUND, errs


@pytest.mark.gpu
@pytest.mark.parametrize("route,size", CHUNKS)
def test_weight_gradients_of_a_chunk(route, size):
    L, H = size[0], size[2]
    cfg, prob = _chunk_problem(size)
    res, dp = _run(cfg, prob, route)
    want, dW = _chunk_gradients(size, prob, _planes(0)), dp.split_dW(res["dW"])
    errs = {"dW": rel_l2(dW[-1], want["dW"]), "db": rel_l2(res["db"].reshape(L, 4 * H)[-1], want["db"]),
            "dW_out": rel_l2(res["dW_out"], want["dW_out"].ravel())}
    print(size, {k: "%.1e" % v for k, v in errs.items()})
    assert max(errs.values()) < CHUNK_BOUND, errs
    assert not any(w.any() for w in dW[:-1])


@pytest.mark.parametrize("problem,gradients,bound,size", [(_carried_problem, _carried_gradients, BOUND, s) for _, s in SIZES] +
                         [(_chunk_problem, _chunk_gradients, CHUNK_BOUND, s) for _, s in CHUNKS])
def test_a_dropped_plane_would_be_noticed(problem, gradients, bound, size):
    """The same gradients from operands cut to fewer planes (in the oracle) miss the bound."""
    prob = problem(size)[1]
    whole, three = gradients(size, prob, _planes(0)), gradients(size, prob, _planes(3))
    for planes in (1, 2):
        cut = gradients(size, prob, _planes(planes))
        for name in whole:
            if not name.startswith("db"):          # (sums of the gradients themselves)
                assert rel_l2(cut[name], whole[name]) > 1.5 * bound, (name, planes, rel_l2(cut[name], whole[name]))
                assert rel_l2(three[name], whole[name]) < 0.1 * bound
