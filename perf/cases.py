"""The calls whose speed counts for a user of this library, and their exact values.

A case names one call (`kind`) of the binding and its sizes:
  step         api.SomaExperts.step: one SPSA step (estimate, then SGD), dense probes
  adam         api.SomaExperts.adam_step: the paper's optimizer step, sparse probes
  eval         api.SomaExperts.eval: the unperturbed loss of every expert
  routed       api.mixture_nll: routed inference over k experts per request
  update       api.spsa_update: the SGD update alone, from given coefficients
  adam_update  api.adam_update: the Adam update alone, sparse probes
  body_step    api.SomaBodies.step: SPSA step of the paper's expert body
  body_adam    api.SomaBodies.adam_step: its optimizer step
  body_eval    api.SomaBodies.eval: its unperturbed loss
Parameters and byte streams are the seeded synthetic ones of
paper_2609_37899_gb300.inputs (scaled-normal weights, order-2 Zipf Markov
bytes), the same that the tests and the benchmark use.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2609_37899_gb300 import api, inputs

V = 256
EPS = 1e-3
ADAM = dict(beta1=0.9, beta2=0.999, delta=1e-8, weight_decay=1e-4)
ADAM_T = 20  # the optimizer cases stand in the middle of a run: moments are not zero


def listed():
    return [
        # the smallest call: one expert of a unit-test or sweep size, all latency
        dict(name="tiny_step", kind="step", N=1, E=32, H=64, n=8, B=4, T=64, lr=1e-2),
        # the headline workload: two 4.2M-parameter experts
        dict(name="n2_step", kind="step", N=2, E=64, H=960, n=64, B=32, T=256, lr=1e-3),
        # the monolithic control with 1,024 probes
        dict(name="mono_step", kind="step", N=1, E=64, H=1376, n=1024, B=32, T=256, lr=1e-3),
        # eight experts under the paper's optimizer, two accumulation batches
        dict(name="n8_adam", kind="adam", N=8, E=64, H=480, n=64, B=32, T=256, lr=1e-3, A=2),
        # many small experts, whole recurrences on chip
        dict(name="n256_step", kind="step", N=256, E=32, H=48, n=64, B=16, T=512, lr=1e-3),
        # no size a multiple of anything, and a batch of more than 64 sequences
        dict(name="ragged_step", kind="step", N=3, E=50, H=200, n=37, B=70, T=48, lr=1e-3),
        # held-out loss of the eight experts
        dict(name="n8_eval", kind="eval", N=8, E=64, H=480, n=1, B=256, T=512),
        # serving: 1,024 requests, four experts each, the first 128 bytes are context
        dict(name="n8_routed", kind="routed", N=8, E=64, H=480, R=1024, k=4, T=512, t0=128),
        # the paper's expert body, its N = 256 ensemble with its own probe law
        dict(name="body_n256_step", kind="body_step", N=256, D=2, n=64, B=16, T=512, lr=1e-3),
        # a few bodies on a ragged batch, two accumulation batches
        dict(name="body_ragged_adam", kind="body_adam", N=5, D=2, n=12, B=21, T=70, lr=1e-3, A=2),
        # the update over 1,024 probes, coefficients given (a coordinator that
        # gathered them, or a replay of recorded coefficients)
        dict(name="mono_update", kind="update", N=1, E=64, H=1376, n=1024, lr=1e-3),
        # the Adam update of four recorded accumulation batches
        dict(name="n2_adam_update", kind="adam_update", N=2, E=64, H=960, n=64, A=4, lr=1e-3),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


# The most work a drawn case may have, in flops: at the least efficient sizes
# this stays below the largest listed case.
_DRAW_FLOPS = {"step": 1.5e12, "adam": 1.5e12, "eval": 2e12, "routed": 2e12, "update": 1.8e10,
               "adam_update": 1.8e10, "body_step": 3e12, "body_adam": 3e12, "body_eval": 2e12}


def draw(rng):
    while True:
        kind = rng.choice(["step", "step", "step", "adam", "adam", "eval", "routed", "update",
                           "adam_update", "body_step", "body_adam", "body_eval"])
        c = dict(kind=kind)
        if kind.startswith("body"):
            c.update(N=_log_int(rng, 1, 256), D=rng.choice([1, 2, 2]),
                     n=1 if kind == "body_eval" else _log_int(rng, 2, 64),
                     B=_log_int(rng, 1, 64), T=_log_int(rng, 8, 512))
        elif kind == "routed":
            small = rng.random() < 0.4
            N = _log_int(rng, 2, 256 if small else 8)
            T = _log_int(rng, 16, 512)
            c.update(N=N, E=rng.choice([16, 32, 40, 64]),
                     H=_log_int(rng, 24, 64) if small else _log_int(rng, 65, 960),
                     R=_log_int(rng, 16, 1024), k=rng.randint(1, min(4, N)), T=T,
                     t0=rng.choice([0, T // 4]))
        elif kind in ("update", "adam_update"):
            c.update(N=_log_int(rng, 1, 64), E=rng.choice([16, 32, 50, 64]),
                     H=_log_int(rng, 24, 1376), n=_log_int(rng, 4, 1024))
        else:
            small = rng.random() < 0.4
            c.update(N=_log_int(rng, 1, 256 if small else 8), E=rng.choice([16, 32, 40, 64]),
                     H=_log_int(rng, 16, 64) if small else _log_int(rng, 65, 1376),
                     n=1 if kind == "eval" else _log_int(rng, 2, 128),
                     B=_log_int(rng, 1, 24) if small else _log_int(rng, 2, 96),
                     T=_log_int(rng, 16, 512))
        if kind in ("adam", "body_adam", "adam_update"):
            c["A"] = rng.choice([1, 2, 4])
        if kind not in ("eval", "body_eval", "routed"):
            c["lr"] = 1e-3
        if work(c)["flops"] <= _DRAW_FLOPS[kind]:
            return c


def _params_of(c):
    if c["kind"].startswith("body"):
        return inputs.body_param_count(32, c["D"])
    return inputs.param_count(c["E"], c["H"])


def work(c):
    kind, N = c["kind"], c["N"]
    P, A = _params_of(c), c.get("A", 1)
    # multiply-adds of one token through one expert (direct form)
    if kind.startswith("body"):
        per_token = 2 * (16 * 32 * 32 * c["D"] + V * 32)
    else:
        per_token = 2 * (4 * c["H"] * (c["E"] + c["H"]) + V * c["H"])
    theta = 4.0 * N * P
    if kind == "routed":
        tokens = c["R"] * c["k"] * c["T"]
        return {"bytes": theta + c["R"] * (c["T"] + 1) + 4.0 * c["R"] * (c["T"] - c["t0"]),
                "flops": float(tokens * per_token)}
    if kind in ("eval", "body_eval"):
        return {"bytes": theta + N * c["B"] * (c["T"] + 1) + 4.0 * N,
                "flops": float(N * c["B"] * c["T"] * per_token)}
    moved = theta * (6 if "adam" in kind else 2)      # theta (and m, v) in and out
    gather = 2.0 * A * c["n"] * N * P                 # sum_i c_i z_i
    if kind in ("update", "adam_update"):
        return {"bytes": moved + 4.0 * A * N * c["n"], "flops": gather}
    tokens = A * N * c["n"] * 2 * c["B"] * c["T"]
    return {"bytes": moved + A * N * c["B"] * (c["T"] + 1) + 12.0 * A * N * c["n"],
            "flops": tokens * per_token + gather}


# --------------------------------------------------------------------------
# Inputs
# --------------------------------------------------------------------------

def _host_params(c, seed):
    if c["kind"].startswith("body"):
        return inputs.init_body(c["N"], 32, c["D"], seed)
    return inputs.init_params(c["N"], c["E"], c["H"], seed)


def _host_bytes(c, seed):
    """A uint8 batches [N, B, T + 1] (requests [R, T + 1] for routed)."""
    if c["kind"] == "routed":
        return [inputs.expert_batch(1, c["R"], c["T"], 2, seed, 0)[0]]
    return [inputs.expert_batch(c["N"], c["B"], c["T"], 2, seed, a) for a in range(c.get("A", 1))]


def _host_routes(c, seed):
    rng = np.random.default_rng([seed & 0xFFFFFFFF, 0x707E])
    order = rng.random((c["R"], c["N"])).argsort(axis=1)
    return np.ascontiguousarray(order[:, :c["k"]], dtype=np.int32)


def _host_coef(c, seed):
    rng = np.random.default_rng([seed & 0xFFFFFFFF, 0xC0EF])
    return rng.standard_normal((c.get("A", 1), c["N"], c["n"])).astype(np.float32)


def _moments(c, seed, device="cuda"):
    """Adam moments of a run in progress, on the device."""
    g = torch.Generator(device=device).manual_seed(int(seed) + 11)
    shape = (c["N"], _params_of(c))
    m = 0.02 * torch.randn(shape, generator=g, device=device)
    v = 0.0025 * torch.rand(shape, generator=g, device=device) + 1e-4
    return m, v


def prepare(c, seed):
    kind, dev = c["kind"], "cuda"
    st = dict(case=c, seed=seed)
    theta = torch.from_numpy(_host_params(c, seed)).to(dev)
    if kind in ("update", "adam_update"):
        st["params"] = theta
        coef = torch.from_numpy(_host_coef(c, seed)).to(dev)
        st["coef"] = coef if kind == "adam_update" else coef[0].contiguous()
        if kind == "adam_update":
            st["m"], st["v"] = _moments(c, seed)
        return st
    st["bytes"] = [torch.from_numpy(b).to(dev) for b in _host_bytes(c, seed)]
    if kind == "routed":
        st["params"] = theta
        st["routes"] = _host_routes(c, seed)
        st["out"] = torch.empty(c["R"], c["T"] - c["t0"], device=dev)
        st["workspace"] = torch.empty(
            api.mixture_workspace_bytes(c["E"], c["H"], c["N"], st["routes"], c["T"]),
            dtype=torch.uint8, device=dev)
        return st
    if kind.startswith("body"):
        m = api.SomaBodies(c["N"], c["n"], c["B"], c["T"], 32, c["D"])
        m.head.copy_(torch.from_numpy(inputs.init_head(32, seed)))
    else:
        m = api.SomaExperts(c["N"], c["E"], c["H"], c["n"], c["B"], c["T"])
    m.params.copy_(theta)
    if kind.endswith("adam"):
        m.m, m.v = _moments(c, seed)
    st["model"] = m
    return st


def run(st):
    c, kind, seed = st["case"], st["case"]["kind"], st["seed"]
    if kind == "update":
        api.spsa_update(st["params"], c["E"], c["H"], c["lr"], seed, 3, st["coef"])
        return {"params": st["params"]}
    if kind == "adam_update":
        api.adam_update(st["params"], st["m"], st["v"], c["E"], c["H"], "sparse", seed,
                        list(range(c["A"])), st["coef"], c["lr"], t=ADAM_T, **ADAM)
        return {"params": st["params"], "m": st["m"], "v": st["v"]}
    if kind == "routed":
        api.mixture_nll(st["params"], st["bytes"][0], c["E"], c["H"], st["routes"], c["t0"],
                        st["out"], st["workspace"])
        return {"nll": st["out"]}
    m = st["model"]
    if kind in ("eval", "body_eval"):
        return {"loss": m.eval(st["bytes"][0])}
    if kind == "step":
        losses, coef = m.step(st["bytes"][0], EPS, c["lr"], seed, 0)
        return {"losses": losses, "coef": coef, "params": m.params}
    if kind == "body_step":
        losses, coef = m.step(st["bytes"][0], EPS, c["lr"], seed, 0, kind="sparse")
        return {"losses": losses, "coef": coef, "params": m.params}
    losses, coef = m.adam_step(st["bytes"], EPS, seed, list(range(c["A"])), ADAM_T, c["lr"],
                               kind="sparse", **ADAM)
    return {"losses": losses, "coef": coef, "params": m.params, "m": m.m, "v": m.v}


# --------------------------------------------------------------------------
# Exact values: plain torch in float64
# --------------------------------------------------------------------------

_M32 = 0xFFFFFFFF
_EXACT_FLOPS = 6e12  # float64 work of one exact evaluation that stays within seconds


def _mulhilo(a, x):
    p = x * a  # wraps modulo 2^64: both 32-bit halves are right
    return (p >> 32) & _M32, p & _M32


def _philox(c0, c1, c2, c3, seed):
    k0, k1 = seed & _M32, (seed >> 32) & _M32
    for _ in range(10):
        ha, la = _mulhilo(0xD2511F53, c0)
        hb, lb = _mulhilo(0xCD9E8D57, c2)
        c0, c1, c2, c3 = hb ^ c1 ^ k0, lb, ha ^ c3 ^ k1, la
        k0, k1 = (k0 + 0x9E3779B9) & _M32, (k1 + 0xBB67AE85) & _M32
    return c0, c1, c2, c3


def _bits(P, probes, step, expert, seed, p0=0):
    """bool [len(probes), P - p0]: the Philox bits of parameters p0 .. P - 1 (p0 % 128 == 0)."""
    blk = torch.arange(p0 // 128, (P + 127) // 128, device="cuda", dtype=torch.int64)[None, :]
    w = _philox(blk.expand(probes.numel(), -1), probes[:, None].expand(-1, blk.shape[1]),
                torch.full_like(blk, step), torch.full_like(blk, expert), seed)
    w = torch.stack(torch.broadcast_tensors(*w), dim=-1)  # [probes, blocks, 4]
    o = torch.arange(32, device="cuda")
    bit = (w[..., None] >> ((o >> 1) + 16 * (o & 1))) & 1
    return bit.reshape(probes.numel(), -1)[:, :P - p0].bool()


def _probes(P, probes, step, expert, seed, sparse, dense_from, p0=0):
    """z [len(probes), P - p0] float64."""
    z = 1.0 - 2.0 * _bits(P, probes, step, expert, seed, p0).double()
    if sparse:
        act = _bits(P, probes | 0x80000000, step, expert, seed, p0)
        act[:, max(0, dense_from - p0):] = True
        z *= act
    return z


def _f32(x):
    return float(np.float32(x))


def _lstm_nll(th, y, E, H):
    """NLL [lanes, B, T] of the one-layer LSTM; th [lanes, P] float64, y [B or lanes, B, T + 1]."""
    o = inputs.param_offsets(E, H)
    L = th.shape[0]
    emb = th[:, :o["w_ih"]].reshape(L, V, E)
    wi = th[:, o["w_ih"]:o["w_hh"]].reshape(L, 4 * H, E)
    wh = th[:, o["w_hh"]:o["b"]].reshape(L, 4 * H, H)
    b = th[:, o["b"]:o["w_out"]][:, None]
    wo = th[:, o["w_out"]:o["b_out"]].reshape(L, V, H)
    bo = th[:, o["b_out"]:][:, None]
    w = torch.cat([wi, wh], 2).transpose(1, 2)
    B, T = y.shape[1], y.shape[2] - 1
    rows = torch.arange(L, device=th.device)[:, None]
    h = th.new_zeros(L, B, H)
    cell = torch.zeros_like(h)
    out = th.new_empty(L, B, T)
    for t in range(T):
        a = torch.baddbmm(b, torch.cat([emb[rows, y[:, :, t].expand(L, -1)], h], 2), w)
        i, f, g, og = a.split(H, dim=2)
        cell = torch.sigmoid(f) * cell + torch.sigmoid(i) * torch.tanh(g)
        h = torch.sigmoid(og) * torch.tanh(cell)
        z = torch.baddbmm(bo, h, wo.transpose(1, 2))
        out[:, :, t] = torch.logsumexp(z, 2) - z.gather(2, y[:, :, t + 1].expand(L, -1)[..., None])[..., 0]
    return out


def _ln(x, gain):
    return torch.nn.functional.layer_norm(x, (32,), None, None, 1e-5) * gain


def _body_nll(th, head, y, D):
    o = inputs.body_offsets(32, D)
    L, B, T = th.shape[0], y.shape[1], y.shape[2] - 1

    def part(k, rows, cols):
        return th[:, o[k]:o[k] + rows * cols].reshape(L, rows, cols).transpose(1, 2)

    def gain(k):
        return th[:, o[k]:o[k] + 32][:, None]
    wih = [part(f"w_ih{k}", 128, 32) for k in range(D)]
    whh = [part(f"w_hh{k}", 128, 32) for k in range(D)]
    w1 = [part(f"w1{k}", 128, 32) for k in range(D)]
    w2 = [part(f"w2{k}", 32, 128) for k in range(D)]
    h = [th.new_zeros(L, B, 32) for _ in range(D)]
    cell = [th.new_zeros(L, B, 32) for _ in range(D)]
    out = th.new_empty(L, B, T)
    for t in range(T):
        x = head[y[:, :, t]].expand(L, -1, -1)
        for k in range(D):
            a = _ln(x, gain(f"ga{k}")) @ wih[k] + h[k] @ whh[k]
            i, f, g, og = a.split(32, dim=2)
            cell[k] = torch.sigmoid(f) * cell[k] + torch.sigmoid(i) * torch.tanh(g)
            h[k] = torch.sigmoid(og) * torch.tanh(cell[k])
            x = x + h[k]
            x = x + torch.nn.functional.gelu(_ln(x, gain(f"gb{k}")) @ w1[k]) @ w2[k]
        z = _ln(x, gain("gf")) @ head.T
        out[:, :, t] = torch.logsumexp(z, 2) - z.gather(2, y[:, :, t + 1].expand(L, -1)[..., None])[..., 0]
    return out


def exact(c, seed):
    kind, N = c["kind"], c["N"]
    body = kind.startswith("body")
    P, A = _params_of(c), c.get("A", 1)
    if work(c)["flops"] > (2e10 if "update" in kind else _EXACT_FLOPS):
        return None
    if kind in ("step", "adam") and (c["E"] + c["H"]) < 256 and work(c)["flops"] > 5e11:
        return None  # small matrices run far below the float64 rate
    if body and work(c)["flops"] > 3e11:
        return None
    theta = torch.from_numpy(_host_params(c, seed)).cuda().double()
    sparse = kind in ("adam", "adam_update", "body_step", "body_adam")
    dense_from = 16 * 32 * 32 * c["D"] if body else P
    head = torch.from_numpy(inputs.init_head(32, seed)).cuda().double() if body else None
    eps, lr = _f32(EPS), _f32(c.get("lr", 0.0))

    def nll(th, y):
        return _body_nll(th, head, y, c["D"]) if body else _lstm_nll(th, y, c["E"], c["H"])

    if kind == "routed":
        y = torch.from_numpy(_host_bytes(c, seed)[0]).cuda().long()
        routes = torch.from_numpy(_host_routes(c, seed)).cuda().long()
        per = theta.new_empty(c["k"], c["R"], c["T"])
        for e in range(N):
            r, j = (routes == e).nonzero(as_tuple=True)
            if r.numel():
                per[j, r] = nll(theta[e:e + 1], y[r][None])[0]
        return {"nll": (math.log(c["k"]) - torch.logsumexp(-per, 0))[:, c["t0"]:].contiguous()}
    if kind in ("update", "adam_update"):
        coef = torch.from_numpy(_host_coef(c, seed)).cuda().double()
        steps = list(range(A)) if kind == "adam_update" else [3]
        losses = None
    else:
        batches = [torch.from_numpy(b).cuda().long() for b in _host_bytes(c, seed)]
        if kind in ("eval", "body_eval"):
            return {"loss": torch.stack([nll(theta[e:e + 1], batches[0][e:e + 1]).mean()
                                         for e in range(N)])}
        steps = list(range(A))
        losses = theta.new_empty(A, N, c["n"], 2)
        group = max(1, int(4e8 // P))
        for a in range(A):
            for e in range(N):
                for i0 in range(0, c["n"], group):
                    pr = torch.arange(i0, min(c["n"], i0 + group), device="cuda")
                    z = _probes(P, pr, steps[a], e, seed, sparse, dense_from)
                    th = torch.cat([theta[e] + eps * z, theta[e] - eps * z])
                    del z
                    L = nll(th, batches[a][e:e + 1]).mean(dim=(1, 2))
                    losses[a, e, i0:i0 + pr.numel()] = L.reshape(2, -1).T
        coef = (losses[..., 0] - losses[..., 1]) / (2 * eps)
    ghat = torch.zeros_like(theta)
    span = 1 << 17
    for a in range(A):
        for e in range(N):
            for i0 in range(0, c["n"], 256):
                pr = torch.arange(i0, min(c["n"], i0 + 256), device="cuda")
                for p0 in range(0, P, span):
                    p1 = min(P, p0 + span)
                    z = _probes(p1, pr, steps[a], e, seed, sparse, dense_from, p0)
                    ghat[e, p0:p1] += coef[a, e, pr] @ z
    ghat /= A * c["n"]
    if kind in ("update", "step", "body_step"):
        res = {"params": theta - lr * ghat}
        return res if losses is None else {"losses": losses[0], "coef": coef[0], **res}
    b1, b2 = _f32(ADAM["beta1"]), _f32(ADAM["beta2"])
    m, v = (x.double() for x in _moments(c, seed))
    g = ghat + _f32(ADAM["weight_decay"]) * theta
    m = b1 * m + (1 - b1) * g
    v = b2 * v + (1 - b2) * g * g
    mh, vh = m / (1 - b1 ** ADAM_T), v / (1 - b2 ** ADAM_T)
    res = {"params": theta - lr * mh / (vh.sqrt() + _f32(ADAM["delta"])), "m": m, "v": v}
    return res if losses is None else {"losses": losses, "coef": coef, **res}
