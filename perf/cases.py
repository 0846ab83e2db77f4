"""Performance cases: whole M-AVG rounds and meta-updates as a program that uses the engine calls
them, over the sizes of this repository's workloads (paper_2110_00625_b200/workloads.py), its
examples and its tests.

A case is one of three kinds, named after the handle's objective:
  "mlp"   one round (K local minibatch-SGD steps of P learners, then the meta-update) of an MLP
          dims[0]-...-dims[-1] given as a text "3072-512-512-10".  gemm: 0 = fp32 arithmetic,
          1 = bf16 operands on the tensor cores, 2 = bf16 operands on the CUDA cores (widths or batch
          sizes that mode 1 refuses).  x_bf16: the dataset is kept as bf16 on the device.  defer:
          deferred re-broadcast.  beta: learner-level momentum.  host: the model lives in pinned host
          memory (mavg_round_host).  loss: the program reads the round's mean loss each round.
  "pg"    one round of K seeded pseudo-gradient steps on P replicas of n parameters
  "meta"  one meta-update over P replicas of n parameters that the program wrote itself

run() is one call of that entry point; what comes back is the whole updated state: the global
model w, the momentum buffer v, the replica array, the learner momentum buffers where there are
any, and the mean loss where the program asked for it.
"""
import math

import numpy as np
import torch

import paper_2110_00625_b200 as m


def _mlp(dims, gemm, P, K, B, samples, lr=0.002, mu=0.9, x_bf16=False, defer=False, beta=0.0,
         host=False, loss=False):
    return dict(kind="mlp", dims=dims, gemm=gemm, P=P, K=K, B=B, samples=samples, lr=lr, mu=mu,
                x_bf16=x_bf16, defer=defer, beta=beta, host=host, loss=loss)


def _pg(n, P, K, mu=0.9, defer=True, beta=0.0):
    return dict(kind="pg", n=n, P=P, K=K, lr=0.05, mu=mu, sigma=math.sqrt(1e-3), defer=defer,
                beta=beta)


def _meta(n, P, mu=0.9, defer=False):
    return dict(kind="meta", n=n, P=P, mu=mu, defer=defer)


def listed():
    return [
        # The smallest workload: a tiny fp32 model trained on a small tabular dataset, the loss
        # printed every round.  Launch count and latency are all there is.
        dict(_mlp("32-64-10", 0, 4, 4, 32, 4096, lr=0.05, loss=True), name="tiny_fp32_round"),
        # A true-fp32 model of ordinary size with a batch size that is no power of two: the engine's
        # default arithmetic (gemm_bf16 = 0), e.g. the full-precision control run of a study.
        dict(_mlp("3072-512-512-10", 0, 4, 4, 100, 50000, lr=0.01, loss=True),
             name="cifar_fp32_round"),
        # bf16 operands with widths, batch and class count that the tensor-core path refuses.
        dict(_mlp("1000-333-100", 2, 6, 4, 50, 20000), name="odd_bf16_round"),
        # The CIFAR-shaped workload: latency chain of medium products, state about L2-sized.
        dict(_mlp("3072-512-512-10", 1, 8, 8, 128, 50000, x_bf16=True, defer=True),
             name="cifar_bf16_round"),
        # The same model in a sweep over the number of learners (48, the largest of the study).
        dict(_mlp("3072-512-512-10", 1, 48, 8, 64, 50000, mu=0.7, x_bf16=True),
             name="sweep_p48_round"),
        # The same model driven by a program that keeps it in host memory between rounds.
        dict(_mlp("3072-512-512-10", 1, 8, 8, 128, 50000, host=True), name="cifar_host_round"),
        # The large MLP: the flagship workload, masters stream through HBM every step.
        dict(_mlp("3072-2048-2048-2048-10", 1, 32, 16, 64, 50000, x_bf16=True, defer=True),
             name="large_round"),
        # The large MLP with learner-level momentum, fewer learners and steps.
        dict(_mlp("3072-2048-2048-2048-10", 1, 8, 4, 64, 50000, x_bf16=True, defer=True, beta=0.9),
             name="large_momentum_round"),
        # A full round at the size of a 25.6 M-parameter model with seeded gradients, averaging after
        # every step and after 64 steps.
        dict(_pg(25_600_000, 16, 1), name="pseudograd_k1_round"),
        dict(_pg(25_600_000, 16, 64), name="pseudograd_k64_round"),
        # The meta-update alone on an 11.2 M-parameter vector, few and many replicas.
        dict(_meta(11_200_000, 4), name="meta_p4"),
        dict(_meta(11_200_000, 64), name="meta_p64"),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _eight(v):
    return max(8, v // 8 * 8)


def draw(rng):
    kind = rng.choice(["tiny", "fp32", "odd", "tc", "tc", "tc_large", "pg", "meta"])
    if kind == "tiny":       # small fp32 models, any widths
        dims = [rng.randint(8, 80)] + [rng.randint(8, 128) for _ in range(rng.choice([1, 1, 2]))]
        dims.append(rng.randint(2, 16))
        return _mlp("-".join(map(str, dims)), 0, rng.randint(1, 8), rng.randint(1, 8),
                    rng.randint(1, 48), 4096, lr=0.05, mu=rng.choice([0.0, 0.9]), loss=rng.random() < 0.5,
                    defer=rng.random() < 0.3, beta=rng.choice([0.0, 0.0, 0.9]))
    if kind in ("fp32", "odd"):   # CUDA-core arithmetic at ordinary sizes, any widths
        gemm = 0 if kind == "fp32" else 2
        dims = [_log(rng, 300, 3072)] + [_log(rng, 100, 800) for _ in range(rng.choice([0, 1, 2]))]
        dims.append(rng.randint(2, 100))
        return _mlp("-".join(map(str, dims)), gemm, rng.randint(1, 8), rng.randint(1, 4),
                    rng.randint(16, 160), 20000, lr=0.01 if gemm == 0 else 0.002,
                    mu=rng.choice([0.0, 0.9]), loss=rng.random() < 0.5, x_bf16=gemm == 2 and rng.random() < 0.5, defer=rng.random() < 0.5)
    if kind == "tc":         # the CIFAR-shaped family
        width = _eight(_log(rng, 128, 800))
        dims = [_eight(_log(rng, 512, 3072))] + [width] * rng.choice([1, 2, 2])
        dims.append(rng.randint(2, 32))
        return _mlp("-".join(map(str, dims)), 1, _log(rng, 2, 48), _log(rng, 1, 16),
                    16 * rng.randint(1, 16), 30000, mu=rng.choice([0.0, 0.5, 0.9]),
                    x_bf16=rng.random() < 0.5, defer=rng.random() < 0.5,
                    beta=rng.choice([0.0, 0.0, 0.0, 0.9]), host=rng.random() < 0.2)
    if kind == "tc_large":   # the large-MLP family: masters larger than the L2
        width = _eight(_log(rng, 1000, 2048))
        dims = [_eight(_log(rng, 2000, 3072))] + [width] * rng.choice([2, 3]) + [10]
        return _mlp("-".join(map(str, dims)), 1, rng.randint(8, 32), rng.randint(2, 8),
                    16 * rng.randint(2, 8), 30000, x_bf16=True, defer=rng.random() < 0.7)
    n = _log(rng, 100_000, 25_600_000)
    if kind == "pg":
        return _pg(n, _log(rng, 2, 16), _log(rng, 1, 64), mu=rng.choice([0.0, 0.9]),
                   defer=rng.random() < 0.5, beta=rng.choice([0.0, 0.0, 0.9]))
    return _meta(min(n, 11_200_000), _log(rng, 2, 64), mu=rng.choice([0.0, 0.9]),
                 defer=rng.random() < 0.3)


# --------------------------------------------------------------------------------------- inputs

def _dims(case):
    return [int(d) for d in case["dims"].split("-")]


def _n(case):
    if case["kind"] != "mlp":
        return case["n"]
    d = _dims(case)
    return sum(d[l + 1] * d[l] + d[l + 1] for l in range(len(d) - 1))


def _gen(seed):
    return torch.Generator(device="cuda").manual_seed(1 + seed)


def _inputs(case, seed):
    """Device tensors: initial model w1 and, by kind, the dataset (x, y) or the replicas."""
    g = _gen(seed)

    def randn(*shape):
        return torch.randn(*shape, generator=g, device="cuda")

    if case["kind"] == "pg":
        return dict(w1=0.05 * randn(case["n"]))
    if case["kind"] == "meta":
        w1 = 0.05 * randn(case["n"])
        rep = randn(case["P"], case["n"]).mul_(0.1).add_(w1)
        return dict(w1=w1, rep=rep)
    d, S = _dims(case), case["samples"]
    parts = []
    for l in range(len(d) - 1):
        parts += [(randn(d[l + 1] * d[l]) * math.sqrt(2.0 / d[l])), torch.zeros(d[l + 1], device="cuda")]
    w1 = torch.cat(parts)
    if d[0] <= 80:           # unit-variance clusters with means N(0, 4)
        means = 2.0 * randn(d[-1], d[0])
        y = torch.randint(0, d[-1], (S,), generator=g, device="cuda")
        x = means[y] + randn(S, d[0])
    else:                    # N(0, 1) inputs labelled by a fixed random ReLU teacher
        x = randn(S, d[0])
        t1, t2 = randn(d[0], 256) / math.sqrt(d[0]), randn(256, d[-1])
        y = (torch.relu(x @ t1) @ t2).argmax(1)
    if case["x_bf16"]:
        x = x.bfloat16()
    return dict(w1=w1, x=x, y=y.to(torch.int32))


def prepare(case, seed):
    inp = _inputs(case, seed)
    if case["kind"] == "meta":
        g = m.Mavg(inp["w1"], P=case["P"], K=1, local_lr=0.1, mu=case["mu"],
                   objective=m.OBJ_NONE, defer_broadcast=case["defer"])
        g.replicas[:, :g.n] = inp["rep"]
        return dict(case=case, g=g)
    if case["kind"] == "pg":
        g = m.Mavg(inp["w1"], P=case["P"], K=case["K"], local_lr=case["lr"], mu=case["mu"],
                   seed=seed, objective=m.OBJ_PSEUDOGRAD, sigma=case["sigma"],
                   defer_broadcast=case["defer"], learner_momentum=case["beta"])
        return dict(case=case, g=g)
    g = m.Mavg(inp["w1"], P=case["P"], K=case["K"], local_lr=case["lr"], mu=case["mu"],
               B=case["B"], seed=seed, objective=m.OBJ_MLP, dims=_dims(case),
               gemm_bf16=case["gemm"], x=inp["x"], y=inp["y"], x_bf16=case["x_bf16"],
               defer_broadcast=case["defer"], learner_momentum=case["beta"])
    state = dict(case=case, g=g)
    if case["host"]:
        state["w"] = inp["w1"].cpu().pin_memory()
        state["v"] = torch.zeros(g.n).pin_memory()
    return state


def run(state):
    case, g = state["case"], state["g"]
    out = dict(w=g.w, v=g.v, replicas=g.replicas[:, :g.n])
    if case["kind"] == "meta":
        g.meta_update()
        return out
    if case["kind"] == "pg":
        g.round()
    elif case["host"]:
        out["loss"] = g.round_host(state["w"], state["v"])
        out["w"], out["v"] = state["w"], state["v"]
    elif case["loss"]:
        out["loss"] = g.round(want_loss=True)
    else:
        g.round()
    if g.u is not None:
        out["u"] = g.u[:, :g.n]
    return out


def work(case):
    n, P = _n(case), case["P"]
    byts = 16 * n                                      # w and v, read and written
    if case["kind"] == "meta":
        return dict(bytes=byts + 4 * P * n * (1 if case["defer"] else 2), flops=2 * P * n)
    byts += 4 * P * n                                  # the replica array, written
    if case["beta"]:
        byts += 8 * P * n                              # learner momentum, read and written
    if case["kind"] == "pg":
        return dict(bytes=byts, flops=2 * P * n * case["K"])
    d = _dims(case)
    rows = P * case["K"] * case["B"]
    byts += rows * (d[0] * (2 if case["x_bf16"] else 4) + 4)
    products = [d[l] * d[l + 1] for l in range(len(d) - 1)]
    return dict(bytes=byts, flops=2 * rows * (3 * sum(products) - products[0]))


def _open_branches(case):
    """Whether a round has so many (sample, hidden unit) pairs that one of them is likely to have a
    pre-activation that is zero to within fp32 rounding.  ReLU'(0) is a jump: that unit's weight row
    then differs by one sample's contribution between two equally correct fp32 sums (measured on
    cifar_fp32_round: v moves by 4e-4 to 1e-3 in the 2-norm, from 6e-6 without such a pair), and no
    single 64-bit value of w, v or the replicas exists to be compared with."""
    return case["P"] * case["K"] * case["B"] * sum(_dims(case)[1:-1]) > 1e5


def tolerance(case):
    if case["kind"] != "mlp":
        return {"rel": 4e-6, "max": 4e-5}
    if case["gemm"] == 0:
        # open ReLU branches as described above, else sums of a few thousand fp32 terms
        return {"rel": 4e-3, "max": 4e-1} if _open_branches(case) else {"rel": 2e-5, "max": 2e-3}
    # Two schedules of the library that differ in the order of their fp32 sums only: v differs by
    # 1e-3 to 6e-3 (largest element 2e-2 to 9e-2) after one and two rounds, the compound effect of
    # bf16 roundings and ReLU branches that fall the other way over K steps.
    return {"rel": 2e-2, "max": 4e-1}


# ----------------------------------------------------------------------- the same in 64 bits
# Algorithm 1 in plain torch float64 (integers for the index and gradient streams, which are
# defined by SplitMix64 as a counter-based generator, see include/mavg.h).

_G, _M = 0x9E3779B97F4A7C15, (1 << 64) - 1


def _mix(z):
    z = ((z ^ (z >> 30)) * 0xBF58476D1CE4E5B9) & _M
    z = ((z ^ (z >> 27)) * 0x94D049BB133111EB) & _M
    return z ^ (z >> 31)


def _fold(s, c):
    return _mix((s + (c + 1) * _G) & _M)


def _step_key(seed, tag, j, k, round_=1):
    return _fold(_fold(_fold(_fold(seed, tag), round_), j), k)


def _signed(v):
    return v - (1 << 64) if v >> 63 else v


def _shr(z, s):
    return (z >> s) & ((1 << (64 - s)) - 1)


def _variates(key, i, scale):
    """Irwin-Hall(4) variates of the elements i (int64 tensor), as float64."""
    z = (i + 1) * _signed(_G) + _signed(key)
    z = (z ^ _shr(z, 30)) * _signed(0xBF58476D1CE4E5B9)
    z = (z ^ _shr(z, 27)) * _signed(0x94D049BB133111EB)
    z = z ^ _shr(z, 31)
    s = (z & 65535) + (_shr(z, 16) & 65535) + (_shr(z, 32) & 65535) + _shr(z, 48)
    return (s - 131070).double() * scale


def _grad(d, w, x, y):
    """Mean loss of the batch and its gradient with respect to the flat parameters w."""
    L, off, layers, a = len(d) - 1, 0, [], [x]
    for l in range(L):
        W = w[off:off + d[l + 1] * d[l]].view(d[l + 1], d[l])
        off += W.numel()
        layers.append(W)
        z = a[-1] @ W.T + w[off:off + d[l + 1]]
        off += d[l + 1]
        a.append(torch.relu(z) if l < L - 1 else z)
    logp = torch.log_softmax(a[-1], 1)
    rows = torch.arange(len(y), device=y.device)
    loss = -logp[rows, y].mean()
    dz = logp.exp()
    dz[rows, y] -= 1.0
    dz /= len(y)
    parts = []
    for l in range(L - 1, -1, -1):
        parts += [dz.sum(0), (dz.T @ a[l]).reshape(-1)]
        if l:
            dz = (dz @ layers[l]) * (a[l] > 0)
    return loss, torch.cat(parts[::-1])


def exact(case, seed):
    open_ = case["kind"] == "mlp" and case["gemm"] == 0 and _open_branches(case)
    if open_ and not case["loss"]:
        return None
    inp = _inputs(case, seed)
    w1, P, n = inp["w1"].double(), case["P"], _n(case)
    mu = float(np.float32(case["mu"]))
    total = torch.zeros_like(w1)
    # replicas of a case that re-broadcasts are w itself; otherwise each learner's own result
    own = torch.empty(P, n, dtype=torch.float64, device="cuda") if case["defer"] else None
    us, losses = None, []
    if case["kind"] == "meta":
        for j in range(P):
            total += inp["rep"][j].double() - w1
            if own is not None:
                own[j] = inp["rep"][j].double()
    else:
        lr, beta = float(np.float32(case["lr"])), float(np.float32(case["beta"]))
        us = torch.empty(P, n, dtype=torch.float64, device="cuda") if beta else None
        if case["kind"] == "pg":
            i = torch.arange(n, device="cuda")
            sd = math.sqrt(4.0 * (65536.0 * 65536.0 - 1.0) / 12.0)
            scale = float(np.float32(float(np.float32(case["sigma"])) / sd))
        else:
            d, B, S = _dims(case), case["B"], case["samples"]
            x, y = inp["x"], inp["y"].long()
        for j in range(P):
            w, u = w1.clone(), torch.zeros_like(w1) if beta else None
            for k in range(1, case["K"] + 1):
                if case["kind"] == "pg":
                    g = _variates(_step_key(seed, 2, j, k), i, scale)
                else:
                    lo, hi = j * S // P, (j + 1) * S // P
                    key = _step_key(seed, 1, j, k)
                    idx = torch.tensor([lo + (((_fold(key, s) >> 32) * (hi - lo)) >> 32)
                                        for s in range(B)], device="cuda")
                    loss, g = _grad(d, w, x[idx].double(), y[idx])
                    losses.append(loss)
                if beta:
                    u.mul_(beta).sub_(g, alpha=lr)
                    w += u
                else:
                    w.sub_(g, alpha=lr)
            total += w - w1
            if own is not None:
                own[j] = w
            if beta:
                us[j] = u
    v = total / P                                      # the momentum buffer starts at zero
    w = w1 + v
    out = dict(w=w, v=v, replicas=own if own is not None else w.expand(P, n))
    if case["kind"] == "mlp" and (case["host"] or case["loss"]):
        out["loss"] = torch.stack(losses).mean().item()
    if us is not None:
        out["u"] = us
    if open_:
        out.update(dict.fromkeys(set(out) - {"loss"}))
    return out
