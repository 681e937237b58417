"""Workloads by which the speed of this framework is judged.

Each case is a call (or a short sequence of calls) that a VMC program makes on
one GPU through `paper_2310_04166_gb300`: the local energies of a sample set,
the gradient, the amplitudes, the connected set, or one whole pass.  Networks
are random-init (Gaussian weights of variance 1/fan_in, small biases) and the
Hamiltonians seeded integrals of molecular shape.  The sample sets follow the
network's own Born distribution: they are drawn here by a plain torch
autoregressive sampler, and the most frequent determinants are kept.

`exact` evaluates the same quantities in float64 with plain torch.
"""
from __future__ import annotations

import math
import random

import numpy as np
import torch

DEV = "cuda"
EVEN = 0x5555555555555555


# ---------------------------------------------------------------------------
# the cases
# ---------------------------------------------------------------------------

def _mlp(n, na, nb, form, width=128, hidden=3, **k):
    return dict(net="mlp", form=form, n=n, na=na, nb=nb, width=width, hidden=hidden, du=0, **k)


def _tf(n, na, nb, form, d, heads, blocks, **k):
    return dict(net="tf", form=form, n=n, na=na, nb=nb, d=d, heads=heads, blocks=blocks, du=0, **k)


def listed():
    return [
        # Local energies of a small molecule (water in a minimal basis: 14 qubits, nearly the whole
        # 441-determinant sector in the sample): a few thousand cheap amplitudes, launch and latency bound.
        _mlp(7, 5, 5, "bf16", call="energy", n_x=441, name="energy_mlp16_h2o"),
        # The largest sample set of the 16-bit MLP: 28 qubits at half filling (the largest problems of a batch),
        # about 1e8 connected determinants.
        _mlp(14, 7, 7, "bf16", call="energy", n_x=30000, name="energy_mlp16_28q"),
        # A medium molecule with the transformer ansatz (nitrogen in a minimal basis: 20 qubits), most of the sector
        # in the sample, as after a pass with 1e6 draws.
        _tf(10, 7, 7, "bf16", 64, 4, 2, call="energy", n_x=10816, name="energy_tf16_n2"),
        # Few samples of a large active space: 52 qubits, 33,507 connected determinants per sample, hardly any of them
        # in the sample set, deep transformer.
        _tf(26, 9, 9, "bf16", 128, 8, 4, call="energy", n_x=64, name="energy_tf16_52q"),
        # The plain FP32 form, as used to check the 16-bit one, with an odd sector and the DU pruning of the last slots.
        dict(_mlp(9, 4, 3, "fp32", call="energy", n_x=1500, name="energy_mlp32_du"), du=2),
        # The per-qubit complex NADE (FP32 only).
        dict(net="nade", form="fp32", n=7, na=5, nb=5, width=64, du=0, call="energy", n_x=441, name="energy_nade_h2o"),
        # Local energies of several independent problems of unequal sizes in one batched call.
        dict(call="batch", net="mlp", form="bf16", n_lo=6, n_hi=13, problems=8, n_x=4000, pick=5, width=128, hidden=3,
             name="energy_batch8"),
        # VMC gradient of the 16-bit MLP over a large sample set.
        _mlp(12, 6, 6, "bf16", call="grad", n_x=20000, name="grad_mlp16_24q"),
        # VMC gradient of the transformer over the nitrogen-shaped sample set.
        _tf(10, 7, 7, "bf16", 64, 4, 2, call="grad", n_x=10816, name="grad_tf16_n2"),
        # Connected determinants and matrix elements alone (a selected-CI step, or a user's own estimator).
        dict(call="connected", n=26, na=9, nb=9, n_x=256, name="connected_52q"),
        # One pass of the small molecule, as each iteration of a training run makes it: weights packed, samples drawn,
        # local energies and their statistics, gradient.
        _mlp(7, 5, 5, "bf16", call="step", n_samples=100000, n_x=0, name="step_mlp16_h2o"),
        # The same pass with the transformer and 1e6 draws.
        _tf(10, 7, 7, "bf16", 64, 4, 2, call="step", n_samples=1000000, n_x=0, name="step_tf16_n2"),
    ]


def _log_int(rng, lo, hi):
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng: random.Random):
    kind = rng.choice(["energy_mlp16", "energy_mlp16", "energy_tf16", "energy_tf16w", "energy_fp32", "energy_nade",
                       "batch", "grad_mlp16", "grad_tf16", "connected", "step", "logpsi"])

    def sector(lo, hi):
        n = rng.randint(lo, hi)
        na = rng.randint(1, n - 1)
        return n, na, na if rng.random() < 0.5 else rng.randint(1, n - 1)

    def rows(n, na, nb, lo, hi, most):  # samples such that the connected set stays below `most` determinants
        return _log_int(rng, lo, max(lo, min(hi, int(most / max(1, n_connected(n, na, nb))))))

    if kind == "energy_mlp16":
        n, na, nb = sector(4, 14)
        c = _mlp(n, na, nb, "bf16", rng.choice([64, 128]), rng.choice([2, 3]), call="energy",
                 n_x=rows(n, na, nb, 16, 30000, 1e8))
        c["du"] = rng.choice([0, 0, 0, 2])
        return c
    if kind == "energy_tf16":
        n, na, nb = sector(6, 14)
        heads = rng.choice([2, 4])
        return _tf(n, na, nb, "bf16", 64, heads, rng.choice([1, 2, 3]), call="energy",
                   n_x=rows(n, na, nb, 16, 11000, 5e6))
    if kind == "energy_tf16w":
        n, na, nb = sector(12, 26)
        return _tf(n, na, nb, "bf16", 128, rng.choice([4, 8]), rng.choice([2, 4]), call="energy",
                   n_x=rows(n, na, nb, 3, 300, 5e5))
    if kind == "energy_fp32":
        n, na, nb = sector(4, 10)
        if rng.random() < 0.5:
            c = _mlp(n, na, nb, "fp32", rng.choice([64, 128]), 2, call="energy", n_x=rows(n, na, nb, 16, 2000, 3e5))
            c["du"] = rng.choice([0, 1, 2])
            return c
        return _tf(n, na, nb, "fp32", rng.choice([32, 64]), 4, 2, call="energy", n_x=rows(n, na, nb, 16, 1000, 3e5))
    if kind == "energy_nade":
        n, na, nb = sector(4, 10)
        return dict(net="nade", form="fp32", n=n, na=na, nb=nb, width=rng.choice([32, 64]), du=0, call="energy",
                    n_x=rows(n, na, nb, 16, 1000, 2e5))
    if kind == "batch":
        return dict(call="batch", net="mlp", form="bf16", n_lo=6, n_hi=rng.randint(10, 13),
                    problems=rng.randint(2, 8), n_x=_log_int(rng, 100, 4000), pick=rng.randint(0, 999), width=128,
                    hidden=3)
    if kind == "grad_mlp16":
        n, na, nb = sector(4, 14)
        return _mlp(n, na, nb, "bf16", 128, rng.choice([2, 3]), call="grad", n_x=_log_int(rng, 33, 20000))
    if kind == "grad_tf16":
        n, na, nb = sector(6, 12)
        return _tf(n, na, nb, "bf16", 64, 4, rng.choice([1, 2]), call="grad", n_x=_log_int(rng, 33, 8000))
    if kind == "connected":
        n, na, nb = sector(4, 26)
        return dict(call="connected", n=n, na=na, nb=nb, n_x=rows(n, na, nb, 16, 20000, 8e6))
    if kind == "step":
        n, na, nb = sector(6, 10)
        return _mlp(n, na, nb, "bf16", call="step", n_samples=_log_int(rng, 10000, 500000), n_x=0)
    n, na, nb = sector(6, 14)
    if rng.random() < 0.5:
        return _mlp(n, na, nb, "bf16", call="logpsi", n_x=_log_int(rng, 100, 100000))
    return _tf(n, na, nb, "bf16", rng.choice([64, 128]), 4, 2, call="logpsi", n_x=_log_int(rng, 100, 20000))


# ---------------------------------------------------------------------------
# sizes
# ---------------------------------------------------------------------------

def n_connected(n, na, nb):
    sa, sb = na * (n - na), nb * (n - nb)
    c = math.comb
    return sa + sb + c(na, 2) * c(n - na, 2) + c(nb, 2) * c(n - nb, 2) + sa * sb


def _batch_problems(case):
    r = random.Random(case["pick"])
    out = []
    for _ in range(case["problems"]):
        n = r.randint(case["n_lo"], case["n_hi"])
        na = r.randint(1, n - 1)
        out.append(dict(_mlp(n, na, na, case["form"], case["width"], case["hidden"], call="energy", n_x=case["n_x"])))
    return out


def _position_flops(case):
    """FLOP of one slot's (or position's) network for one prefix, averaged over the slots."""
    n = case["n"]
    if case["net"] == "mlp":
        w = case["width"]
        return 2.0 * (2.0 * (n - 1) * w + (case["hidden"] - 1) * w * w + 8 * w)
    if case["net"] == "nade":
        w = case["width"]
        return 3 * (8.0 * w * w + 16 * w + 2 * n * w)
    d = case["d"]
    return case["blocks"] * (24.0 * d * d + 2.0 * (n + 1) * d) + 16 * d


def _param_count(case):
    n = case["n"]
    if case["net"] == "mlp":
        w, h = case["width"], case["hidden"]
        return sum(4 * p * w + w + (h - 1) * (w * w + w) + 8 * w + 8 for p in range(n))
    if case["net"] == "nade":
        w = case["width"]
        return sum(2 * (w * i + w + w * w + w + 2 * w + 2) for i in range(2 * n))
    d = case["d"]
    return 5 * d + n * d + case["blocks"] * (12 * d * d + 13 * d) + 2 * d + 8 * d + 8


def work(case):
    """What one pass cannot do without.  A local energy needs the amplitude of every distinct determinant of the
    samples' connected sets once (counted as if the sets fell at random into the sector), and of each at least one
    network position that no other shares; then one complex term per connected determinant."""
    if case["call"] == "batch":
        ws = [work(c) for c in _batch_problems(case)]
        return {k: sum(w[k] for w in ws) for k in ("bytes", "flops")}
    n, na, nb = case["n"], case["na"], case["nb"]
    K = n_connected(n, na, nb)
    sector = math.comb(n, na) * math.comb(n, nb)
    if case["call"] == "connected":
        m = case["n_x"]
        return {"bytes": m * K * 17.0 + m * 16.0 + 8.0 * n**4, "flops": 2.0 * m * K}
    P = 4.0 * _param_count(case)
    n_x = min(case["n_x"] or case["n_samples"], sector)
    f = _position_flops(case)
    if case["call"] == "logpsi":
        return {"bytes": P + 16.0 * n_x, "flops": f * n_x}
    if case["call"] == "grad":
        return {"bytes": 2 * P + 32.0 * n_x, "flops": 3 * f * n_x}
    distinct = sector * -math.expm1(-n_x * (K + 1.0) / sector)
    energy = {"bytes": P + 32.0 * n_x + 8.0 * n**4, "flops": f * distinct + 8.0 * n_x * K}
    if case["call"] == "energy":
        return energy
    return {"bytes": energy["bytes"] + P + 16.0 * n_x, "flops": energy["flops"] + 3 * f * n_x}


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------

def _integrals(rng, n):
    h = np.zeros((n, n))
    iu = np.triu_indices(n, 1)
    h[iu] = rng.normal(0.0, 0.05, len(iu[0]))
    h = h + h.T
    h[np.diag_indices(n)] = np.linspace(-2.0, 1.0, n)
    B = rng.normal(0.0, 0.1, (2 * n, n, n))
    B = np.triu(B) + np.triu(B, 1).transpose(0, 2, 1)
    B = B.reshape(2 * n, n * n)
    return h, (B.T @ B).reshape(n, n, n, n)


def _bf16(a):
    return torch.tensor(a, dtype=torch.float32).to(torch.bfloat16).to(torch.float32).numpy()


def _params(rng, case):
    """Flat float32 parameters of a random-init network (the transformer's are bfloat16 values)."""
    n, parts = case["n"], []
    if case["net"] == "mlp":
        w = case["width"]
        for p in range(n):
            for k in range(case["hidden"] + 1):
                o, i = (w if k < case["hidden"] else 8), (4 * p if k == 0 else w)
                if i:
                    parts.append(rng.normal(0, 1 / math.sqrt(i), o * i))
                parts.append(rng.normal(0, 0.2, o))
        return np.concatenate(parts).astype(np.float32)
    if case["net"] == "nade":
        w = case["width"]
        for i in range(2 * n):
            for o, k in ((w, i), (w, w), (2, w)):
                parts.append(rng.normal(0, 1 / math.sqrt(2 * max(k, 1)), 2 * o * k))
                parts.append(rng.normal(0, 0.1, 2 * o))
        return np.concatenate(parts).astype(np.float32)
    d = case["d"]
    parts += [rng.normal(0, 1, 5 * d), rng.normal(0, 1, n * d)]
    for _ in range(case["blocks"]):
        parts += [1 + rng.normal(0, 0.1, d), rng.normal(0, 0.1, d)]
        for _ in range(4):
            parts += [rng.normal(0, 1 / math.sqrt(d), d * d), rng.normal(0, 0.1, d)]
        parts += [1 + rng.normal(0, 0.1, d), rng.normal(0, 0.1, d)]
        parts += [rng.normal(0, 1 / math.sqrt(d), 4 * d * d), rng.normal(0, 0.1, 4 * d)]
        parts += [rng.normal(0, 1 / math.sqrt(4 * d), 4 * d * d), rng.normal(0, 0.1, d)]
    parts += [1 + rng.normal(0, 0.1, d), rng.normal(0, 0.1, d)]
    parts += [rng.normal(0, 1 / math.sqrt(d), 8 * d), rng.normal(0, 0.1, 8)]
    return _bf16(np.concatenate(parts))


def _samples(case, flat, seed):
    """Unique determinants drawn from the network's Born distribution, the most frequent `n_x` of them in the order in
    which a tree sampler emits them, and their counts."""
    n, na, nb = case["n"], case["na"], case["nb"]
    sector = math.comb(n, na) * math.comb(n, nb)
    draws = 1000000 if case["n_x"] > sector // 3 else max(4096, 4 * case["n_x"])
    net = _Net(case, flat.to(torch.float32))
    gen = torch.Generator(device=DEV)
    gen.manual_seed(seed + 77)
    x = torch.zeros(draws, dtype=torch.int64, device=DEV)
    with torch.no_grad():
        for p in range(n):
            uniq, inv = torch.unique(x, return_inverse=True)
            out = net.slot(uniq, p)
            logit = torch.where(_physical(case, uniq, p), out[:, :4], torch.full_like(out[:, :4], -math.inf))
            c = torch.softmax(logit.double(), -1).cumsum(-1)
            u = torch.rand(draws, generator=gen, device=DEV, dtype=torch.float64)
            ok = _physical(case, uniq, p)
            v = (u[:, None] * c[inv, -1:] >= c[inv, :3]).sum(-1)
            last = 3 - ok.flip(-1).to(torch.int64).argmax(-1)  # rounding never picks a masked outcome
            v = torch.minimum(v, last[inv])
            x = x | (v << (2 * p))
    x, cnt = torch.unique(x, return_counts=True)
    want = min(case["n_x"], sector)
    if x.numel() > want:
        keep = torch.sort(cnt, descending=True, stable=True).indices[:want]
        x, cnt = x[keep], cnt[keep]
    elif x.numel() < want:  # a longer pass would also have met these, once
        strings = [torch.combinations(torch.arange(n, device=DEV), ne) for ne in (na, nb)]
        a, b = ((1 << (2 * c + s)).sum(1) for s, c in enumerate(strings))
        rest = (a[:, None] + b).reshape(-1)
        rest = rest[~torch.isin(rest, x)][:want - x.numel()]
        x, cnt = torch.cat([x, rest]), torch.cat([cnt, torch.ones_like(rest)])
    key = torch.zeros_like(x)
    for p in range(n):
        key = key * 4 + ((x >> (2 * p)) & 3)
    order = torch.argsort(key)
    return x[order].contiguous(), cnt[order].contiguous()


def _random_determinants(case, seed):
    n, gen = case["n"], torch.Generator(device=DEV)
    gen.manual_seed(seed + 55)
    x = torch.zeros(case["n_x"], dtype=torch.int64, device=DEV)
    bias = torch.linspace(1.5, -1.5, n, device=DEV)
    for s, ne in ((0, case["na"]), (1, case["nb"])):
        g = bias - torch.log(-torch.log(torch.rand(case["n_x"], n, generator=gen, device=DEV)))
        x += (1 << (2 * torch.topk(g, ne, dim=1).indices + s)).sum(1)
    return x


def _inputs(case, seed):
    rng = np.random.default_rng(seed)
    h, g = _integrals(rng, case["n"])
    if case["call"] == "connected":
        return dict(h=h, g=g, x=_random_determinants(case, seed))
    flat = torch.tensor(_params(rng, case), device=DEV)
    d = dict(h=h, g=g, flat=flat)
    if case["call"] != "step":
        d["x"], d["cnt"] = _samples(case, flat, seed)
    if case["call"] == "grad":  # local energies such as the samples of a partly trained network have
        gen = torch.Generator(device=DEV)
        gen.manual_seed(seed + 99)
        m = d["x"].numel()
        e = torch.randn(2, m, generator=gen, device=DEV, dtype=torch.float64)
        d["ere"], d["eim"] = -6.0 + 0.8 * e[0], 0.5 * e[1]
        d["stats"] = _stats(torch.complex(d["ere"], d["eim"]), d["cnt"])
    return d


def _stats(e, cnt):
    w = cnt.double() / cnt.sum()
    mean = (w * e).sum()
    var = (w * (e - mean).abs() ** 2).sum()
    return torch.stack([mean.real, mean.imag, var, cnt.sum().double()])


def _model(A, case, flat):
    if case["net"] == "mlp":
        return A.Model.mlp(case["n"], case["width"], case["hidden"], flat, case["form"])
    if case["net"] == "nade":
        return A.Model.nade(case["n"], case["width"], flat)
    return A.Model.transformer(case["n"], case["d"], case["heads"], case["blocks"], flat, case["form"])


def _ham(A, case, d):
    ham = A.Hamiltonian(d["h"], d["g"], 0.0, case["na"], case["nb"])
    return ham.set_pruning(case["du"]) if case.get("du") else ham


def prepare(case, seed):
    import paper_2310_04166_gb300 as A

    if case["call"] == "batch":
        items = []
        for k, c in enumerate(_batch_problems(case)):
            d = _inputs(c, seed + 1009 * k)
            items.append(dict(model=_model(A, c, d["flat"]), ham=_ham(A, c, d), x=d["x"], counts=d["cnt"]))
        batch = A.EnergyBatch(len(items))
        return dict(A=A, call="batch", batch=batch, items=items)
    d = _inputs(case, seed)
    state = dict(A=A, call=case["call"], ham=_ham(A, case, d), **{k: d[k] for k in d if k not in ("h", "g", "flat")})
    if case["call"] != "connected":
        state["model"] = _model(A, case, d["flat"])
    if case["call"] == "step":  # the buffers that a training loop keeps from one iteration to the next
        model, ham, m = state["model"], state["ham"], case["n_samples"]
        cap = min(m, ham.sector_dim)
        i64, f64 = dict(dtype=torch.int64, device=DEV), dict(dtype=torch.float64, device=DEV)
        state.update(n_samples=m, seed=seed, x=torch.zeros(cap, **i64), cnt=torch.zeros(cap, **i64),
                     nu=torch.zeros(1, **i64), ere=torch.zeros(cap, **f64), eim=torch.zeros(cap, **f64),
                     stats=torch.zeros(4, **f64), g=torch.zeros(model.n_params, device=DEV),
                     ws_s=torch.empty(A.sample_workspace_bytes(model, ham, m), dtype=torch.uint8, device=DEV),
                     ws_e=torch.empty(A.local_energy_workspace_bytes(model, ham, cap), dtype=torch.uint8, device=DEV),
                     ws_g=torch.empty(A.grad_workspace_bytes(model, ham, cap), dtype=torch.uint8, device=DEV))
    return state


def run(state):
    A, call = state["A"], state["call"]
    if call == "batch":
        return state["batch"].local_energy(state["items"])
    if call == "connected":
        return A.connected(state["ham"], state["x"])
    if call == "logpsi":
        return A.logpsi(state["model"], state["ham"], state["x"])
    if call == "energy":
        return A.local_energy(state["model"], state["ham"], state["x"], state["cnt"])
    if call == "grad":
        return A.grad(state["model"], state["ham"], state["x"], state["cnt"], state["ere"], state["eim"],
                      state["stats"])
    model, ham, x, cnt, nu = (state[k] for k in ("model", "ham", "x", "cnt", "nu"))
    model.sync()  # the weights changed: an optimiser step lies between two passes
    A.sample_into(model, ham, state["n_samples"], state["seed"], 0, x, cnt, nu, state["ws_s"])
    out = state["ere"], state["eim"], state["stats"]
    A.local_energy(model, ham, x, cnt, workspace=state["ws_e"], n_dev=nu, out=out)
    A.grad(model, ham, x, cnt, *out, workspace=state["ws_g"], n_dev=nu, out=state["g"])
    return (nu, x, cnt) + out + (state["g"],)


# ---------------------------------------------------------------------------
# the same quantities in float64
# ---------------------------------------------------------------------------

def _popc(x):
    """Set bits of non-negative int64 values."""
    x = x - ((x >> 1) & EVEN)
    x = (x & 0x3333333333333333) + ((x >> 2) & 0x3333333333333333)
    x = (x + (x >> 4)) & 0x0F0F0F0F0F0F0F0F
    return (x * 0x0101010101010101 >> 56) & 0xFF


def _physical(case, x, p):
    """[B, 4]: the outcomes of slot p that can still reach the sector after the prefix of x."""
    n, na, nb = case["n"], case["na"], case["nb"]
    below = x & ((1 << (2 * p)) - 1)
    a, b = _popc(below & EVEN), _popc((below >> 1) & EVEN)
    v = torch.arange(4, device=x.device)
    a, b, left = a[:, None] + (v & 1), b[:, None] + (v >> 1), n - 1 - p
    return (a <= na) & (b <= nb) & (a + left >= na) & (b + left >= nb)


class _Net:
    """The three ansatz networks in plain torch, in the dtype of the flat parameters."""

    def __init__(self, case, flat):
        self.case, self.dt, self.off, self.flat = case, flat.dtype, 0, flat
        n = case["n"]
        if case["net"] == "mlp":
            w, h = case["width"], case["hidden"]
            self.slots = [[(self._take(w if k < h else 8, 4 * p if k == 0 else w), self._take(w if k < h else 8))
                           for k in range(h + 1)] for p in range(n)]
        elif case["net"] == "nade":
            w = case["width"]
            self.qubits = [[(self._ctake(o, k), self._ctake(o)) for o, k in ((w, i), (w, w), (2, w))]
                           for i in range(2 * n)]
        else:
            d = case["d"]
            self.tok, self.pos, self.layers = self._take(5, d), self._take(n, d), []
            for _ in range(case["blocks"]):
                L = dict(g1=self._take(d), s1=self._take(d))
                for k in "qkvo":
                    L["w" + k], L["b" + k] = self._take(d, d), self._take(d)
                L["g2"], L["s2"] = self._take(d), self._take(d)
                L["w1"], L["b1"], L["w2"], L["b2"] = self._take(4 * d, d), self._take(4 * d), self._take(d, 4 * d), self._take(d)
                self.layers.append(L)
            self.gf, self.sf, self.wh, self.bh = self._take(d), self._take(d), self._take(8, d), self._take(8)

    def _take(self, *shape):
        k = math.prod(shape)
        self.off += k
        return self.flat[self.off - k:self.off].view(*shape)

    def _ctake(self, *shape):
        return torch.view_as_complex(self._take(*shape, 2))

    def slot(self, x, p):
        """[B, 8] outputs of slot p for the prefixes of x (the NADE's already masked and normalised)."""
        if self.case["net"] == "mlp":
            v = (x[:, None] >> (2 * torch.arange(p, device=x.device))) & 3
            z = torch.nn.functional.one_hot(v, 4).reshape(x.numel(), 4 * p).to(self.dt)
            for k, (W, b) in enumerate(self.slots[p]):
                z = z @ W.T + b
                if k < self.case["hidden"]:
                    z = torch.tanh(z)
            return z
        if self.case["net"] == "tf":
            return torch.cat([self.positions(c, p + 1)[:, p] for c in torch.split(x, 16384)])
        bits = (x[:, None] >> torch.arange(2 * p, device=x.device)) & 1
        cdt = torch.complex128 if self.dt == torch.float64 else torch.complex64
        ok = _physical(self.case, x, p)

        def qubit(i, bits, allowed):
            (W1, b1), (W2, b2), (W3, b3) = self.qubits[i]
            z = torch.tanh(bits.to(cdt) @ W1.T + b1) @ W2.T + b2
            z = torch.complex(torch.nn.functional.leaky_relu(z.real, 0.01), torch.nn.functional.leaky_relu(z.imag, 0.01))
            z = z @ W3.T + b3
            re = torch.where(allowed, z.real, torch.full_like(z.real, -math.inf))
            lse = 0.5 * torch.logsumexp(2 * re, -1, keepdim=True)
            return re - torch.where(torch.isfinite(lse), lse, torch.zeros_like(lse)), z.imag

        r0, i0 = qubit(2 * p, bits, torch.stack([ok[:, 0] | ok[:, 2], ok[:, 1] | ok[:, 3]], 1))
        cols = [None] * 8
        for a in (0, 1):
            col = torch.full_like(x[:, None], a)
            r1, i1 = qubit(2 * p + 1, torch.cat([bits, col], 1), torch.stack([ok[:, a], ok[:, a + 2]], 1))
            for b in (0, 1):
                cols[a + 2 * b], cols[4 + a + 2 * b] = 2 * (r0[:, a] + r1[:, b]), i0[:, a] + i1[:, b]
        return torch.stack(cols, 1)

    def positions(self, x, T):
        """[B, T, 8] outputs of the transformer's first T positions."""
        d, H, B = self.case["d"], self.case["heads"], x.numel()
        tok = torch.full((B, T), 4, dtype=torch.int64, device=x.device)
        if T > 1:
            tok[:, 1:] = (x[:, None] >> (2 * torch.arange(T - 1, device=x.device))) & 3
        h = self.tok[tok] + self.pos[:T]
        ln = lambda h, g, s: torch.nn.functional.layer_norm(h, (d,), g, s, 1e-5)
        causal = torch.ones(T, T, dtype=torch.bool, device=x.device).tril()
        for L in self.layers:
            a = ln(h, L["g1"], L["s1"])
            q, k, v = ((a @ L["w" + c].T + L["b" + c]).view(B, T, H, d // H).transpose(1, 2) for c in "qkv")
            s = (q @ k.transpose(-1, -2)) / math.sqrt(d // H)
            s = torch.softmax(s.masked_fill(~causal, -math.inf), -1)
            h = h + (s @ v).transpose(1, 2).reshape(B, T, d) @ L["wo"].T + L["bo"]
            h = h + torch.relu(ln(h, L["g2"], L["s2"]) @ L["w1"].T + L["b1"]) @ L["w2"].T + L["b2"]
        return ln(h, self.gf, self.sf) @ self.wh.T + self.bh

    def terms(self, x, out, p):
        """log|psi_p(v_p)| and its phase for rows x with outputs out of slot p."""
        ok = _physical(self.case, x, p)
        v = ((x >> (2 * p)) & 3)[:, None]
        if self.case["net"] == "nade":
            return 0.5 * out.gather(1, v)[:, 0], out.gather(1, v + 4)[:, 0]
        norm = ok if p < self.case["n"] - self.case["du"] else torch.ones_like(ok)
        lse = torch.logsumexp(torch.where(norm, out[:, :4], torch.full_like(out[:, :4], -math.inf)), -1)
        return 0.5 * (out[:, :4].gather(1, v)[:, 0] - lse), out.gather(1, v + 4)[:, 0]

    def log_psi(self, x):
        """log|psi| and phase of sector determinants; every distinct prefix is evaluated once."""
        n, la, ph = self.case["n"], 0.0, 0.0
        if self.case["net"] == "tf":
            las, phs = [], []
            for c in torch.split(x, 8192):
                out = self.positions(c, n)
                t = [self.terms(c, out[:, p], p) for p in range(n)]
                las.append(sum(a for a, _ in t))
                phs.append(sum(b for _, b in t))
            return torch.cat(las), torch.cat(phs)
        for p in range(n):
            uniq, inv = torch.unique(x & ((1 << (2 * p)) - 1), return_inverse=True)
            out = torch.cat([self.slot(c, p) for c in torch.split(uniq, 1 << 17)])
            tl, tp = self.terms(x, out[inv], p)
            la, ph = la + tl, ph + tp
        return la, ph


def _connected(case, h, g, x):
    """x' [B, K], H_xx' [B, K], the first differing slot [B, K] and H_xx [B] in the library's order."""
    n, B, dev = case["n"], x.numel(), x.device
    q = torch.arange(2 * n, device=dev)
    occ = (x[:, None] >> q) & 1
    below = torch.cumsum(occ, 1) - occ  # occupied spin-orbitals below q
    order, part = [], []
    for s, ne in ((0, case["na"]), (1, case["nb"])):
        o = torch.argsort(1 - occ[:, s::2], dim=1, stable=True)
        order.append((o[:, :ne], o[:, ne:]))
    J = torch.einsum("iijj->ij", g)
    X = torch.einsum("ijji->ij", g)
    diag = torch.zeros(B, dtype=torch.float64, device=dev)
    for s in (0, 1):
        o = order[s][0]
        diag += h.diagonal()[o].sum(1)
        for t in (0, 1):
            u = order[t][0]
            diag += 0.5 * J[o[:, :, None], u[:, None, :]].sum((1, 2))
            if s == t:
                diag -= 0.5 * X[o[:, :, None], u[:, None, :]].sum((1, 2))
    Jaij = torch.einsum("aijj->aij", g).contiguous()
    Xaij = torch.einsum("ajji->aij", g).contiguous()

    def count(idx):  # occupied spin-orbitals below idx [B, k]
        return below.gather(1, idx)

    for s in (0, 1):
        o, v = order[s]
        i = o[:, :, None].expand(B, o.shape[1], v.shape[1]).reshape(B, -1)
        a = v[:, None, :].expand(B, o.shape[1], v.shape[1]).reshape(B, -1)
        val = h[a, i].clone()
        for t in (0, 1):
            for k in range(order[t][0].shape[1]):
                j = order[t][0][:, k:k + 1].expand_as(i)
                val += Jaij[a, i, j]
                if t == s:
                    val -= Xaij[a, i, j]
        I, A = 2 * i + s, 2 * a + s
        sg = count(I) + count(A) - (I < A).to(torch.int64)
        part.append((x[:, None] ^ (1 << I) ^ (1 << A), torch.where(sg % 2 == 1, -val, val), torch.minimum(i, a)))

    def doubles(i, j, a, b, I, Jq, Aq, Bq, val):
        lt = lambda u, w: (u < w).to(torch.int64)
        sg = count(I) + count(Jq) - lt(I, Jq) + count(Bq) - lt(I, Bq) - lt(Jq, Bq)
        sg = sg + count(Aq) - lt(I, Aq) - lt(Jq, Aq) + lt(Bq, Aq)
        first = torch.minimum(torch.minimum(i, j), torch.minimum(a, b))
        part.append((x[:, None] ^ (1 << I) ^ (1 << Jq) ^ (1 << Aq) ^ (1 << Bq),
                     torch.where(sg % 2 == 1, -val, val), first))

    for s in (0, 1):
        o, v = order[s]
        po, pv = torch.combinations(torch.arange(o.shape[1], device=dev), 2), torch.combinations(
            torch.arange(v.shape[1], device=dev), 2)
        if len(po) == 0 or len(pv) == 0:
            continue
        io = po.repeat_interleave(len(pv), 0)
        iv = pv.repeat(len(po), 1)
        i, j, a, b = o[:, io[:, 0]], o[:, io[:, 1]], v[:, iv[:, 0]], v[:, iv[:, 1]]
        doubles(i, j, a, b, 2 * i + s, 2 * j + s, 2 * a + s, 2 * b + s, g[a, i, b, j] - g[a, j, b, i])
    (oa, va), (ob, vb) = order
    grid = torch.cartesian_prod(*(torch.arange(t.shape[1], device=dev) for t in (oa, va, ob, vb)))
    if len(grid):
        i, a, j, b = oa[:, grid[:, 0]], va[:, grid[:, 1]], ob[:, grid[:, 2]], vb[:, grid[:, 3]]
        doubles(i, j, a, b, 2 * i, 2 * j + 1, 2 * a, 2 * b + 1, g[a, i, b, j])
    return tuple(torch.cat(t, 1) for t in zip(*part)) + (diag,)


def _exact_energy(case, d):
    h, g = (torch.tensor(d[k], device=DEV) for k in ("h", "g"))
    x = d["x"]
    net = _Net(case, d["flat"].double())
    step = max(1, int(3e6 / max(1, n_connected(case["n"], case["na"], case["nb"]))))
    chunks = torch.split(x, step)
    uniq = torch.unique(x)
    for k in range(0, len(chunks), 8):
        uniq = torch.unique(torch.cat([uniq] + [torch.unique(_connected(case, h, g, c)[0]) for c in chunks[k:k + 8]]))
    la, ph = net.log_psi(uniq)
    out = []
    for c in chunks:
        xp, hv, _, diag = _connected(case, h, g, c)
        r, o = torch.searchsorted(uniq, xp.reshape(-1)).view(xp.shape), torch.searchsorted(uniq, c)
        dl, dp = la[r] - la[o][:, None], ph[r] - ph[o][:, None]
        w = hv * torch.exp(dl)
        out.append(torch.complex(diag + (w * torch.cos(dp)).sum(1), (w * torch.sin(dp)).sum(1)))
    e = torch.cat(out)
    return e.real.contiguous(), e.imag.contiguous(), _stats(e, d["cnt"])


def _affordable(case):
    """Whether the float64 evaluation stays within a few seconds."""
    if case["call"] == "step":
        return False
    m = case["n_x"] * (n_connected(case["n"], case["na"], case["nb"]) if case["call"] == "energy" else 1)
    sector = math.comb(case["n"], case["na"]) * math.comb(case["n"], case["nb"])
    if case.get("net") == "tf":
        return min(m, sector) * case["n"] * _position_flops(case) < 5e12
    return m < 2e8


def exact(case, seed):
    if case["call"] == "batch":
        cs = _batch_problems(case)
        return [_exact_energy(c, _inputs(c, seed + 1009 * k)) for k, c in enumerate(cs)]
    if not _affordable(case):
        return None
    d = _inputs(case, seed)
    if case["call"] == "connected":
        h, g = (torch.tensor(d[k], device=DEV) for k in ("h", "g"))
        parts = [_connected(case, h, g, c) for c in torch.split(d["x"], 64)]
        _, hv, _, diag = (torch.cat(t) for t in zip(*parts))
        return None, hv, None, diag
    if case["call"] == "energy":
        return _exact_energy(case, d)
    with torch.no_grad():
        if case["call"] == "logpsi":
            return _Net(case, d["flat"].double()).log_psi(d["x"])
    flat = d["flat"].double().requires_grad_(True)
    w = 2.0 * d["cnt"].double() / d["stats"][3]
    total = torch.zeros_like(flat)
    for k in torch.split(torch.arange(d["x"].numel(), device=DEV), 4096):
        la, ph = _Net(case, flat).log_psi(d["x"][k])
        loss = (w[k] * (d["ere"][k] - d["stats"][0]) * la).sum() + (w[k] * (d["eim"][k] - d["stats"][1]) * ph).sum()
        total += torch.autograd.grad(loss, flat)[0]
    return total
