"""What is measured: passes through the public entry points of the trial-loop library, over the
range of networks, sample counts and calls that training programs use.

A case is a network with its data and one kind of call:

* "run"       a training job of n trials from given parameters: mca_set_params (a checkpoint, the
              next mini-batch's handle or a fresh start; it recomputes every cached field with a full
              forward pass), mca_run, the updated parameters and the loss. Starting every pass from
              the same parameters keeps the work of a pass the same.
* "eval"      mca_eval_candidates: the loss changes of n given single-weight changes, no commit
              (a caller with its own acceptance rule, or looking at the loss landscape)
* "trials"    mca_eval_trials: one shard's step of a chain whose samples are split over handles
* "channels"  mca_set_params, then n multi-weight channel trials (a full forward pass each)

Inputs are drawn on the GPU from the seed alone: images with 20 % non-zero pixels, labels of a
random teacher net, symbols of an order-2 Markov chain.
"""
import math

import numpy as np
import torch

from paper_2607_08406_gb300 import mca
from paper_2607_08406_gb300 import workloads as W

DENSITY = 0.2          # share of non-zero input features

# transfer functions, loss, weight storage and initial weights of the networks in use
STYLES = {
    "tanh_mse": dict(act="tanh", out="sigmoid", loss="mse_onehot", wkind="fp32", init=0.1),
    "tanh_ce": dict(act="tanh", out="identity", loss="softmax_ce", wkind="fp32", init=0.05),
    "relu_ce": dict(act="relu", out="identity", loss="softmax_ce", wkind="fp32", init=0.05),
    "ternary": dict(act="gaussian", out="sigmoid", loss="mse_onehot", wkind="ternary_i8", init=0.0),
    "masked": dict(act="gaussian", out="sigmoid", loss="mse_onehot", wkind="masked_fp32", init=0.0),
}


def _mlp(call, style, N, hidden, depth=1, D=784, C=10, K=64, n=64, op="replace", beta=0.0):
    """beta = 0: the greedy rule."""
    return {"net": "mlp", "call": call, "style": style, "N": N, "hidden": hidden, "depth": depth,
            "D": D, "C": C, "K": K, "n": n, "op": op, "beta": beta}


def _tfm(call, B, n, vocab=65, ctx=64, d=128, layers=2, heads=4, ff=512, act="gelu", K=64):
    return {"net": "tfm", "call": call, "B": B, "n": n, "vocab": vocab, "ctx": ctx, "d": d,
            "layers": layers, "heads": heads, "ff": ff, "act": act, "K": K}


def listed():
    out = []

    def add(name, case):
        out.append(dict(case, name=name))

    # one batch of a sharded chain on the smallest net: latency and launches
    add("trials_small", _mlp("trials", "tanh_mse", 1000, 64, K=16, n=16))
    # a short job of the smallest net
    add("run_small", _mlp("run", "tanh_mse", 1000, 64, K=16, n=2000))
    # the wide net of the benchmark: a stretch of its job, and explicit candidates on it
    add("run_wide", _mlp("run", "tanh_ce", 60000, 16384, n=4000))
    add("eval_wide", _mlp("eval", "tanh_ce", 60000, 16384, n=64))
    # discrete weights at full size
    add("run_ternary", _mlp("run", "ternary", 60000, 4096, n=4000))
    # pruning of an odd-sized net
    add("run_masked_ragged", _mlp("run", "masked", 12347, 1001, D=391, C=7, K=33, n=3000))
    # half of the training set as a mini-batch, ReLU, small perturbations, Metropolis rule
    add("run_minibatch_relu", _mlp("run", "relu_ce", 30000, 2048, n=2000, op="perturb", beta=1e5))
    # the 24-layer net; a small net of another width
    add("run_deep", _mlp("run", "tanh_ce", 10000, 256, depth=24, K=128, n=96))
    add("run_deep_narrow", _mlp("run", "tanh_ce", 3001, 100, depth=5, K=32, n=64))
    # multi-weight trials of the 24-layer net: the full forward pass
    add("channels_deep", _mlp("channels", "tanh_ce", 10000, 256, depth=24, n=8))
    # the character-level Transformer, and a small one of other sizes
    add("run_tfm", _tfm("run", 256, 128))
    add("run_tfm_ragged", _tfm("run", 33, 48, vocab=50, ctx=48, d=96, layers=1, ff=200, K=16))
    return out


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    fam = rng.choice(["mlp2", "mlp2", "mlp2", "deep", "deep", "tfm"])
    call = rng.choice(["run", "run", "run", "eval", "trials"])
    if fam == "mlp2":
        style = rng.choice(["tanh_mse", "tanh_ce", "relu_ce", "ternary", "masked"])
        N = _log_int(rng, 1000, 60000)
        H = _log_int(rng, 64, 16384)
        if rng.random() < 0.5:
            H = max(64, H // 64 * 64)
        beta = _log_int(rng, 1000, 1000000) if rng.random() < 0.3 else 0.0
        op = "perturb" if rng.random() < 0.3 else "replace"
        n = _log_int(rng, 200, 4000) if call == "run" else rng.randint(8, 128)
        return _mlp(call, style, N, H, D=rng.choice([784, 784, rng.randint(100, 784)]),
                    C=rng.choice([10, 10, rng.randint(2, 14)]), K=rng.choice([16, 64, 128]), n=n,
                    op=op, beta=float(beta))
    if fam == "deep":
        # mostly the 256-wide nets; other widths are small nets
        if rng.random() < 0.7:
            H, depth, N = 256, rng.randint(2, 24), _log_int(rng, 500, 10000)
            n = _log_int(rng, 16, 96) if call == "run" else rng.randint(8, 64)
        else:
            H, depth, N = rng.randint(32, 255), rng.randint(2, 6), _log_int(rng, 500, 4000)
            n = _log_int(rng, 16, 64)
        if rng.random() < 0.2:
            call, n = "channels", rng.randint(2, 8)
        return _mlp(call, "tanh_ce", N, H, depth=depth, K=rng.choice([32, 128]), n=n)
    if rng.random() < 0.75:
        n = _log_int(rng, 16, 128) if call == "run" else rng.randint(8, 32)
        return _tfm(call, 2 * _log_int(rng, 4, 128), n, vocab=rng.randint(40, 128),
                    layers=rng.randint(1, 2), ff=128 * rng.randint(1, 4),
                    act=rng.choice(["gelu", "gelu", "gaussian"]))
    n = _log_int(rng, 16, 48) if call == "run" else rng.randint(8, 16)
    heads = rng.choice([2, 4])
    return _tfm(call, _log_int(rng, 5, 48), n, vocab=rng.randint(30, 90), ctx=rng.randint(16, 63),
                d=heads * rng.randint(8, 24), layers=1, heads=heads, ff=rng.randint(64, 256), K=16)


# ------------------------------------------------------------------------------------ inputs

def _layers(case):
    s = STYLES[case["style"]]
    dims = [case["D"]] + [case["hidden"]] * case["depth"] + [case["C"]]
    L = len(dims) - 1
    g = 1.0 if s["act"] == "gaussian" else 0.0
    scale = [2.0 ** -4, 2.0 ** -6] if s["wkind"] == "ternary_i8" else [1.0] * L
    return [W.Layer(dims[m], dims[m + 1], s["act"] if m < L - 1 else s["out"],
                    g if m < L - 1 else 0.0, s["wkind"], scale[m]) for m in range(L)]


def _domain(case):
    beta = case.get("beta", 0.0)
    return W.Domain(op=case.get("op", "replace"), delta=0.05, beta=beta if beta else float("inf"))


def _spec(case):
    return W.TfmSpec(vocab=case["vocab"], ctx=case["ctx"], d_model=case["d"],
                     n_layer=case["layers"], n_head=case["heads"], d_ff=case["ff"],
                     act=case["act"])


def _mlp_inputs(case, seed):
    """X [N, D], labels and initial parameters, on the GPU."""
    g = torch.Generator(device="cuda").manual_seed(seed)
    N, D, C = case["N"], case["D"], case["C"]

    def uni(shape, a):
        return (torch.rand(shape, generator=g, device="cuda") * 2.0 - 1.0) * a

    keep = torch.rand((N, D), generator=g, device="cuda") < DENSITY
    if STYLES[case["style"]]["init"] == 0.0:      # discrete / pruning nets: inputs k / 256
        X = torch.randint(1, 256, (N, D), generator=g, device="cuda").float() / 256.0
    else:
        X = torch.rand((N, D), generator=g, device="cuda")
    X = torch.where(keep, X, torch.zeros((), device="cuda")).contiguous()
    t1 = uni((32, D), math.sqrt(3.0 / D)).double()
    t2 = uni((C, 32), math.sqrt(3.0 / 32)).double()
    y = torch.argmax(torch.tanh(X.double() @ t1.T) @ t2.T, dim=1).to(torch.int32)
    parts = []
    for m, L in enumerate(_layers(case)):
        n = L.n_in * L.n_out
        if L.wkind == "ternary_i8":
            parts.append(torch.randint(-1, 2, (n,), generator=g, device="cuda").float())
        elif L.wkind == "masked_fp32":
            parts.append(torch.randint(-64, 65, (n,), generator=g, device="cuda").float() /
                         (512.0 if m == 0 else 1024.0))
        else:
            a = math.sqrt(3.0 / L.n_in) if case["depth"] > 1 else STYLES[case["style"]]["init"]
            parts.append(uni((n,), a))
    return X, y, torch.cat(parts).contiguous()


def _tfm_inputs(case, seed):
    """Token windows [B, ctx + 1] and parameters some ten thousand trials into a job (2 % of the
    initial values replaced by mutations), on the GPU."""
    r = np.random.default_rng([seed, 6])
    sp = _spec(case)
    V, B = sp.vocab, case["B"]
    cdf = np.cumsum(r.dirichlet(np.full(V, 0.1), size=V * V), axis=1)
    cdf[:, -1] = 1.0
    a, b = r.integers(0, V, B), r.integers(0, V, B)
    cols = []
    for _ in range(sp.ctx + 1):
        a, b = b, np.minimum((cdf[a * V + b] <= r.random(B)[:, None]).sum(axis=1), V - 1)
        cols.append(b)
    tokens = torch.from_numpy(np.stack(cols, axis=1).astype(np.int32)).cuda()
    init = W.tfm_init(r, sp)
    moved = r.random(init.size) < 0.02
    init[moved] = r.uniform(-1.0, 1.0, int(moved.sum())).astype(np.float32)
    return tokens, torch.from_numpy(init).cuda()


def _key(case):
    """Philox key of the trials: the first whose n trials touch no key bias of a Transformer. (A key
    bias shifts all scores of a query alike, so the loss does not depend on it and rounding alone
    would decide such a trial.)"""
    if case["net"] == "mlp":
        return 0
    o, spans = 0, []
    for name, shape in _spec(case).blocks():
        if name.endswith(".bk"):
            spans.append((o, o + shape[0]))
        o += int(np.prod(shape))
    for key in range(1000):
        idx = (_words(key, np.arange(case["n"]))[:, 0] * np.uint64(o)) >> np.uint64(32)
        if not any(((idx >= a) & (idx < b)).any() for a, b in spans):
            return key
    raise ValueError("no key found")


def _candidates(case, seed, P):
    r = np.random.default_rng([seed, 8])
    idx = r.integers(0, P, case["n"]).astype(np.uint32)
    return idx, r.uniform(-1.0, 1.0, case["n"]).astype(np.float32)


def prepare(case, seed):
    if case["net"] == "mlp":
        X, y, init = _mlp_inputs(case, seed)
        h = mca.mca_create(_layers(case), STYLES[case["style"]]["loss"], _domain(case), X, y, init,
                           K=case["K"])
    else:
        tokens, init = _tfm_inputs(case, seed)
        h = mca.mca_create_transformer(_spec(case), _domain(case), tokens, init, K=case["K"])
    state = {"h": h, "init": init, "call": case["call"], "n": case["n"], "key": _key(case),
             "out": torch.empty_like(init)}
    if case["call"] == "eval":
        state["idx"], state["new"] = _candidates(case, seed, init.numel())
    return state


def _bits(params):
    """Updated weights as whole values: a kept trial's weight is one given fp32 number."""
    return params.view(torch.int32)


def run(s):
    h, n = s["h"], s["n"]
    if s["call"] == "eval":
        return {"dS": mca.mca_eval_candidates(h, s["idx"], s["new"])}
    if s["call"] == "trials":
        r = mca.mca_eval_trials(h, s["key"], 0, n)
        return {"idx": r["idx"].astype(np.int64), "new": r["new_w"], "dS": r["dS"]}
    mca.mca_set_params(h, s["init"])
    if s["call"] == "channels":
        acc, dS = mca.mca_run_channels(h, n, s["key"], "he")
        return {"accepted": acc, "dS": dS,
                "params": _bits(mca.mca_get_params(h, s["init"].numel(), s["out"]))}
    mca.mca_run(h, n, s["key"])
    return {"params": _bits(mca.mca_get_params(h, s["init"].numel(), s["out"])),
            "loss": mca.mca_loss(h)}


# ------------------------------------------------------------------------------------ work

def _mlp_work(case):
    """(bytes, flops) of a full forward pass, and of one candidate evaluation on average over the
    uniformly drawn parameter. Cached fields are read and written once; the first layer costs only
    the non-zeros of X."""
    L = _layers(case)
    N, nnz = case["N"], DENSITY * case["N"] * case["D"]
    fwd_f = 2 * nnz * L[0].n_out + sum(2.0 * N * m.n_in * m.n_out for m in L[1:])
    fwd_b = 8 * nnz + 4 * sum(N * m.n_out + m.n_in * m.n_out for m in L)
    P = float(sum(m.n_in * m.n_out for m in L))
    b = f = 0.0
    for l, m in enumerate(L):
        share = m.n_in * m.n_out / P
        if l == 0 and len(L) == 2:          # the non-zeros of one input feature
            cb, cf = DENSITY * N * 12, DENSITY * N * (2 + 2 * case["C"])
        else:
            cb, cf = 8.0 * N, 2.0 * N
            if l + 1 < len(L):
                cf += 2.0 * N * L[l + 1].n_out
                cb += 4.0 * N * L[l + 1].n_out
            for q in range(l + 2, len(L)):
                cf += 2.0 * N * L[q].n_in * L[q].n_out
                cb += 4.0 * (N * L[q].n_out + L[q].n_in * L[q].n_out)
        b += share * cb
        f += share * cf
    return fwd_b, fwd_f, b, f


def _tfm_work(case):
    """The same for the Transformer: a parameter of a block recomputes its block's remainder and
    everything after it, one of a feed-forward hidden unit only the following blocks."""
    sp = _spec(case)
    B, T, d, F, V = case["B"], sp.ctx, sp.d_model, sp.d_ff, sp.vocab
    attn = B * (8.0 * T * d * d + 2.0 * T * T * d)
    ffn = B * 4.0 * T * d * F
    head = B * 2.0 * T * d * V
    stream = 4.0 * B * T * d
    n = sp.n_layer
    P = float(sp.n_params)
    f = (V + T) * d / P * (n * (attn + ffn) + head)
    for b in range(n):
        after = (n - 1 - b) * (attn + ffn) + head
        f += (4 * d * d + 6 * d) / P * (attn + ffn + after)
        f += (2 * d * F + d + F) / P * after
    f += (2 * d + V * d + V) / P * head
    return 4.0 * P + stream * (2 * n + 1), n * (attn + ffn) + head, 4.0 * P + stream, f


def work(case):
    fb, ff, cb, cf = _mlp_work(case) if case["net"] == "mlp" else _tfm_work(case)
    n = case["n"]
    if case["call"] in ("eval", "trials"):
        return {"bytes": n * cb, "flops": n * cf}
    if case["call"] == "channels":
        return {"bytes": n * fb, "flops": n * ff}
    return {"bytes": fb + n * cb, "flops": ff + n * cf}


def _params(case):
    if case["net"] == "tfm":
        return _spec(case).n_params
    return sum(m.n_in * m.n_out for m in _layers(case))


def tolerance(case):
    """Loss changes are differences of sums of fp32 losses: their error is that of the fields and
    losses, not of the (much smaller) change. Against 64 bits: up to 7e-5 of their norm for single-
    hidden-layer nets, 2.4e-4 for deep nets and the Transformer; the mean loss up to 6.5e-7. Of the
    kept trials, one whose loss change is within that error of its threshold may go either way
    (about one in 10000 for the discrete nets, one in 200 where the Transformer's attention weights
    still matter little), which moves the mean loss by up to 8e-6 of itself through the later trials."""
    if case["call"] in ("eval", "trials"):
        return {"rel": 3e-4 if case["net"] == "mlp" and case["depth"] == 1 else 1e-3}
    ties = 4 + (0.001 if case["net"] == "mlp" else 0.02) * case["n"]
    return {"rel": 1e-3 if case["call"] == "channels" else 5e-5,
            "differ": min(0.01, ties / _params(case))}


# ------------------------------------------------------------------------------------ in 64 bits

def _words(seed, taus, c2=0, c3=0):
    """Philox4x32-10 words [len(taus), 4], key = seed, counter = (tau, c2, c3)."""
    t = np.asarray(taus, dtype=np.uint64)
    M = np.uint64(0xFFFFFFFF)
    s = np.uint64(32)
    c = [t & M, t >> s, np.full_like(t, c2), np.full_like(t, c3)]
    k0, k1 = np.uint64(seed & 0xFFFFFFFF), np.uint64(seed >> 32)
    for _ in range(10):
        p0, p1 = np.uint64(0xD2511F53) * c[0], np.uint64(0xCD9E8D57) * c[2]
        c = [(p1 >> s) ^ c[1] ^ k0, p1 & M, (p0 >> s) ^ c[3] ^ k1, p0 & M]
        k0, k1 = (k0 + np.uint64(0x9E3779B9)) & M, (k1 + np.uint64(0xBB67AE85)) & M
    return np.stack(c, axis=1)


def _act(name, z, g=1.0):
    if name == "tanh":
        return torch.tanh(z)
    if name == "sigmoid":
        return torch.sigmoid(z)
    if name == "relu":
        return torch.relu(z)
    if name == "gaussian":
        return torch.exp(-g * z * z)
    if name == "gelu":
        return 0.5 * z * (1.0 + torch.erf(z * math.sqrt(0.5)))
    return z


class _Mlp64:
    """Fields of every layer [n_out, N] in fp64, the effective weights, and one changed weight."""

    def __init__(self, case, seed):
        self.L = _layers(case)
        X, y, init = _mlp_inputs(case, seed)
        self.XT, self.y = X.T.double().contiguous(), y.long()
        self.loss = STYLES[case["style"]]["loss"]
        self.W, self.off, o = [], [], 0
        self.base = init.cpu().numpy()            # fixed values of masked layers
        for m in self.L:
            n = m.n_in * m.n_out
            w = init[o:o + n].double().view(m.n_out, m.n_in)
            self.W.append(w * m.scale if m.wkind == "ternary_i8" else w.clone())
            self.off.append(o)
            o += n
        self.P = o
        self.forward()

    def forward(self):
        self.Z, a = [], self.XT
        for m, w in zip(self.L, self.W):
            self.Z.append(w @ a)
            a = _act(m.act, self.Z[-1], m.act_param) if m is not self.L[-1] else None
        self.S = self.sum_loss(self.Z[-1])

    def sum_loss(self, z):
        a = _act(self.L[-1].act, z, self.L[-1].act_param)
        one = (torch.arange(a.shape[0], device=a.device)[:, None] == self.y[None, :]).to(a.dtype)
        if self.loss == "mse_onehot":
            return float(((a - one) ** 2).sum())
        return float((torch.logsumexp(a, dim=0) - (a * one).sum(dim=0)).sum())

    def find(self, idx):
        l = max(q for q in range(len(self.L)) if self.off[q] <= idx)
        return (l,) + divmod(idx - self.off[l], self.L[l].n_in)

    def change(self, idx, new):
        """(loss sum, updates) with weight idx at its new effective value."""
        L = self.L
        l, j, i = self.find(idx)
        d = float(new) - float(self.W[l][j, i])
        a = self.XT[i] if l == 0 else _act(L[l - 1].act, self.Z[l - 1][i], L[l - 1].act_param)
        row = self.Z[l][j] + d * a
        up = [(l, j, row)]
        if l == len(L) - 1:
            z = self.Z[l].clone()
            z[j] = row
        else:
            g = L[l].act_param
            da = _act(L[l].act, row, g) - _act(L[l].act, self.Z[l][j], g)
            z = self.Z[l + 1] + self.W[l + 1][:, j:j + 1] * da[None, :]
            up.append((l + 1, None, z))
            for m in range(l + 2, len(L)):
                z = self.W[m] @ _act(L[m - 1].act, z, L[m - 1].act_param)
                up.append((m, None, z))
        return self.sum_loss(z), up

    def keep(self, idx, new, S, up):
        l, j, i = self.find(idx)
        self.W[l][j, i] = float(new)
        for m, r, z in up:
            if r is None:
                self.Z[m] = z
            else:
                self.Z[m][r] = z
        self.S = S

    def value(self, idx):
        l, j, i = self.find(idx)
        return float(self.W[l][j, i])

    def proposal(self, idx, r1, dom):
        m = self.L[self.find(idx)[0]]
        if m.wkind == "ternary_i8":
            return m.scale * float(((int(r1) * 3) >> 32) - 1)
        if m.wkind == "masked_fp32":              # toggles between its fixed value and 0
            fixed = float(self.base[idx])
            return 0.0 if self.value(idx) != 0.0 else fixed
        return _new_value(self.value(idx), r1, dom)

    def flat(self):
        return torch.cat([w.reshape(-1) for w in self.W])


class _Tfm64:
    """The Transformer's loss sum by a full fp64 forward pass of every sequence."""

    def __init__(self, case, seed):
        self.sp = _spec(case)
        tokens, init = _tfm_inputs(case, seed)
        self.inp, self.tgt = tokens[:, :-1].long(), tokens[:, 1:].long()
        self.p = init.double().clone()
        self.P = init.numel()
        self.S = self.forward()

    def forward(self):
        sp, v, o = self.sp, {}, 0
        for name, shape in sp.blocks():
            n = int(np.prod(shape))
            v[name] = self.p[o:o + n].view(*shape)
            o += n
        B, T = self.inp.shape
        d, H = sp.d_model, sp.n_head

        def ln(x, k):
            return torch.nn.functional.layer_norm(x, (d,), v[k + ".g"], v[k + ".b"], sp.ln_eps)

        x = v["tok_emb"][self.inp] + v["pos_emb"][:T]
        mask = torch.full((T, T), -math.inf, device=x.device, dtype=x.dtype).triu(1)
        for b in range(sp.n_layer):
            q = "b%d." % b
            a = ln(x, q + "ln1")
            qkv = [(a @ v[q + "w" + c].T + v[q + "b" + c]).view(B, T, H, d // H).transpose(1, 2)
                   for c in "qkv"]
            pr = torch.softmax(qkv[0] @ qkv[1].transpose(2, 3) / math.sqrt(d // H) + mask, dim=-1)
            x = x + (pr @ qkv[2]).transpose(1, 2).reshape(B, T, d) @ v[q + "wo"].T + v[q + "bo"]
            u = ln(x, q + "ln2") @ v[q + "w1"].T + v[q + "b1"]
            x = x + _act(sp.act, u, sp.act_param) @ v[q + "w2"].T + v[q + "b2"]
        z = ln(x, "lnf") @ v["w_head"].T + v["b_head"]
        return float(torch.nn.functional.cross_entropy(z.view(B * T, -1), self.tgt.reshape(-1),
                                                       reduction="sum"))

    def change(self, idx, new):
        old = float(self.p[idx])
        self.p[idx] = float(new)
        S = self.forward()
        self.p[idx] = old
        return S, None

    def keep(self, idx, new, S, up):
        self.p[idx] = float(new)
        self.S = S

    def proposal(self, idx, r1, dom):
        return _new_value(float(self.p[idx]), r1, dom)

    def flat(self):
        return self.p


def _new_value(old, r1, dom):
    f = np.float32
    u = f(int(r1) >> 8) * f(2.0 ** -24)
    if dom.op == "perturb":
        return float(f(old) + f(dom.delta) * (f(2.0) * u - f(1.0)))
    return float(f(dom.lo) + (f(dom.hi) - f(dom.lo)) * u)


def exact(case, seed):
    net = (_Mlp64 if case["net"] == "mlp" else _Tfm64)(case, seed)
    n, dom = case["n"], _domain(case)
    terms = case["N"] if case["net"] == "mlp" else case["B"] * case["ctx"]
    if case["call"] == "eval":
        idx, new = _candidates(case, seed, net.P)
        return {"dS": np.array([net.change(int(i), w)[0] - net.S for i, w in zip(idx, new)])}
    if case["call"] == "channels":
        return _exact_channels(net, n, _key(case))
    r = _words(_key(case), np.arange(n))
    index = (r[:, 0] * np.uint64(net.P)) >> np.uint64(32)
    if case["call"] == "trials":
        new = [net.proposal(int(i), q, dom) for i, q in zip(index, r[:, 1])]
        dS = [net.change(int(i), w)[0] - net.S for i, w in zip(index, new)]
        return {"idx": index.astype(np.int64), "new": np.array(new), "dS": np.array(dS)}
    for t in range(n):
        idx = int(index[t])
        new = net.proposal(idx, r[t, 1], dom)
        S, up = net.change(idx, new)
        theta = -(terms / dom.beta) * math.log((float(r[t, 3]) + 0.5) * 2.0 ** -32)
        if S - net.S <= theta:
            net.keep(idx, new, S, up)
    return {"params": _bits(net.flat().float()), "loss": net.S / terms}


def _exact_channels(net, n, key):
    L, acc, dS = net.L, [], []
    dims = [L[0].n_in] + [m.n_out for m in L]
    for t in range(n):
        v = np.concatenate([_words(key, [t], 2, q)[0] for q in range(2 * len(dims))])
        node = [(int(v[m]) * dims[m]) >> 32 for m in range(len(dims))]
        old, S0 = [w.clone() for w in net.W], net.S
        for m, ly in enumerate(L):
            a = np.float32(math.sqrt(6.0 / ly.n_in))
            u = np.float32(int(v[len(dims) + m]) >> 8) * np.float32(2.0 ** -24)
            net.W[m][node[m + 1], node[m]] = float(a * (np.float32(2.0) * u - np.float32(1.0)))
        net.forward()
        dS.append(net.S - S0)
        acc.append(dS[-1] <= 0.0)
        if not acc[-1]:
            net.W = old
            net.forward()
    return {"accepted": np.array(acc), "dS": np.array(dS),
            "params": _bits(net.flat().float())}
