"""Performance cases of the framework: what its users have it compute, by kind.

  apply    interaction scores of value vectors that are already on the GPU
           (``Plan.apply``): the smallest call, the batches of the paper's
           data sets, the headline batch, a large game in float32, and an odd
           size with another index;
  batch    uneven games in one call (``Batch.apply``);
  values   the masked-model value function over all coalitions, in float64,
           in float32 and on the tensor cores, with one baseline or with
           background rows;
  train    training steps of the amortised explainer, and the state after them;
  screen   the amortised explainer's scores of many instances and their
           residual check against the model.

A case names its kind and its sizes.  Inputs are drawn from the seed on the
GPU; models, plans and batches are built in ``prepare`` as a program that
uses them more than once would.
"""
import math
from fractions import Fraction

import numpy as np
import torch

import paper_2601_01903_gb300 as fsi
from paper_2601_01903_gb300 import student as student_mod
from paper_2601_01903_gb300 import synthetic

DEV = "cuda"
F64 = torch.float64


def listed():
    return [
        # one small game, interactively explained: latency of a single call
        dict(name="apply_d8_l2", kind="apply", d=8, ell=2, B=1, arith="exact", index="fsi"),
        # a batch of instances of a mid-size tabular model
        dict(name="apply_d14_l2_b64", kind="apply", d=14, ell=2, B=64, arith="exact", index="fsi"),
        # the benchmark's workload: 16 instances of a 20-feature model, order 3
        dict(name="apply_d20_l3_b16", kind="apply", d=20, ell=3, B=16, arith="exact", index="fsi"),
        # an odd size and batch with another index, whose weights need 64 bits
        dict(name="apply_d19_l3_b3_ksii", kind="apply", d=19, ell=3, B=3, arith="exact", index="ksii"),
        # the largest single game, in float32
        dict(name="apply_d24_l2_f32", kind="apply", d=24, ell=2, B=1, arith="f32", index="fsi"),
        # many games of uneven size and order at once
        dict(name="batch_96", kind="batch", n=96, d_lo=10, d_hi=20, shapes=3, arith="exact"),
        # value vectors in full precision for the exact scores of 64 instances
        dict(name="values_f64_d14_h64", kind="values", path="f64", d=14, h1=64, h2=64, B=64, n_bg=1),
        # value vectors in float32 from the wider model
        dict(name="values_f32_d16_h128", kind="values", path="f32", d=16, h1=128, h2=128, B=8, n_bg=1),
        # training labels of the amortised explainer: dense values on the tensor cores
        dict(name="values_tc_d16_b64", kind="values", path="tc", d=16, h1=128, h2=128, B=64, n_bg=1),
        # the interventional value function with 100 background rows
        dict(name="values_tc_d12_bg100", kind="values", path="tc", d=12, h1=128, h2=128, B=8, n_bg=100),
        # a pass over resident batches of training data, then the state
        dict(name="train_16x4096", kind="train", d=16, ell=2, hidden=1024, B=4096, steps=16),
        # scores of many instances, each checked at 64 coalitions of the model
        dict(name="screen_6000", kind="screen", d=16, ell=2, hidden=1024, n=6000, batch=4096),
    ]


# Work of the largest listed case of each kind, which no drawn case exceeds.
MAX_COALITIONS = 1 << 24
MAX_VALUE_MACS = {"f64": 64 << 26, "f32": 8 << 30, "tc": 64 << 30}


def _log_int(rng, lo, hi):
    """An integer in [lo, hi], spread evenly over its logarithm."""
    return min(hi, max(lo, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    kind = rng.choice(["apply"] * 5 + ["batch"] + ["values"] * 4 + ["train", "screen"])
    if kind == "apply":
        arith = rng.choice(["exact"] * 4 + ["f32"])
        d = rng.randint(6, 24) if arith == "exact" else rng.randint(13, 24)
        ell = rng.randint(1, min(4, 3 if d > 20 else 4))
        B = _log_int(rng, 1, max(1, min(512, MAX_COALITIONS >> d)))
        index = rng.choice(["fsi"] * 4 + ["sii", "bii", "ksii"]) if d <= 20 else "fsi"
        return dict(kind=kind, d=d, ell=ell, B=B, arith=arith, index=index)
    if kind == "batch":
        d_hi = rng.randint(13, 20)
        return dict(kind=kind, n=_log_int(rng, 8, 96), d_lo=rng.randint(8, 10), d_hi=d_hi,
                    shapes=rng.randint(0, 999), arith=rng.choice(["exact", "exact", "f32"]))
    if kind == "values":
        path = rng.choice(["f64", "f32", "tc", "tc"])
        h1, h2 = (128, 128) if path == "tc" else (rng.randint(16, 128), rng.randint(16, 128))
        n_bg = rng.choice([1, 1, _log_int(rng, 2, 100)]) if path == "tc" else rng.choice([1, 1, 1, rng.randint(2, 5)])
        most = MAX_VALUE_MACS[path] // (h1 * h2 * n_bg)
        d = rng.randint(8, max(8, min(18, most.bit_length() - 1)))
        return dict(kind=kind, path=path, d=d, h1=h1, h2=h2, B=_log_int(rng, 1, max(1, min(256, most >> d))), n_bg=n_bg)
    d = 8 * rng.randint(1, 3)
    hidden = 8 * rng.randint(16, 128)
    if kind == "train":
        return dict(kind=kind, d=d, ell=2, hidden=hidden, B=_log_int(rng, 256, 4096), steps=rng.randint(4, 16))
    return dict(kind=kind, d=16, ell=2, hidden=hidden, n=_log_int(rng, 100, 6000), batch=4096)


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------
def _gen(seed, device=DEV):
    return torch.Generator(device=device).manual_seed(int(seed))


def _randn(g, *shape, dtype=F64):
    return torch.randn(*shape, generator=g, device=DEV, dtype=dtype)


def _model_games(g, d, B, hidden=6):
    """Values of B small masked networks on every coalition, [B, 2^d]:
    smooth games with interactions of every order, as masked models give."""
    v = torch.empty(B, 1 << d, device=DEV, dtype=F64)
    step = max(1, (1 << 24) >> d)
    for b0 in range(0, B, step):
        n = min(step, B - b0)
        delta = _randn(g, n, hidden, d) / math.sqrt(d)
        pre = 0.3 * _randn(g, n, hidden, 1)
        out = 0.5 * _randn(g, n, hidden, 1)
        for i in range(d):
            pre = torch.cat([pre, pre + 2.0 * delta[:, :, i:i + 1]], dim=2)
        acc = v[b0:b0 + n].zero_()
        for k in range(hidden):
            acc += out[:, k] * torch.tanh_(pre[:, k])
    return v


def _popcounts(d):
    pc = torch.zeros(1, device=DEV, dtype=torch.int64)
    for _ in range(d):
        pc = torch.cat([pc, pc + 1])
    return pc


def _sparse_game(g, d, density=0.01, max_order=5):
    """A Moebius-sparse game: each T with 1 <= |T| <= max_order kept with
    probability ``density``, its coefficient normal."""
    pc = _popcounts(d)
    keep = (torch.rand(1 << d, generator=g, device=DEV) < density) & (pc >= 1) & (pc <= max_order)
    v = torch.where(keep, _randn(g, 1 << d), torch.zeros((), device=DEV, dtype=F64))
    for i in range(d):
        w = v.view(-1, 2, 1 << i)
        w[:, 1] += w[:, 0]
    return v


def _batch_shapes(case):
    """The games of a batch, (d, ell, v_offset, phi_offset) each, and the
    number of values and scores of all."""
    shape = synthetic.Stream(case["shapes"], synthetic.TAG_GAME_SHAPE)
    ds = shape.integers(case["d_lo"], case["d_hi"], case["n"])
    ds[0] = case["d_hi"]  # at least one game of the largest size
    ells = shape.integers(1, 3, case["n"])
    games, vo, po = [], 0, 0
    for d, ell in zip(ds, ells):
        games.append((int(d), int(ell), vo, po))
        vo += 1 << int(d)
        po += synthetic.n_scores(int(d), int(ell))
    return games, vo, po


def _batch_values(case, games, seed):
    g = _gen(seed)
    v = torch.cat([_sparse_game(g, d) for d, _, _, _ in games])
    return v.float() if case["arith"] == "f32" else v


def _mlp(case, seed):
    m = synthetic.random_mlp(case["d"], case["h1"], case["h2"], seed)
    st = synthetic.Stream(seed, 77)
    m.b1, m.b2, m.b3 = 0.1 * st.normal(case["h1"]), 0.1 * st.normal(case["h2"]), 0.1 * st.normal(1)
    return m


def _value_inputs(case, seed):
    g = _gen(seed)
    x = _randn(g, case["B"], case["d"])
    bg = _randn(g, case["n_bg"], case["d"]) if case["n_bg"] > 1 else torch.zeros(case["d"], device=DEV, dtype=F64)
    return _mlp(case, seed), x, bg


def _train_inputs(case, seed):
    """Initial weights and Adam state in the middle of a run, and the batches."""
    d, H, B = case["d"], case["hidden"], case["B"]
    n_out = synthetic.n_scores(d, case["ell"])
    g = _gen(seed)
    params = student_mod.init_params(d, H, n_out, seed, out_scale=0.3)
    n = min(4, case["steps"])
    x = _randn(g, n, B, d, dtype=torch.float32)
    # labels that a model of the instance gives: single scores of order 0.3,
    # interactions smaller, all of them functions of x
    w = _randn(g, d, n_out, dtype=torch.float32) / math.sqrt(d)
    scale = torch.full((n_out,), 0.05, device=DEV)
    scale[:d + 1] = 0.3
    labels = torch.tanh((x.double() @ w.double()).float()) * scale
    labels[:, :, 0] = 0.1
    target = labels[:, :, 1:].double().sum(2).float()
    p = torch.as_tensor(params, device=DEV)
    gr = _student_grads(p.double(), x[0].double(), labels[0].double(), target[0].double(), 0.1, d, H, n_out)[0]
    m0, v0, o = torch.empty_like(gr), torch.empty_like(gr), 0
    for size in (H * d, H, H * H, H, n_out * H, n_out):
        part = gr[o:o + size]
        v0[o:o + size] = part.square().mean() + 1e-16
        m0[o:o + size] = 0.3 * part
        o += size
    return params, m0.float().cpu().numpy(), v0.float().cpu().numpy(), x, labels, target, n_out


# ---------------------------------------------------------------------------
# a case's state and one pass over it
# ---------------------------------------------------------------------------
def prepare(case, seed):
    kind = case["kind"]
    if kind == "apply":
        v = _model_games(_gen(seed), case["d"], case["B"])
        v = v.float() if case["arith"] == "f32" else v
        return dict(kind=kind, v=v, plan=fsi.Plan(case["d"], case["ell"], case["arith"], max_batch=case["B"],
                                                  index=case["index"]))
    if kind == "batch":
        games, _, n_phi = _batch_shapes(case)
        v = _batch_values(case, games, seed)
        return dict(kind=kind, v=v, batch=fsi.Batch(games, case["arith"]),
                    phi=torch.zeros(n_phi, device=DEV, dtype=v.dtype))
    if kind == "values":
        mlp, x, bg = _value_inputs(case, seed)
        return dict(kind=kind, path=case["path"], n_bg=case["n_bg"], mlp=fsi.DeviceMLP(mlp), x=x, bg=bg)
    if kind == "train":
        params, m0, v0, x, labels, target, n_out = _train_inputs(case, seed)
        st = student_mod.Student(case["d"], case["hidden"], n_out, case["B"], params)
        st.load_state(params, m0, v0, 1000)
        return dict(kind=kind, student=st, x=x, labels=labels, target=target, steps=case["steps"])
    mlp = synthetic.random_mlp(case["d"], 128, 128, seed)
    ex = student_mod.Explainer(mlp, case["ell"], hidden=case["hidden"], batch=min(case["batch"], case["n"]), seed=seed)
    x = _randn(_gen(seed), case["n"], case["d"], dtype=torch.float32)
    return dict(kind=kind, ex=ex, x=x, target=ex.targets(x.double()))


def run(state):
    kind = state["kind"]
    if kind == "apply":
        return state["plan"].apply(state["v"])
    if kind == "batch":
        return state["batch"].apply(state["v"], state["phi"])
    if kind == "values":
        if state["path"] == "tc":
            return fsi.masked_game_tc(state["mlp"], state["x"], state["bg"])
        dtype = F64 if state["path"] == "f64" else torch.float32
        if state["n_bg"] > 1:
            return fsi.masked_game_interventional(state["mlp"], state["x"], state["bg"], dtype=dtype)
        return fsi.masked_game(state["mlp"], state["x"], state["bg"], dtype=dtype)
    if kind == "train":
        st, x, labels, target = state["student"], state["x"], state["labels"], state["target"]
        for k in range(state["steps"]):
            b = k % x.shape[0]
            loss = st.train_step(x[b], labels[b], target[b], 0.1)
        return dict(loss=loss, params=st.state()[0])
    ex = state["ex"]
    phi = ex.predict_raw(state["x"], state["target"])
    return dict(phi=phi, residual=ex.residuals(state["x"], phi))


def work(case):
    kind = case["kind"]
    if kind == "apply":
        e = 4 if case["arith"] == "f32" else 8
        n, s = case["B"] << case["d"], case["B"] * synthetic.n_scores(case["d"], case["ell"])
        # one subtraction per coalition and two players: the Moebius step alone
        return dict(bytes=e * (n + s), flops=n * case["d"] / 2)
    if kind == "batch":
        games, n, n_phi = _batch_shapes(case)
        return dict(bytes=(4 if case["arith"] == "f32" else 8) * (n + n_phi),
                    flops=sum((1 << d) * d / 2 for d, _, _, _ in games))
    if kind == "values":
        n = case["B"] << case["d"]
        return dict(bytes=(8 if case["path"] == "f64" else 4) * n, flops=2.0 * n * case["n_bg"] * case["h2"] * (case["h1"] + 1))
    d, H = case["d"], case["hidden"]
    n_out = synthetic.n_scores(d, case["ell"])
    weights = H * d + H * H + n_out * H
    if kind == "train":
        return dict(bytes=case["steps"] * (4 * case["B"] * (d + n_out) + 24 * weights),
                    flops=case["steps"] * 6.0 * case["B"] * weights)
    n = case["n"]
    return dict(bytes=4.0 * n * (d + n_out), flops=2.0 * n * (weights + 64 * 128 * 129))


# ---------------------------------------------------------------------------
# the same outputs in 64 bits
# ---------------------------------------------------------------------------
def _weights(d, ell, index):
    """W[s][t], the weight of the Moebius coefficient of T in the score of S,
    |S| = s <= ell, |T| = t, S a subset of T."""
    bern = [Fraction(1)]
    for n in range(1, ell + 1):
        bern.append(-sum(Fraction(math.comb(n + 1, k)) * bern[k] for k in range(n)) / (n + 1))
    W = [[0.0] * (d + 1) for _ in range(ell + 1)]
    for s in range(ell + 1):
        for t in range(s, d + 1):
            w = Fraction(1 if t == s else 0)
            if index == "sii":
                w = Fraction(1, t - s + 1)
            elif index == "bii":
                w = Fraction(1, 1 << (t - s))
            elif index == "fsi" and t > ell:
                w = Fraction((-1) ** (ell - s) * s * math.comb(ell, s) * math.comb(t - 1, ell),
                             (ell + s) * math.comb(t + ell - 1, ell + s))
            elif index == "ksii" and t > ell and s > 0:
                w = sum(math.comb(t - s, j) * bern[j] / (t - s - j + 1) for j in range(ell - s + 1))
            W[s][t] = float(w)
    return W


def _scores(v, d, ell, index):
    """The scores of value vectors v [B, 2^d] in float64."""
    B = v.shape[0]
    a = v.double().clone()
    for i in range(d):
        w = a.view(B, -1, 2, 1 << i)
        w[:, :, 1] -= w[:, :, 0]
    pc = _popcounts(d)
    masks = torch.as_tensor([sum(1 << i for i in c) for s in range(ell + 1) for c in _subsets(d, s)], device=DEV)
    out = torch.empty(B, len(masks), device=DEV, dtype=F64)
    for s, row in enumerate(_weights(d, ell, index)):
        z = a * torch.as_tensor(row, device=DEV, dtype=F64)[pc]
        for i in range(d):
            w = z.view(B, -1, 2, 1 << i)
            w[:, :, 0] += w[:, :, 1]
        at = torch.nonzero(pc[masks] == s).flatten()
        out[:, at] = z[:, masks[at]]
    return out


def _subsets(d, s):
    import itertools
    return itertools.combinations(range(d), s)


def _gelu(z):
    return 0.5 * z * (1.0 + torch.erf(z * math.sqrt(0.5)))


def _forward(mlp, z):
    f = lambda a: torch.as_tensor(np.asarray(a, dtype=np.float64), device=DEV)
    h = _gelu(z @ f(mlp.W1).T + f(mlp.b1))
    h = _gelu(h @ f(mlp.W2).T + f(mlp.b2))
    return h @ f(mlp.W3).reshape(-1) + f(mlp.b3).reshape(-1)[0]


def _values(mlp, x, bg):
    B, d = x.shape
    bits = ((torch.arange(1 << d, device=DEV)[:, None] >> torch.arange(d, device=DEV)) & 1).bool()
    rows = bg.reshape(-1, d)
    v = torch.zeros(B, 1 << d, device=DEV, dtype=F64)
    for b in range(B):
        for c in range(0, 1 << d, 1 << 16):
            on = bits[c:c + (1 << 16)]
            for r in rows:
                v[b, c:c + (1 << 16)] += _forward(mlp, torch.where(on, x[b], r)) / len(rows)
    return v


def _split_params(p, d, H, n_out):
    shapes, o, got = [(H, d), (H,), (H, H), (H,), (n_out, H), (n_out,)], 0, []
    for s in shapes:
        n = math.prod(s)
        got.append(p[o:o + n].view(s))
        o += n
    return got


def _student_raw(p, x, d, H, n_out):
    W1, b1, W2, b2, W3, b3 = _split_params(p, d, H, n_out)
    return _gelu(_gelu(x @ W1.T + b1) @ W2.T + b2) @ W3.T + b3


def _project(y, target, v_empty):
    shift = (target - y[:, 1:].sum(1)) / (y.shape[1] - 1)
    return torch.cat([torch.full_like(y[:, :1], v_empty), y[:, 1:] + shift[:, None]], dim=1)


def _student_grads(p, x, labels, target, v_empty, d, H, n_out):
    p = p.detach().clone().requires_grad_(True)
    phi = _project(_student_raw(p, x, d, H, n_out), target, v_empty)
    loss = (phi - labels).square().mean()
    loss.backward()
    return p.grad, loss.detach()


def exact(case, seed):
    kind = case["kind"]
    if kind == "apply":
        v = _model_games(_gen(seed), case["d"], case["B"])
        v = v.float() if case["arith"] == "f32" else v
        step = max(1, (1 << 24) >> case["d"])
        return torch.cat([_scores(v[b:b + step], case["d"], case["ell"], case["index"])
                          for b in range(0, case["B"], step)])
    if kind == "batch":
        games, _, _ = _batch_shapes(case)
        v = _batch_values(case, games, seed)
        return torch.cat([_scores(v[o:o + (1 << d)].unsqueeze(0), d, ell, "fsi")[0] for d, ell, o, _ in games])
    if kind == "values":
        return _values(*_value_inputs(case, seed))
    if kind == "train":
        params, m0, v0, x, labels, target, n_out = _train_inputs(case, seed)
        p, m, v = (torch.as_tensor(a, device=DEV).double() for a in (params, m0, v0))
        for k in range(case["steps"]):
            b = k % x.shape[0]
            g, loss = _student_grads(p, x[b].double(), labels[b].double(), target[b].double(), float(np.float32(0.1)),
                                     case["d"], case["hidden"], n_out)
            m, v, t = 0.9 * m + 0.1 * g, 0.999 * v + 0.001 * g * g, 1001 + k
            p = p - 1e-3 * (m / (1 - 0.9 ** t)) / ((v / (1 - 0.999 ** t)).sqrt() + 1e-8)
        return dict(loss=loss.reshape(1), params=p)
    mlp = synthetic.random_mlp(case["d"], 128, 128, seed)
    d, n, batch = case["d"], case["n"], min(case["batch"], case["n"])
    n_out = synthetic.n_scores(d, case["ell"])
    x = _randn(_gen(seed), n, d, dtype=torch.float32).double()
    zero = torch.zeros(1, d, device=DEV, dtype=F64)
    v_empty = float(_forward(mlp, zero)[0])
    target = _forward(mlp, x) - v_empty
    p = torch.as_tensor(student_mod.init_params(d, case["hidden"], n_out, seed), device=DEV).double()
    phi = _project(_student_raw(p, x, d, case["hidden"], n_out), target, v_empty)
    pool = student_mod.sample_coalitions(batch, d, 64, seed).astype(np.int64)
    coal = torch.as_tensor(pool, device=DEV)[torch.arange(n, device=DEV) % batch]
    masks = torch.as_tensor([sum(1 << i for i in c) for s in range(case["ell"] + 1) for c in _subsets(d, s)], device=DEV)
    res = torch.empty(n, device=DEV, dtype=F64)
    for b in range(0, n, 512):
        c = coal[b:b + 512]
        inside = ((c[:, :, None] & masks) == masks).double()
        got = torch.einsum("bkm,bm->bk", inside, phi[b:b + 512])
        on = ((c[:, :, None] >> torch.arange(d, device=DEV)) & 1).bool()
        val = _forward(mlp, torch.where(on, x[b:b + 512, None, :], torch.zeros((), device=DEV, dtype=F64)))
        res[b:b + 512] = (got - val).square().mean(1).sqrt()
    return dict(phi=phi, residual=res)
