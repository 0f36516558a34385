"""Work that a program using this library has it do, as measurable cases.

Kinds of work (each through the binding's public entry points):

- "run": a tabu search from a start point: BestShift.set_state, BestShift.run
  (chap_tabu_run), the state read back into device buffers.
- "pass": one best-shift pass at a mid-search checkpoint with every variable's
  value, score and violation change written to device buffers.
- "steps": a host-driven search: a start point loaded, then chap_bs_step with
  the move returned to the host after each, and the residuals at the end.
- "batch": independent chains over several uneven instances (BatchChains).
- "learned": the learned tabu loop (chap_learned_run).
- "log": one training record and one proposal (refresh, features, targets,
  predictions, top-k list).
- "train": minibatch steps (loss gradient, Adam) and a validation forward pass
  of the proposal network.

Instance families (drawn from the seed on the GPU, the shapes of
paper_2605_05086_gb300/instances.py): "setcover" (binary, >= rows of 8),
"general" (binary / integer / continuous, Zipf row lengths, integral and N(0,1)
rows), "skewed" (short columns and a few dense integer ones), "hubs" (a few
continuous and wide-domain integer variables in thousands of rows each).

exact() restates the pass, the search and the network in plain torch (float64 /
int64) from the definition: every half's penalty at every candidate value by a
sorted prefix sum over its change points.
"""
import ctypes
import math

import numpy as np
import torch

from paper_2605_05086_gb300 import chap, instances as inst, learn

TENURE = 10
FEAS_TOL = 1e-9
F, H = 12, 64


# ------------------------------------------------------------------ the cases

def listed():
    return [
        # the smallest search a user starts: a set cover of 2,000 variables to
        # feasibility (default limits); every iteration is launch latency
        dict(name="run_setcover_2k", kind="run", family="setcover", n=2000, m=1000, iters=1000, stop=True, near=False),
        # a large sparse cover, thousands of cheap iterations
        dict(name="run_setcover_200k", kind="run", family="setcover", n=200_000, m=100_000, iters=2000, stop=True,
             near=False),
        # the headline: a general integer MIP of 200k variables from x0
        dict(name="run_general_200k", kind="run", family="general", n=200_000, m=100_000, cap=5000, iters=256,
             stop=True, near=False),
        # a repair search from a nearly feasible point (ragged sizes): few
        # violated rows, weight updates between the moves
        dict(name="run_general_21k_near", kind="run", family="general", n=20_983, m=10_007, cap=600, iters=384,
             stop=True, near=True),
        # millions of short columns and 50 dense integer ones
        dict(name="run_skewed_2m", kind="run", family="skewed", n=2_000_000, m=1_000_000, dense=50,
             dense_len=100_000, iters=64, stop=True, near=False),
        # every variable's best shift for the caller (bounds for another solver)
        dict(name="pass_general_200k", kind="pass", family="general", n=200_000, m=100_000, cap=5000),
        # the same on long breakpoint lists (merge sort, CTA sort)
        dict(name="pass_hubs_7x9k", kind="pass", family="hubs", n=6007, hubs=7, hub_rows=9001),
        # a search driven move by move from the host
        dict(name="steps_general_55k", kind="steps", family="general", n=54_321, m=26_001, cap=1500, steps=8,
             near=False),
        # 64 chains over 16 uneven instances until feasible
        dict(name="batch_16x4", kind="batch", instances=16, n_min=1000, n_max=50_000, chains_per=4, iters=1000),
        # the learned loop on a large cover
        dict(name="learned_setcover_200k", kind="learned", family="setcover", n=200_000, m=100_000, topk=4096,
             exact_every=50, iters=400),
        # training pairs logged and one proposal on a general instance
        dict(name="log_general_90k", kind="log", family="general", n=90_001, m=45_000, cap=2000, topk=4096),
        # the network's training: 8 minibatches and a validation pass
        dict(name="train_8x8192", kind="train", batch=8192, steps=8, val=100_003),
    ]


def _logu(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["run", "run", "run", "pass", "pass", "steps", "batch", "learned", "log", "train"])
    if kind == "train":
        return dict(kind=kind, batch=_logu(rng, 1000, 8192), steps=rng.randint(2, 8), val=_logu(rng, 1000, 100_003))
    if kind == "batch":
        return dict(kind=kind, instances=rng.randint(2, 16), n_min=1000, n_max=_logu(rng, 2000, 50_000),
                    chains_per=rng.randint(1, 4), iters=_logu(rng, 100, 1000))
    if kind == "learned":
        n = _logu(rng, 10_000, 200_000)
        return dict(kind=kind, family="setcover", n=n, m=n // 2, topk=_logu(rng, 256, 4096),
                    exact_every=rng.choice([20, 50]), iters=_logu(rng, 100, 400))
    if kind == "log":
        n = _logu(rng, 5000, 90_001)
        return dict(kind=kind, family="general", n=n, m=n // 2, cap=_logu(rng, 50, 2000), topk=_logu(rng, 64, 4096))
    family = rng.choice(["setcover", "general", "skewed"] if kind == "run" else
                        ["general", "skewed", "hubs"] if kind == "pass" else ["setcover", "general"])
    c = dict(kind=kind, family=family)
    if family == "setcover":
        c["n"] = _logu(rng, 2000, 200_000)
        c["m"] = c["n"] // rng.choice([1, 2, 3]) + 1
    elif family == "general":
        c["n"] = _logu(rng, 2000, 200_000)
        c["m"] = c["n"] // 2 + rng.randint(0, 99)
        c["cap"] = min(5000, max(30, c["n"] // rng.choice([40, 100, 400])))
    elif family == "skewed":
        c["n"] = _logu(rng, 60_000, 2_000_000)
        c["m"] = c["n"] // 2 + rng.randint(0, 99)
        c["dense"] = rng.randint(1, 50)
        c["dense_len"] = max(500, c["m"] // rng.randint(10, 40))
    else:
        c["n"] = _logu(rng, 500, 6007)
        c["hubs"] = rng.randint(1, 7)
        c["hub_rows"] = _logu(rng, 300, 9001)
    if kind == "run":
        c["iters"] = _logu(rng, 64, 1000) if family == "setcover" else _logu(rng, 32, 256 if family == "general" else 64)
        c["stop"] = True
        c["near"] = rng.random() < 0.4
    if kind == "steps":
        c["steps"] = rng.randint(1, 8)
        c["near"] = rng.random() < 0.4
    return c


# ------------------------------------------------- instances, drawn on the GPU

def _gen(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed) * 1_000_003 + 17)
    return g


def _rand(g, n):
    return torch.rand(n, generator=g, device="cuda", dtype=torch.float64)


def _randint(g, lo, hi, n):
    return torch.randint(lo, hi, (n,), generator=g, device="cuda", dtype=torch.int64)


def _zipf(seed, a, size, lo, hi):
    return torch.from_numpy(np.clip(np.random.default_rng(seed).zipf(a, size=size), lo, hi).astype(np.int64)).cuda()


def _senses(g, m):
    """40% <=, 40% >=, 20% = (exactly, in random order)."""
    k = torch.arange(m, device="cuda") * 5 // max(m, 1)
    return torch.div(k, 2, rounding_mode="floor")[torch.randperm(m, generator=g, device="cuda")]


def _nonzero(g, n, mag):
    """Uniform in {-mag..mag} without 0."""
    return (_randint(g, 1, mag + 1, n) * (1 - 2 * _randint(g, 0, 2, n))).to(torch.float64)


def _row_sums(m, rows, v):
    """Sums per row, in index order on the host: the same doubles every time."""
    return torch.from_numpy(np.bincount(rows.cpu().numpy(), weights=v.cpu().numpy(), minlength=m)).cuda()


def _rhs(g, m, rows, cols, vals, xs, sense, integral):
    """a.x* plus (<=) or minus (>=) a slack, integer on integral rows."""
    ax = _row_sums(m, rows, vals * xs[cols])
    ax = torch.where(integral, ax.round(), ax)
    s = torch.where(integral, _randint(g, 0, 11, m).to(torch.float64), _rand(g, m))
    return ax + torch.where(sense == 0, s, torch.where(sense == 1, -s, torch.zeros_like(s)))


def _problem(n, m, rows, cols, vals, lb, ub, rhs, vtype, sense, g):
    """CSR and CSC host copies of triplets already sorted by (row, column)."""
    rp = torch.zeros(m + 1, dtype=torch.int64, device="cuda")
    rp[1:] = torch.cumsum(torch.bincount(rows, minlength=m), 0)
    order = torch.argsort(cols, stable=True)
    cp = torch.zeros(n + 1, dtype=torch.int64, device="cuda")
    cp[1:] = torch.cumsum(torch.bincount(cols, minlength=n), 0)
    obj = _randint(g, 1, 11, n).to(torch.float64)
    h = lambda t, d: t.to(d).cpu().numpy()  # noqa: E731
    i32, f64, i64, u8 = torch.int32, torch.float64, torch.int64, torch.uint8
    lb, ub = h(lb, f64), h(ub, f64)
    return inst.Problem(
        name="case", n=n, m=m, row_ptr=h(rp, i64), col_idx=h(cols, i32), row_val=h(vals, f64), col_ptr=h(cp, i64),
        row_idx=h(rows[order], i32), col_val=h(vals[order], f64), lb=lb, ub=ub, obj=h(obj, f64), rhs=h(rhs, f64),
        vtype=h(vtype, u8), sense=h(sense, u8), x0=np.clip(np.zeros(n), lb, ub))


def _setcover(n, m, seed, k=8):
    g = _gen(seed)
    key = torch.unique(torch.arange(m, device="cuda").repeat_interleave(k) * n + _randint(g, 0, n, m * k))
    rows, cols = key // n, key % n
    vals = _randint(g, 1, 6, len(key)).to(torch.float64)
    rhs = torch.ceil(0.3 * _row_sums(m, rows, vals))
    z = torch.zeros(n, dtype=torch.float64, device="cuda")
    p = _problem(n, m, rows, cols, vals, z, z + 1, rhs, z, torch.ones(m, device="cuda"), g)
    # a point that meets about nine rows in ten
    return p, (_rand(g, n) < 0.5).to(torch.float64).cpu().numpy()


def _general(n, m, cap, seed):
    """70% binary, 20% integer in [0, 100], 10% continuous in [0, 1000]; half of
    the rows integral (no continuous variable), half N(0, 1)."""
    g = _gen(seed)
    perm = torch.randperm(n, generator=g, device="cuda")
    vtype = torch.zeros(n, dtype=torch.int64, device="cuda")
    nb, ni = int(0.7 * n), int(0.2 * n)
    vtype[perm[nb:nb + ni]] = 1
    vtype[perm[nb + ni:]] = 2
    ub = torch.tensor([1.0, 100.0, 1000.0], dtype=torch.float64, device="cuda")[vtype]
    sense = _senses(g, m)
    length = _zipf(seed, 1.5, m, 2, cap)
    integral = _rand(g, m) < 0.5
    row = torch.arange(m, device="cuda").repeat_interleave(length)
    pool = perm[:nb + ni]
    u = _rand(g, len(row))
    col = torch.where(integral[row], pool[(u * len(pool)).long()], (u * n).long())
    key = torch.unique(row * n + col)
    rows, cols = key // n, key % n
    vals = torch.where(integral[rows], _nonzero(g, len(key), 20),
                       torch.randn(len(key), generator=g, device="cuda", dtype=torch.float64))
    xs = torch.floor(_rand(g, n) * (ub + 1)).clamp(max=ub)
    xs = torch.where(vtype == 2, _rand(g, n) * 1000.0, xs)
    rhs = _rhs(g, m, rows, cols, vals, xs, sense, integral)
    z = torch.zeros(n, dtype=torch.float64, device="cuda")
    return _problem(n, m, rows, cols, vals, z, ub, rhs, vtype, sense, g), xs.cpu().numpy()


def _skewed(n, m, dense, dense_len, seed):
    """90% binary, 10% integer in [0, 1000]; column lengths Zipf(1.3) up to 14
    and `dense` integer columns of about dense_len entries; integral rows."""
    g = _gen(seed)
    perm = torch.randperm(n, generator=g, device="cuda")
    nb = int(0.9 * n)
    vtype = torch.zeros(n, dtype=torch.int64, device="cuda")
    vtype[perm[nb:]] = 1
    ub = torch.where(vtype == 0, 1.0, 1000.0).to(torch.float64)
    length = _zipf(seed, 1.3, n, 1, 14)
    length[perm[nb:nb + dense]] = dense_len
    col = torch.arange(n, device="cuda").repeat_interleave(length)
    key = torch.unique(_randint(g, 0, m, len(col)) * n + col)
    rows, cols = key // n, key % n
    vals = _nonzero(g, len(key), 50)
    sense = _senses(g, m)
    xs = torch.floor(_rand(g, n) * (ub + 1)).clamp(max=ub)
    rhs = _rhs(g, m, rows, cols, vals, xs, sense, torch.ones(m, dtype=torch.bool, device="cuda"))
    z = torch.zeros(n, dtype=torch.float64, device="cuda")
    return _problem(n, m, rows, cols, vals, z, ub, rhs, vtype, sense, g), xs.cpu().numpy()


def _hubs(n, hubs, hub_rows, seed):
    """`hubs` variables (continuous in [0, 1024] and integer in [0, 10^6] in
    turn), each in hub_rows rows with one or two of the other variables (a
    third each binary, integer in [0, 20], continuous in [0, 16]); the hubs'
    breakpoints are spread over their domains."""
    g = _gen(seed)
    m = hubs * hub_rows
    vtype = _randint(g, 0, 3, n)
    vtype[:hubs] = 2 - torch.arange(hubs, device="cuda") % 2
    ub = torch.tensor([1.0, 20.0, 16.0], dtype=torch.float64, device="cuda")[vtype]
    ub[:hubs] = torch.where(vtype[:hubs] == 2, 1024.0, 1e6).to(torch.float64)
    hub = torch.arange(m, device="cuda") // hub_rows
    i = torch.arange(m, device="cuda")
    key = torch.unique(torch.cat([i * n + hub, i * n + _randint(g, hubs, n, m), i[::2] * n + _randint(g, hubs, n, len(i[::2]))]))
    rows, cols = key // n, key % n
    vals = torch.where(vtype[hub[rows]] == 2, torch.randn(len(key), generator=g, device="cuda", dtype=torch.float64),
                       _nonzero(g, len(key), 3))
    xs = torch.where(vtype == 2, _rand(g, n) * ub, torch.floor(_rand(g, n) * (ub + 1)).clamp(max=ub))
    spread = _rand(g, m) * ub[hub]
    spread = torch.where(vtype[hub] == 2, spread, spread.floor())
    at = torch.where(cols == hub[rows], spread[rows], xs[cols])
    ax = _row_sums(m, rows, vals * at)
    rhs = torch.where(vtype[hub] == 2, ax, ax.floor()) + _randint(g, -2, 3, m)
    z = torch.zeros(n, dtype=torch.float64, device="cuda")
    return _problem(n, m, rows, cols, vals, z, ub, rhs, vtype, _senses(g, m), g), xs.cpu().numpy()


def _instance(case, seed):
    f = case["family"]
    if f == "setcover":
        return _setcover(case["n"], case["m"], seed)
    if f == "general":
        return _general(case["n"], case["m"], case["cap"], seed)
    if f == "skewed":
        return _skewed(case["n"], case["m"], case["dense"], case["dense_len"], seed)
    return _hubs(case["n"], case["hubs"], case["hub_rows"], seed)


def _start(case, prob, xs, seed):
    """The start point: x0, or the hidden point with 1% of its values redrawn."""
    if not case.get("near"):
        return prob.x0.copy()
    rng = np.random.default_rng(seed + 5)
    x = xs.copy()
    j = rng.choice(prob.n, size=max(1, prob.n // 100), replace=False)
    v = prob.lb[j] + rng.random(len(j)) * (prob.ub[j] - prob.lb[j])
    x[j] = np.where(prob.vtype[j] == 2, v, np.floor(v + 0.5))
    return np.minimum(x, prob.ub)


def _batch_sizes(case):
    rng = np.random.default_rng(case["instances"] + case["n_max"])
    return [int(round(math.exp(rng.uniform(math.log(case["n_min"]), math.log(case["n_max"])))))
            for _ in range(case["instances"])]


def _batch(case, seed):
    probs = [_setcover(n, max(1, 10 * n // 8), 64 * seed + k)[0] for k, n in enumerate(_batch_sizes(case))]
    chain_prob = [k for k in range(len(probs)) for _ in range(case["chains_per"])]
    tenures = [(5, 20, 35, 50)[c % case["chains_per"]] for c in range(len(chain_prob))]
    return probs, chain_prob, tenures


def _checkpoint(prob, xs, m_norm, seed):
    """A mid-search state: the hidden point with a tenth of its values redrawn,
    grown weights, some tabu stamps still active."""
    rng = np.random.default_rng(seed + 9)
    x = _start(dict(near=True), prob, xs, seed)
    j = rng.choice(prob.n, size=prob.n // 10, replace=False)
    v = prob.lb[j] + rng.random(len(j)) * (prob.ub[j] - prob.lb[j])
    x[j] = np.minimum(np.where(prob.vtype[j] == 2, v, np.floor(v + 0.5)), prob.ub[j])
    ti, td = np.zeros(prob.n, np.int64), np.zeros(prob.n, np.int64)
    k = rng.choice(prob.n, size=min(prob.n // 2, 40), replace=False)
    ti[k[::2]] = 500 + rng.integers(-5, 12, size=len(k[::2]))
    td[k[1::2]] = 500 + rng.integers(-5, 12, size=len(k[1::2]))
    return dict(x=x, w=np.minimum(rng.geometric(0.5, size=m_norm), 9).astype(np.int32), tabu_inc=ti, tabu_dec=td,
                iter=500, best_nviol=1 << 40)


def _train_data(case, seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed + 3)
    n = case["batch"] * case["steps"]
    x = torch.rand(n + case["val"], F, generator=g, device="cuda")
    x[:, 9] = (x[:, 9] < 0.7).float()
    x[:, 10] = (x[:, 10] < 0.2).float()
    t = (x[:, 4] - x[:, 5] * x[:, 0] + 0.3 * x[:, 6])[:n] + 0.01 * torch.randn(n, generator=g, device="cuda")
    return x.to(torch.bfloat16), t.contiguous()


# --------------------------------------------------------- prepare, run, work

def _buffers(n, m_norm):
    d = dict(device="cuda")
    return dict(x=torch.empty(n, dtype=torch.float64, **d), w=torch.empty(m_norm, dtype=torch.int32, **d),
                tabu_inc=torch.empty(n, dtype=torch.int64, **d), tabu_dec=torch.empty(n, dtype=torch.int64, **d))


def prepare(case, seed):
    kind = case["kind"]
    if kind == "train":
        x, t = _train_data(case, seed)
        n = case["batch"] * case["steps"]
        w32 = torch.tensor(learn.init_params(seed), device="cuda")
        z = torch.zeros_like
        return dict(case=case, x=x[:n].view(torch.int16).contiguous(), t=t, xv=x[n:].view(torch.int16).contiguous(),
                    w0=w32, w32=w32.clone(), wbf=learn.to_bf16_bits(w32).contiguous(), m=z(w32), v=z(w32), g=z(w32),
                    loss=torch.zeros(1, device="cuda"), y=torch.empty(case["val"], device="cuda"))
    if kind == "batch":
        probs, chain_prob, tenures = _batch(case, seed)
        b = chap.BatchChains(probs, chain_prob, tenures)
        b.autotune(iters=3)
        return dict(case=case, b=b)
    prob, xs = _instance(case, seed)
    bs = chap.BestShift(prob, tenure=TENURE, feas_tol=FEAS_TOL)
    s = dict(case=case, bs=bs, n=prob.n)
    if kind in ("pass", "log"):
        ck = _checkpoint(prob, xs, bs.m_norm, seed)
        bs.set_checkpoint(ck)
    else:
        s["x"] = _start(case, prob, xs, seed)
    if kind == "pass":
        d = dict(device="cuda")
        s["out"] = (torch.empty(prob.n, dtype=torch.float64, **d), torch.empty(prob.n, dtype=torch.int64, **d),
                    torch.empty(prob.n, dtype=torch.int32, **d))
    if kind in ("run", "learned"):
        s["state"] = _buffers(prob.n, bs.m_norm)
    if kind == "steps":
        s["r"] = torch.empty(bs.m_norm, dtype=torch.float64, device="cuda")
    if kind in ("learned", "log"):
        s["weights"] = learn.to_bf16_bits(torch.tensor(learn.init_params(seed), device="cuda")).contiguous()
    if kind == "log":
        d = dict(device="cuda")
        s["feat"] = torch.empty((prob.n, F), dtype=torch.int16, **d)
        s["target"] = torch.empty(prob.n, **d)
        s["list"] = torch.empty(min(case["topk"], prob.n), dtype=torch.int32, **d)
        s["pred"] = torch.empty(prob.n, **d)
    return s


def _read_state(bs, t):
    """The search state into the caller's device buffers, and its counters."""
    sc = np.zeros(6, np.int64)
    p = lambda a: ctypes.c_void_p(a.data_ptr())  # noqa: E731
    st = chap.load().chap_bs_get_state(bs.h, p(t["x"]), p(t["w"]), p(t["tabu_inc"]), p(t["tabu_dec"]),
                                       sc.ctypes.data_as(ctypes.c_void_p), chap.CHAP_MEM_DEVICE)
    if st != chap.CHAP_OK:
        raise chap.ChapError(st, "chap_bs_get_state")
    return dict(t, counters=sc)


def run(s):
    case, kind = s["case"], s["case"]["kind"]
    if kind == "run":
        bs = s["bs"]
        bs.set_state(s["x"])
        r = bs.run(max_iters=case["iters"], stop_at_feasible=1 if case["stop"] else 0)
        return dict(_read_state(bs, s["state"]), objective=r.objective,
                    result=np.array([r.iters, r.moves, r.feasible_iter, r.final_nviol, r.best_nviol]))
    if kind == "pass":
        xh, sh, dc = s["out"]
        _, _, _, mv = chap.chap_bs_best_shift(s["bs"].h, s["n"], xh, sh, dc, mem=chap.CHAP_MEM_DEVICE)
        return dict(xhat=xh, score=sh, dnviol=dc, move=np.array([mv.var, mv.dnviol, mv.score_half]),
                    value=mv.new_value)
    if kind == "steps":
        bs = s["bs"]
        bs.set_state(s["x"])
        mv = [bs.step() for _ in range(case["steps"])]
        chap.chap_bs_residuals(bs.h, bs.m_norm, s["r"], mem=chap.CHAP_MEM_DEVICE)
        return dict(moves=np.array([[m.var, m.dnviol, m.score_half] for m in mv]),
                    values=np.array([m.new_value for m in mv]), r=s["r"])
    if kind == "batch":
        b = s["b"]
        b.reset()
        res, _ = b.run(max_iters=case["iters"], stop_at_feasible=True)
        per = case["chains_per"]
        best = [min(range(k * per, (k + 1) * per), key=lambda c: (res[c].best_nviol, res[c].iters))
                for k in range(case["instances"])]
        return dict(res=np.array([[r.iters, r.moves, r.feasible_iter, r.final_nviol, r.best_nviol] for r in res]),
                    x={str(k): b.x(c) for k, c in enumerate(best)})
    if kind == "learned":
        bs = s["bs"]
        bs.set_state(s["x"])
        r = chap.chap_learned_run(bs.h, s["weights"], topk=case["topk"], exact_every=case["exact_every"],
                                  max_iters=case["iters"])
        return dict(_read_state(bs, s["state"]),
                    result=np.array([r.iters, r.moves, r.feasible_iter, r.final_nviol, r.best_nviol, r.exact_passes,
                                     r.misses]))
    if kind == "log":
        h = s["bs"].h
        chap.chap_bs_refresh_features(h)
        chap.chap_bs_features(h, s["feat"], s["target"])
        chap.chap_bs_propose(h, s["weights"], case["topk"], s["list"], s["pred"])
        return dict(feat=s["feat"].view(torch.bfloat16), target=s["target"], list=s["list"], pred=s["pred"])
    s["w32"].copy_(s["w0"])
    s["wbf"].copy_(s["w0"].to(torch.bfloat16).view(torch.int16))
    s["m"].zero_()
    s["v"].zero_()
    s["loss"].zero_()
    nb = case["batch"]
    for k in range(case["steps"]):
        chap.chap_mlp_loss_grad(s["wbf"], s["x"][k * nb:(k + 1) * nb], s["t"][k * nb:(k + 1) * nb], s["g"], s["loss"])
        chap.chap_mlp_adam(s["w32"], s["wbf"], s["m"], s["v"], s["g"], k + 1, 1e-3)
    chap.chap_mlp_forward(s["wbf"], s["xv"], s["y"])
    return dict(w32=s["w32"], m=s["m"], v=s["v"], loss=s["loss"], y=s["y"])


def _zipf_mean(a, lo, hi):
    """Mean of a Zipf(a) draw clipped to [lo, hi]."""
    k = np.arange(1, 2_000_001, dtype=np.float64)
    p = k ** -a
    tail = 2_000_000.5 ** (1 - a) / (a - 1)
    return float((p * np.clip(k, lo, hi)).sum() + tail * hi) / (float(p.sum()) + tail)


def _shape(case):
    """(variables, rows, expected nonzeros) of the case's instance(s)."""
    f = case.get("family")
    if f == "setcover":
        return case["n"], case["m"], 8 * case["m"]
    if f == "general":
        return case["n"], case["m"], case["m"] * _zipf_mean(1.5, 2, case["cap"])
    if f == "skewed":
        return case["n"], case["m"], case["n"] * _zipf_mean(1.3, 1, 14) + case["dense"] * case["dense_len"]
    if f == "hubs":
        m = case["hubs"] * case["hub_rows"]
        return case["n"], m, 2.5 * m
    n = case["instances"] * (case["n_max"] - case["n_min"]) / max(1e-9, math.log(case["n_max"] / case["n_min"]))
    return n, 1.25 * n, 10 * n


def work(case):
    """Bytes of a pass: the matrix once (a 4-byte row and a 4- or 8-byte
    coefficient per nonzero, 10 on average where both kinds occur), the row
    states and the variables' state once, the outputs once.  A search adds, per
    iteration, the moved column's rows; operations: one penalty term per
    nonzero of an evaluation."""
    kind = case["kind"]
    if kind == "train":
        rows = case["batch"] * case["steps"]
        mac = F * H + H * H + H
        return dict(bytes=24.0 * (rows + case["val"]) + 4.0 * (rows + case["val"]) + 8 * 4 * 5057.0 * case["steps"],
                    flops=2.0 * mac * (3 * rows + case["val"]))
    n, m, nnz = _shape(case)
    entry = 10.0 if case.get("family") in ("general", "hubs") else 8.0
    once = entry * nnz + 32.0 * m + 41.0 * n
    if kind == "pass":
        return dict(bytes=once + 20.0 * n, flops=10.0 * nnz)
    if kind == "batch":
        c = case["chains_per"]
        return dict(bytes=8.0 * nnz + c * (16.0 * m + n / 8.0 + 8.0 * n) + 8.0 * n, flops=10.0 * nnz * c)
    if kind == "log":
        return dict(bytes=once + n * (24.0 + 24.0 + 8.0), flops=10.0 * nnz + 2.0 * n * (F * H + H * H + H))
    its = case.get("iters", case.get("steps", 1))
    return dict(bytes=once + 8.0 * n + 28.0 * n + 4.0 * m + its * (nnz / max(n, 1)) * (entry + 64.0), flops=10.0 * nnz)


def tolerance(case):
    if case["kind"] == "train":
        # sums over the minibatch in FP32 (atomics in any order); a weight whose
        # gradient is near zero turns Adam's normalised step by a part of it
        return dict(rel=2e-4, max=0.05)
    if case["kind"] == "log":
        # BF16 features and predictions; a tie at the k-th prediction may move
        return dict(rel=1e-2, max=0.2, differ=5e-3)
    if case.get("family") in ("general", "hubs"):
        # breakpoints and residuals of N(0, 1) rows: sums of up to 5,000 doubles
        return dict(rel=1e-9, max=1e-7)
    return "exact"


# ------------------------------------------------------- the 64-bit statement

class _Ref:
    """The instance and the search state in plain torch (float64 / int64)."""

    def __init__(self, prob):
        d = lambda a, t: torch.from_numpy(np.ascontiguousarray(a)).cuda().to(t)  # noqa: E731
        f64, i64 = torch.float64, torch.int64
        self.n, self.m = prob.n, prob.m
        rp = d(prob.row_ptr, i64)
        rows, cols = torch.arange(prob.m, device="cuda").repeat_interleave(rp[1:] - rp[:-1]), d(prob.col_idx, i64)
        sense, vals = d(prob.sense, i64), d(prob.row_val, f64)
        self.lb, self.ub, self.vt = d(prob.lb, f64), d(prob.ub, f64), d(prob.vtype, i64)
        sgn = torch.where(sense == 1, -1.0, 1.0).to(f64)
        rhs = d(prob.rhs, f64)
        # integral rows have no tolerance
        bad = torch.zeros(prob.m, dtype=i64, device="cuda")
        bad.index_add_(0, rows, ((vals != vals.round()) | (self.vt[cols] == 2)).to(i64))
        integral = (bad == 0) & (rhs == rhs.round())
        eps = torch.where(integral, 0.0, FEAS_TOL * rhs.abs().clamp(min=1.0))
        # normalised rows: "=" rows give (a, b) and (-a, -b)
        nhalf = 1 + (sense == 2).to(i64)
        base = torch.cumsum(nhalf, 0) - nhalf
        self.mn = int(nhalf.sum())
        self.b = torch.empty(self.mn, dtype=f64, device="cuda")
        self.eps = torch.empty_like(self.b)
        self.b[base], self.eps[base] = sgn * rhs, eps
        eq = sense == 2
        self.b[base[eq] + 1], self.eps[base[eq] + 1] = -rhs[eq], eps[eq]
        e2 = eq[rows]
        i = torch.cat([base[rows], base[rows[e2]] + 1])
        j = torch.cat([cols, cols[e2]])
        a = torch.cat([sgn[rows] * vals, -vals[e2]])
        o = torch.argsort(j, stable=True)
        self.i, self.j, self.a = i[o], j[o], a[o]
        cnt = torch.bincount(self.j, minlength=self.n)
        self.cp = torch.zeros(self.n + 1, dtype=i64, device="cuda")
        self.cp[1:] = torch.cumsum(cnt, 0)
        isb = (self.vt == 0)[self.j]
        self.hb, self.hn = torch.nonzero(isb).flatten(), torch.nonzero(~isb).flatten()
        # the halves of the binary and of the other columns, side by side
        self.ib, self.jb, self.ab = self.i[self.hb], self.j[self.hb], self.a[self.hb]
        self.in_, self.jn, self.an = self.i[self.hn], self.j[self.hn], self.a[self.hn]

    def load(self, x, w=None, ti=None, td=None, it=0, best=None):
        d = lambda a, t: torch.from_numpy(np.ascontiguousarray(a)).cuda().to(t)  # noqa: E731
        self.x = d(x, torch.float64).clone()
        i64 = torch.int64
        self.w = torch.ones(self.mn, dtype=i64, device="cuda") if w is None else d(w, i64)
        self.ti = torch.zeros(self.n, dtype=i64, device="cuda") if ti is None else d(ti, i64).clone()
        self.td = torch.zeros(self.n, dtype=i64, device="cuda") if td is None else d(td, i64).clone()
        self.r = torch.zeros(self.mn, dtype=torch.float64, device="cuda").index_add_(0, self.i, self.a * self.x[self.j]) - self.b
        self.it, self.moves = it, 0
        self.nv = int((self.r > self.eps).sum())
        self.best = self.nv if best is None else best
        self.feas = it if self.nv == 0 else -1

    def shifts(self):
        """Every variable's best admissible shift (x̂, score in half weights, violation change)."""
        n, i64 = self.n, torch.int64
        xh, sc, dv = self.x.clone(), torch.zeros(n, dtype=i64, device="cuda"), torch.zeros(n, dtype=i64, device="cuda")
        free_i, free_d = self.ti <= self.it, self.td <= self.it
        # binary flips
        up = self.x == 0
        r, w = self.r[self.ib], self.w[self.ib]
        m = self.eps[self.ib] - r
        ad = torch.where(up[self.jb], self.ab, -self.ab)
        v0, v1 = m < 0, ad > m
        f = 2 * (v0.to(i64) - v1.to(i64)) + torch.where(v0 & v1, torch.where(ad < 0, 1, -1), 0)
        sb = torch.zeros(n, dtype=i64, device="cuda").index_add_(0, self.jb, f * w)
        db = torch.zeros(n, dtype=i64, device="cuda").index_add_(0, self.jb, v1.to(i64) - v0.to(i64))
        ok = (self.vt == 0) & (self.lb < self.ub) & (sb > 0)
        ok &= torch.where(up, free_i, free_d) | (self.nv + db < self.best)
        xh = torch.where(ok, torch.where(up, 1.0, 0.0).to(torch.float64), xh)
        sc, dv = torch.where(ok, sb, sc), torch.where(ok, db, dv)
        if not len(self.jn):
            return xh, sc, dv
        # other columns: change points of every half's penalty as x_j runs from -inf
        j, a = self.jn, self.an
        r, w, eps = self.r[self.in_], self.w[self.in_], self.eps[self.in_]
        x, l, u, isint = self.x[j], self.lb[j], self.ub[j], self.vt[j] == 1
        live = l < u
        j, a, r, w, eps, x, l, u, isint = (t[live] for t in (j, a, r, w, eps, x, l, u, isint))
        m = eps - r
        v0, pos = m < 0, a > 0
        q = m / a
        tb = x + torch.where(isint, torch.where(pos, torch.floor(q), torch.ceil(q)), q)
        base = torch.where(pos, torch.where(v0, 2, 0), torch.where(v0, -1, -2)) * w
        bcnt = torch.where(pos, -v0.to(i64), (~v0).to(i64))
        # the half's status changes at tb: from tb on (a < 0), after tb (a > 0)
        del_ = torch.where(pos, torch.where(v0, -1, -2), torch.where(v0, 1, 2)) * w
        dcnt = torch.where(pos, 1, -1)
        # a half that stays violated grows instead of falling across x
        cross = torch.where(v0, torch.where(pos, -2, 2), 0) * w
        left, inside = tb < l, (tb >= l) & (tb <= u)
        z = lambda: torch.zeros(n, dtype=i64, device="cuda")  # noqa: E731
        beta = z().index_add_(0, j, base + torch.where(left, del_, 0))
        bc = z().index_add_(0, j, bcnt + torch.where(left, dcnt, 0))
        alpha = z().index_add_(0, j, cross)
        # candidates: breakpoints (integer), tight points (continuous), finite bounds
        near0 = (r.abs() <= eps) & ~isint
        t = torch.where(isint, tb, x - r / a)
        cand = (t >= l) & (t <= u) & (t != x) & ~near0
        jl = torch.nonzero((self.vt != 0) & (self.lb < self.ub)).flatten()
        kt = torch.cat([tb[inside], t[cand], self.lb[jl], self.ub[jl]])
        kj = torch.cat([j[inside], j[cand], jl, jl])
        nc = int(cand.sum()) + 2 * len(jl)
        order = torch.cat([torch.where(pos[inside], 2, 0), torch.ones(nc, dtype=i64, device="cuda")])
        kd = torch.cat([del_[inside], torch.zeros(nc, dtype=i64, device="cuda")])
        kc = torch.cat([dcnt[inside], torch.zeros(nc, dtype=i64, device="cuda")])
        fin = torch.isfinite(kt)
        kt, kj, order, kd, kc = (t_[fin] for t_ in (kt, kj, order, kd, kc))
        o = torch.argsort(order, stable=True)
        o = o[torch.argsort(kt[o], stable=True)]
        o = o[torch.argsort(kj[o], stable=True)]
        kt, kj, order, kd, kc = (t_[o] for t_ in (kt, kj, order, kd, kc))
        ps, pc = torch.cumsum(kd, 0), torch.cumsum(kc, 0)
        first = torch.ones_like(kj, dtype=torch.bool)
        first[1:] = kj[1:] != kj[:-1]
        seg = torch.cumsum(first.to(i64), 0) - 1
        ps = ps - (ps - kd)[first][seg]
        pc = pc - (pc - kc)[first][seg]
        right = kt > self.x[kj]
        s = beta[kj] + ps + torch.where(right, alpha[kj], 0)
        c = bc[kj] + pc
        good = (order == 1) & (kt != self.x[kj]) & (s > 0)
        good &= torch.where(right, free_i[kj], free_d[kj]) | (self.nv + c < self.best)
        s, c, t, jj = s[good], c[good], kt[good], kj[good]
        # largest score, then smallest distance, then smallest value
        top = z().index_reduce_(0, jj, s, "amax")
        k = s == top[jj]
        s, c, t, jj = s[k], c[k], t[k], jj[k]
        inf = torch.full((n,), math.inf, dtype=torch.float64, device="cuda")
        dist = (t - self.x[jj]).abs()
        k = dist == inf.clone().index_reduce_(0, jj, dist, "amin")[jj]
        s, c, t, jj = s[k], c[k], t[k], jj[k]
        k = t == inf.clone().index_reduce_(0, jj, t, "amin")[jj]
        xh[jj[k]], sc[jj[k]], dv[jj[k]] = t[k], s[k], c[k]
        return xh, sc, dv

    def step(self):
        """One iteration; (variable, violation change, score, value) of its move."""
        xh, sc, dv = self.shifts()
        top, j = sc.max(), -1
        mv = (-1, 0, 0, 0.0)
        if int(top) > 0:
            j = int(torch.nonzero(sc == top)[0])
            v, old = float(xh[j]), float(self.x[j])
            mv = (j, int(dv[j]), int(top), v)
            e0, e1 = int(self.cp[j]), int(self.cp[j + 1])
            i = self.i[e0:e1]
            self.r[i] = self.r[i] + self.a[e0:e1] * (v - old)
            self.x[j] = v
            (self.td if v > old else self.ti)[j] = self.it + 1 + TENURE
            self.moves += 1
        else:
            self.w = self.w + (self.r > self.eps).to(torch.int64)
        self.nv = int((self.r > self.eps).sum())
        self.it += 1
        self.best = min(self.best, self.nv)
        if self.nv == 0 and self.feas < 0:
            self.feas = self.it
        return mv

    def search(self, iters):
        """Iterations until feasible or the limit."""
        while self.it < iters and self.nv > 0:
            self.step()


def _mlp64(p, x):
    o = [0, F * H, F * H + H, F * H + H + H * H, F * H + 2 * H + H * H, F * H + 3 * H + H * H, F * H + 3 * H + H * H + 1]
    W1, b1, W2, b2, w3, b3 = (p[o[k]:o[k + 1]] for k in range(6))
    h1 = torch.relu(x @ W1.view(F, H) + b1)
    return torch.relu(h1 @ W2.view(H, H) + b2) @ w3 + b3[0]


def _exact_train(case, seed):
    x, t = _train_data(case, seed)
    x = x.double()
    w = torch.tensor(learn.init_params(seed), device="cuda").double()
    m, v = torch.zeros_like(w), torch.zeros_like(w)
    loss = torch.zeros(1, dtype=torch.float64, device="cuda")
    nb = case["batch"]
    for k in range(case["steps"]):
        p = w.to(torch.float32).to(torch.bfloat16).double().requires_grad_()
        e = _mlp64(p, x[k * nb:(k + 1) * nb]) - t[k * nb:(k + 1) * nb].double()
        g, = torch.autograd.grad((e * e).mean(), p)
        loss += (e * e).sum().detach()
        m, v = 0.9 * m + 0.1 * g, 0.999 * v + 0.001 * g * g
        w = w - 1e-3 * (m / (1 - 0.9 ** (k + 1))) / ((v / (1 - 0.999 ** (k + 1))).sqrt() + 1e-8)
    y = _mlp64(w.to(torch.float32).to(torch.bfloat16).double(), x[case["batch"] * case["steps"]:])
    return dict(w32=w, m=m, v=v, loss=loss, y=y)


def exact(case, seed):
    kind = case["kind"]
    if kind == "train":
        return _exact_train(case, seed)
    if kind in ("batch", "learned"):
        return None  # whole numbers and 0/1 values only
    if kind == "run" and case["family"] == "setcover":
        return None  # the same
    prob, xs = _instance(case, seed)
    ref = _Ref(prob)
    if kind == "pass":
        ck = _checkpoint(prob, xs, ref.mn, seed)
        ref.load(ck["x"], ck["w"], ck["tabu_inc"], ck["tabu_dec"], ck["iter"], ck["best_nviol"])
        xh, sc, dv = ref.shifts()
        return dict(xhat=xh, score=sc, dnviol=dv, move=None, value=None)
    if kind == "log":
        ck = _checkpoint(prob, xs, ref.mn, seed)
        ref.load(ck["x"], ck["w"], ck["tabu_inc"], ck["tabu_dec"], ck["iter"], ck["best_nviol"])
        sc = ref.shifts()[1]
        return dict(feat=None, target=sc.double() / (1.0 + float(sc.max())), list=None, pred=None)
    ref.load(_start(case, prob, xs, seed))
    if kind == "steps":
        mv = [ref.step() for _ in range(case["steps"])]
        return dict(moves=np.array([m[:3] for m in mv]), values=np.array([m[3] for m in mv]), r=ref.r)
    if case["iters"] * (2.0 * len(ref.jb) + 8.0 * len(ref.jn)) > 1.2e10:
        return None
    ref.search(case["iters"])
    return dict(x=ref.x, w=ref.w, tabu_inc=ref.ti, tabu_dec=ref.td, counters=None, result=None,
                objective=float((torch.from_numpy(prob.obj).cuda() * ref.x).sum()))
