"""The kept-score search of chap_tabu_run against the plain iteration
(chap_bs_step evaluates every score from scratch): the same state, counters
and moves after the same number of iterations."""
import numpy as np
import pytest

from oracle.oracle import Oracle
from paper_2605_05086_gb300 import instances as inst

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def chap():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_2605_05086_gb300 import chap as c
    c.load()
    return c


def binary_rows(seed, n, m, k, fp=False, name="binrows"):
    """m rows of k entries over n binaries, all senses; fp: every other row N(0,1)."""
    rng = np.random.default_rng(seed)
    sense = rng.choice([0, 1, 2], size=m, p=[0.4, 0.4, 0.2]).astype(np.uint8)
    xs = rng.integers(0, 2, size=n)
    rows, cols, vals, rhs = [], [], [], []
    for i in range(m):
        js = np.sort(rng.choice(n, size=min(k, n), replace=False))
        a = rng.integers(1, 5, size=len(js)) * np.where(rng.random(len(js)) < 0.5, -1, 1).astype(float)
        if fp and i % 2:
            a = rng.standard_normal(len(js))
        rows.append(np.full(len(js), i)); cols.append(js); vals.append(a)
        rhs.append(float(a @ xs[js]) + (1.0 if sense[i] == 0 else -1.0 if sense[i] == 1 else 0.0))
    return inst.from_triplets(name, n, m, np.concatenate(rows), np.concatenate(cols), np.concatenate(vals),
                              np.zeros(n), np.ones(n), np.ones(n), np.array(rhs), np.full(n, inst.VAR_BIN), sense,
                              x0=np.zeros(n))


INSTANCES = {
    # one CTA: blocks of 256 positions and rows, and one past them
    "cover_256": lambda: inst.gen_setcover(seed=1, n=256, m=256, k=4),
    "cover_257": lambda: inst.gen_setcover(seed=2, n=257, m=257, k=6),
    "cover_20k": lambda: inst.gen_setcover(seed=3, n=20_000, m=10_000, k=8),
    # "=" rows and N(0,1) rows
    "mixed_rows": lambda: binary_rows(4, 900, 500, 7, fp=True),
    "tiny": lambda: binary_rows(5, 5, 4, 3, fp=True),
    # rows of one chunk and one entry more; long rows (a cluster runs the search)
    "chunk_edge": lambda: binary_rows(6, 600, 40, 257, fp=True),
    "long_rows": lambda: binary_rows(7, 4000, 300, 900, fp=True),
    # every move changes all rows: the walk goes to the whole GPU
    "dense": lambda: binary_rows(8, 18_000, 70, 18_000, fp=True),
}


def integers_long_columns(seed, n_hub=5, rows_per=200, dom=300, n_other=120):
    """Integer hubs of more than 128 entries (counting-sorted columns) beside
    short binary, integer and continuous columns, an unbounded integer among
    them; integral and N(0,1) rows, all senses."""
    rng = np.random.default_rng(seed)
    n = n_hub + n_other
    vt = np.concatenate([np.full(n_hub, inst.VAR_INT), rng.integers(0, 3, size=n_other)]).astype(np.uint8)
    ub = np.where(vt == inst.VAR_BIN, 1.0, np.where(vt == inst.VAR_INT, 25.0, 8.0))
    ub[:n_hub] = dom
    lb = np.zeros(n)
    lb[n_hub + 1::7] = np.where(vt[n_hub + 1::7] == inst.VAR_BIN, 0.0, -3.0)
    free = n - 1
    vt[free], lb[free], ub[free] = inst.VAR_INT, -np.inf, np.inf
    m = n_hub * rows_per
    rows, cols, vals, rhs = [], [], [], []
    sense = rng.choice([0, 1, 2], size=m, p=[0.4, 0.4, 0.2]).astype(np.uint8)
    for i in range(m):
        js = np.unique(np.concatenate([[i % n_hub], rng.integers(n_hub, n, size=4)]))
        a = rng.integers(1, 9, size=len(js)) * np.where(rng.random(len(js)) < 0.5, -1, 1).astype(float)
        if i % 3 == 0:
            a = rng.standard_normal(len(js))
        x = np.array([rng.integers(0, dom) if j < n_hub else rng.integers(0, 2) for j in js], dtype=float)
        rows.append(np.full(len(js), i)); cols.append(js); vals.append(a)
        rhs.append(float(a @ x) if i % 3 == 0 else float(np.round(a @ x)))
    return inst.from_triplets("hubs", n, m, np.concatenate(rows), np.concatenate(cols), np.concatenate(vals), lb, ub,
                              np.ones(n), np.array(rhs), vt, sense, x0=np.clip(np.zeros(n), lb, ub))


def nearly_feasible(prob):
    """The instance with the right-hand sides moved so that the start point
    violates at most every 20th row."""
    x0 = np.clip(0.0, prob.lb, prob.ub)
    rows = np.repeat(np.arange(prob.m), np.diff(prob.row_ptr))
    act = np.bincount(rows, weights=prob.row_val * x0[prob.col_idx], minlength=prob.m)
    prob.rhs = np.where(np.arange(prob.m) % 20 == 0, prob.rhs, act)
    return prob


INSTANCES.update({
    # non-binary columns: bounds and kept results, short lists and long ones
    "general": lambda: inst.gen_general(seed=1, n=6_000, m=3_000, len_cap=300),
    "general_long": lambda: inst.gen_general(seed=2, n=3_001, m=5_003, len_cap=200),
    "tiny_mixed": lambda: inst.gen_tiny_mixed(3, n=9, m=8, cont_frac=0.3),
    "no_binary": lambda: inst.gen_tiny_mixed(8, n=300, m=200, dom=30, cont_frac=1.0),
    # counting-sorted columns; their own moves (more rows than one record list)
    "hubs": lambda: integers_long_columns(4),
    "hubs_700": lambda: integers_long_columns(5, n_hub=3, rows_per=700),
    "skewed": lambda: inst.gen_skewed(seed=6, n=40_000, m=20_000, n_dense=6, dense_len=6_000),
    # the two forms in which a search with counting-sorted columns starts by
    # itself: many nonzeros, or few violated rows (else the iteration graph runs)
    "skewed_many_nonzeros": lambda: inst.gen_skewed(seed=6, n=320_000, m=160_000, n_dense=6, dense_len=20_000),
    "skewed_near": lambda: nearly_feasible(inst.gen_skewed(seed=6, n=40_000, m=20_000, n_dense=6, dense_len=6_000)),
    "hubs_near": lambda: nearly_feasible(integers_long_columns(4)),
    "hubs_700_near": lambda: nearly_feasible(integers_long_columns(5, n_hub=3, rows_per=700)),
})


def _same_state(a, b):
    for k in ("x", "w", "tabu_inc", "tabu_dec"):
        assert np.array_equal(a[k], b[k]), k
    for k in ("iter", "nviol", "best_nviol", "feasible_iter", "moves", "weight_updates"):
        assert a[k] == b[k], k


# 1: the search whatever the size and the state, 0: the library's choice
@pytest.mark.parametrize("run_scores", [1, 0])
@pytest.mark.parametrize("which", sorted(INSTANCES))
@pytest.mark.parametrize("tenure", [0, 25])
def test_search_equals_steps(chap, which, tenure, run_scores):
    prob = INSTANCES[which]()
    a = chap.BestShift(prob, tenure=tenure, run_scores=run_scores)
    assert a.info.kept_scores == 1 or not run_scores
    b = chap.BestShift(prob, tenure=tenure)
    rng = np.random.default_rng(11)
    lo, hi = np.maximum(prob.lb, -5.0), np.minimum(prob.ub, 40.0)
    x = np.where(prob.vtype == inst.VAR_CONT, lo + rng.random(prob.n) * (hi - lo),
                 np.floor(lo + rng.random(prob.n) * (hi - lo + 1)))
    starts = [None, np.minimum(x, prob.ub)]
    for x in starts:
        w = None if x is None else rng.integers(1, 6, size=a.m_norm).astype(np.int32)
        a.set_state(x, w)
        b.set_state(x, w)
        for iters in (1, 2, 37, 60):
            a.run(max_iters=iters, stop_at_feasible=0)
            for _ in range(iters):
                b.step()
            sa, sb = a.state(), b.state()
            sb["feasible_iter"] = sa["feasible_iter"]   # a run counts from its own start
            _same_state(sa, sb)
            assert np.array_equal(a.residuals(), b.residuals())
    a.close()
    b.close()


def test_search_follows_the_oracle_to_feasibility(chap):
    """A cover searched until feasible, weight updates included."""
    prob = inst.gen_setcover(seed=9, n=1500, m=900, k=7)
    bs = chap.BestShift(prob, tenure=6)
    orc = Oracle(prob)
    ost = orc.initial_state()
    orc.run(ost, tenure=6, n_iters=4000, stop_at_feasible=True)
    r = bs.run(max_iters=4000, stop_at_feasible=1)
    st = bs.state()
    assert np.array_equal(st["x"], ost["x"]) and np.array_equal(st["w"], ost["w"])
    assert st["iter"] == ost["iter"] == r.iters and r.feasible_iter == (r.iters if r.final_nviol == 0 else -1)
    bs.close()


@pytest.mark.parametrize("mixed", [False, True])
def test_checkpointed_tabu_and_aspiration(chap, mixed):
    """Loaded stamps that make the best flips tabu (the admissible scan; kept
    results of columns with a tabu direction not used), and a best count that
    lets aspiration through."""
    prob = integers_long_columns(12) if mixed else binary_rows(12, 700, 400, 6, fp=True)
    a = chap.BestShift(prob, tenure=5, run_scores=1)
    b = chap.BestShift(prob, tenure=5)
    rng = np.random.default_rng(3)
    for slack in (0, 3, 1000):
        x = rng.integers(0, 2, size=prob.n).astype(float)
        st = dict(x=x, w=rng.integers(1, 9, size=a.m_norm), tabu_inc=rng.integers(0, 140, size=prob.n),
                  tabu_dec=rng.integers(0, 140, size=prob.n), iter=100, best_nviol=0)
        a.set_checkpoint(st)
        st["best_nviol"] = a.state()["nviol"] - 1 + slack
        a.set_checkpoint(st)
        b.set_checkpoint(st)
        for _ in range(3):
            a.run(max_iters=20, stop_at_feasible=0)
            for _ in range(20):
                b.step()
            sa, sb = a.state(), b.state()
            sb["feasible_iter"] = sa["feasible_iter"]
            _same_state(sa, sb)
    a.close()
    b.close()


@pytest.mark.parametrize("stop", [False, True])
def test_chains_default_schedule(chap, stop):
    """A batch on its default schedule (each chain a search of its own where the
    instances allow it) follows the single handle over split runs and a reset;
    one instance of long columns keeps the whole batch on the other schedules."""
    probs = [inst.gen_setcover(seed=5, n=257, m=256, k=6), binary_rows(21, 900, 513, 7),
             inst.gen_setcover(seed=6, n=3000, m=1500, k=8)]
    for extra in ([], [binary_rows(22, 40, 700, 30)]):
        ps = probs + extra
        chain_prob = [k for k in range(len(ps)) for _ in range(2)]
        tenures = [0, 12] * len(ps)
        b = chap.BatchChains(ps, chain_prob, tenures)
        for again in range(2):
            if again:
                b.reset()
            for iters in (1, 60, 150):
                res, _ = b.run(max_iters=iters, stop_at_feasible=stop)
            for c, (k, t) in enumerate(zip(chain_prob, tenures)):
                bs = chap.BestShift(ps[k], tenure=t)
                for iters in (1, 60, 150):
                    bs.run(max_iters=iters, stop_at_feasible=1 if stop else 0)
                st = bs.state()
                bs.close()
                assert (res[c].iters, res[c].moves, res[c].final_nviol, res[c].best_nviol) == \
                    (st["iter"], st["moves"], st["nviol"], st["best_nviol"]), c
                assert np.array_equal(b.x(c), st["x"]), c
        b.close()


@pytest.mark.parametrize("n,lanes", [(8_000, 32), (20_000, 16), (60_000, 8)])
def test_short_column_lanes_fill_the_gpu(chap, n, lanes):
    """Short non-binary columns at every lane count the library picks, far from
    and near a feasible point (short lists, and lists longer than a group's):
    scores and violation changes equal the oracle's, values within the rounding
    of a breakpoint (two roundings of 1e-16, asserted at 1e-9)."""
    prob = inst.gen_general(seed=17, n=n, m=n // 2, len_cap=n // 100)
    bs = chap.BestShift(prob, tenure=5)
    assert bs.info.nb_lanes == lanes
    orc = Oracle(prob)
    rng = np.random.default_rng(1)
    pick = np.sort(rng.choice(np.flatnonzero(prob.vtype != inst.VAR_BIN), size=1500, replace=False)).astype(np.int32)
    for run in (0, 400):
        if run:
            bs.run(max_iters=run, stop_at_feasible=0)
        bs.set_checkpoint(bs.state())
        st = bs.state()
        g = bs.best_shift()
        o = orc.best_shift(st["x"], st["w"], st["tabu_inc"], st["tabu_dec"], st["iter"], st["nviol"], st["best_nviol"],
                           vars=pick)
        assert np.array_equal(g[1][pick], o[1]) and np.array_equal(g[2][pick], o[2])
        assert np.allclose(g[0][pick], o[0], rtol=1e-9, atol=1e-9)
    bs.close()


def _run_equals_steps(chap, prob, start, tenure=0, feas_tol=1e-9, iters=(1, 2, 9, 30), kept=1):
    """Runs of the search and single steps from `start` (x, w) give the same state."""
    a = chap.BestShift(prob, tenure=tenure, feas_tol=feas_tol, run_scores=1)
    assert a.info.kept_scores == kept
    b = chap.BestShift(prob, tenure=tenure, feas_tol=feas_tol)
    a.set_state(*start)
    b.set_state(*start)
    for k in iters:
        a.run(max_iters=k, stop_at_feasible=0)
        for _ in range(k):
            b.step()
        sa, sb = a.state(), b.state()
        sb["feasible_iter"] = sa["feasible_iter"]
        _same_state(sa, sb)
    a.close()
    b.close()
    return sa


@pytest.mark.parametrize("vt", [inst.VAR_CONT, inst.VAR_INT])
def test_column_without_a_candidate_on_its_unbounded_side(chap, vt):
    """y in [0, inf) at 5, z binary at 0; y <= 3 (weight 1), y >= 5 (3),
    y - 10 z >= -4 (1), z >= 1 (2).  At first y's candidates 3 and 0 score -4
    while every value right of 5 scores -1; z flips, and then y moves to 6
    with score 1 (two gained on the third row, one lost on the first)."""
    prob = inst.from_triplets("open_side", 2, 4, [0, 1, 2, 2, 3], [0, 0, 0, 1, 1], [1.0, 1.0, 1.0, -10.0, 1.0],
                              [0.0, 0.0], [np.inf, 1.0], [1.0, 1.0], [3.0, 5.0, -4.0, 1.0], [vt, inst.VAR_BIN],
                              [inst.ROW_LE, inst.ROW_GE, inst.ROW_GE, inst.ROW_GE], x0=[5.0, 0.0])
    st = _run_equals_steps(chap, prob, (np.array([5.0, 0.0]), np.array([1, 3, 1, 2], np.int32)), tenure=3, iters=(2,))
    assert st["x"].tolist() == [6.0, 1.0] and st["moves"] == 2


def open_bounds(seed, finite=0.3):
    """Short rows over binaries, integers and continuous columns, most of the
    latter in [0, inf) or free; "=" rows and a third of the others tight at the
    start point, uneven right-hand sides elsewhere."""
    rng = np.random.default_rng(seed)
    n, m = int(rng.integers(6, 60)), int(rng.integers(6, 70))
    vt = rng.choice(np.array([inst.VAR_BIN, inst.VAR_INT, inst.VAR_CONT], np.uint8), size=n, p=[0.4, 0.2, 0.4])
    lb, ub = np.zeros(n), np.where(vt == inst.VAR_BIN, 1.0, np.inf)
    other = vt != inst.VAR_BIN
    lb[other & (rng.random(n) < 0.3)] = -np.inf
    fin = other & (rng.random(n) < finite)
    ub[fin] = rng.integers(3, 12, size=int(fin.sum()))
    x0 = np.where(vt == inst.VAR_CONT, rng.integers(0, 25, size=n) / 8.0, rng.integers(0, 4, size=n)).astype(float)
    x0 = np.where(vt == inst.VAR_BIN, rng.integers(0, 2, size=n), x0).astype(float)
    rows, cols, vals = [], [], []
    for i in range(m):
        js = rng.choice(n, size=int(rng.integers(1, min(6, n) + 1)), replace=False)
        rows += [i] * len(js); cols += sorted(js.tolist())
        vals += rng.choice([-4, -2, -1, -0.5, 0.5, 1, 2, 4, 8], size=len(js)).tolist()
    act = np.bincount(rows, weights=np.array(vals) * x0[cols], minlength=m)
    sense = rng.choice([0, 1, 2], size=m, p=[0.4, 0.4, 0.2]).astype(np.uint8)
    off = np.where((sense == 2) & (rng.random(m) < 0.7) | (rng.random(m) < 0.33), 0.0, rng.integers(-12, 13, size=m) / 4.0)
    w = rng.integers(1, 7, size=int(m + (sense == 2).sum())).astype(np.int32)
    return inst.from_triplets(f"open_{seed}", n, m, rows, cols, vals, lb, ub, np.ones(n), act + off, vt, sense, x0=x0), x0, w


@pytest.mark.parametrize("seed", range(240))
def test_unbounded_columns_equal_steps(chap, seed):
    """Dyadic data (exact sums), tolerances 0, 1e-9 and a quarter (whose windows
    between boundary and tight point hold other rows' candidates)."""
    prob, x, w = open_bounds(seed, finite=(0.3, 1.0)[seed % 2])
    _run_equals_steps(chap, prob, (x, w), tenure=seed % 5, feas_tol=(0.0, 1e-9, 0.25, 0.25)[seed // 2 % 4])


def test_reverse_flip_on_an_absorbed_residual(chap):
    """feas_tol 0: 0.1 x + 0.2 y + z <= 0.3 (weight 3) with x = y = 1 fixed has
    residual 5.6e-17 at z = 0, violated; z >= 1 (weight 2).  z rises with score
    -3 + 4; at z = 1 the first row's residual rounds to 1, and back at 0 it is
    satisfied: the flip back scores 6 - 4, not -1."""
    prob = inst.from_triplets("absorbed", 3, 2, [0, 0, 0, 1], [0, 1, 2, 2], [0.1, 0.2, 1.0, 1.0], [1.0, 1.0, 0.0],
                              [1.0, 1.0, 1.0], [1.0] * 3, [0.3, 1.0], [inst.VAR_BIN] * 3, [inst.ROW_LE, inst.ROW_GE],
                              x0=[1.0, 1.0, 0.0])
    st = _run_equals_steps(chap, prob, (np.array([1.0, 1.0, 0.0]), np.array([3, 2], np.int32)), feas_tol=0.0, iters=(2,))
    assert st["x"].tolist() == [1.0, 1.0, 0.0] and st["moves"] == 2


def absorbing_rows(seed, n, m, k):
    """Binary rows of decimal coefficients, some of them with one coefficient of
    1e8 whose rounding exceeds the tolerance; many rows tight at a hidden point."""
    rng = np.random.default_rng(seed)
    xs = rng.integers(0, 2, size=n).astype(float)
    rows, cols, vals, rhs = [], [], [], []
    sense = rng.choice([0, 1, 2], size=m, p=[0.4, 0.4, 0.2]).astype(np.uint8)
    for i in range(m):
        js = np.sort(rng.choice(n, size=min(k, n), replace=False))
        a = rng.integers(1, 30, size=len(js)) * np.where(rng.random(len(js)) < 0.5, -0.1, 0.1)
        if i % 3 == 0:
            a[rng.integers(0, len(js))] = rng.choice([-1e8, 1e8])
        rows.append(np.full(len(js), i)); cols.append(js); vals.append(a)
        rhs.append(float(a[::-1] @ xs[js[::-1]]) + rng.choice([0.0, 0.0, 5e-9, -5e-9, 0.3]))
    return inst.from_triplets("absorb", n, m, np.concatenate(rows), np.concatenate(cols), np.concatenate(vals), np.zeros(n),
                              np.ones(n), np.ones(n), np.array(rhs), np.full(n, inst.VAR_BIN), sense, x0=xs)


@pytest.mark.parametrize("feas_tol", [0.0, 1e-9])
@pytest.mark.parametrize("n,m,k", [(40, 30, 5), (500, 400, 6), (600, 60, 400), (700, 600, 500)])
def test_reverse_flips_on_rounded_rows(chap, n, m, k, feas_tol):
    """Every form in which a move is applied: one CTA, a cluster, the whole GPU
    (more rows than one record list)."""
    for seed in range(4):
        prob = absorbing_rows(seed, n, m, k)
        rng = np.random.default_rng(seed)
        x = np.where(rng.random(n) < 0.05, 1.0 - prob.x0, prob.x0)
        w = rng.integers(1, 5, size=int(m + (prob.sense == 2).sum())).astype(np.int32)
        _run_equals_steps(chap, prob, (x, w), tenure=seed, feas_tol=feas_tol, iters=(1, 2, 37, 60))


def wide_mixed(n, n_bin):
    """n_bin binary, the rest integer in [0, 9], every variable in one row of 8."""
    rng = np.random.default_rng(n)
    m = n // 8
    vt = np.where(np.arange(n) < n_bin, inst.VAR_BIN, inst.VAR_INT).astype(np.uint8)
    ub = np.where(vt == inst.VAR_BIN, 1.0, 9.0)
    cols = rng.permutation(n)[:8 * m]
    a = rng.integers(1, 6, size=8 * m).astype(float)
    return inst.from_triplets("wide", n, m, np.repeat(np.arange(m), 8), cols, a, np.zeros(n), ub, np.ones(n),
                              np.ceil(0.3 * (a * ub[cols]).reshape(m, 8).sum(axis=1)), vt, np.full(m, inst.ROW_GE, np.uint8))


# 70% binary up to where the flip bits and the candidate lists share a CTA's
# memory, where only the lists fit, and past those; many integers
@pytest.mark.parametrize("n,n_bin,kept", [(620_000, 434_000, 1), (700_000, 490_000, 1), (760_000, 532_000, 1),
                                          (1_200_000, 840_000, 0), (400_000, 40_000, 0), (5_000, 3_500, 1)])
def test_driver_by_size(chap, n, n_bin, kept):
    """chap_info.kept_scores on both sides of what a cluster's shared memory
    holds, and a run against steps on either driver."""
    prob = wide_mixed(n, n_bin)
    bs = chap.BestShift(prob, tenure=3)
    assert bs.info.kept_scores == kept
    bs.close()
    _run_equals_steps(chap, prob, (prob.x0,), tenure=3, iters=(1, 12), kept=kept)


def test_driver_of_other_handles(chap):
    """kept_scores by option and by kind and size of the instance: tiny mixed ones
    and those with counting-sorted columns from nearly feasible states, small
    dense mixed ones never, large or sparse ones always."""
    def kept(prob, **opts):
        bs = chap.BestShift(prob, **opts)
        k = bs.info.kept_scores
        bs.close()
        return k

    cover, hubs = inst.gen_setcover(seed=1, n=257, m=257, k=6), integers_long_columns(4)
    for opts, want in [({}, 1), (dict(run_scores=1), 1), (dict(run_scores=2), 0), (dict(run_scores=7), 1),
                       (dict(lazy_binary=1), 0), (dict(bin_kernel=2), 0), (dict(static_scratch_only=1), 0)]:
        assert kept(cover, **opts) == want, opts
    assert (kept(hubs), kept(hubs, run_scores=1), kept(hubs, run_scores=2)) == (2, 1, 0)
    # 4,992 and 5,000 nonzeros
    assert (kept(wide_mixed(4_992, 3_000)), kept(wide_mixed(5_000, 3_000))) == (2, 1)
    sparse = inst.gen_general(seed=1, n=6_000, m=3_000, len_cap=300)
    assert kept(sparse) == 1
    rng = np.random.default_rng(0)
    n, m, k = 2_000, 60, 300   # 18,000 nonzeros, a move meets an eighth of them
    cols = np.concatenate([np.sort(rng.choice(n, size=k, replace=False)) for _ in range(m)])
    vt = np.where(np.arange(n) % 2, inst.VAR_INT, inst.VAR_BIN).astype(np.uint8)
    dense = inst.from_triplets("dense_mixed", n, m, np.repeat(np.arange(m), k), cols, rng.integers(1, 9, m * k).astype(float),
                               np.zeros(n), np.where(vt == inst.VAR_BIN, 1.0, 9.0), np.ones(n), np.full(m, 900.0), vt,
                               np.full(m, inst.ROW_GE, np.uint8))
    assert (kept(dense), kept(dense, run_scores=1)) == (0, 1)
    a, b = chap.BestShift(dense, tenure=3), chap.BestShift(dense, tenure=3)
    a.run(max_iters=50, stop_at_feasible=0)
    for _ in range(50):
        b.step()
    assert np.array_equal(a.state()["x"], b.state()["x"])
    a.close()
    b.close()
