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


def _same_state(a, b):
    for k in ("x", "w", "tabu_inc", "tabu_dec"):
        assert np.array_equal(a[k], b[k]), k
    for k in ("iter", "nviol", "best_nviol", "feasible_iter", "moves", "weight_updates"):
        assert a[k] == b[k], k


@pytest.mark.parametrize("which", sorted(INSTANCES))
@pytest.mark.parametrize("tenure", [0, 25])
def test_search_equals_steps(chap, which, tenure):
    prob = INSTANCES[which]()
    a = chap.BestShift(prob, tenure=tenure)
    b = chap.BestShift(prob, tenure=tenure)
    rng = np.random.default_rng(11)
    starts = [None, rng.integers(0, 2, size=prob.n).astype(float)]
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


def test_checkpointed_tabu_and_aspiration(chap):
    """Loaded stamps that make the best flips tabu (the admissible scan), and a
    best count that lets aspiration through."""
    prob = binary_rows(12, 700, 400, 6, fp=True)
    a = chap.BestShift(prob, tenure=5)
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
