"""Row residuals, weights and the violated count after set_state, at the edges of
the residual kernel's split: rows of 0, 7 to 9 and 63 to 65 entries, partly
filled groups of 32 short rows, integral and floating-point rows mixed."""
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


@pytest.mark.parametrize("m", [1, 31, 32, 33, 700])
@pytest.mark.parametrize("lens", [(8,), (0, 1, 7, 8, 9, 63, 64), (64, 65), (3, 200)])
@pytest.mark.parametrize("fp_rows", [0.0, 0.3])
def test_residuals(chap, m, lens, fp_rows):
    rng = np.random.default_rng(1000 * m + len(lens) + int(10 * fp_rows))
    n = 400
    vt = rng.choice([inst.VAR_BIN, inst.VAR_INT], n)
    ub = np.where(vt == inst.VAR_BIN, 1.0, 9.0)
    rows, cols, vals = [], [], []
    for i in range(m):
        k = lens[i % len(lens)]
        rows += [i] * k
        cols += list(rng.choice(n, k, replace=False))
        fp = rng.random() < fp_rows
        vals += list(rng.standard_normal(k) if fp else rng.integers(1, 9, k) * rng.choice([-1.0, 1.0], k))
    kind = rng.choice([inst.ROW_LE, inst.ROW_GE, inst.ROW_EQ], m)
    prob = inst.from_triplets("residuals", n, m, rows, cols, vals, np.zeros(n), ub, np.ones(n),
                              rng.integers(-4, 5, m).astype(float), vt, kind)
    orc = Oracle(prob)
    bs = chap.BestShift(prob, tenure=3)
    for _ in range(2):
        x = np.floor(rng.random(n) * (ub + 1))
        bs.set_state(x)
        r, _, nv = orc.residuals(x)
        assert np.array_equal(bs.residuals(), r)
        assert bs.state()["nviol"] == nv
    bs.close()


@pytest.mark.parametrize("m", [456 * 16, 456 * 16 + 1, 456 * 16 + 33])
@pytest.mark.parametrize("lens", [(8,), (0, 1, 7, 8, 9, 63, 64, 65, 130)])
def test_residuals_of_many_rows(chap, m, lens):
    """Integral rows alone, one per warp and, from one row more than the grid has
    warps, short ones 32 to a warp."""
    rng = np.random.default_rng(m + len(lens))
    n = 700
    vt = rng.choice([inst.VAR_BIN, inst.VAR_INT], n)
    ub = np.where(vt == inst.VAR_BIN, 1.0, 9.0)
    k = np.array(lens)[np.arange(m) % len(lens)]
    rows = np.repeat(np.arange(m), k)
    at = np.arange(len(rows)) - np.repeat(np.cumsum(k) - k, k)
    cols = (np.repeat(rng.integers(0, n, m), k) + 5 * at) % n     # distinct: 140 places before one comes again
    prob = inst.from_triplets("many", n, m, rows, cols, rng.integers(1, 9, len(rows)) * rng.choice([-1.0, 1.0], len(rows)),
                              np.zeros(n), ub, np.ones(n), rng.integers(-4, 5, m).astype(float), vt,
                              rng.choice([inst.ROW_LE, inst.ROW_GE, inst.ROW_EQ], m))
    orc = Oracle(prob)
    bs = chap.BestShift(prob, tenure=3)
    w = rng.integers(1, 9, size=bs.m_norm).astype(np.int32)
    for _ in range(2):
        x = np.floor(rng.random(n) * (ub + 1))
        bs.set_state(x, w)
        r, _, nv = orc.residuals(x)
        assert np.array_equal(bs.residuals(), r)
        st = bs.state()
        assert st["nviol"] == nv and np.array_equal(st["w"], w)
    bs.close()


# the least sizes on either side of the device's check, and a last partial block
@pytest.mark.parametrize("n", [16383, 16384, 20001])
def test_refused_states(chap, n):
    rng = np.random.default_rng(n)
    vt = np.array([inst.VAR_BIN, inst.VAR_INT, inst.VAR_CONT])[np.arange(n) % 3]
    lb, ub = np.zeros(n), np.where(vt == inst.VAR_BIN, 1.0, 9.0)
    ub[4] = np.inf
    m = 50
    rows = np.repeat(np.arange(m), 6)
    prob = inst.from_triplets("states", n, m, rows, rng.integers(0, n, 6 * m), np.ones(6 * m), lb, ub, np.ones(n),
                              np.full(m, 2.0), vt, np.full(m, inst.ROW_LE))
    bs = chap.BestShift(prob, tenure=3)
    good = np.floor(rng.random(n) * (np.minimum(ub, 9.0) + 1))
    bs.set_state(good)
    before = bs.state()
    bounds, frac = "x out of bounds at variable %d", "fractional value of integer variable %d"
    for changes, msg in [({n - 1: -1.0}, bounds % (n - 1)), ({0: np.nan}, bounds % 0), ({1: 0.5}, frac % 1),
                         ({2: 9.5, 3: 0.5}, bounds % 2), ({9: 0.5, 10: 100.0}, frac % 9), ({4: np.inf}, frac % 4)]:
        x = good.copy()
        for j, v in changes.items():
            x[j] = v
        with pytest.raises(chap.ChapError, match=msg):
            bs.set_state(x)
        st = bs.state()
        assert all(np.array_equal(st[k], before[k]) for k in before)
    x = good.copy()
    x[2] = 3.25          # a continuous variable takes any value in its bounds
    bs.set_state(x)
    assert np.array_equal(bs.state()["x"], x)
    bs.close()


def test_column_longer_than_the_apply_grid(chap):
    # 152 CTAs of 1,024 threads apply a move: this column has more entries
    m = 152 * 1024 + 77
    rows = np.concatenate([np.arange(m), [0, 1]])
    cols = np.concatenate([np.zeros(m, np.int64), [1, 2]])
    prob = inst.from_triplets("long_column", 3, m, rows, cols, np.ones(m + 2), np.zeros(3), np.ones(3), np.ones(3),
                              np.ones(m), np.full(3, inst.VAR_BIN), np.full(m, inst.ROW_GE))
    bs = chap.BestShift(prob, tenure=3)
    assert bs.state()["nviol"] == m
    mv = bs.step()
    assert (mv.var, mv.dnviol) == (0, -m)
    st = bs.state()
    assert st["nviol"] == 0 and np.array_equal(bs.residuals(), Oracle(prob).residuals(st["x"])[0])
    bs.close()
