"""chap_info.launches_per_step against the kernels of a step: flips (two kernels
where they are row-blocked), short columns, counting-sorted columns, long lists
(ranked: 2; merged: generation, one per merge round, tile sums, scan), the kept
binary scores' two extra kernels, one apply kernel."""
import numpy as np
import pytest

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


def long_column(rows, count=1):
    """`count` continuous columns in every row, beside 40 others."""
    rng = np.random.default_rng(rows)
    n = count + 40
    r = np.repeat(np.arange(rows), count + 1)
    c = np.concatenate([np.tile(np.arange(count), (rows, 1)), rng.integers(count, n, size=(rows, 1))], axis=1).ravel()
    return inst.from_triplets("long", n, rows, r, c, rng.standard_normal(len(r)), np.zeros(n), np.full(n, 50.0), np.ones(n),
                              rng.standard_normal(rows) * 20, np.full(n, inst.VAR_CONT), np.zeros(rows, np.uint8))


CASES = {
    "flips": (lambda: inst.gen_setcover(seed=1, n=2000, m=1000, k=8), {}, 2),
    "flips_kept": (lambda: inst.gen_setcover(seed=1, n=2000, m=1000, k=8), dict(lazy_binary=1), 4),
    "short": (lambda: inst.gen_general(seed=1, n=3000, m=1500, len_cap=100), {}, 3),
    "short_blocked": (lambda: inst.gen_general(seed=1, n=60_000, m=30_000, len_cap=600), {}, 4),
    "counting": (lambda: inst.gen_skewed(seed=6, n=40_000, m=20_000, n_dense=6, dense_len=6_000), {}, 5),
    "ranked": (lambda: long_column(9_000), {}, 4),
    "merged": (lambda: long_column(40_000), {}, 11),   # 40 chunks: 6 merge rounds
    # 48 runs are ranked where there is one long column, 64 where there are 17
    "ranked_longest": (lambda: long_column(24_384), {}, 4),
    "merged_shortest": (lambda: long_column(24_385), {}, 10),
    "ranked_longest_17": (lambda: long_column(32_512, 17), {}, 4),
    "merged_shortest_17": (lambda: long_column(32_513, 17), {}, 10),
}


@pytest.mark.parametrize("which", sorted(CASES))
def test_launches_per_step(chap, which):
    make, options, launches = CASES[which]
    bs = chap.BestShift(make(), tenure=10, **options)
    assert bs.info.launches_per_step == launches
    bs.close()
