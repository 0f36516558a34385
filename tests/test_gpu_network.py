"""The network's tile kernels and the proposal's selection at the edges of their
tiles, against the FP64 oracle (oracle/mlp.py)."""
import numpy as np
import pytest

from oracle import mlp
from paper_2605_05086_gb300 import instances as inst

pytestmark = pytest.mark.gpu

U32 = 2.0 ** -24


@pytest.fixture(scope="module")
def env():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_2605_05086_gb300 import chap, learn
    chap.load()
    return torch, chap, learn


def _bf16(torch, a):
    return torch.tensor(a, dtype=torch.float32).to(torch.bfloat16)


# one row, a tile less / exactly / plus one row, more tiles than CTAs (both kernels)
@pytest.mark.parametrize("rows", [1, 63, 64, 65, 152 * 2 * 64 + 1, 152 * 4 * 64 + 65])
def test_tiles_match_oracle(env, rows):
    torch, chap, learn = env
    rng = np.random.default_rng(rows)
    pb, xb = _bf16(torch, mlp.init_params(2)), _bf16(torch, rng.standard_normal((rows, 12)))
    p, x = pb.double().numpy(), xb.double().numpy()
    t = rng.standard_normal(rows).astype(np.float32)
    w_d, x_d = pb.view(torch.int16).cuda(), xb.view(torch.int16).cuda()
    y = torch.full((rows + 8,), 7.0, dtype=torch.float32, device="cuda")
    chap.chap_mlp_forward(w_d, x_d, y[:rows])
    assert torch.all(y[rows:] == 7.0)
    # FP32 sums of 12, 64 and 64 products in a fixed order: every rounding is at
    # most U32 of the sum of absolute terms, (12 + 64 + 64 + 5) of them in a row
    q = mlp.unpack(np.abs(p))
    mag = ((np.abs(x) @ q["W1"] + q["b1"]) @ q["W2"] + q["b2"]) @ q["w3"] + q["b3"][0]
    assert np.all(np.abs(y[:rows].cpu().numpy() - mlp.forward(p, x)) <= 145 * U32 * mag)
    g = torch.zeros(mlp.N_PARAMS, dtype=torch.float32, device="cuda")
    loss = torch.zeros(1, dtype=torch.float32, device="cuda")
    chap.chap_mlp_loss_grad(w_d, x_d, torch.tensor(t, device="cuda"), g, loss)
    l_ref, g_ref = mlp.loss_and_grad(p, x, t.astype(np.float64))
    gg = g.double().cpu().numpy()
    # a unit at its kink may fall on the other side in FP32: the bound is on the
    # whole vector, as for the 1,000-row case of the general test
    assert np.linalg.norm(gg - g_ref) <= 1e-3 * np.linalg.norm(g_ref)
    assert abs(loss.item() / rows - l_ref) <= 1e-4 * l_ref


# a warp's 32 variables less / exactly / plus one, one CTA's worth, several rounds
@pytest.mark.parametrize("n", [31, 32, 33, 257, 152 * 2 * 256 + 33])
@pytest.mark.parametrize("weights", ["drawn", "constant"])
def test_selection_edges(env, n, weights):
    torch, chap, learn = env
    prob = inst.gen_setcover(seed=n, n=n, m=max(8, n // 2), k=min(6, n))
    bs = chap.BestShift(prob, tenure=10)
    chap.chap_bs_refresh_features(bs.h)
    p = mlp.init_params(5)
    if weights == "constant":
        p[:] = 0.0          # every prediction equal: the first k variables
    w = learn.to_bf16_bits(torch.tensor(p, device="cuda"))
    for k in sorted({1, n // 3, n - 1, n}):
        lst = torch.empty(k, dtype=torch.int32, device="cuda")
        pred = torch.empty(n, dtype=torch.float32, device="cuda")
        chap.chap_bs_propose(bs.h, w, k, lst, pred)
        got = np.sort(lst.cpu().numpy())
        assert np.array_equal(got, mlp.topk(pred.cpu().numpy(), k)), k
        if weights == "constant":
            assert np.array_equal(got, np.arange(k))
    bs.close()
