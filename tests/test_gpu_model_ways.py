"""The two ways of the batched model: records on either side of the short way's
limits, records of both sides in one warp, and the same bits from every kernel
that evaluates a record."""
import numpy as np
import pytest

import oracle as O
import synthetic as S

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

N_SM = 152
THETA = O.prior_theta(N_SM).astype(np.float32).astype(np.float64)
# M N at, just below and above 2^41; K at, just below and above 2^24; (M + N) K at,
# just below and above 2^48; the largest extents
SHAPES = [(1 << 20, 1 << 20, 1 << 20), (1 << 21, (1 << 20) - 1, 64), (1 << 21, 1 << 20, 64), (2 ** 31 - 1, 1023, 96),
          (2 ** 31 - 1, 1024, 96), (2 ** 31 - 1, 1025, 96), (1023, 2 ** 31 - 1, 33), (300, 500, (1 << 24) - 1),
          (300, 500, 1 << 24), (300, 500, (1 << 24) + 1), (300, 500, 2 ** 31 - 1), ((1 << 24) - 64, 64, 1 << 24),
          ((1 << 24) - 65, 64, 1 << 24), ((1 << 24) - 63, 64, 1 << 24), (64, (1 << 25) - 64, (1 << 23) - 1),
          (2 ** 31 - 1, 2 ** 31 - 1, 2 ** 31 - 1), (1, 2 ** 31 - 1, 1), (16, 16, 16)]


def space_cfgs(n, seed, shapes):
    """Records of the search space (both TMEM strategies) over the shapes."""
    r = np.random.default_rng(seed)
    pick = lambda v: r.choice(np.array(v), n)
    s = np.array(shapes, dtype=np.int64)[np.arange(n) % len(shapes)]
    c = dict(M=s[:, 0], N=s[:, 1], K=s[:, 2], BM=pick((64, 128, 256)), BN=pick((64, 128, 256)), BK=pick((32, 64, 128)),
             stages=pick((2, 3, 4, 5, 6)), cta_group=pick((1, 2)), dtype=pick((0, 1, 2)), kind=np.zeros(n),
             tmem_a=pick((0, 0, 0, 1)))
    return {k: np.asarray(v).astype(np.int32) for k, v in c.items()}


def check_against_oracle(lib, c, n, n_sm, seed):
    t_o, gi = O.model_batch(c, THETA, n_sm, grad=True)
    dev = lib.cfg_tensor(c)
    t = torch.empty(n, dtype=torch.float32, device="cuda")
    lib.pm_model_predict(dev, n, THETA, n_sm, t)
    assert np.all(np.abs(t.cpu().numpy() - t_o) <= 1e-5 * t_o)
    t_meas = (t_o * np.exp(0.3 * (S.uniform01_f64(seed, n) - 0.5))).astype(np.float32).astype(np.float64)
    L_o, g_o = O.model_loss_grad(c, THETA, n_sm, t_meas)
    r = np.log(t_o) - np.log(t_meas)
    scale = (2.0 / n) * np.sum(np.abs(r[:, None] * gi / t_o[:, None]), axis=0)
    ws = torch.empty(lib.pm_model_grad_workspace(n) // 8, dtype=torch.float64, device="cuda")
    out = torch.empty(lib.N_GRAD_OUT, dtype=torch.float64, device="cuda")
    lib.pm_model_grad(dev, n, THETA, n_sm, torch.from_numpy(t_meas.astype(np.float32)).cuda(), ws, out)
    o = out.cpu().numpy()
    assert o[0] == pytest.approx(L_o, rel=1e-4, abs=1e-9)
    assert np.all(np.abs(o[1:] - g_o) <= 1e-4 * scale + 1e-30)
    lib.pm_model_grad_f64(dev, n, THETA, n_sm, torch.from_numpy(t_meas).cuda(), ws, out)
    o = out.cpu().numpy()
    assert o[0] == pytest.approx(L_o, rel=1e-10)
    assert np.all(np.abs(o[1:] - g_o) <= 1e-10 * scale + 1e-300)


# one table of many rounds and one of a part of a warp
@pytest.mark.parametrize("n_sm", [152, 3])
@pytest.mark.parametrize("n", [54000, 7])
def test_extents_at_the_limits_of_the_short_way(lib, reading, n, n_sm):
    check_against_oracle(lib, space_cfgs(n, 80, SHAPES), n, n_sm, 81)


@pytest.mark.parametrize("outside", [2, 37])
def test_records_of_both_ways_in_a_warp(lib, reading, outside):
    n = 40011
    c = space_cfgs(n, 82, [(300, 500, 4096), (4096, 4096, 512), (16, 8192, 64)])
    odd = np.arange(n) % outside == 1
    c["BM"][odd], c["BN"][odd], c["tmem_a"][odd] = 192, 96, 0
    probe = np.arange(n) % 41 == 5
    c["kind"][probe], c["M"][probe], c["N"][probe], c["BN"][probe] = 3, 2048, 2048, 64
    check_against_oracle(lib, c, n, N_SM, 83)


# up to six shapes per SM go to the kernel that evaluates every tile by the general
# way, more to the one that tabulates the tile terms
@pytest.mark.parametrize("dt", [0, 1, 2])
@pytest.mark.parametrize("n", [200, 3000])
def test_tuner_and_prediction_give_the_same_bits(lib, reading, dt, n):
    k = 16
    r = np.random.default_rng(84 + dt)
    mnk = np.exp(r.uniform(np.log(1.0), np.log(2.0e6), (n, 3))).astype(np.int32)
    mnk[::2] = 16 * (mnk[::2] // 16 + 1)
    picks = torch.empty(n * k * 24, dtype=torch.uint8, device="cuda")
    t_tune = torch.empty(n * k, dtype=torch.float32, device="cuda")
    lib.pm_autotune_topk(torch.from_numpy(mnk).cuda(), n, dt, THETA, N_SM, k, picks, t_tune)
    t = torch.empty(n * k, dtype=torch.float32, device="cuda")
    lib.pm_model_predict(picks, n * k, THETA, N_SM, t)
    assert torch.all(torch.isfinite(t_tune))
    assert torch.equal(t.view(torch.int32), t_tune.view(torch.int32))
