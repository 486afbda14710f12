"""The model's kernels at the sizes where their work split changes, against the
FP64 CPU oracle."""
import numpy as np
import pytest

import oracle as O
import synthetic as S

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

N_SM = 152
THETA = O.prior_theta(N_SM).astype(np.float32).astype(np.float64)


# one group is dealt plainly; 32 groups make one vote piece, 113 one pass of the
# tuner's candidates, 256 one round of the evaluation's threads, 1024 is the limit
@pytest.mark.parametrize("G", [1, 2, 32, 33, 113, 114, 256, 257, 1024])
def test_grouped_schedule_sizes(lib, reading, G):
    Mg = S.grouped_m(G, 3 + G)
    N, K = 1024, 512
    t_g, bm, bn, launch = lib.pm_grouped_autotune(Mg, N, K, 1, THETA, N_SM)
    t_o, _, _, _ = O.grouped_autotune(Mg, N, K, 1, THETA, N_SM)
    assert t_g == pytest.approx(t_o, rel=1e-5)
    # mixed tiles, so that the list is not the caller's order
    bm = [(64, 256, 128)[q % 3] for q in range(G)]
    bn = [(128, 64, 256)[(q // 2) % 3] for q in range(G)]
    for launch in ((64, 3, 1), (64, 4, 2)):
        b_m = [b if O.cfg_valid(b, n, *launch, 1) else 64 for b, n in zip(bm, bn)]
        t_o, g_o = O.grouped_predict_grad(Mg, N, K, b_m, bn, *launch, 1, THETA, N_SM)
        assert lib.pm_grouped_predict(Mg, N, K, b_m, bn, *launch, 1, THETA, N_SM) == pytest.approx(t_o, rel=1e-5)
        t_g, g_g = lib.pm_grouped_grad(Mg, N, K, b_m, bn, *launch, 1, THETA, N_SM)
        assert t_g == pytest.approx(t_o, rel=1e-12)
        assert np.all(np.abs((g_g - g_o) * THETA) <= 1e-10 * np.abs(g_o * THETA).max())


def test_grouped_calls_on_streams_and_threads(lib):
    # the calls keep one block of host memory per thread, and wait for their
    # kernel: threads on streams of their own, and a shutdown in between
    import threading
    cases = [(S.grouped_m(g, g), 64 * g, 512) for g in (3, 17, 40, 70)]
    want = [lib.pm_grouped_autotune(M, N, K, 1, THETA, N_SM) for M, N, K in cases]
    got = [None] * len(cases)

    def work(i):
        s = torch.cuda.Stream()
        for _ in range(5):
            got[i] = lib.pm_grouped_autotune(*cases[i], 1, THETA, N_SM, stream=s)
            lib.pm_shutdown()

    th = [threading.Thread(target=work, args=(i,)) for i in range(len(cases))]
    [t.start() for t in th]
    [t.join() for t in th]
    assert got == want


# one shape; the last number of shapes that gets a block each and the first that
# goes through the table (six per SM); one more than the table's warps
@pytest.mark.parametrize("dt", [0, 1, 2])
def test_autotune_splits_agree_with_oracle(lib, reading, dt):
    sms = lib.sm_count()
    n_all = 32 * sms + 1
    r = S.splitmix64(41, 3 * n_all).reshape(n_all, 3)
    MNK = np.where(r[:, :1] % np.uint64(2) == 0, 1 + (r >> np.uint64(50)), 16 * (1 + (r >> np.uint64(54)))).astype(np.int32)
    MNK[3] = (0, 64, 64)                            # no time for an empty product
    dev = torch.from_numpy(MNK.ravel()).cuda()
    idx = np.r_[0:3, 4:64]
    _, t_o = O.autotune(MNK[idx], dt, THETA, N_SM)
    whole = None
    for n in (n_all, 6 * sms + 1, 6 * sms, 1):
        for k in (1, 16):
            picks = torch.empty(n * k * 24, dtype=torch.uint8, device="cuda")
            t = torch.empty(n * k, dtype=torch.float32, device="cuda")
            lib.pm_autotune_topk(dev, n, dt, THETA, N_SM, k, picks, t)
            t, picks = t.cpu().numpy().reshape(n, k), picks.cpu().numpy().view(lib.CFG_DTYPE).reshape(n, k)
            if n > 1:
                assert np.all(np.abs(t[idx, 0] - t_o) <= 1e-5 * t_o)
                assert np.all(np.isinf(t[3])) and np.all(picks[3]["BM"] == 0)
            assert np.all(t[:, 1:] >= t[:, :-1])
            if k == 16:
                if whole is None:
                    whole = (t, picks)
                # the same numbers whichever way the work is split
                assert np.array_equal(t.view(np.uint32), whole[0][:n].view(np.uint32))
                assert picks.tobytes() == whole[1][:n].tobytes()
            else:
                first = (t, picks) if n == n_all else first
                assert picks.tobytes() == first[1][:n].tobytes()
        one_t = torch.empty(n, dtype=torch.float32, device="cuda")
        one_p = torch.empty(n * 24, dtype=torch.uint8, device="cuda")
        lib.pm_autotune_pick(dev, n, dt, THETA, N_SM, one_p, one_t)
        assert one_p.cpu().numpy().tobytes() == first[1][:n].tobytes()


def test_autotune_nan_parameters(lib):
    # both splits treat times that are not numbers alike: a NaN launch time
    # leaves no tile, a NaN drain rate leaves the double-buffered ones
    MNK = torch.tensor([4096, 4096, 4096] * 1000, dtype=torch.int32, device="cuda")
    for j in (0, 14, 17):
        th = THETA.copy()
        th[j] = np.nan
        got = []
        for n in (1, 1000):
            p = torch.empty(n * 24, dtype=torch.uint8, device="cuda")
            t = torch.empty(n, dtype=torch.float32, device="cuda")
            lib.pm_autotune_pick(MNK, n, 1, th, N_SM, p, t)
            rec = p.cpu().numpy().view(lib.CFG_DTYPE)
            got.append((rec[-1].tobytes(), float(t[-1])))
            assert np.all(rec["BM"] == 0) == (j == 0)
            assert bool(torch.isnan(t).all()) == (j == 0)
        assert got[0][0] == got[1][0] and (j == 0 or got[0][1] == got[1][1])


# one warp of a record, a whole record and one row more, the last number of
# records that FP64 spreads over clusters (two thirds of the SMs) and one more
@pytest.mark.parametrize("rows", [1, 31, 33, 256, 257, "clusters", "clusters+1"])
def test_gradient_record_sizes(lib, rows):
    limit = 256 * (2 * lib.sm_count() // 3)
    n = {"clusters": limit, "clusters+1": limit + 1}.get(rows, rows)
    c = S.model_config_batch(n, seed=50)
    c["kind"] = np.zeros(n, dtype=np.int32)
    c["tmem_a"] = np.zeros(n, dtype=np.int32)
    t_true, gi = O.model_batch(c, THETA, N_SM, grad=True)
    t_meas = (t_true * np.exp(0.3 * (S.uniform01_f64(51, n) - 0.5))).astype(np.float32).astype(np.float64)
    L_o, g_o = O.model_loss_grad(c, THETA, N_SM, t_meas)
    r = np.log(t_true) - np.log(t_meas)
    scale = (2.0 / n) * np.sum(np.abs(r[:, None] * gi / t_true[:, None]), axis=0)
    dev = lib.cfg_tensor(c)
    ws = torch.empty(lib.pm_model_grad_workspace(n) // 8, dtype=torch.float64, device="cuda")
    out = torch.empty(lib.N_GRAD_OUT, dtype=torch.float64, device="cuda")
    for _ in range(2):                              # the workspace is written before it is read
        lib.pm_model_grad_f64(dev, n, THETA, N_SM, torch.from_numpy(t_meas).cuda(), ws, out)
        o = out.cpu().numpy()
        assert o[0] == pytest.approx(L_o, rel=1e-10)
        assert np.all(np.abs(o[1:] - g_o) <= 1e-10 * scale + 1e-300)
        ws.fill_(float("nan"))
    lib.pm_model_grad(dev, n, THETA, N_SM, torch.from_numpy(t_meas.astype(np.float32)).cuda(), ws, out)
    o = out.cpu().numpy()
    assert o[0] == pytest.approx(L_o, rel=1e-4, abs=1e-9)
    assert np.all(np.abs(o[1:] - g_o) <= 1e-4 * scale + 1e-30)


def test_gradient_in_a_captured_graph(lib):
    # the two launches of a call, the second set up during the first, replayed
    n = 3000
    c = S.model_config_batch(n, seed=52)
    c["kind"] = np.zeros(n, dtype=np.int32)
    dev = lib.cfg_tensor(c)
    t = torch.full((n,), 1e-4, dtype=torch.float64, device="cuda")
    ws = torch.empty(lib.pm_model_grad_workspace(n) // 8, dtype=torch.float64, device="cuda")
    want = torch.empty(lib.N_GRAD_OUT, dtype=torch.float64, device="cuda")
    lib.pm_model_grad_f64(dev, n, THETA, N_SM, t, ws, want)
    got = torch.zeros_like(want)
    s, g = torch.cuda.Stream(), torch.cuda.CUDAGraph()
    torch.cuda.synchronize()
    with torch.cuda.graph(g, stream=s):
        lib.pm_model_grad_f64(dev, n, THETA, N_SM, t, ws, got, stream=s)
    for _ in range(3):
        g.replay()
    torch.cuda.synchronize()
    assert torch.equal(got, want)


def edge_cfgs(n, seed):
    """Records on both sides of every limit of the model's short way: tile extents, stages and extents inside and
    just outside the search space, probe kinds and TMEM strategy B."""
    r = np.random.default_rng(seed)
    pick = lambda v: r.choice(np.array(v), n)
    ext = (1, 63, 64, 65, 255, 16384, (1 << 20) - 1, 1 << 20, (1 << 20) + 1, 3000017)
    c = dict(M=pick(ext), N=pick(ext), K=pick(ext), BM=pick((32, 64, 128, 192, 256, 320, 512)),
             BN=pick((32, 64, 128, 192, 256, 384, 512)), BK=pick((16, 32, 48, 64, 96, 128, 160, 256)),
             stages=pick((1, 2, 3, 6, 7, 8)), cta_group=pick((1, 2)), dtype=pick((0, 1, 2)),
             kind=pick((0, 0, 0, 0, 0, 0, 1, 2, 3)), tmem_a=pick((0, 0, 0, 1)))
    # strategy B copies A in 32-byte slices: a K-step of part of one is no tile
    c["tmem_a"][c["BK"] % 32 != 0] = 0
    return {k: v.astype(np.int32) for k, v in c.items()}


def test_short_way_agrees_with_the_general_one(lib, reading):
    n = 60000
    c = edge_cfgs(n, 60)
    t_o, gi = O.model_batch(c, THETA, N_SM, grad=True)
    dev = lib.cfg_tensor(c)
    t = torch.empty(n, dtype=torch.float32, device="cuda")
    lib.pm_model_predict(dev, n, THETA, N_SM, t)
    assert np.all(np.abs(t.cpu().numpy() - t_o) <= 1e-5 * t_o)
    t_meas = (t_o * np.exp(0.3 * (S.uniform01_f64(61, n) - 0.5))).astype(np.float32).astype(np.float64)
    L_o, g_o = O.model_loss_grad(c, THETA, N_SM, t_meas)
    r = np.log(t_o) - np.log(t_meas)
    scale = (2.0 / n) * np.sum(np.abs(r[:, None] * gi / t_o[:, None]), axis=0)
    ws = torch.empty(lib.pm_model_grad_workspace(n) // 8, dtype=torch.float64, device="cuda")
    out = torch.empty(lib.N_GRAD_OUT, dtype=torch.float64, device="cuda")
    lib.pm_model_grad(dev, n, THETA, N_SM, torch.from_numpy(t_meas.astype(np.float32)).cuda(), ws, out)
    o = out.cpu().numpy()
    assert o[0] == pytest.approx(L_o, rel=1e-4, abs=1e-9)
    assert np.all(np.abs(o[1:] - g_o) <= 1e-4 * scale + 1e-30)
    # what the model cannot evaluate stays without a time
    bad = {f: v.copy() for f, v in c.items()}
    for f, v in (("M", 0), ("BM", -64), ("stages", 0), ("cta_group", 3), ("dtype", 3), ("kind", 7), ("tmem_a", 2)):
        bad[f][:] = v
        lib.pm_model_predict(lib.cfg_tensor(bad), n, THETA, N_SM, t)
        wrong = np.ones(n, bool) if f in ("M", "kind") else c["kind"] == 0
        assert np.all(np.isnan(t.cpu().numpy()[wrong])), f
        bad[f][:] = c[f]


@pytest.mark.parametrize("n_sm", [152, 3])
@pytest.mark.parametrize("w0", [None, 0.0])
def test_fp64_short_ways_agree_with_oracle(lib, reading, n_sm, w0):
    # every kind of record in one table; without the L2 blend the general way
    n = 20000
    c = edge_cfgs(n, 70)
    probes = np.arange(n) >= n - 600
    c["kind"][~probes] = 0
    c["kind"][probes] = 1 + np.arange(600) // 200
    th = O.prior_theta(N_SM, reading=reading)
    if w0 is not None:
        th[3] = w0
    t_o, gi = O.model_batch(c, th, n_sm, grad=True)
    t_meas = t_o * np.exp(0.3 * (S.uniform01_f64(71, n) - 0.5))
    L_o, g_o = O.model_loss_grad(c, th, n_sm, t_meas)
    r = np.log(t_o) - np.log(t_meas)
    scale = (2.0 / n) * np.sum(np.abs(r[:, None] * gi / t_o[:, None]), axis=0)
    ws = torch.empty(lib.pm_model_grad_workspace(n) // 8, dtype=torch.float64, device="cuda")
    out = torch.empty(lib.N_GRAD_OUT, dtype=torch.float64, device="cuda")
    lib.pm_model_grad_f64(lib.cfg_tensor(c), n, th, n_sm, torch.from_numpy(t_meas).cuda(), ws, out)
    o = out.cpu().numpy()
    assert o[0] == pytest.approx(L_o, rel=1e-10)
    assert np.all(np.abs(o[1:] - g_o) <= 1e-10 * scale + 1e-300)
