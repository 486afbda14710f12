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
