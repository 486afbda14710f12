"""Chains of overlapping launches with nothing between them: the same calls, with a
synchronisation after each, give the reference bit for bit.  Every step has its own
inputs, scales and result, and the products are long (many K-steps, few tiles), so
that a preparation or a product that did not wait would read or write too early."""
import numpy as np
import pytest

import oracle as O
import synthetic as S

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

TILES = {0: (128, 128, 32, 2, 1), 1: (128, 128, 64, 4, 2), 2: (64, 64, 128, 6, 1)}
N_SM = 152
THETA = O.prior_theta(N_SM).astype(np.float32).astype(np.float64)


def normal(shape, factor, seed):
    g = torch.Generator(device="cuda").manual_seed(seed)
    return torch.randn(shape, device="cuda", generator=g) * factor


def run_both(calls, outputs):
    """Runs calls(step) with step() between any two calls: once synchronising there, twice not, once as a
    replayed graph; outputs() are compared after each."""
    s = torch.cuda.Stream()

    def clean():
        for t in outputs():
            t.view(torch.uint8).fill_(0xFF)              # NaN in every float type
        torch.cuda.synchronize()

    clean()
    calls(s, torch.cuda.synchronize)
    torch.cuda.synchronize()
    want = [t.clone() for t in outputs()]
    for _ in range(2):
        clean()
        calls(s, lambda: None)
        torch.cuda.synchronize()
        for t, w in zip(outputs(), want):
            assert torch.equal(t.view(torch.uint8), w.view(torch.uint8))
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, stream=s):
        calls(s, lambda: None)
    for _ in range(2):
        clean()
        g.replay()
        torch.cuda.synchronize()
        for t, w in zip(outputs(), want):
            assert torch.equal(t.view(torch.uint8), w.view(torch.uint8))


# the second product's operands overwrite what the first is still reading
@pytest.mark.parametrize("dt", [0, 1, 2])
def test_products_through_one_operand_buffer(lib, dt):
    M, N, K = 192, 256, 8192
    steps = [(normal((M, K), f, 10 + i), normal((K, N), 1 / (1 + i), 20 + i)) for i, f in
             enumerate((1.0, 37.0, 0.02, 5.0))]
    C = [torch.empty(M, N, device="cuda") for _ in steps]
    ops = lib.GemmOperands(dt, M, N, K)
    c = lib.cfg(M, N, K, *TILES[dt], dtype=dt)

    def calls(s, step):
        for (A, B), out in zip(steps, C):
            ops.prepare(A, B, stream=s)
            step()
            ops.run(c, out, stream=s)
            step()

    run_both(calls, lambda: C + [ops.A_op, ops.B_op] + ([ops.scales] if dt == 2 else []))
    assert all(torch.isfinite(t).all() for t in C)


# a product's result is the next preparation's input, as in a stack of layers
@pytest.mark.parametrize("dt", [0, 1, 2])
def test_result_straight_into_the_next_preparation(lib, dt):
    M, W = 128, 4096
    X0 = normal((M, W), 3.0, 30)
    weights = [normal((W, W), f / 64, 31 + i) for i, f in enumerate((1.0, 2.5, 0.3))]
    X = [torch.empty(M, W, device="cuda") for _ in weights]
    ops = [lib.GemmOperands(dt, M, W, W) for _ in range(2)]
    c = lib.cfg(M, W, W, *TILES[dt], dtype=dt)

    def calls(s, step):
        x = X0
        for i, w in enumerate(weights):
            ops[i % 2].prepare(x, w, stream=s)
            step()
            ops[i % 2].run(c, X[i], stream=s)
            step()
            x = X[i]

    run_both(calls, lambda: X)
    assert all(torch.isfinite(t).all() for t in X)


# a long product and a short one write one C; the later one's values stay
@pytest.mark.parametrize("dt", [0, 1, 2])
def test_two_products_into_one_result(lib, dt):
    M, N = 192, 256
    probs = []
    for K, seed in ((16384, 50), (256, 52)):
        ops = lib.GemmOperands(dt, M, N, K)
        ops.prepare(normal((M, K), 1.0, seed), normal((K, N), 7.0, seed + 1))
        probs.append((ops, lib.cfg(M, N, K, *TILES[dt], dtype=dt)))
    C = torch.empty(M, N, device="cuda")

    def calls(s, step):
        for ops, c in probs * 3:
            ops.run(c, C, stream=s)
            step()

    run_both(calls, lambda: [C])


# the sums are read only after the partial records of the same call are written
@pytest.mark.parametrize("n", [300, 3000, 200003])
@pytest.mark.parametrize("f64", [False, True])
def test_gradients_in_a_row(lib, n, f64):
    ws = torch.empty(lib.pm_model_grad_workspace(n) // 8, dtype=torch.float64, device="cuda")
    tables = []
    for i in range(3):
        c = S.model_config_batch(n, seed=60 + i)
        c["kind"] = np.zeros(n, dtype=np.int32)
        t = torch.full((n,), 1e-4 * (i + 1), dtype=torch.float64 if f64 else torch.float32, device="cuda")
        tables.append((lib.cfg_tensor(c), t, torch.empty(lib.N_GRAD_OUT, dtype=torch.float64, device="cuda")))
    grad = lib.pm_model_grad_f64 if f64 else lib.pm_model_grad

    def calls(s, step):
        for dev, t, out in tables:
            grad(dev, n, THETA, N_SM, t, ws, out, stream=s)
            step()

    run_both(calls, lambda: [t[2] for t in tables] + [ws])
    assert all(torch.isfinite(t[2]).all() for t in tables)
