"""Kernels that are set up during the previous kernel of their stream: every
operand, workspace and result is settled before it is read or overwritten, in
chains of dependent calls, between other libraries' kernels, on several streams
and in captured graphs."""
import numpy as np
import pytest

import oracle as O
import synthetic as S

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

TILES = {0: (128, 128, 32, 2, 1), 1: (128, 128, 64, 4, 2), 2: (64, 64, 128, 6, 1)}


def problem(lib, dt, M, N, K, seed):
    A, B = S.integer_matrix(seed, M, K), S.integer_matrix(seed + 1, K, N)
    d = dict(A=torch.from_numpy(A).cuda(), B=torch.from_numpy(B).cuda(), ops=lib.GemmOperands(dt, M, N, K),
             C=torch.empty(M, N, dtype=torch.float32, device="cuda"), cfg=lib.cfg(M, N, K, *TILES[dt], dtype=dt))
    return d, O.gemm_f64(A, B)


def close(C, ref, dt):
    C = C.cpu().numpy().astype(np.float64)
    return np.all(np.abs(C - ref) <= 2.0 ** -23 * np.abs(ref)) if dt == 2 else np.array_equal(C, ref)


@pytest.mark.parametrize("dt", [0, 1, 2])
def test_chain_reuses_its_buffers(lib, dt):
    # one operand and result buffer for a chain of different products: a
    # preparation overwrites what the previous GEMM reads, a copy of C runs
    # between two GEMMs that write it
    M, N, K = 260, 196, 512
    d, _ = problem(lib, dt, M, N, K, 5)
    inputs = [problem(lib, dt, M, N, K, 7 + 2 * i) for i in range(6)]
    got = []
    for e, _ in inputs:
        d["ops"].prepare(e["A"], e["B"])
        d["ops"].run(d["cfg"], d["C"])
        got.append(d["C"].clone())
        d["ops"].run(d["cfg"], d["C"])
        got.append(d["C"].clone())
    for i, C in enumerate(got):
        assert close(C, inputs[i // 2][1], dt)
    assert lib.pm_device_status(True) == lib.PM_OK


@pytest.mark.parametrize("dt", [0, 1, 2])
def test_streams_and_graphs(lib, dt):
    M, N, K = 129, 260, 256
    probs = [problem(lib, dt, M, N, K, 40 + 2 * i) for i in range(3)]
    streams = [torch.cuda.Stream() for _ in probs]
    torch.cuda.synchronize()
    for _ in range(3):
        for (d, _), s in zip(probs, streams):
            d["ops"].prepare(d["A"], d["B"], stream=s)
            d["ops"].run(d["cfg"], d["C"], stream=s)
    torch.cuda.synchronize()
    assert all(close(d["C"], ref, dt) for d, ref in probs)
    # the same calls as one graph: three chains one after another, replayed
    g, s = torch.cuda.CUDAGraph(), torch.cuda.Stream()
    for d, _ in probs:
        d["C"].fill_(float("nan"))
    torch.cuda.synchronize()
    with torch.cuda.graph(g, stream=s):
        for d, _ in probs:
            d["ops"].prepare(d["A"], d["B"], stream=s)
            d["ops"].run(d["cfg"], d["C"], stream=s)
    for _ in range(3):
        g.replay()
    torch.cuda.synchronize()
    assert all(close(d["C"], ref, dt) for d, ref in probs)


def test_inputs_from_another_kernel(lib):
    # A is written by a kernel of PyTorch right before the call and overwritten
    # by one right after it
    M, N, K = 512, 512, 512
    d, ref = problem(lib, 1, M, N, K, 60)
    A0 = d["A"].clone()
    out = []
    for i in range(8):
        torch.mul(A0, float(2 ** (i % 4)), out=d["A"])
        d["ops"].prepare(d["A"], d["B"])
        d["A"].zero_()
        d["ops"].run(d["cfg"], d["C"])
        out.append(d["C"].clone())
        d["C"].zero_()
    for i, C in enumerate(out):
        assert close(C, ref * 2 ** (i % 4), 1)
