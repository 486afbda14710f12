"""Operand preparation at the edges of its tiles and vector rules, bit-exact
against the CPU oracle's conversions: extents around the 64 x 64 tile and the
4096-element piece, rows that are not multiples of four elements, and matrices
whose base is only 4-byte aligned."""
import numpy as np
import pytest

import oracle as O
import synthetic as S

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

SHAPES = [(1, 1, 1), (3, 5, 7), (64, 64, 64), (65, 63, 66), (64, 128, 192), (127, 4, 4), (1, 4096, 4), (33, 65, 4100),
          (1023, 260, 1040)]


def prepared(lib, dt, A, B, shift):
    """Codes as (A planes, B planes) and scales, the FP32 inputs `shift` floats off their allocation."""
    M, K = A.shape
    N = B.shape[1]
    dev = []
    for X in (A, B):
        buf = torch.full((X.size + shift,), float("nan"), dtype=torch.float32, device="cuda")
        buf[shift:] = torch.from_numpy(X.ravel()).cuda()
        dev.append(buf)
    ops = lib.GemmOperands(dt, M, N, K)
    ops.A_op.fill_(0xA5)
    ops.B_op.fill_(0xA5)
    ops.prepare(dev[0].data_ptr() + 4 * shift, dev[1].data_ptr() + 4 * shift)
    return ops.A_op.cpu().numpy(), ops.B_op.cpu().numpy(), ops.scales.cpu().numpy()


@pytest.mark.parametrize("shift", [0, 1])
@pytest.mark.parametrize("dt", [0, 1, 2])
@pytest.mark.parametrize("M,N,K", SHAPES)
def test_prepare_bit_exact_at_tile_edges(lib, M, N, K, dt, shift):
    A, B = S.gemm_operands(M, N, K, seed=5 + dt, dist="uniform" if dt == 0 else "normal")
    a, b, scales = prepared(lib, dt, A, B, shift)
    for got, X in ((a, A), (b, B.T.copy())):
        if dt == 0:
            hi, lo = O.tf32_split(X)
            want = np.concatenate([hi.ravel(), lo.ravel()]).view(np.uint32)
            assert np.array_equal(got.view(np.uint32), want)
        elif dt == 1:
            codes = got.view(np.uint16).astype(np.uint32) << 16
            assert np.array_equal(codes.view(np.float32).reshape(X.shape), O.to_bf16(X))
        else:
            s = O.fp8_scale(X)
            assert scales[0 if X.shape == A.shape and got is a else 1] == s
            assert np.array_equal(got.reshape(X.shape), O.to_e4m3(X * s))


def test_prepare_fp8_zero_and_repeated(lib):
    # an all-zero operand keeps scale 1, and a second call starts its maxima anew
    A, B = S.gemm_operands(130, 70, 96, seed=9, dist="normal")
    ops = lib.GemmOperands(2, 130, 70, 96)
    ops.prepare(torch.from_numpy(1000 * A).cuda(), torch.from_numpy(B).cuda())
    ops.prepare(torch.from_numpy(A).cuda(), torch.zeros(96, 70, device="cuda"))
    sc = ops.scales.cpu().numpy()
    assert sc[0] == O.fp8_scale(A) and sc[1] == 1.0
    assert not ops.B_op.any()
