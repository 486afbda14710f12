"""Three-pass TF32 on two-stage rings, whose low planes arrive on a barrier of their
own: integers of 14 bits in one operand (their low plane is not zero) against small
ones in the other, so that every product and sum is exact in FP32."""
import numpy as np
import pytest

import oracle as O

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

# one and two row blocks, one and two swizzle atoms along K, CTA pairs, and the
# 256 x 256 accumulator that is released in halves
TILES = [(64, 64, 32, 2, 1), (128, 128, 32, 2, 1), (128, 256, 32, 2, 1), (128, 64, 64, 2, 1), (64, 64, 32, 2, 2),
         (256, 128, 32, 2, 2), (256, 256, 32, 2, 2)]
SHAPES = [(1, 1, 16), (130, 70, 32), (300, 201, 80), (700, 516, 144), (1500, 1003, 256)]


@pytest.mark.parametrize("t", TILES, ids=["-".join(map(str, t)) for t in TILES])
def test_low_planes_of_two_stage_rings_are_exact(lib, t):
    rng = np.random.default_rng(5)
    for M, N, K in SHAPES:
        for wide_a in (True, False):
            hi, lo = 2 ** 13, 3                     # |sum| < 2^13 * 2 * 256 = 2^22
            A = rng.integers(-hi + 1, hi, (M, K)) if wide_a else rng.integers(-2, lo, (M, K))
            B = rng.integers(-2, lo, (K, N)) if wide_a else rng.integers(-hi + 1, hi, (K, N))
            A, B = A.astype(np.float32), B.astype(np.float32)
            ops = lib.GemmOperands(0, M, N, K)
            ops.prepare(torch.from_numpy(A).cuda(), torch.from_numpy(B).cuda())
            C = torch.full((M, N), -7.5, dtype=torch.float32, device="cuda")
            ops.run(lib.cfg(M, N, K, *t, dtype=0), C)
            torch.cuda.synchronize()
            assert lib.pm_device_status(True) == lib.PM_OK
            assert np.array_equal(C.cpu().numpy().astype(np.float64), O.gemm_f64(A, B)), (M, N, K, wide_a)
