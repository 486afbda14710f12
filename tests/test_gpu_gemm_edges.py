"""The GEMM epilogue at ragged edges: exact integer products where C has odd row
lengths, partial row chunks and every accumulator layout, with and without room
for the staging buffers."""
import numpy as np
import pytest

import oracle as O
import synthetic as S

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

# dtype and (BM, BN, BK, stages, cta_group): one row per lane, 64 rows on one SM
# (16 rows per warp) and on a pair (rows split over lanes), two row blocks; the
# five-stage 256 x 64 and 64 x 256 rings leave no room for staging
TILES = [(1, (128, 128, 64, 4, 1)), (1, (64, 128, 64, 4, 1)), (1, (64, 256, 64, 3, 2)), (1, (256, 256, 64, 3, 1)),
         (1, (256, 128, 64, 4, 2)), (1, (256, 64, 64, 5, 1)), (1, (64, 256, 64, 5, 1)), (2, (256, 256, 128, 3, 1)),
         (2, (64, 64, 64, 6, 2)), (0, (128, 128, 32, 2, 1)), (0, (64, 64, 32, 3, 2))]
SHAPES = [(1, 1, 16), (300, 201, 64), (33, 31, 128), (129, 1003, 64), (500, 260, 64), (31, 100, 64), (257, 128, 48),
          (1000, 66, 64)]


@pytest.mark.parametrize("dt,t", TILES, ids=["-".join(map(str, (d,) + t)) for d, t in TILES])
def test_ragged_products_are_exact_and_stay_inside_c(lib, dt, t):
    for M, N, K in SHAPES:
        A, B = S.integer_matrix(11, M, K), S.integer_matrix(12, K, N)
        ref = O.gemm_f64(A, B)
        ops = lib.GemmOperands(dt, M, N, K)
        ops.prepare(torch.from_numpy(A).cuda(), torch.from_numpy(B).cuda())
        # C in the middle of a guarded buffer, at offsets that allow and forbid 16-byte stores
        for off in (64, 65):
            buf = torch.full((M * N + 256,), -7.5, dtype=torch.float32, device="cuda")
            if off == 65 and N % 4 == 0 and M > 400:
                continue
            lib.pm_gemm_run(lib.cfg(M, N, K, *t, dtype=dt), ops.A_op, ops.B_op, buf.data_ptr() + 4 * off, ops.scales)
            torch.cuda.synchronize()
            assert lib.pm_device_status(True) == lib.PM_OK
            got = buf.cpu().numpy()
            assert np.all(got[:off] == -7.5) and np.all(got[off + M * N:] == -7.5), (M, N, K)
            C = got[off:off + M * N].reshape(M, N).astype(np.float64)
            if dt == 2:
                assert np.all(np.abs(C - ref) <= 2.0 ** -23 * np.abs(ref)), (M, N, K)
            else:
                assert np.array_equal(C, ref), (M, N, K)


@pytest.mark.parametrize("N", [260, 201])
@pytest.mark.parametrize("launch", [(64, 3, 1), (64, 3, 2)])
def test_grouped_ragged_rows_do_not_cross_groups(lib, launch, N):
    # partial row chunks at the end of a group are followed by another group's
    # rows, except in the last one, whose chunks the tensor map clips
    Ms = [33, 257, 1, 100, 45]
    K = 128
    A_list = [S.integer_matrix(31 + q, m, K) for q, m in enumerate(Ms)]
    B_list = [S.integer_matrix(91 + q, K, N) for q in range(len(Ms))]
    sum_m = sum(Ms)
    A_op = torch.empty(sum_m * K * 2, dtype=torch.uint8, device="cuda")
    B_op = torch.empty(len(Ms) * N * K * 2, dtype=torch.uint8, device="cuda")
    row = 0
    for q, (A, B) in enumerate(zip(A_list, B_list)):
        lib.pm_gemm_prepare(1, torch.from_numpy(A).cuda(), torch.from_numpy(B).cuda(), Ms[q], N, K,
                            A_op.data_ptr() + row * K * 2, B_op.data_ptr() + q * N * K * 2)
        row += Ms[q]
    for bm, bn in (([64, 256, 64, 128, 64], [64, 128, 256, 128, 64]), ([128] * 5, [128] * 5)):
        buf = torch.full((sum_m * N + 128,), -7.5, dtype=torch.float32, device="cuda")
        lib.pm_grouped_gemm_run(Ms, N, K, bm, bn, *launch, A_op, B_op, buf.data_ptr() + 256)
        torch.cuda.synchronize()
        got = buf.cpu().numpy()
        assert np.all(got[:64] == -7.5) and np.all(got[64 + sum_m * N:] == -7.5)
        C = got[64:64 + sum_m * N].reshape(sum_m, N).astype(np.float64)
        row = 0
        for A, B in zip(A_list, B_list):
            assert np.array_equal(C[row:row + A.shape[0]], O.gemm_f64(A, B))
            row += A.shape[0]
