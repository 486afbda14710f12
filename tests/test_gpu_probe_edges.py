"""Copy, triad and stencil probes at the edges of their blocks, bit-exact against
the CPU references, with guards around the outputs."""
import numpy as np
import pytest

import oracle as O
import synthetic as S

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

GUARD = 64


def guarded(n):
    buf = torch.full((n + 2 * GUARD,), -7.5, dtype=torch.float32, device="cuda")
    return buf, buf.data_ptr() + 4 * GUARD


def inside(buf, n):
    got = buf.cpu().numpy()
    assert np.all(got[:GUARD] == -7.5) and np.all(got[GUARD + n:] == -7.5)
    return got[GUARD:GUARD + n]


# fewer than a vector, a vector, half a block of 512 vectors, a block, one more
@pytest.mark.parametrize("n", [1, 3, 4, 5, 1023, 1024, 2047, 2048, 2049, 2052, 4099, 300000])
def test_copy_and_triad_block_edges(lib, n):
    x, y = S.normal(1, n), S.uniform_pm1(2, n)
    xd, yd = torch.from_numpy(x).cuda(), torch.from_numpy(y).cuda()
    buf, p = guarded(n)
    lib.pm_probe_launch(lib.probe_args(lib.PM_PROBE_COPY, n=n), xd, p)
    assert np.array_equal(inside(buf, n).view(np.uint32), x.view(np.uint32))
    buf, p = guarded(n)
    lib.pm_probe_launch(lib.probe_args(lib.PM_PROBE_TRIAD, n=n, scalar=3.0), p, xd, yd)
    assert np.array_equal(inside(buf, n).view(np.uint32), O.triad_f32(x, y, 3.0).view(np.uint32))
    # in place: every element is read before it is written
    lib.pm_probe_launch(lib.probe_args(lib.PM_PROBE_TRIAD, n=n, scalar=3.0), xd, xd, yd)
    assert np.array_equal(xd.cpu().numpy().view(np.uint32), O.triad_f32(x, y, 3.0).view(np.uint32))


# one and two rows per thread (below and from one block of the latter per SM),
# rows that end inside a thread's, a warp's and a block's, one warp of columns and less
@pytest.mark.parametrize("rows", [1, 2, 3, 7, 8, 9, 15, 16, 17, 33, 2431, 2432])
@pytest.mark.parametrize("cols", [8, 12, 124, 128, 132, 260])
def test_stencil_block_edges(lib, rows, cols):
    x = S.normal(rows * cols, rows * cols).reshape(rows, cols)
    buf, p = guarded(rows * cols)
    lib.pm_probe_launch(lib.probe_args(lib.PM_PROBE_STENCIL, rows=rows, cols=cols), torch.from_numpy(x).cuda(), p)
    want = O.stencil5_f32(x)
    assert np.array_equal(inside(buf, rows * cols).view(np.uint32), want.ravel().view(np.uint32))
