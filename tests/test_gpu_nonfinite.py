"""Lines of one field are independent: a NaN or an infinity in one of them
leaves every other line's result as it is without it, bit for bit -- wherever
along the line it sits, for lines shorter and longer than what both walls reach,
with and without 16-byte rows.  The same for a right-hand side at the points
that no line and no viscous stencil connects with the bad one, and for the
filter.  Within the bad line, the explicit rows next to the walls depend on the
points of their closure alone."""
import numpy as np
import pytest

import nopcs_synth as S
from gpu_util import binding, stream_ptr, to_dev

pytestmark = pytest.mark.gpu

BAD = [float("nan"), float("inf")]


def _places(n):
    return [0, n // 2, n - 1]


@pytest.mark.parametrize("N", [13, 25, 31, 32, 40, 41, 64, 101])
@pytest.mark.parametrize("axis", [0, 1, 2])
def test_derivative_lines_are_independent(axis, N):
    import torch
    B = binding()
    n = [6, 7, 7]
    n[axis] = N
    p = S.box_params(n, sub_n=(16, 16, 16), perturb_amp=0.0)
    ctx = B.nopcs_init([p], prec=B.NOPCS_MIXED, form=B.NOPCS_FORM_THOMAS, stream=stream_ptr())
    try:
        f = np.random.default_rng(N).uniform(0.5, 1.0, n[::-1]).astype(np.float32)
        fd = to_dev(f)

        def run(order):
            out = torch.empty_like(fd)
            B.nopcs_derivative(ctx, 0, axis, order, 1, fd.data_ptr(), out.data_ptr(), stream_ptr())
            return out.movedim(2 - axis, -1).clone()

        lines = fd.movedim(2 - axis, -1)  # [a][b][along]
        for order in (1, 2, 3):
            clean = run(order)
            assert torch.isfinite(clean).all()
            for bad in BAD:
                for at in _places(N):
                    keep = lines[3, 2, at].clone()
                    lines[3, 2, at] = bad
                    got = run(order)
                    lines[3, 2, at] = keep
                    assert not torch.isfinite(got[3, 2]).all()
                    got[3, 2] = clean[3, 2]
                    diff = (got != clean).any(-1).nonzero().tolist()
                    assert not diff, (order, bad, at, diff)
    finally:
        B.nopcs_destroy(ctx)


@pytest.mark.parametrize("compact", [0, 1])
@pytest.mark.parametrize("nx", [29, 40, 41])
def test_rhs_of_unconnected_points(nx, compact):
    """Explicit viscous terms: the points that share a line with the bad one, and
    those within four nodes of it along every axis (two stencils of two, three
    next to a wall), may change; compact ones pass it on along two axes."""
    import torch
    B = binding()
    n = (nx, 14, 15)
    p = S.box_params(n, sub_n=(0, 0, 0), base_subtract=1, perturb_amp=1e-3, seed=4, visc_compact=compact)
    ctx = B.nopcs_init([p], prec=B.NOPCS_MIXED, form=B.NOPCS_FORM_THOMAS, stream=stream_ptr())
    try:
        q = torch.empty((5,) + n[::-1], dtype=torch.float64, device="cuda")
        B.nopcs_get_state(ctx, 0, q.data_ptr())

        def run():
            r = torch.empty(q.shape, dtype=torch.float32, device="cuda")
            B.nopcs_rhs(ctx, 0, q.data_ptr(), r.data_ptr())
            return r

        clean = run()
        assert torch.isfinite(clean).all()
        # with y0 the last line of a plane, the next line in memory order is of
        # the next plane
        z0, y0 = 7, (n[1] - 1 if compact else 6)
        z, y, x = np.ogrid[:n[2], :n[1], :n[0]]
        for bad in BAD:
            for x0 in _places(nx):
                keep = q[:, z0, y0, x0].clone()
                q[0 if bad != bad else 4, z0, y0, x0] = bad
                got = run()
                q[:, z0, y0, x0] = keep
                same = [x == x0, y == y0, z == z0]
                if compact:
                    free = ~(same[0] | same[1] | same[2])
                else:
                    free = ~((same[0] & same[1]) | (same[0] & same[2]) | (same[1] & same[2]))
                free = free & ~((abs(x - x0) <= 4) & (abs(y - y0) <= 4) & (abs(z - z0) <= 4))
                assert not torch.isfinite(got).all()
                diff = ((got != clean).any(0).cpu().numpy() & free).nonzero()
                assert diff[0].size == 0, (bad, x0, [d[:5] for d in diff])
    finally:
        B.nopcs_destroy(ctx)


@pytest.mark.parametrize("nx", [13, 25, 31, 40, 41, 64])
def test_filter_of_unconnected_lines(nx):
    """Six points along y and z: the filter leaves all of them as they are, so it
    acts along x alone."""
    import torch
    B = binding()
    n = (nx, 6, 6)
    p = S.box_params(n, sub_n=(16, 0, 0), base_subtract=1, perturb_amp=1e-3, seed=4)
    ctx = B.nopcs_init([p], prec=B.NOPCS_MIXED, form=B.NOPCS_FORM_THOMAS, stream=stream_ptr())
    try:
        q = torch.empty((5,) + n[::-1], dtype=torch.float64, device="cuda")
        B.nopcs_get_state(ctx, 0, q.data_ptr())

        def run():
            out = torch.empty_like(q)
            B.nopcs_set_state(ctx, 0, q.data_ptr())
            B.nopcs_filter(ctx, 0)
            B.nopcs_get_state(ctx, 0, out.data_ptr())
            return out

        clean = run()
        assert torch.isfinite(clean).all() and not torch.equal(clean, q)
        for bad in BAD:
            for at in _places(nx):
                keep = q[:, 2, 3, at].clone()
                q[:, 2, 3, at] = bad
                got = run()
                q[:, 2, 3, at] = keep
                got[:, 2, 3] = clean[:, 2, 3]
                diff = (got != clean).any(0).nonzero().tolist()
                assert not diff, (bad, at, diff[:5])
    finally:
        B.nopcs_destroy(ctx)


@pytest.mark.parametrize("dtype", [0, 1])
@pytest.mark.parametrize("N", [13, 26, 40, 41, 64, 101])
@pytest.mark.parametrize("axis", [0, 1, 2])
def test_explicit_rows_of_the_bad_line(axis, N, dtype):
    """The rows next to the walls are explicit, with taps on the five points from
    the wall at most: a bad value beyond these leaves them as they are (first
    derivative and compact second derivative)."""
    import torch
    B = binding()
    n = [6, 7, 7]
    n[axis] = N
    p = S.box_params(n, sub_n=(16, 16, 16), perturb_amp=0.0)
    ctx = B.nopcs_init([p], prec=B.NOPCS_MIXED, form=B.NOPCS_FORM_THOMAS, stream=stream_ptr())
    try:
        f = np.random.default_rng(N).uniform(0.5, 1.0, n[::-1])
        fd = to_dev(f, np.float32 if dtype else np.float64)

        def run(order):
            out = torch.empty_like(fd)
            B.nopcs_derivative(ctx, 0, axis, order, dtype, fd.data_ptr(), out.data_ptr(), stream_ptr())
            return out.movedim(2 - axis, -1)[3, 2].clone()

        line = fd.movedim(2 - axis, -1)[3, 2]
        rows = [0, 1, N - 2, N - 1]
        for order in (1, 3):
            clean = run(order)
            for bad in BAD:
                for at in (5, N // 2, N - 6):
                    keep = line[at].clone()
                    line[at] = bad
                    got = run(order)
                    line[at] = keep
                    assert not torch.isfinite(got).all()
                    assert torch.equal(got[rows], clean[rows]), (order, bad, at, got[rows], clean[rows])
    finally:
        B.nopcs_destroy(ctx)
