"""FP32 flux sweeps (recurrences along the lines, csrc/sweep32.cuh) at the sizes
where their pieces end: lines shorter and longer than what both walls reach,
lengths around multiples of the 8-point chunks and of a segment, with and
without 16-byte rows, every gravity axis; one mixed-form right-hand side
against the FP64 oracle.

Tolerance: a derivative of values f by a line operator with taps of at most
1.6 / h carries binary32 rounding of a few ulps of max |f| / h, and the tap
cut-off of 1e-8 less; the bound allows 32 ulps of the largest flux over h (sum
of the three axes) on top of 1e-6 of the field's maximum."""
import numpy as np
import pytest

import nopcs_synth as S
import oracle
from gpu_util import binding, stream_ptr, to_dev

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("ga", [0, 1, 2])
@pytest.mark.parametrize("n", [(5, 31, 33), (31, 9, 64), (32, 40, 27), (33, 98, 10), (36, 34, 97), (104, 17, 41),
                               (209, 8, 130), (13, 300, 16), (12, 15, 301)])
def test_rhs_at_piece_ends(n, ga):
    import torch
    N = binding()
    p = S.box_params(n, sub_n=(0, 0, 0), base_subtract=1, perturb_amp=1e-3, seed=3, gravity_axis=ga)
    ctx = N.nopcs_init([p], prec=N.NOPCS_MIXED, form=N.NOPCS_FORM_THOMAS, stream=stream_ptr())
    try:
        orc = oracle.Solver(p)
        Q = orc.initial_state()
        rng = np.random.default_rng(5)
        Q[0] *= 1 + 1e-4 * rng.standard_normal(Q[0].shape)
        Q[4] *= 1 + 1e-4 * rng.standard_normal(Q[4].shape)
        ref = orc.rhs(Q)
        for ax in (1, 2, 3):
            for end in (0, -1):
                ref[1:4].swapaxes(1, ax)[:, end] = 0
        r = torch.empty(Q.shape, dtype=torch.float32, device="cuda")
        N.nopcs_rhs(ctx, 0, to_dev(Q).data_ptr(), r.data_ptr())
        got = r.cpu().numpy().astype(np.float64)
        # largest fluxes: rho u; rho u u + p' ; H u
        u = np.abs(Q[1:4] / Q[0]).max()
        pr = (p["gamma"] - 1) * (Q[4] - 0.5 * (Q[1] ** 2 + Q[2] ** 2 + Q[3] ** 2) / Q[0])
        rest = oracle.Solver(dict(p, perturb_amp=0.0)).initial_state()
        dp = np.abs(pr - (p["gamma"] - 1) * rest[4]).max()
        flux = np.array([Q[0].max() * u] + 3 * [Q[0].max() * u * u + dp] + [(Q[4] + pr).max() * u])
        h = p["len"][0] / (n[0] - 1)
        err = np.abs(got - ref).reshape(5, -1).max(1)
        tol = 3 * 32 * 2.0 ** -24 * flux / h + 1e-6 * np.abs(ref).reshape(5, -1).max(1)
        assert np.all(err <= tol), (err / tol)
    finally:
        N.nopcs_destroy(ctx)


@pytest.mark.parametrize("n", [(41, 6, 50), (65, 40, 9), (72, 33, 64), (24, 57, 30)])
@pytest.mark.parametrize("order", [1, 3])
def test_equal_lines_give_equal_bits(n, order):
    """A field that varies along one axis only: every line along it has the bits
    of the first, wherever its points fall in a warp or a block, and the FP32
    result is within its rounding of the FP64 one (order 1: 32 ulps of max |f|
    times the largest tap, 1.6 / h; order 3: 64 ulps times 4 / h^2)."""
    import torch
    N = binding()
    p = S.box_params(n, sub_n=(16, 12, 24), perturb_amp=0.0)
    ctx = N.nopcs_init([p], prec=N.NOPCS_MIXED, form=N.NOPCS_FORM_THOMAS, stream=stream_ptr())
    try:
        h = p["len"][0] / (n[0] - 1)
        for axis in range(3):
            v = np.random.default_rng(axis).uniform(0.5, 1.0, n[axis])
            shape = [1, 1, 1]
            shape[2 - axis] = n[axis]
            f = np.broadcast_to(v.astype(np.float32).reshape(shape), n[::-1]).copy()
            res = []
            for dtype, fd in ((1, to_dev(f, np.float32)), (0, to_dev(f.astype(np.float64)))):
                out = torch.empty_like(fd)
                N.nopcs_derivative(ctx, 0, axis, order, dtype, fd.data_ptr(), out.data_ptr(), stream_ptr())
                torch.cuda.synchronize()
                res.append(np.moveaxis(out.cpu().numpy(), 2 - axis, -1).reshape(-1, n[axis]))
            assert np.array_equal(res[0], np.broadcast_to(res[0][:1], res[0].shape)), axis
            tol = 32 * 2.0 ** -24 * 1.6 / h if order == 1 else 64 * 2.0 ** -24 * 4.0 / h ** 2
            assert np.abs(res[0][0] - res[1][0]).max() <= tol, axis
    finally:
        N.nopcs_destroy(ctx)
