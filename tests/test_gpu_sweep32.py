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
