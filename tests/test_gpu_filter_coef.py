"""Mixed-form filter over the accepted coefficients, |alpha| < 1/2, against the
FP64 oracle: below and above the coefficient (0.287) beyond which the FP32
recurrences would need more start-up rows than they have and the sub-domain
sweep takes over, and far from it; x lines shorter and longer than 32 points,
several sub-domains along every axis.

Tolerance: per axis and point, 8 roundings of the right-hand side, 3 of the two
recurrences, 1 of the input and 1 for the cut tails (1e-8), each of at most 2^-24
times 2 max |D| (the weights' moduli sum to less than 2), amplified by the
tridiagonal inverse, 1 / (1 - 2 |alpha|) at most; three axes."""
import numpy as np
import pytest

import nopcs_synth as S
import oracle
from gpu_util import binding, stream_ptr, to_dev

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("alpha", [-0.45, -0.29, -0.28, 0.0, 1e-9, 0.135, 0.28, 0.29, 0.4, 0.45])
@pytest.mark.parametrize("n", [(29, 41, 36), (70, 27, 33)])
def test_mixed_filter_coefficients(n, alpha):
    import torch
    N = binding()
    p = S.box_params(n, sub_n=(12, 16, 10), base_subtract=1, filter_alpha=alpha, perturb_amp=1e-3, seed=2)
    orc = oracle.Solver(p)
    Q = orc.initial_state()
    rest = oracle.Solver(dict(p, perturb_amp=0.0)).initial_state()
    rng = np.random.default_rng(11)
    Q[0] *= 1 + 1e-4 * rng.standard_normal(Q[0].shape)
    Q[4] *= 1 + 1e-4 * rng.standard_normal(Q[4].shape)
    ref = orc.filter(Q.copy())
    ctx = N.nopcs_init([p], prec=N.NOPCS_MIXED, form=N.NOPCS_FORM_THOMAS, stream=stream_ptr())
    try:
        N.nopcs_set_state(ctx, 0, to_dev(Q).data_ptr())
        N.nopcs_filter(ctx, 0)
        out = torch.empty(Q.shape, dtype=torch.float64, device="cuda")
        N.nopcs_get_state(ctx, 0, out.data_ptr())
        got = out.cpu().numpy()
    finally:
        N.nopcs_destroy(ctx)
    dev = np.abs(Q - rest).reshape(5, -1).max(1)
    err = np.abs(got - ref).reshape(5, -1).max(1)
    change = np.abs(ref - Q).reshape(5, -1).max(1)
    tol = 3 * 13 * 2 * 2.0 ** -24 / (1 - 2 * abs(alpha)) * dev
    assert np.all(change > 50 * tol), (change, tol)
    assert np.all(err <= tol), err / tol
