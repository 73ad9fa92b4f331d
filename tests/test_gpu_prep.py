"""Primitive recovery of the mixed form on either side of the sizes (rows of 64
points, 152 rows) that pick hardware or integer conversions: a run interrupted by
get_state and set_state (which recovers the primitives anew, by either kernel)
continues bit for bit like one that is not (whose stage kernel recovered them).
The state holds momenta that binary32 has as subnormals, zeros of both signs and
values below its range."""
import numpy as np
import pytest

import nopcs_synth as S
import oracle
from gpu_util import binding, stream_ptr, to_dev

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [(5, 12, 14), (64, 16, 11), (65, 16, 11), (65, 5, 6), (97, 8, 19), (257, 12, 13)])
@pytest.mark.parametrize("ga", [0, 2])
def test_recovered_primitives_have_the_same_bits(n, ga):
    import torch
    N = binding()
    p = S.box_params(n, sub_n=(0, 0, 0), perturb_amp=1e-3, gravity_axis=ga, base_subtract=1, filter_every=2)
    Q = oracle.Solver(p).initial_state()
    inner = Q[1:4, 1:-1, 1:-1, 1:-1]
    odd = np.array([0.0, -0.0, 1e-40, -3e-42, 1e-300, -1e-46])
    inner[:] = np.where(np.arange(inner.size).reshape(inner.shape) % 3 == 0,
                        odd[np.arange(inner.size).reshape(inner.shape) % 6], inner)
    ctx = N.nopcs_init([p], prec=N.NOPCS_MIXED, stream=stream_ptr())
    try:
        out = []
        for cut in (False, True):
            N.nopcs_set_state(ctx, 0, to_dev(Q).data_ptr())
            N.nopcs_set_step(ctx, 0, 0)
            q = torch.empty(Q.shape, dtype=torch.float64, device="cuda")
            for _ in range(4):
                N.nopcs_rk_step(ctx, 1)
                N.nopcs_get_state(ctx, 0, q.data_ptr())
                if cut:
                    N.nopcs_set_state(ctx, 0, q.data_ptr())
            out.append(q.cpu().numpy())
    finally:
        N.nopcs_destroy(ctx)
    assert np.array_equal(out[0], out[1])
    assert not np.array_equal(out[0], Q)
