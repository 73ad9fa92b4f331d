"""Wall nodes of the smallest boxes, where the edge nodes that the corners read
overlap from both ends of an edge and the remaining edge nodes are few or none,
against the FP64 oracle: every wall, edge and corner node after one RK step of a
state whose temperature varies from node to node by 1e-3.  Gates: those of
test_gpu_rk.py, 1e-12 (FP64 form) and 1e-5 (mixed form)."""
import numpy as np
import pytest

import nopcs_synth as S
import oracle
from gpu_util import binding, field_rel, state_err, stream_ptr, to_dev

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec,launch", [(0, 0), (1, 0), (1, 1)])
@pytest.mark.parametrize("n,ga", [((5, 6, 7), 2), ((7, 5, 6), 1), ((6, 7, 5), 0), ((9, 5, 40), 2)])
def test_walls_of_small_boxes(prec, launch, n, ga):
    import torch
    N = binding()
    p = S.box_params(n, sub_n=(0, 0, 0), base_subtract=prec, gravity_axis=ga, dt=1e-6, filter_every=0)
    orc = oracle.Solver(p)
    Q = orc.initial_state()
    rng = np.random.default_rng(3)
    Q[0] *= 1 + 1e-3 * rng.standard_normal(Q[0].shape)
    Q[4] *= 1 + 1e-3 * rng.standard_normal(Q[4].shape)
    ref = orc.step(Q.copy(), 1)
    ctx = N.nopcs_init([p], prec=prec, stream=stream_ptr())
    try:
        if launch:
            N.nopcs_set_launch(ctx, launch)
        N.nopcs_set_state(ctx, 0, to_dev(Q).data_ptr())
        N.nopcs_rk_step(ctx, 1)
        out = torch.empty(Q.shape, dtype=torch.float64, device="cuda")
        N.nopcs_get_state(ctx, 0, out.data_ptr())
        got = out.cpu().numpy()
        inner = (slice(None), slice(1, -1), slice(1, -1), slice(1, -1))
        got[inner] = ref[inner]
        if prec == 0:
            assert np.all(state_err(got, ref, p) <= 1e-12), state_err(got, ref, p)
        else:
            assert np.all(field_rel(got, ref)[[0, 4]] <= 1e-5), field_rel(got, ref)
            assert np.all(got[1:4][ref[1:4] == 0] == 0)
    finally:
        N.nopcs_destroy(ctx)
