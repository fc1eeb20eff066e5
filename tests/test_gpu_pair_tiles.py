"""Two-point CCZ4 tiles at the edges of their shapes.

Patches of any size on the one-float row offset layout go in tiles of 32 x 16 x
1, 32 x 8 x 2 or 16 x 8 x 4 points, whichever covers them in the least time.  Sizes: one tile, one point less and more along each
axis, odd widths and depths, and sizes that take each shape; through
sf_substep, through a batch that mixes them and through batches of equal patches.  One RK4 step on NaN-filled
scratch against the FP64 oracle, within the float bound of the 1/dx^2 stencils
(64 rounding terms of |U| over 12 dx^2, four stages of dt, floor 1e-2); the
batch gives the same bits as the per-patch launches.
"""
import numpy as np
import pytest
import torch

import oracle
from paper_1806_04182_gb300 import build, capi, inputs
from paper_1806_04182_gb300.state import PatchState

pytestmark = pytest.mark.gpu
SIZES = [(3, 3, 3), (16, 8, 4), (15, 7, 3), (17, 9, 5), (32, 8, 2 + 1), (33, 8, 4), (31, 9, 7),
         (48, 16, 4), (20, 17, 6), (64, 15, 3), (32, 16, 1 + 2), (36, 41, 5), (33, 17, 3)]


@pytest.fixture(scope="module", autouse=True)
def lib():
    assert torch.cuda.is_available(), "GPU tests need CUDA"
    build.build()
    return capi.lib()


def _state(n, q):
    U0, dx = inputs.z4_perturbed(n, seed=q, amp=0.03)
    st = PatchState(capi.SF_Z4, n, dx, 0.25 * min(dx), precision=capi.SF_FP32_BULK_DW,
                    x_pitch=(n[0] + 7 + 3) // 4 * 4, x_offset=1)
    st.upload(U0)
    for a in (st.B, st.C, st.D):
        a.fill_(float("nan"))
    return st, U0, dx


def _check(st, U0, dx, got):
    G = oracle.ghosted(U0.copy())
    oracle.rk4_step(oracle.Z4, G, dx, st.dt, oracle.params())
    want = oracle.interior(G)
    bound = 4 * 64 / 12 * float(np.finfo(np.float32).eps) * st.dt / min(dx) ** 2 / 1e-2
    for f in range(25):
        e = np.abs(got[f] - want[f]).max() / max(np.abs(want[f]).max(), 1e-2)
        assert e < bound, (st.n, f, e, bound)


@pytest.mark.parametrize("n", SIZES)
def test_patch(n):
    st, U0, dx = _state(n, 3)
    st.step(1)
    g = st.A[:, :, :n[1] + 6, 1:n[0] + 7]
    assert torch.isfinite(g).all()
    # the ghost shell is the periodic image of the interior
    ref = g.clone()
    st.fill_ghosts(st.A)
    assert torch.equal(ref, g)
    _check(st, U0, dx, st.fields().cpu().numpy())
    assert capi.sf_get_device_status() == capi.SF_OK


@pytest.mark.parametrize("sizes", [SIZES] + [[n] * 3 for n in ((36, 41, 5), (32, 8, 4), (48, 16, 4))])
def test_batch(sizes):
    one = [_state(n, q) for q, n in enumerate(sizes)]
    many = [_state(n, q) for q, n in enumerate(sizes)]
    b = capi.sf_batch_create(capi.params(), [s.patch(s.B, s.A, s.C) for s, _, _ in many])
    try:
        assert capi.sf_batch_launches_per_step(b) == 4
        for stage in range(4):
            capi.sf_batch_substep(b, stage, torch.cuda.current_stream().cuda_stream)
        torch.cuda.synchronize()
    finally:
        capi.sf_batch_destroy(b)
    for (s, U0, dx), (m, _, _) in zip(one, many):
        s.step(1)
        assert torch.equal(s.interior(), m.interior()), s.n
