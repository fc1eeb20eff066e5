"""The marching wave kernel (float, patches of 200,000 points and more) against
the per-point kernel.

Both evaluate the same arithmetic, so the stages agree bit for bit; the
right-hand side output of sf_rhs always takes the per-point kernel, from which
the stage combination is formed here in float.  Sizes at the edges of its
32 x 8 columns and around the threshold, odd depths, padded rows, forward and
adjoint, with and without fused ghosts.
"""
import pytest
import torch

from paper_1806_04182_gb300 import build, capi
from paper_1806_04182_gb300.state import PatchState

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def lib():
    assert torch.cuda.is_available(), "GPU tests need CUDA"
    build.build()
    return capi.lib()


SIZES = [(64, 64, 49), (65, 57, 61), (33, 101, 67), (96, 8, 300), (31, 9, 801), (256, 33, 24)]


@pytest.mark.parametrize("n", SIZES)
@pytest.mark.parametrize("adjoint", [False, True])
def test_stages_equal_the_per_point_kernel(n, adjoint):
    assert n[0] * n[1] * n[2] >= 200000
    g = torch.Generator(device="cuda").manual_seed(sum(n))
    U = torch.rand(5, n[2], n[1], n[0], generator=g, device="cuda") - 0.5
    dx = (0.1, 0.2, 0.4)
    st = PatchState(capi.SF_WAVE, n, dx, 0.01, precision=capi.SF_FP32_BULK, x_pitch=n[0] + 9)
    st.upload(U)
    st.C.fill_(float("nan"))
    h = torch.cuda.current_stream().cuda_stream
    # a slab of the same data thin enough for the per-point kernel gives the stage's reference
    for s in range(4):
        us, nx = st.roles(s)
        un, acc, kah = st.A.clone(), st.D.clone(), st.E.clone()
        (capi.sf_adjoint_substep if adjoint else capi.sf_substep)(st.prm, st.stage_patch(s), s, h)
        z0, nz = n[2] // 2 - 4, 8 if n[0] * n[1] * 8 < 200000 else 1
        ref = PatchState(capi.SF_WAVE, (n[0], n[1], nz), dx, 0.01, precision=capi.SF_FP32_BULK,
                         x_pitch=n[0] + 9, prm=capi.params(ghosts=capi.SF_GHOSTS_NONE))
        cut = slice(z0, z0 + nz + 6)
        src = un if s == 0 else us
        arr = {k: torch.zeros_like(ref.A) for k in ("us", "un", "nx")}
        arr["us"].copy_(src[:, cut])
        arr["un"].copy_(un[:, cut])
        ref.D.copy_(acc[:, cut])
        ref.E.copy_(kah[:, cut])
        p = ref.patch(arr["un"] if s == 0 else arr["us"], arr["un"], arr["nx"])
        (capi.sf_adjoint_substep if adjoint else capi.sf_substep)(ref.prm, p, s, h)
        inner = (slice(None), slice(3, -3), slice(3, -3), slice(3, 3 + n[0]))
        got = nx[:, cut]
        assert torch.equal(arr["nx"][inner], got[inner]), (s, "next stage")
        assert torch.equal(ref.D[inner], st.D[:, cut][inner]), (s, "accumulator")
        assert torch.equal(ref.E[inner], st.E[:, cut][inner]), (s, "compensation")
        box = nx[:, :, :, :n[0] + 6].clone()
        st.fill_ghosts(nx)
        assert torch.equal(box, nx[:, :, :, :n[0] + 6]), (s, "ghost shell")


def test_ghosts_left_to_the_caller_and_flagged_values():
    n = (64, 64, 50)
    st = PatchState(capi.SF_WAVE, n, (0.1,) * 3, 0.01, precision=capi.SF_FP32_BULK,
                    prm=capi.params(ghosts=capi.SF_GHOSTS_NONE, check_finite=1))
    st.A.normal_()
    st.B.fill_(7.0)
    st.stage(0)
    shell = st.B.clone()
    shell[:, 3:-3, 3:-3, 3:-3] = 7.0
    assert bool((shell == 7.0).all())
    assert capi.sf_get_device_status() == capi.SF_OK
    st.A[2, 20, 30, 40] = float("inf")
    st.stage(0)
    assert capi.sf_get_device_status() == capi.SF_ENONFINITE
