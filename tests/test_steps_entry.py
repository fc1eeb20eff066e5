"""sf_steps: argument errors (nothing is launched, no GPU needed), and on the
GPU the same bits as the stages called one by one."""
import pytest
import torch

from paper_1806_04182_gb300 import build, capi
from paper_1806_04182_gb300.state import PatchState


@pytest.fixture(scope="module", autouse=True)
def lib():
    build.build()
    return capi.lib()


def _geom(**kw):
    g = capi.sf_patch()
    g.n[:] = kw.pop("n", (8, 8, 8))
    g.ghost = 3
    g.dx[:] = (0.1, 0.1, 0.1)
    g.dt = 0.01
    for k, v in kw.items():
        setattr(g, k, v)
    return g


def _state(**kw):
    b = 1 << 20
    d = dict(u=b, s1=2 * b, s2=3 * b, acc=4 * b, kahan=5 * b)
    d.update(kw)
    return capi.sf_state(**d)


@pytest.mark.parametrize("prm,geom,state,nsteps,adjoint", [
    ({}, {}, {}, -1, False),
    (dict(rk=7), {}, {}, 1, False),
    ({}, dict(system=9), {}, 1, False),
    ({}, dict(n=(2, 8, 8)), {}, 1, False),
    ({}, {}, dict(u=None), 1, False),
    ({}, {}, dict(s1=None), 1, False),
    ({}, {}, dict(s2=None), 1, False),
    ({}, {}, dict(acc=None), 1, False),
    ({}, {}, dict(s1=1 << 20), 1, False),
    ({}, {}, dict(s2=2 << 20), 1, False),
    ({}, dict(precision=capi.SF_FP32_BULK), dict(kahan=None), 1, False),
    ({}, dict(system=capi.SF_Z4, cfl_rate=1 << 20), {}, 1, False),
    ({}, dict(system=capi.SF_Z4), {}, 1, True),
    (dict(rk=capi.SF_SSPRK3), {}, {}, 1, True),
])
def test_refused(prm, geom, state, nsteps, adjoint):
    before = capi.sf_launch_count()
    with pytest.raises(capi.SfError):
        capi.sf_steps(capi.params(**prm), _geom(**geom), _state(**state), nsteps, adjoint)
    assert capi.sf_launch_count() == before


@pytest.mark.gpu
@pytest.mark.parametrize("system,precision,rk", [
    (capi.SF_WAVE, capi.SF_FP64, capi.SF_RK4), (capi.SF_WAVE, capi.SF_FP32_BULK, capi.SF_RK4),
    (capi.SF_WAVE, capi.SF_FP64, capi.SF_SSPRK3), (capi.SF_MHD, capi.SF_FP32_BULK, capi.SF_SSPRK3),
    (capi.SF_MHD, capi.SF_FP64, capi.SF_RK4), (capi.SF_Z4, capi.SF_FP32_BULK_DW, capi.SF_RK4)])
def test_steps_equal_stages(system, precision, rk):
    n = (11, 9, 7)
    sts = [PatchState(system, n, (0.1,) * 3, 1e-3, precision=precision, prm=capi.params(rk=rk)) for _ in range(2)]
    g = torch.Generator(device="cuda").manual_seed(1)
    U = 0.01 * torch.rand(sts[0].nf, n[2], n[1], n[0], generator=g, device="cuda", dtype=torch.float64)
    for f in {capi.SF_MHD: (0, 4), capi.SF_Z4: (0, 1, 4, 6, 18)}.get(system, ()):
        U[f] += 1.0
    for s in sts:
        s.upload(U)
    sts[0].step(3)
    for _ in range(3):
        for q in range(sts[1].nstages):
            sts[1].stage(q)
    assert torch.equal(sts[0].A, sts[1].A)
    assert torch.isfinite(sts[0].A).all()
    if system == capi.SF_WAVE and rk == capi.SF_RK4:
        sts[0].adjoint_step(2)
        h = torch.cuda.current_stream().cuda_stream
        for _ in range(2):
            for q in range(4):
                capi.sf_adjoint_substep(sts[1].prm, sts[1].stage_patch(q), q, h)
        assert torch.equal(sts[0].A, sts[1].A)
