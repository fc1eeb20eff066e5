"""sf_batch_tune times the kernel that the batch then runs.

A batch with CCZ4 patches that have no tiles of their own (FP64) runs its wave
patches in the persistent kernel beside them, so their work shapes are to be
measured there, not in the kernel of batches whose remaining patches are all
wave patches.  The kernels are read from a profile.
"""
import pytest
import torch

from paper_1806_04182_gb300 import build, capi, inputs
from paper_1806_04182_gb300.state import PatchState

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def lib():
    assert torch.cuda.is_available(), "GPU tests need CUDA"
    build.build()
    with torch.profiler.profile(activities=[torch.profiler.ProfilerActivity.CUDA]):  # (the first one may see nothing)
        torch.zeros(1, device="cuda").add_(1)
        torch.cuda.synchronize()
    return capi.lib()


def _tuned(systems):
    """Names of the batch kernels that tuning a batch of these systems launches."""
    states = []
    for q, system in enumerate(systems):
        n = (12, 10, 9)
        U0, dx = inputs.wave_plane(n, seed=q) if system == capi.SF_WAVE else inputs.z4_perturbed(n, seed=q, amp=0.01)
        st = PatchState(system, n, dx, 0.1 * min(dx), precision=capi.SF_FP64)
        st.upload(U0)
        states.append(st)
    b = capi.sf_batch_create(capi.params(), [s.patch(s.B, s.A, s.C) for s in states])
    try:
        torch.cuda.synchronize()
        with torch.profiler.profile(activities=[torch.profiler.ProfilerActivity.CUDA]) as prof:
            capi.sf_batch_tune(b, torch.cuda.current_stream().cuda_stream)
            torch.cuda.synchronize()
    finally:
        capi.sf_batch_destroy(b)
    names = [e.key for e in prof.key_averages() if "batch_" in e.key and "kernel" in e.key]
    if not names:
        pytest.skip("no kernel names from the profiler")
    return {k for k in ("batch_wave_kernel", "batch_stage_kernel") if any(k in n for n in names)}


def test_mixed_batch():
    assert _tuned([capi.SF_WAVE, capi.SF_Z4, capi.SF_WAVE]) == {"batch_stage_kernel"}


def test_wave_batch():
    assert _tuned([capi.SF_WAVE] * 3) == {"batch_wave_kernel"}
