"""Which tile shape a launch of two-point CCZ4 tiles takes.

A launch takes rounds of one tile per SM, so a shape of fewer but slower tiles
pays only where it saves a round.  The shape is read from the kernels' names in
a profile; the outputs are compared with the FP64 oracle (as in
test_gpu_pair_tiles) and, for batches, with the patches' own launches.
"""
import numpy as np
import pytest
import torch

import oracle
from paper_1806_04182_gb300 import build, capi, inputs
from paper_1806_04182_gb300.state import PatchState

pytestmark = pytest.mark.gpu
SHAPES = {"flat": (32, 16, 1), "wide": (32, 8, 2), "deep": (16, 8, 4)}


@pytest.fixture(scope="module", autouse=True)
def lib():
    assert torch.cuda.is_available(), "GPU tests need CUDA"
    build.build()
    with torch.profiler.profile(activities=[torch.profiler.ProfilerActivity.CUDA]):  # (the first one may see nothing)
        torch.zeros(1, device="cuda").add_(1)
        torch.cuda.synchronize()
    return capi.lib()


def _state(n, q):
    U0, dx = inputs.z4_perturbed(n, seed=q, amp=0.03)
    st = PatchState(capi.SF_Z4, n, dx, 0.25 * min(dx), precision=capi.SF_FP32_BULK_DW,
                    x_pitch=(n[0] + 7 + 3) // 4 * 4, x_offset=1)
    st.upload(U0)
    for a in (st.B, st.C, st.D):
        a.fill_(float("nan"))
    return st, U0, dx


def _kernels(fn):
    """Names of the two-point kernels that fn launches."""
    torch.cuda.synchronize()
    with torch.profiler.profile(activities=[torch.profiler.ProfilerActivity.CUDA]) as prof:
        fn()
        torch.cuda.synchronize()
    names = {e.key for e in prof.key_averages() if "z4_pair" in e.key}
    if not names:
        pytest.skip("no kernel names from the profiler")
    return names


def _shapes(names):
    """The shapes in the kernels' template arguments."""
    return {k for k, t in SHAPES.items() for m in names if "PairShape<%d, %d, %d," % t in m}


@pytest.mark.skipif(torch.cuda.is_available() and
                    torch.cuda.get_device_properties(0).multi_processor_count != 152, reason="sizes for 152 SMs")
@pytest.mark.parametrize("n,shape", [((80, 24, 23), "flat"), ((48, 48, 48), "flat"), ((60, 20, 88), "wide"),
                                     ((70, 50, 61), "deep")])
def test_patch(n, shape):
    st, U0, dx = _state(n, 3)
    assert _shapes(_kernels(lambda: st.step(1))) == {shape}
    G = oracle.ghosted(U0.copy())
    oracle.rk4_step(oracle.Z4, G, dx, st.dt, oracle.params())
    want, got = oracle.interior(G), st.fields().cpu().numpy()
    bound = 4 * 64 / 12 * float(np.finfo(np.float32).eps) * st.dt / min(dx) ** 2 / 1e-2
    for f in range(25):
        e = np.abs(got[f] - want[f]).max() / max(np.abs(want[f]).max(), 1e-2)
        assert e < bound, (f, e, bound)


@pytest.mark.skipif(torch.cuda.is_available() and
                    torch.cuda.get_device_properties(0).multi_processor_count != 152, reason="sizes for 152 SMs")
@pytest.mark.parametrize("sizes,shapes", [([(32, 24, 8)] * 3, {"flat"}), ([(32, 24, 8)] * 24, {"wide"}),
                                          ([(48, 48, 12)] * 8, {"deep"}),
                                          ([(32, 8, 10)] * 60 + [(16, 8, 12)] * 60, {"wide", "deep"})])
def test_batch(sizes, shapes):
    one = [_state(n, q)[0] for q, n in enumerate(sizes)]
    many = [_state(n, q)[0] for q, n in enumerate(sizes)]
    b = capi.sf_batch_create(capi.params(), [s.patch(s.B, s.A, s.C) for s in many])
    stream = torch.cuda.current_stream().cuda_stream
    try:
        assert _shapes(_kernels(lambda: [capi.sf_batch_substep(b, k, stream) for k in range(4)])) == shapes
    finally:
        capi.sf_batch_destroy(b)
    for s, m in zip(one, many):
        s.step(1)
        assert torch.equal(s.interior(), m.interior()), s.n
