"""CCZ4 monitors of float states whose values take the slow branches.

The monitor kernel widens floats by moving their bits and evaluates ln det by a
series near det = 1.  Planted here: subnormal values (widened by the conversion
instruction instead), signed zeros, determinants far from 1 (log() instead of
the series), and the values next to the series' limit.  Against the FP64
oracle on the same values, relative 1e-10 as for the other monitors; a value
that is not finite must still be counted and reach the sums.
"""
import numpy as np
import pytest
import torch

import oracle
from paper_1806_04182_gb300 import build, capi, inputs
from paper_1806_04182_gb300.state import PatchState

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def lib():
    assert torch.cuda.is_available(), "GPU tests need CUDA"
    build.build()
    return capi.lib()


@pytest.mark.parametrize("stretch", [1.0, 1.02, 1.021, 1.3, 0.7])
@pytest.mark.parametrize("precision", [capi.SF_FP64, capi.SF_FP32_BULK])
def test_monitors(stretch, precision):
    n = (21, 9, 7)
    U, dx = inputs.z4_perturbed(n, seed=4, amp=0.02)
    U[[1, 4, 6]] *= stretch
    U[[2, 9, 17], 2, 3, 4:9] = 1e-40
    U[[3, 8, 15], 1, 2, ::2] = -0.0
    st = PatchState(capi.SF_Z4, n, dx, 0.01, precision=precision)
    st.upload(U)
    V = st.fields().cpu().numpy()
    if precision != capi.SF_FP64:
        assert (np.abs(st.A[17].cpu().numpy()) == np.float32(1e-40)).any()
    d = st.diagnostics().cpu().numpy()
    assert d[4] == 0
    m = oracle.z4_monitors(oracle.ghosted(V), dx)
    np.testing.assert_allclose(np.sqrt(d[:4] / np.prod(n)), m, rtol=1e-10)


@pytest.mark.parametrize("value", [float("inf"), float("nan")])
@pytest.mark.parametrize("precision", [capi.SF_FP64, capi.SF_FP32_BULK])
def test_nonfinite(value, precision):
    n = (12, 8, 5)
    U, dx = inputs.z4_perturbed(n, seed=5, amp=0.02)
    st = PatchState(capi.SF_Z4, n, dx, 0.01, precision=precision)
    st.upload(U)
    st.A[17, 5, 6, 7] = value
    d = st.diagnostics().cpu().numpy()
    assert d[4] == 1 and not np.isfinite(d[0]) and np.isfinite(d[1:4]).all()
