"""FP64 CCZ4 right-hand side and stages away from flat space, against the
oracle, on both sides of its launch rule.

Metrics whose determinant is near 1 (series logarithm) and not (log), a small
chi, every slicing / shift / advection option, and sizes with at most two
blocks of 32 x 4 points for each of 152 SMs and with more.  Tolerance: FP64
1e-12 of each field's scale, as for the other FP64 stages (about 2500
operations of half an ulp, on terms up to 100 times the largest result).
"""
import numpy as np
import pytest
import torch

import oracle
from paper_1806_04182_gb300 import build, capi, inputs
from paper_1806_04182_gb300.state import PatchState

pytestmark = pytest.mark.gpu
TOL = 1e-12


@pytest.fixture(scope="module", autouse=True)
def lib():
    assert torch.cuda.is_available(), "GPU tests need CUDA"
    build.build()
    return capi.lib()


def _oracle_params(prm):
    return oracle.params(slicing=prm.slicing, shift_frozen=prm.shift_frozen, lopsided=prm.lopsided)


@pytest.mark.parametrize("n", [(33, 5, 7), (40, 12, 50), (64, 40, 30)])
@pytest.mark.parametrize("slicing,frozen,lop", [(0, 0, 0), (1, 1, 0), (1, 0, 1)])
def test_rhs_and_step(n, slicing, frozen, lop):
    U0, dx = inputs.z4_perturbed(n, seed=sum(n), amp=0.05)
    U0[0] *= 0.3                       # chi
    U0[1:7] *= 1.4 if lop else 1.0     # ln det about 1
    prm = capi.params(slicing=slicing, shift_frozen=frozen, lopsided=lop)
    dt = 0.1 * min(dx)
    st = PatchState(capi.SF_Z4, n, dx, dt, prm=prm)
    st.upload(U0)
    G = oracle.ghosted(U0.copy())
    got = st.rhs().cpu().numpy()
    want = oracle.rhs(oracle.Z4, G, dx, _oracle_params(prm))
    for f in range(25):
        e = np.abs(got[f] - want[f]).max() / max(np.abs(want[f]).max(), 1e-3)
        assert e < TOL, (f, e)
    want = oracle.rk4_step(oracle.Z4, G, dx, dt, _oracle_params(prm), stages=True)
    for s in range(st.nstages):
        got = st.fields(st.stage(s)).cpu().numpy()
        for f in range(25):
            e = np.abs(got[f] - want[s][f]).max() / max(np.abs(want[s][f]).max(), 1e-3)
            assert e < TOL, (s, f, e)
