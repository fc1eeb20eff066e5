"""MHD stage kernel (reconstruction of the evolved fields) at the edges of its
tiles, against the FP64 oracle.

A block owns 32 x 15 or 32 x 7 columns and marches a number of planes that
the host picks with the tile; cells and faces that a tile needs from outside
come from the block's last warp.  Sizes: one cell less and more than a tile
and exactly a tile in x and y, several chunks in z, and sizes that take each
tile ((33, 21, 40) and (33, 7, 160) the 32 x 7 one on 152 SMs).  Tolerances as
for the other MHD stages: FP64 1e-12 of each field's scale, float 32 eps32
(ten roundings per flux, six fluxes, dt S / dx <= 0.3).
"""
import numpy as np
import pytest
import torch

import oracle
from paper_1806_04182_gb300 import build, capi, inputs
from paper_1806_04182_gb300.state import PatchState

pytestmark = pytest.mark.gpu
TOL = {capi.SF_FP64: 1e-12, capi.SF_FP32_BULK: 32 * float(np.finfo(np.float32).eps)}


@pytest.fixture(scope="module", autouse=True)
def lib():
    assert torch.cuda.is_available(), "GPU tests need CUDA"
    build.build()
    return capi.lib()


def _oracle_params(prm):
    return oracle.params(gamma_eos=prm.gamma_eos, weno_eps=prm.weno_eps, weno_q=prm.weno_q,
                         weno_variant=prm.weno_variant)


def _check(n, precision, prm, floor, U0, dx):
    dt = 0.3 / oracle.mhd_max_rate(oracle.ghosted(U0), dx)
    st = PatchState(capi.SF_MHD, n, dx, dt, precision=precision, prm=prm)
    st.upload(U0)
    step = oracle.rk4_step if prm.rk == capi.SF_RK4 else oracle.ssprk3_step
    want = step(oracle.MHD, oracle.ghosted(U0.copy()), dx, dt, _oracle_params(prm), stages=True)
    for s in range(st.nstages):
        got = st.fields(st.stage(s)).cpu().numpy()
        for f in range(8):
            e = np.abs(got[f] - want[s][f]).max() / max(np.abs(want[s][f]).max(), floor[f])
            assert e < TOL[precision], (n, s, f, e / TOL[precision])


SIZES = [(31, 14, 4), (32, 15, 4), (33, 16, 4), (64, 30, 3), (65, 31, 5), (3, 8, 3), (33, 21, 40),
         (33, 7, 160)]
EVEN = [(129, 50, 50), (352, 210, 3)]


@pytest.mark.parametrize("precision", [capi.SF_FP64, capi.SF_FP32_BULK])
@pytest.mark.parametrize("n", SIZES)
def test_tile_edges(n, precision):
    U0, dx = inputs.mhd_blast(n, seed=sum(n), radius=0.3)
    _check(n, precision, capi.params(rk=capi.SF_SSPRK3), [1e-3] * 8, U0, dx)


# sizes at which double blocks take even shares of all columns on 152 SMs:
# shares that start inside a column, and shares of more than one column
@pytest.mark.parametrize("n", EVEN)
def test_even_shares(n):
    U0, dx = inputs.mhd_blast(n, seed=sum(n), radius=0.3)
    _check(n, capi.SF_FP64, capi.params(rk=capi.SF_SSPRK3), [1e-3] * 8, U0, dx)


@pytest.mark.parametrize("precision", [capi.SF_FP64, capi.SF_FP32_BULK])
@pytest.mark.parametrize("variant,q,rk", [(1, 2.0, capi.SF_SSPRK3), (1, 1.0, capi.SF_SSPRK3),
                                          (1, 1.5, capi.SF_SSPRK3), (2, 2.0, capi.SF_SSPRK3),
                                          (0, 2.0, capi.SF_RK4)])
def test_weights_and_rk(variant, q, rk, precision):
    n = (33, 9, 5)
    U0, dx = inputs.mhd_blast(n, seed=8, radius=0.3)
    _check(n, precision, capi.params(rk=rk, weno_variant=variant, weno_q=q), [1e-3] * 8, U0, dx)


# The equations keep their form when density, momentum and energy scale by s
# and B by sqrt(s); the smoothness indicators then scale by s^2 against a
# fixed epsilon, so that the weights' products span the range of a float.
@pytest.mark.parametrize("precision", [capi.SF_FP64, capi.SF_FP32_BULK])
@pytest.mark.parametrize("variant", [0, 1, 2])
@pytest.mark.parametrize("s", [1e-4, 1e6])
def test_units(s, variant, precision):
    n = (33, 9, 5)
    U0, dx = inputs.mhd_blast(n, seed=9, radius=0.3)
    scale = np.array([s] * 5 + [s ** 0.5] * 3)
    U0 = U0 * scale[:, None, None, None]
    _check(n, precision, capi.params(rk=capi.SF_SSPRK3, weno_variant=variant), list(1e-3 * scale), U0, dx)
