"""MHD right-hand side beside strong jumps, against the FP64 oracle.

Random states near 1 (10%), scaled by J in half of the box: density, momentum
and energy by J, B by sqrt(J), so that velocities and signal speeds stay of
order one on both sides.  A cell is compared relative to the largest value
among itself and its six neighbours, the cells whose edge values its faces
use: a jump that its stencils only touch must not leave an error of its own
size.  Bound: an edge value takes eight roundings of that size and a flux of
it twelve more, at signal speeds up to 3, half the sum of two states per face,
two faces per direction: 20 eps x 3 x scale x sum_d 2 / dx_d, twice that for
the oracle's own in double.
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


def _states(n, axis, J, seed, noise=0.1):
    """(8, nz, ny, nx) conserved fields, the upper half along `axis` (0: x) scaled by J."""
    r = np.random.default_rng(seed).uniform(-noise, noise, (8, n[2], n[1], n[0]))
    U = inputs.mhd_primitive_to_conserved(1 + r[0], list(r[1:4]), 1 + r[4], [0.3 + r[5], r[6], 0.2 + r[7]], 5 / 3)
    half = np.arange(n[axis]) >= n[axis] // 2
    s = np.where(half, J, 1.0).reshape([-1 if d == 2 - axis else 1 for d in range(3)])
    return U * np.stack([s] * 5 + [np.sqrt(s)] * 3)


def _local(a):
    """Largest value among a cell and its six neighbours (periodic)."""
    m = a.copy()
    for ax in range(3):
        for o in (-1, 1):
            m = np.maximum(m, np.roll(a, o, ax))
    return m


def _check(U, dx, precision, speed_err=0.0, **kw):
    n = U.shape[:0:-1]
    eps = float(np.finfo(np.float64 if precision == capi.SF_FP64 else np.float32).eps)
    if precision != capi.SF_FP64:
        U = U.astype(np.float32).astype(np.float64)
    st = PatchState(capi.SF_MHD, n, dx, 1e-3, precision=precision, prm=capi.params(rk=capi.SF_SSPRK3, **kw))
    st.upload(U)
    got = st.rhs().double().cpu().numpy()
    want = oracle.rhs(oracle.MHD, oracle.ghosted(U.copy()), dx, oracle.params(**kw))
    hydro, mag = (_local(np.abs(U[a]).max(0)) for a in (slice(0, 5), slice(5, 8)))
    tol = ((40 if precision == capi.SF_FP64 else 20) * eps * 3 + 0.5 * speed_err) * sum(2 / h for h in dx)
    for f in range(8):
        e = np.abs(got[f] - want[f]) / (tol * (hydro if f < 5 else mag))
        assert np.isfinite(e).all() and e.max() < 1, (f, np.nanmax(e), np.isnan(e).sum())


# blocks of 32 x 15 or 32 x 7 columns: one tile and its edges crossed along each axis
@pytest.mark.parametrize("precision", [capi.SF_FP64, capi.SF_FP32_BULK])
@pytest.mark.parametrize("n,axis", [((40, 9, 5), 0), ((34, 18, 4), 1), ((9, 8, 16), 2)])
@pytest.mark.parametrize("variant,J", [(0, 1e3), (0, 1e6), (0, 1e8), (1, 1e3), (1, 1e6), (2, 1e6)])
def test_jump(n, axis, variant, J, precision):
    U = _states(n, axis, J, seed=axis)
    _check(U, tuple(1.0 / v for v in n), precision, weno_variant=variant)


# the smoothness indicators are squares of up to 1e12, their products of squares
# beyond a float
@pytest.mark.parametrize("precision", [capi.SF_FP64, capi.SF_FP32_BULK])
@pytest.mark.parametrize("n,axis", [((40, 9, 5), 0), ((34, 18, 4), 1), ((9, 8, 16), 2)])
@pytest.mark.parametrize("J", [4e9, 1e12])
def test_js_range(n, axis, J, precision):
    _check(_states(n, axis, J, seed=axis), tuple(1.0 / v for v in n), precision, weno_variant=0)


# the weights' products with the differences go with the fifth power of a jump
@pytest.mark.parametrize("precision", [capi.SF_FP64, capi.SF_FP32_BULK])
@pytest.mark.parametrize("n,axis", [((40, 9, 5), 0), ((34, 18, 4), 1), ((9, 8, 16), 2)])
@pytest.mark.parametrize("J", [1e8, 4e9, 1e12])
def test_weno3_range(n, axis, J, precision):
    _check(_states(n, axis, J, seed=axis), tuple(1.0 / v for v in n), precision, weno_variant=2)


# WENO-Z: the ratio of the indicators beside a jump is its square over epsilon
# where the state is uniform; its q-th power leaves a float from jumps of 1e5 on
@pytest.mark.parametrize("precision", [capi.SF_FP64, capi.SF_FP32_BULK])
@pytest.mark.parametrize("n,axis", [((40, 9, 5), 0), ((34, 18, 4), 1), ((9, 8, 16), 2)])
@pytest.mark.parametrize("J,noise,q", [(1e6, 0.0, 2.0), (1e6, 0.0, 1.5), (1e8, 0.1, 2.0), (1e12, 0.1, 2.0)])
def test_z_range(n, axis, J, noise, q, precision):
    U = _states(n, axis, J, seed=axis, noise=noise)
    _check(U, tuple(1.0 / v for v in n), precision, weno_variant=1, weno_q=q)


# Negative gas pressure p and no field along x and y: s = (gamma p + B^2) / rho
# is negative, s + sqrt(s^2) zero, and the signal speed |v_d|; rounding leaves
# up to 2 eps |s| of the sum, a speed of its root.
def _negative_pressure(n, seed, noise, vx=0.0):
    r = np.random.default_rng(seed).uniform(-noise, noise, (5, n[2], n[1], n[0]))
    zero = np.zeros(r.shape[1:])
    rho, p = 1 + r[0], -0.5 + 0.5 * r[4]
    U = inputs.mhd_primitive_to_conserved(rho, [vx + r[1], r[2], r[3]], p, [zero, zero, zero + 0.2], 5 / 3)
    return U, float(np.abs((5 / 3 * p + 0.04) / rho).max())


@pytest.mark.parametrize("precision", [capi.SF_FP64, capi.SF_FP32_BULK])
@pytest.mark.parametrize("n", [(40, 9, 5), (9, 8, 16)])
def test_negative_pressure(n, precision):
    U, s = _negative_pressure(n, 3, 0.1)
    eps = float(np.finfo(np.float64 if precision == capi.SF_FP64 else np.float32).eps)
    _check(U, tuple(1.0 / v for v in n), precision, speed_err=np.sqrt(2 * eps * 1.5 * s))


@pytest.mark.parametrize("precision", [capi.SF_FP64, capi.SF_FP32_BULK])
@pytest.mark.parametrize("fused", [False, True])
def test_negative_pressure_rate(fused, precision):
    """Uniform states, one after the other, moving along x: the rate is |v_x| / dx."""
    n, dx = (3, 3, 3), (0.25, 0.25, 0.25)
    eps = float(np.finfo(np.float64 if precision == capi.SF_FP64 else np.float32).eps)
    for seed in range(24):
        vx = 1.5 + 0.01 * seed
        U, s = _negative_pressure((1, 1, 1), seed, 0.3, vx)
        vx = (U[1] / U[0]).item()
        st = PatchState(capi.SF_MHD, n, dx, 1e-3, precision=precision, prm=capi.params(rk=capi.SF_SSPRK3))
        st.upload(np.broadcast_to(U, (8,) + n[::-1]).copy())
        if fused:  # the rate of the state after a step, which is the same state
            rate = torch.zeros(1, dtype=torch.float64, device="cuda")
            st._steps(1, torch.cuda.current_stream().cuda_stream, rate=rate.data_ptr())
        else:
            rate = st.mhd_max_rate()
        assert abs(rate.item() * dx[0] - vx) < 16 * eps * vx + np.sqrt(2 * eps * s), (seed, rate.item())
