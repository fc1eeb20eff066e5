"""The descriptors that PatchState packs for sf_steps are those that it fills by
name for the single stages (CPU: sf_steps is replaced by a recorder)."""
import ctypes
import struct

import pytest

from paper_1806_04182_gb300 import build, capi, state
from paper_1806_04182_gb300.state import PatchState


@pytest.fixture(scope="module", autouse=True)
def lib():
    build.build()
    return capi.lib()


@pytest.mark.parametrize("system,precision,kw", [
    (capi.SF_WAVE, capi.SF_FP64, {}),
    (capi.SF_Z4, capi.SF_FP32_BULK_DW, dict(x_pitch=16, x_offset=1, plane_rows=12)),
    (capi.SF_MHD, capi.SF_FP32_BULK, {}),
])
def test_same_fields(monkeypatch, system, precision, kw):
    seen = []
    monkeypatch.setattr(capi, "sf_steps", lambda prm, g, s, n, adjoint, h: seen.append((g, s, n, adjoint)))
    st = PatchState(system, (5, 4, 3), (0.1, 0.2, 0.3), 0.07, precision=precision, device="cpu", **kw)
    st._steps(3, 0, rate=4096)
    (g, s, n, adjoint), want = seen[0], st.patch(st.A, st.A, st.B)
    assert (n, adjoint) == (3, False)
    for f in ("ghost", "dt", "system", "precision", "sy", "sz", "sf"):
        assert getattr(g, f) == getattr(want, f), f
    assert (g.n[:], g.dx[:], g.cfl_rate) == (want.n[:], want.dx[:], 4096)
    assert (s.u, s.s1, s.s2) == (st.ptr(st.A), st.ptr(st.B), st.ptr(st.C))
    assert (s.acc, s.kahan) == (want.acc, want.kahan)


@pytest.mark.parametrize("cls", [capi.sf_patch, capi.sf_state])
def test_added_field(cls):
    """A structure with one field more, of the same size or not, takes one value more."""
    values = [0] * (len(state._packer(cls).unpack(bytes(ctypes.sizeof(cls)))))
    state._packer(cls).pack(*values)
    for t in (ctypes.c_int64, ctypes.c_double):
        more = type("more", (ctypes.Structure,), {"_fields_": cls._fields_ + [("extra", t)]})
        with pytest.raises(struct.error):
            state._packer(more).pack(*values)


def test_padding():
    pad = type("pad", (ctypes.Structure,), {"_fields_": [("a", ctypes.c_int32), ("b", ctypes.c_double)]})
    with pytest.raises(TypeError):
        state._packer(pad)


@pytest.mark.parametrize("n", [0, -1])
def test_no_steps(n):
    """No step, no call: a patch that sf_steps would refuse included."""
    st = PatchState(capi.SF_WAVE, (2, 2, 2), (0.1, 0.1, 0.1), 0.01, device="cpu")
    st.step(n, stream=0)
    st.adjoint_step(n, stream=0)
