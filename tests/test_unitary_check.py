"""Caller matrices that hold a NaN or an infinity are refused and the state is left alone."""
import numpy as np
import pytest

from fake_gpu import _fake_library, fake_gpu  # noqa: F401  (fixtures)
from paper_2512_07311_gb300 import capi
from paper_2512_07311_gb300 import circuits as C


@pytest.mark.parametrize("bad", [np.nan, np.inf, -np.inf, 1j * np.nan, 1j * np.inf])
@pytest.mark.parametrize("k", [1, 3, 7])
@pytest.mark.parametrize("where", ["first", "last", "all"])
def test_not_finite(fake_gpu, bad, k, where):  # noqa: F811
    u = np.eye(1 << k, dtype=np.complex128)
    if where == "all":
        u[:] = bad
    else:
        u[(0, -1) if where == "first" else (-1, -1)] = bad
    targets = np.arange(k, dtype=np.int32)
    ctx = capi.rcs_create(8)
    try:
        for items in ([(targets, u)], [(targets, np.eye(1 << k)), (targets, u)]):
            with pytest.raises(capi.RcsError) as e:
                capi.rcs_apply_unitaries(ctx, items)
            assert e.value.code == capi.RCS_ERR_ARG
        assert fake_gpu.launches() == []
        capi.rcs_apply_unitaries(ctx, [(targets, np.eye(1 << k))])
        assert fake_gpu.launches()
    finally:
        capi.rcs_destroy(ctx)


@pytest.mark.parametrize("bad", [np.nan, np.inf, 1j * np.nan])
@pytest.mark.parametrize("kind, d", [(C.U1, 2), (C.U2, 4)])
def test_not_finite_gate(fake_gpu, kind, d, bad):  # noqa: F811
    m = np.eye(d, dtype=np.complex128)
    m[0, -1] = bad
    with pytest.raises(capi.RcsError) as e:
        capi.rcs_plan_build(2, np.array([C.make_gate(kind, 0, 1 if d == 4 else -1)]), umats={0: m})
    assert e.value.code == capi.RCS_ERR_ARG
