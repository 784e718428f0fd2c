"""Single BF16x3 passes on a state so large that a CTA's loader warps work in step: the bits of
the same passes chained (whose loaders do not), and bounded waits when a tile never finishes."""
import numpy as np
import pytest

from paper_2512_07311_gb300 import capi

pytestmark = pytest.mark.gpu

N = 29


class _DeviceArray:
    def __init__(self, ptr, count):
        self.__cuda_array_interface__ = dict(shape=(count,), typestr="<c8", data=(ptr, False), version=3, strides=None)


def _items():
    rng = np.random.default_rng(N)
    out = []
    for t in ([23, 24, 25, 26, 27, 28], [0, 9, 17, 23, 26, 28], [3, 10, 11, 12, 13, 14]):
        q, _ = np.linalg.qr(rng.standard_normal((64, 64)) + 1j * rng.standard_normal((64, 64)))
        out.append((np.array(t, dtype=np.int32), q))
    return out


def test_single_passes_equal_chained_ones():
    torch = pytest.importorskip("torch")
    g = torch.Generator("cuda").manual_seed(1)
    psi = torch.randn(1 << N, dtype=torch.complex64, device="cuda", generator=g) * 2.0 ** (-N / 2)
    items, got, ctxs = _items(), [], []
    try:
        for calls in ([[it] for it in items], [items]):
            ctx = capi.rcs_create(N, capi.RCS_PREC_BF16X3)
            ctxs.append(ctx)
            state = torch.as_tensor(_DeviceArray(capi.rcs_state_device(ctx), 1 << N), device="cuda")
            state.copy_(psi)
            torch.cuda.synchronize()
            for c in calls:
                capi.rcs_apply_unitaries(ctx, c)
                chains = capi.rcs_last_run_launches(ctx)[1]
                assert (chains > 0) == (len(c) > 1)
            capi.rcs_sync(ctx)
            got.append(torch.view_as_real(state).view(torch.int32))
        assert torch.equal(*got)
    finally:
        for ctx in ctxs:
            capi.rcs_destroy(ctx)


def test_wait_limit_reports_timeout():
    ctx = capi.rcs_create(N, capi.RCS_PREC_BF16X3)
    try:
        capi.rcs_tc_test_fault(2, 0.05)
        capi.rcs_apply_unitaries(ctx, _items()[:1])
        with pytest.raises(capi.RcsError) as e:
            capi.rcs_sync(ctx)
        assert e.value.code == capi.RCS_ERR_TIMEOUT
        capi.rcs_tc_test_fault(-1)
        capi.rcs_reset(ctx)
        capi.rcs_apply_unitaries(ctx, _items()[:1])
        capi.rcs_sync(ctx)
        assert abs(capi.rcs_norm(ctx) - 1.0) <= 2e-6  # per pass
    finally:
        capi.rcs_tc_test_fault(-1)
        capi.rcs_destroy(ctx)
