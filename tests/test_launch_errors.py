"""A launch that fails is reported by its own call and by no later one."""
import numpy as np
import pytest

from fake_gpu import _fake_library, fake_gpu  # noqa: F401  (fixtures)
from paper_2512_07311_gb300 import capi
from paper_2512_07311_gb300 import circuits as C

OUT_OF_RESOURCES = 701


@pytest.mark.parametrize("kernel, n, k, precision", [
    ("k_init_zero", 10, 3, capi.RCS_PREC_FP32_FUSED),
    ("k_fused_small", 6, 3, capi.RCS_PREC_FP32_FUSED),
    ("k_fused_simt", 10, 3, capi.RCS_PREC_FP32_FUSED),
    ("k_fused_wide", 10, 6, capi.RCS_PREC_FP32_FUSED),
    ("k_fused_tc", 14, 6, capi.RCS_PREC_BF16X3),
    ("k_fused_tc", 24, 6, capi.RCS_PREC_BF16X3),
])
def test_failed_launch_is_reported_once(fake_gpu, kernel, n, k, precision):  # noqa: F811
    items = [(np.arange(k, dtype=np.int32) + n - k, np.eye(1 << k))] * 2
    gates = np.array([C.make_gate(C.SQRT_X, 0)])
    ctx, plain = capi.rcs_create(n, precision), capi.rcs_create(4, capi.RCS_PREC_FP32_PLAIN)
    try:
        fake_gpu.fail(kernel, OUT_OF_RESOURCES)
        with pytest.raises(capi.RcsError) as e:
            capi.rcs_apply_unitaries(ctx, items)
        assert e.value.code == capi.RCS_ERR_CUDA
        capi.rcs_apply_circuit(plain, gates)
        capi.rcs_apply_unitaries(ctx, items)
    finally:
        capi.rcs_destroy(plain)
        capi.rcs_destroy(ctx)
