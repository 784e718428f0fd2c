"""A fused FP32 pass asks for so much shared memory that no SM takes more than its even share
of the CTAs (they come in while the pass before still holds most SMs, and would crowd onto
the others)."""
import numpy as np
import pytest

from fake_gpu import _fake_library, fake_gpu  # noqa: F401  (fixtures)
from paper_2512_07311_gb300 import capi

SMS, PER_SM, PER_CTA = 152, 228 * 1024, 1024
RESIDENT = {1: 3, 2: 2, 3: 2, 4: 2, 5: 3, 6: 2, 7: 1}  # CTAs on an SM when the card is full


@pytest.mark.parametrize("n", range(12, 24))
@pytest.mark.parametrize("k", range(1, 8))
def test_ctas_spread_over_the_sms(fake_gpu, k, n):  # noqa: F811
    ctx = capi.rcs_create(n)
    try:
        capi.rcs_state_device(ctx)
        fake_gpu.reset()
        capi.rcs_apply_unitary(ctx, np.arange(k, dtype=np.int32), np.eye(1 << k))
        (name, grid, _), = fake_gpu.launches()
        smem = fake_gpu.lib.fake_launch_smem(0)
    finally:
        capi.rcs_destroy(ctx)
    assert "k_fused_simt" in name or "k_fused_wide" in name
    assert smem <= 227 * 1024 and grid <= RESIDENT[k] * SMS
    assert PER_SM // (smem + PER_CTA) == -(-grid // SMS)
