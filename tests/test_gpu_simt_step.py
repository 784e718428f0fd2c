"""Fused FP32 passes of width 4 on a state large enough that the warps of a CTA work in step,
with target sets of both kinds (in step; each warp alone), against complex128 on the device."""
import numpy as np
import pytest

from paper_2512_07311_gb300 import capi

pytestmark = pytest.mark.gpu

N, K = 28, 4


class _DeviceArray:
    def __init__(self, ptr, count):
        self.__cuda_array_interface__ = dict(shape=(count,), typestr="<c8", data=(ptr, False), version=3, strides=None)


@pytest.mark.parametrize("targets", [[24, 25, 26, 27], [5, 6, 7, 8], [0, 9, 18, 27], [0, 2, 3, 4], [1, 9, 18, 27],
                                     [0, 1, 2, 3]])
def test_width_4_on_a_large_state(targets):
    torch = pytest.importorskip("torch")
    rng = np.random.default_rng(7)
    q, _ = np.linalg.qr(rng.standard_normal((16, 16)) + 1j * rng.standard_normal((16, 16)))
    ctx = capi.rcs_create(N, capi.RCS_PREC_FP32_FUSED)
    try:
        psi = torch.as_tensor(_DeviceArray(capi.rcs_state_device(ctx), 1 << N), device="cuda")
        psi.copy_(torch.randn(1 << N, dtype=torch.complex64, device="cuda") * 2.0 ** (-N / 2))
        base = torch.arange(1 << (N - K), device="cuda")
        for t in targets:
            base = ((base >> t) << (t + 1)) | (base & ((1 << t) - 1))
        offs = [sum(((j >> i) & 1) << targets[i] for i in range(K)) for j in range(1 << K)]
        want = torch.as_tensor(q, device="cuda") @ torch.stack([psi[base + o] for o in offs]).to(torch.complex128)
        norm = float(torch.linalg.vector_norm(want))
        torch.cuda.synchronize()
        for _ in range(2):  # the second call walks the same way; U^H between them restores the input
            capi.rcs_apply_unitary(ctx, targets, q)
            capi.rcs_sync(ctx)
            got = torch.stack([psi[base + o] for o in offs])
            # rounding of U and of 2 * 2^k fused multiply-adds, half an ulp (2^-24) each, of the norm; the
            # second time that of the two passes before as well
            err = float(torch.linalg.vector_norm(got.to(torch.complex128) - want))
            assert err <= 3 * (2 * 2 ** K + 1) * 2.0 ** -24 * norm
            del got
            capi.rcs_apply_unitary(ctx, targets, q.conj().T)
    finally:
        capi.rcs_sync(ctx)
        capi.rcs_destroy(ctx)
