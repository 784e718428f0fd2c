"""Fused FP32 passes of width 1 to 4 against a plain complex128 product.

One lane works on one slice of a unit of 32: the sizes are those below one unit (the small
kernel), one unit, a few and many (several per warp, both orders of the walk), with the
lowest target on every bit 0..5 and on bits 0 and 1 together, each its own order in shared
memory and its own stores.
"""
import numpy as np
import pytest

from paper_2512_07311_gb300 import capi

pytestmark = pytest.mark.gpu

LOWS = [(0,), (1,), (2,), (3,), (4,), (5,), (0, 1), (0, 2), (1, 2)]


def _apply(psi, n, targets, u):
    k = len(targets)
    base = np.arange(1 << (n - k))
    for t in sorted(targets):
        base = ((base >> t) << (t + 1)) | (base & ((1 << t) - 1))
    at = np.stack([base + sum(((j >> i) & 1) << targets[i] for i in range(k)) for j in range(1 << k)])
    psi[at] = u @ psi[at]


@pytest.mark.parametrize("k", [1, 2, 3, 4])
@pytest.mark.parametrize("extra", [0, 1, 4, 5, 6, 9, 15])
def test_width_vs_product(k, extra):
    n = k + extra
    rng = np.random.default_rng(10 * n + k)
    psi = rng.standard_normal(1 << n) + 1j * rng.standard_normal(1 << n)
    psi = (psi / np.linalg.norm(psi)).astype(np.complex64)
    want = psi.astype(np.complex128)
    items = []
    for low in LOWS:
        low = [b for b in low if b < n][:k]
        rest = rng.permutation([b for b in range(n) if b not in low and b > max(low, default=-1)] +
                               [b for b in range(n) if b not in low and b < max(low, default=-1)][::-1])
        targets = (low + [int(b) for b in sorted(rest, reverse=True)])[:k]
        q, _ = np.linalg.qr(rng.standard_normal((1 << k,) * 2) + 1j * rng.standard_normal((1 << k,) * 2))
        items.append((np.array(targets, dtype=np.int32), q))
        _apply(want, n, targets, q)
    ctx = capi.rcs_create(n, capi.RCS_PREC_FP32_FUSED)
    try:
        capi.rcs_state_write(ctx, psi)
        capi.rcs_apply_unitaries(ctx, items)
        got = capi.rcs_state_read(ctx)
    finally:
        capi.rcs_destroy(ctx)
    # per pass: rounding of U and of 2 * 2^k fused multiply-adds, half an ulp (2^-24) each, relative
    # to the norm of the state (a dot product's error is at most that of its terms' norms)
    bound = len(LOWS) * (2 * 2 ** k + 1) * 2.0 ** -24
    assert np.linalg.norm(got - want) <= bound
