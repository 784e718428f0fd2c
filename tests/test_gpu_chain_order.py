"""Chains of tensor-core passes on a state whose every chunk holds data.

A chunk that a pass reads before the pass before it has stored it, or that is overwritten
too early, gives other bits here. (From |0...0> most chunks are still zero when a chain
runs, and a chunk read too early gives the right zeros.) 24 qubits have 16 chunks, 25 have
32: more than a pass may be ahead of the next one, so the window holds passes back too.
"""
import numpy as np
import pytest

from paper_2512_07311_gb300 import capi

pytestmark = pytest.mark.gpu

SETS = {
    "pairs": lambda n, rng: rng.permutation(n)[:6],  # three of these fit no chunk
    "threes": lambda n, rng: rng.permutation(np.arange(n - 9, n))[:6],
    "low": lambda n, rng: np.append(rng.permutation(6)[:1], rng.permutation(np.arange(n - 7, n))[:5]),
    "bits_0_1": lambda n, rng: np.append([0, 1], rng.permutation(np.arange(n - 7, n))[:4]),
}


def items_of(n, kind):
    rng = np.random.default_rng(100 + n)
    items = []
    for _ in range(7):
        q, _ = np.linalg.qr(rng.standard_normal((64, 64)) + 1j * rng.standard_normal((64, 64)))
        items.append((SETS[kind](n, rng).astype(np.int32), q))
    return items


@pytest.mark.parametrize("n", [24, 25])
@pytest.mark.parametrize("kind", sorted(SETS))
def test_chain_equals_single_passes_on_a_full_state(n, kind):
    psi = np.random.default_rng(n).standard_normal(2 << n, dtype=np.float32).view(np.complex64)
    psi *= np.float32(2.0 ** (-(n + 1) / 2))
    items = items_of(n, kind)
    got, chains = [], []
    for calls in ([[it] for it in items], [items]):  # a call with one unitary cannot chain
        ctx = capi.rcs_create(n, capi.RCS_PREC_BF16X3)
        try:
            capi.rcs_state_write(ctx, psi)
            for c in calls:
                capi.rcs_apply_unitaries(ctx, c)
            chains.append(capi.rcs_last_run_launches(ctx)[1])
            got.append(capi.rcs_state_read(ctx).view(np.uint64))
        finally:
            capi.rcs_destroy(ctx)
    assert chains[0] == 0 and chains[1] >= 3
    assert np.array_equal(*got)
