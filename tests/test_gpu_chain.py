"""Chains of tensor-core passes: two or three passes in one launch give the bits that the
same passes give one launch each (the single pass is held to the oracle elsewhere).

A call with several unitaries on 24 or more qubits runs them as chains; one unitary per
call cannot. The target sets cover the lowest target on every bit 0..5 (each has its own
order of a block in the stage), targets that share no qubits (the widest chunks), shared
ones (chunks at their least size, three passes), and a sequence that leaves one over.
"""
import numpy as np
import pytest

from paper_2512_07311_gb300 import capi

pytestmark = pytest.mark.gpu


def _unitary(rng):
    q, _ = np.linalg.qr(rng.standard_normal((64, 64)) + 1j * rng.standard_normal((64, 64)))
    return q


SETS = {
    "low": lambda n, rng, i: [i % 6] + [8 + (i * 2 + j) % (n - 8) for j in range(5)],
    "apart": lambda n, rng, i: rng.permutation(n)[:6],
    "shared": lambda n, rng, i: rng.permutation(np.arange(n - 9, n))[:6],
    "two_low": lambda n, rng, i: list(rng.permutation(5)[:2]) + [10, 13, n - 2, n - 1],
    "bits_0_1": lambda n, rng, i: [0, 1, 2 + i % 5, 9, n - 2, n - 1],
}


@pytest.mark.parametrize("n", [24, 25])
@pytest.mark.parametrize("kind", sorted(SETS))
def test_chain_equals_single_passes(n, kind):
    rng = np.random.default_rng(n)
    items = [(np.array(SETS[kind](n, rng, i), dtype=np.int32), _unitary(rng)) for i in range(7)]
    assert all(len(set(t.tolist())) == 6 for t, _ in items)
    got = []
    for calls in ([[it] for it in items], [items]):
        ctx = capi.rcs_create(n, capi.RCS_PREC_BF16X3)
        try:
            for c in calls:
                capi.rcs_apply_unitaries(ctx, c)
            got.append(capi.rcs_state_read(ctx).view(np.uint64))
        finally:
            capi.rcs_destroy(ctx)
    assert np.array_equal(*got)


def test_chain_wait_limit_reports_timeout():
    """A tile whose MMAs never run: every CTA's waits end, the call reports it, the next run works."""
    n, rng = 24, np.random.default_rng(0)
    items = [(np.array([1, 9, 12, 15, 20, 23], dtype=np.int32), _unitary(rng)) for _ in range(2)]
    ctx = capi.rcs_create(n, capi.RCS_PREC_BF16X3)
    try:
        capi.rcs_tc_test_fault(2, 0.05)
        capi.rcs_apply_unitaries(ctx, items)
        with pytest.raises(capi.RcsError) as e:
            capi.rcs_sync(ctx)
        assert e.value.code == capi.RCS_ERR_TIMEOUT
        capi.rcs_tc_test_fault(-1)
        capi.rcs_reset(ctx)
        capi.rcs_apply_unitaries(ctx, items)
        capi.rcs_sync(ctx)
        assert abs(capi.rcs_norm(ctx) - 1.0) <= 4e-6  # 2e-6 per pass
    finally:
        capi.rcs_tc_test_fault(-1)
        capi.rcs_destroy(ctx)
