"""Stored qubit layouts brought back to the caller's order: every amplitude unchanged.

A saved state carries its layout, so a file can name any permutation of the qubits: the
ones a planned circuit chooses (swaps with the lowest bits, one pass of the permutation
kernel) and arbitrary ones (several passes beyond 12 moved bits; states below one tile).
"""
import struct

import numpy as np
import pytest

from paper_2512_07311_gb300 import capi
from paper_2512_07311_gb300 import circuits as C

pytestmark = pytest.mark.gpu


def _save(path, n, phys, amps):
    head = struct.pack("<8sIi64iQ", b"RCSSTATE", 1, n, *phys, *range(n, 64), 1 << n)
    with open(path, "wb") as f:
        f.write(head + amps.tobytes())


def _caller_order(stored, n, phys):
    c = np.arange(1 << n, dtype=np.int64)
    s = np.zeros_like(c)
    for q in range(n):
        s |= ((c >> q) & 1) << int(phys[q])
    return stored[s]


@pytest.mark.parametrize("kind", ["planned", "any"])
@pytest.mark.parametrize("n", [2, 5, 11, 12, 13, 17, 21])
def test_layout_is_restored_exactly(tmp_path, n, kind):
    rng = np.random.default_rng(n)
    phys = np.arange(n)
    if kind == "any":
        phys = rng.permutation(n)
    else:
        for low in range(min(5, n // 2)):
            high = int(rng.integers(n // 2, n))
            i, j = np.flatnonzero(phys == low)[0], np.flatnonzero(phys == high)[0]
            phys[[i, j]] = phys[[j, i]]
    stored = rng.integers(0, 1 << 62, 1 << n).view(np.complex64)  # any bit patterns
    _save(tmp_path / "s", n, phys, stored)
    ctx = capi.rcs_create(n)
    try:
        capi.rcs_state_load(ctx, str(tmp_path / "s"))
        got = capi.rcs_state_read(ctx)
        assert np.array_equal(capi.rcs_qubit_layout(ctx), np.arange(n))
    finally:
        capi.rcs_destroy(ctx)
    assert np.array_equal(got.view(np.uint64), _caller_order(stored, n, phys).view(np.uint64))


def test_batch_state_read_follows_the_caller_order():
    circ = C.generate(C.grid_for_n(14), 8, "EFGH", seed=3)
    ctx = capi.rcs_create(14, capi.RCS_PREC_BF16X3)
    b = capi.rcs_batch_create([(14, circ.gates, 10, 1)], precision=capi.RCS_PREC_BF16X3)
    try:
        plan = capi.rcs_plan_build(14, circ.gates, capi.RCS_PREC_BF16X3)
        assert not np.array_equal(capi.rcs_plan_layout(plan, 14), np.arange(14))  # the case is a permuted one
        capi.rcs_plan_destroy(plan)
        capi.rcs_batch_launch(b)
        capi.rcs_batch_wait(b)
        got = capi.rcs_batch_state_read(b, 0)
        capi.rcs_apply_circuit(ctx, circ.gates)
        want = capi.rcs_state_read(ctx)
    finally:
        capi.rcs_batch_destroy(b)
        capi.rcs_destroy(ctx)
    assert np.array_equal(got.view(np.uint64), want.view(np.uint64))
