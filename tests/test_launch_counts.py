"""The launch counts of a run are what was launched, and the GPU tests of chained passes do
run chains: nearly all of their target sets as two pairs and a three."""
import numpy as np
import pytest

import test_gpu_chain
import test_gpu_chain_order
from fake_gpu import _fake_library, fake_gpu  # noqa: F401  (fixtures)
from paper_2512_07311_gb300 import capi
from paper_2512_07311_gb300 import circuits as C

CHAIN = "k_fused_tcILb0ELb0ELb0ELb1E"


def noted(gpu):
    names = [k for k, _, _ in gpu.launches()]
    return len(names), sum(CHAIN in k for k in names)


@pytest.mark.parametrize("n, precision, flags", [
    (1, capi.RCS_PREC_FP32_PLAIN, 0), (9, capi.RCS_PREC_FP32_PLAIN, 0), (3, capi.RCS_PREC_FP32_FUSED, 0),
    (16, capi.RCS_PREC_FP32_FUSED, 0), (11, capi.RCS_PREC_BF16X3, 0), (19, capi.RCS_PREC_TF32X3, 0),
    (21, capi.RCS_PREC_BF16X3, capi.RCS_OPT_PAIR_PASSES), (24, capi.RCS_PREC_TF32X3, 0),
    (24, capi.RCS_PREC_BF16X3, 0), (25, capi.RCS_PREC_BF16X3, 0)])
def test_counts_are_the_launches(fake_gpu, n, precision, flags):  # noqa: F811
    gates = C.generate(C.grid_for_n(n), 8, "EFGH", seed=n).gates if n > 1 else np.array([C.make_gate(C.SQRT_X, 0)])
    ctx = capi.rcs_create(n, precision, k_max=4 if precision == capi.RCS_PREC_FP32_FUSED else 0, flags=flags)
    plan = capi.rcs_plan_build(n, gates, precision, flags=flags)
    try:
        capi.rcs_plan_upload(ctx, plan)
        for fresh in (True, False):
            for run in (lambda: capi.rcs_apply_circuit(ctx, gates), lambda: capi.rcs_plan_run(ctx, plan)):
                if fresh:
                    capi.rcs_reset(ctx)
                else:
                    capi.rcs_state_device(ctx)  # the caller's order: no layout change in the run
                fake_gpu.reset()
                try:
                    run()
                except capi.RcsError as e:
                    assert not fresh and e.code == capi.RCS_ERR_ARG  # a plan with its own layout
                    continue
                assert capi.rcs_last_run_launches(ctx) == noted(fake_gpu)
    finally:
        capi.rcs_plan_destroy(plan)
        capi.rcs_destroy(ctx)


def chain_items(n, kind):
    """The items of test_gpu_chain's test, drawn as it draws them."""
    rng = np.random.default_rng(n)
    return [(np.array(test_gpu_chain.SETS[kind](n, rng, i), dtype=np.int32), test_gpu_chain._unitary(rng))
            for i in range(7)]


@pytest.mark.parametrize("n", [24, 25])
@pytest.mark.parametrize("items_of, kind", [(f, k) for f, sets in ((chain_items, test_gpu_chain.SETS),
                                                                  (test_gpu_chain_order.items_of, test_gpu_chain_order.SETS))
                                            for k in sorted(sets)])
def test_chain_tests_run_chains(fake_gpu, items_of, kind, n):  # noqa: F811
    items = items_of(n, kind)
    ctx = capi.rcs_create(n, capi.RCS_PREC_BF16X3)
    try:
        capi.rcs_state_device(ctx)
        fake_gpu.reset()
        capi.rcs_apply_unitaries(ctx, items)
        kernels, chains = capi.rcs_last_run_launches(ctx)
        assert (kernels, chains) == noted(fake_gpu)
        assert (kernels, chains) == (3, 3)  # the cheapest split of seven: two pairs and a three
        for item in items:
            capi.rcs_apply_unitaries(ctx, [item])
            assert capi.rcs_last_run_launches(ctx) == (1, 0)
    finally:
        capi.rcs_destroy(ctx)
