"""Chained passes need all their CTAs resident together. Where the process has fewer SMs
than the device reports, the launch is refused and the same passes run one launch each."""
import numpy as np
import pytest

from fake_gpu import _fake_library, fake_gpu  # noqa: F401  (fixtures)
from paper_2512_07311_gb300 import capi

CHAIN, SINGLE = "k_fused_tcILb0ELb0ELb0ELb1E", "k_fused_tcILb0ELb0ELb0ELb0E"
TOO_LARGE, NOT_SUPPORTED, ILLEGAL = 720, 801, 700


def apply(ctx):
    items = [(np.arange(15 + i % 3, 21 + i % 3, dtype=np.int32), np.eye(64)) for i in range(5)]
    capi.rcs_apply_unitaries(ctx, items)


def kernels(gpu):
    names = [k for k, _, _ in gpu.launches()]
    return sum(CHAIN in k for k in names), sum(SINGLE in k for k in names)


@pytest.mark.parametrize("skip", [0, 1])
@pytest.mark.parametrize("code", [TOO_LARGE, NOT_SUPPORTED])
def test_refused_chain_runs_as_single_passes(fake_gpu, code, skip):  # noqa: F811
    ctx = capi.rcs_create(24, capi.RCS_PREC_BF16X3)
    try:
        apply(ctx)
        assert kernels(fake_gpu) == (2, 0)  # five passes: one chain of two, one of three
        fake_gpu.reset()
        fake_gpu.fail(CHAIN, code, skip=skip, times=99)
        apply(ctx)
        chains, singles = kernels(fake_gpu)
        assert chains == skip and singles in ((5,) if skip == 0 else (2, 3))
        assert capi.rcs_last_pass_timing(ctx)[1] == 5
        assert fake_gpu.lib.cudaGetLastError() == 0  # nothing left behind for the next call
    finally:
        capi.rcs_destroy(ctx)


def test_other_launch_errors_are_reported(fake_gpu):  # noqa: F811
    ctx = capi.rcs_create(24, capi.RCS_PREC_BF16X3)
    try:
        fake_gpu.fail(CHAIN, ILLEGAL)
        with pytest.raises(capi.RcsError) as e:
            apply(ctx)
        assert e.value.code == capi.RCS_ERR_CUDA
    finally:
        capi.rcs_destroy(ctx)


def test_fewer_sms_than_passes(fake_gpu):  # noqa: F811
    fake_gpu.reset(sms=1)
    fake_gpu.lib.fake_set_device(2)  # its SM count has not been asked for yet
    ctx = capi.rcs_create(24, capi.RCS_PREC_BF16X3)
    try:
        apply(ctx)
        assert kernels(fake_gpu) == (0, 5)
    finally:
        capi.rcs_destroy(ctx)
