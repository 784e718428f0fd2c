"""A batch belongs to the device that was current when it was made; its state is read there
whatever device the caller has current, and that one stays current."""
from fake_gpu import _fake_library, fake_gpu  # noqa: F401  (fixtures)
from paper_2512_07311_gb300 import capi
from paper_2512_07311_gb300 import circuits as C


def test_state_read_runs_on_the_batch_device(fake_gpu):  # noqa: F811
    circ = C.generate(C.grid_for_n(14), 8, "EFGH", seed=3)  # stored in a permuted layout: read by a kernel
    b = capi.rcs_batch_create([(14, circ.gates, 10, 1)], precision=capi.RCS_PREC_BF16X3)
    try:
        for current in (0, 1):
            fake_gpu.reset()
            fake_gpu.lib.fake_set_device(current)
            capi.rcs_batch_state_read(b, 0)
            assert fake_gpu.lib.fake_device() == current
            assert [device for _, _, device in fake_gpu.launches()] == [0]
            fake_gpu.fail("k_read_mapped", 719)  # a launch that fails hands the device back too
            try:
                capi.rcs_batch_state_read(b, 0)
                raise AssertionError("the failed launch was not reported")
            except capi.RcsError as e:
                assert e.code == capi.RCS_ERR_CUDA
            assert fake_gpu.lib.fake_device() == current
    finally:
        fake_gpu.reset()
        capi.rcs_batch_destroy(b)
