"""A change of the stored layout that stops half way leaves the layout that the state has."""
import struct

import numpy as np
import pytest

from fake_gpu import _fake_library, fake_gpu  # noqa: F401  (fixtures)
from paper_2512_07311_gb300 import capi


def test_failed_pass_keeps_the_passes_before_it(fake_gpu, tmp_path):  # noqa: F811
    n = 18
    phys = np.random.default_rng(4).permutation(n)
    with open(tmp_path / "s", "wb") as f:
        f.write(struct.pack("<8sIi64iQ", b"RCSSTATE", 1, n, *phys, *range(n, 64), 1 << n))
        f.write(np.zeros(1 << n, dtype=np.complex64).tobytes())
    ctx = capi.rcs_create(n)

    def load(fail_at=None):
        capi.rcs_state_load(ctx, str(tmp_path / "s"))
        fake_gpu.reset()
        if fail_at is not None:
            fake_gpu.fail("k_permute", 701, skip=fail_at)

    try:
        load()
        capi.rcs_state_device(ctx)
        passes = len(fake_gpu.launches())
        assert passes >= 2 and np.array_equal(capi.rcs_qubit_layout(ctx), np.arange(n))
        for done in range(passes):
            load(done)
            with pytest.raises(capi.RcsError):
                capi.rcs_state_device(ctx)
            assert len(fake_gpu.launches()) == done
            assert np.array_equal(capi.rcs_qubit_layout(ctx), phys) == (done == 0)
            capi.rcs_state_device(ctx)  # the rest of the passes and no more
            assert len(fake_gpu.launches()) == passes
            assert np.array_equal(capi.rcs_qubit_layout(ctx), np.arange(n))
    finally:
        capi.rcs_destroy(ctx)
