"""FP32 batch engine on circuits around the size where a work item has one slice per thread
(256) and where it has two, every fusion width, against complex128."""
import numpy as np
import pytest

from paper_2512_07311_gb300 import capi
from paper_2512_07311_gb300 import circuits as C

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("k", [2, 3, 4, 5])
def test_small_circuits_vs_oracle(oracle, k):
    circs = [C.generate(C.grid_for_n(n), 8, "EFGH", seed=900 + n, jitter=0.05) for n in range(2, 16)]
    b = capi.rcs_batch_create([(c.n_qubits, c.gates, 0, 1) for c in circs], k_max=k, autotune=0)
    try:
        capi.rcs_batch_launch(b)
        capi.rcs_batch_wait(b)
        for i, c in enumerate(circs):
            want = oracle.simulate(c.n_qubits, c.gates)
            # per pass: rounding of U and of 2 * 2^k fused multiply-adds, half an ulp each, of the norm
            bound = capi.rcs_batch_info(b, i)["n_passes"] * (2 * 2 ** k + 1) * 2.0 ** -24
            assert np.linalg.norm(capi.rcs_batch_state_read(b, i) - want) <= bound
    finally:
        capi.rcs_batch_destroy(b)
