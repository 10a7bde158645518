"""How the gap currents are rounded: products fused into the sums, short chains, compensation."""
import numpy as np
import pytest

from paper_1612_01501_gb300 import inputs
from paper_1612_01501_gb300 import ion

from test_gpu_parity import torch_cuda  # noqa: F401

pytestmark = pytest.mark.gpu


def test_direct_csr_fuses_the_product_into_the_sum(torch_cuda):
    """A ring with linear junctions and one lane per row: I_c = w1 d1 + w2 d2 with the second
    product fused, the sum of one rounded and one exact product rounded once.  Exact products
    and their sum fit 64 bits, so the reference is exact; a second rounded product differs from
    it in about a quarter of the cells."""
    n = 4096
    rp = np.arange(0, 2 * n + 1, 2, dtype=np.int32)
    i = np.arange(n)
    col = np.sort(np.stack([(i - 1) % n, (i + 1) % n], 1), axis=1).astype(np.int32)
    w = inputs.uniform(inputs.stream_seed(n, "ring"), 2 * n, 0.001, 0.01).astype(np.float32).reshape(n, 2)
    S0 = ion.ion_default_state(n)
    S0[0] = (S0[0] + inputs.vdend_jitter(n, 3)).astype(np.float32)
    with ion.Simulation(n, ion.CSR, row_ptr=rp, col=col.ravel(), w=w.ravel(), init_state=S0,
                        flags=ion.FLAG_KAHAN | ion.FLAG_SGJ, tune=dict(csr_staging=1, csr_lanes_per_row=1)) as sim:
        sim.step(1)
        ic = sim.state(18)
    d = (S0[0][:, None] - S0[0][col]).astype(np.float32)
    p = w.astype(np.float64) * d.astype(np.float64)
    fused = (p[:, 0].astype(np.float32).astype(np.float64) + p[:, 1]).astype(np.float32)
    twice = p[:, 0].astype(np.float32) + p[:, 1].astype(np.float32)
    assert (fused != twice).mean() > 0.1
    assert np.array_equal(ic, fused)
