"""A tensor-core wait that runs out: the CTA reports it and stores nothing of its cells."""
import numpy as np
import pytest

from paper_1612_01501_gb300 import inputs
from paper_1612_01501_gb300 import ion

from test_gpu_parity import torch_cuda  # noqa: F401

pytestmark = pytest.mark.gpu


def _weights():
    rng = np.random.default_rng(3)
    p = {"w1": rng.normal(0, 1, (64, 2)), "b1": rng.normal(0, 1, 64), "w2": rng.normal(0, .12, (64, 64)),
         "b2": rng.normal(0, .1, 64), "w3": rng.normal(0, .05, (24, 64)), "b3": np.zeros(24)}
    return ion.weights_from_dict(p, in_shift=(-25.0, 1.5), in_scale=(1 / 75.0, 0.67))


@pytest.mark.parametrize("which", [1, 2, 3, 4, 5, 6])
def test_a_wait_that_runs_out_stores_nothing(torch_cuda, which):
    """The which-th completion of the first CTA is withheld (every wait ends after 0.5 s): its 128
    cells keep every word of the step before, the others advance, the status says timeout, and
    the next handle works."""
    n = 300
    S0 = ion.ion_default_state(n)
    S0[0] = (S0[0] + inputs.vdend_jitter(n, 7)).astype(np.float32)
    with ion.Simulation(n, ion.NO_GJ, init_state=S0, flags=ion.FLAG_KAHAN | ion.FLAG_SURROGATE, surrogate=_weights()) as sim:
        sim.step(1)
        ref = sim.state()
    got = np.zeros_like(S0)
    with ion.Simulation(n, ion.NO_GJ, init_state=S0, flags=ion.FLAG_KAHAN | ion.FLAG_SURROGATE, surrogate=_weights(),
                        debug_delay_ns=which) as sim:
        sim.step(1)
        with pytest.raises(ion.IonError) as e:
            sim.sync()
        assert e.value.status == ion.ERR_TIMEOUT
        rc = ion.lib().ion_read_state(sim.h, ion.FIELD_ALL, got.ctypes.data_as(ion.c_f32p), got.size)
        assert rc == ion.ERR_TIMEOUT
    assert np.array_equal(got[1:, :128], S0[1:, :128])     # (V_dend of step 1 lies in its other slot)
    assert np.array_equal(got[:, 128:], ref[:, 128:])
    with ion.Simulation(n, ion.NO_GJ, init_state=S0, flags=ion.FLAG_KAHAN | ion.FLAG_SURROGATE, surrogate=_weights()) as sim:
        sim.step(1)
        assert np.array_equal(sim.state(), ref)
