"""The dense network with linear junctions: its sums run over 16-byte groups of four chains and,
beyond 16 384 cells, over the partial sums of a first launch while the cells' words are already
being read.  Checked at the edges of the groups, of the CTAs and of the one-launch rule."""
import numpy as np
import pytest

from paper_1612_01501_gb300 import inputs
from paper_1612_01501_gb300 import ion

from helpers import STEP_RTOL
from test_gpu_parity import _sgj_one_step, torch_cuda  # noqa: F401

pytestmark = pytest.mark.gpu


# one step against the oracle, at its bound for one step
@pytest.mark.parametrize("n", [2, 3, 5, 127, 255, 257, 1023, 16383, 16384, 16385, 24577])
def test_one_step(torch_cuda, O, n):
    err = _sgj_one_step(O, n, O.DENSE, g=float(np.float32(inputs.junction_weight(0.04, n))))
    assert err.max() <= STEP_RTOL, err.max(axis=1)


# many steps as programmatic launches in a graph and one ordinary launch after the other: the
# early reads may not change a bit
@pytest.mark.parametrize("n", [1001, 16385, 70001, 1048579])
def test_steps_match_ordinary_launches(torch_cuda, n):
    S0 = ion.ion_default_state(n)
    S0[0] = (S0[0] + inputs.vdend_jitter(n, 5)).astype(np.float32)
    got = []
    for fl in (0, ion.FLAG_NO_PDL | ion.FLAG_NO_GRAPH):
        with ion.Simulation(n, ion.DENSE_UNIFORM, g=float(np.float32(inputs.junction_weight(0.04, n))), init_state=S0,
                            flags=ion.FLAG_KAHAN | ion.FLAG_SGJ | fl) as sim:
            sim.step(67)
            got.append(sim.state())
    np.testing.assert_array_equal(got[0].view(np.uint32), got[1].view(np.uint32))
