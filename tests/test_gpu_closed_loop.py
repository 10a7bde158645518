"""The closed loop's host path: from a handle's fourth small read on, state and status come back
through a pinned buffer and dense inputs are read from it in place.  Both must be what the
copies give, bit for bit, whatever the field, the size and the order of calls."""
import numpy as np
import pytest

from paper_1612_01501_gb300 import inputs
from paper_1612_01501_gb300 import ion

from test_gpu_parity import torch_cuda  # noqa: F401

pytestmark = pytest.mark.gpu


def _make(kind, n):
    S0 = ion.ion_default_state(n)
    S0[0] = (S0[0] + inputs.vdend_jitter(n, 3)).astype(np.float32)
    if kind == "dense":
        return ion.Simulation(n, ion.DENSE_UNIFORM, g=inputs.junction_weight(0.04, n), init_state=S0)
    if kind == "cells":
        return ion.Simulation(n, ion.NO_GJ, init_state=S0)
    rp, col = inputs.random_symmetric_csr(n, 10, 3)
    return ion.Simulation(n, ion.CSR, row_ptr=rp, col=col, w=np.full(len(col), 0.01, np.float32), init_state=S0)


# 862 cells: the largest whole state the buffer holds; 16384: the largest field and input
@pytest.mark.parametrize("kind,n", [("dense", 1), ("dense", 862), ("dense", 863), ("csr", 1000), ("cells", 16384),
                                    ("cells", 16385)])
def test_repeated_small_reads_and_inputs_match_copies(torch_cuda, kind, n):
    rng = np.random.default_rng(n)
    with _make(kind, n) as a, _make(kind, n) as b:
        drive = rng.uniform(0, 4, (12, n)).astype(np.float32)
        for t in range(12):
            a.step(1, dense=drive[t:t + 1])
            if t in (5, 6):                      # two inputs without a read between them
                continue
            v = a.state(t % ion.NFIELDS)
            assert np.array_equal(v, a.state(t % ion.NFIELDS))
        b.step(12, dense=drive)                  # one copy, no read: the plain path
        ref = b.state()
        assert np.array_equal(a.state(), ref)
        for f in range(ion.NFIELDS):
            assert np.array_equal(a.state(f), ref[f])
        assert a.t == b.t == 12


def test_status_is_reported_through_the_pinned_read(torch_cuda):
    n = 50
    with _make("cells", n) as sim:
        for _ in range(6):
            sim.step(1)
            sim.state(2)
        bad = sim.state()
        bad[1, 7] = np.nan
        sim.write(bad)
        sim.step(1)
        with pytest.raises(ion.IonError) as e:
            sim.state(1)
        assert e.value.status == ion.ERR_NONFINITE
