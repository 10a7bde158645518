"""The sliced layout of the staged CSR kernel against the FP64 oracle, at the sizes where its
plan changes: one chunk or two buffers, rows whose state words are staged or not, more CTAs
than SMs, rows far longer than their neighbours, empty rows, per-edge weights, both junctions,
and currents left to a separate update."""
import numpy as np
import pytest

from paper_1612_01501_gb300 import inputs
from paper_1612_01501_gb300 import ion

from helpers import STEP_RTOL
from test_gpu_parity import _one_step_case, _sgj_one_step, torch_cuda  # noqa: F401

pytestmark = pytest.mark.gpu


def _uneven_graph(n, k, seed):
    """A random symmetric graph in which cell 0 touches many cells and the last tenth none."""
    live = max(2, n - n // 10)
    rp, col = inputs.random_symmetric_csr(live, k, seed)
    rows = np.repeat(np.arange(live), np.diff(rp))
    hub = np.arange(1, live, max(1, live // 3000))
    key = np.unique(np.concatenate([rows.astype(np.int64) * n + col, hub, hub.astype(np.int64) * n]))
    r, c = (key // n).astype(np.int64), (key % n).astype(np.int32)
    row_ptr = np.zeros(n + 1, np.int64)
    np.cumsum(np.bincount(r, minlength=n), out=row_ptr[1:])
    return row_ptr.astype(np.int32), c


# n: a few cells; the row rounding; the last one-chunk size and the first with two buffers
# (152 SMs); the last with staged state words and the first without; more CTAs than SMs
@pytest.mark.parametrize("n,k", [(3, 2), (609, 8), (9001, 60), (51968, 8), (51969, 8), (77824, 4), (77900, 4), (160000, 4)])
@pytest.mark.parametrize("weights", ["uniform", "random"])
def test_sliced_step_matches_oracle(torch_cuda, O, n, k, weights):
    rp, col = _uneven_graph(n, k, 51)
    w = np.full(len(col), 0.002, np.float32)
    if weights == "random":
        w = (w * inputs.uniform(inputs.stream_seed(n, "sliced_w"), len(col), 0.5, 1.5)).astype(np.float32)
    err = _one_step_case(O, "csr", n, O.CSR, rp=rp, col=col, w=w, warm=3, tune=dict(csr_staging=2))
    assert err.max() <= STEP_RTOL, err.max(axis=1)


@pytest.mark.parametrize("n,weights", [(700, "random"), (60000, "uniform")])
def test_sliced_linear_junctions(torch_cuda, O, n, weights):
    rp, col = _uneven_graph(n, 12, 53)
    w = np.full(len(col), 0.002, np.float32)
    if weights == "random":
        w = (w * inputs.uniform(inputs.stream_seed(n, "sliced_w"), len(col), 0.5, 1.5)).astype(np.float32)
    err = _sgj_one_step(O, n, O.CSR, rp=rp, col=col, w=w, tune=dict(csr_staging=2))
    assert err.max() <= STEP_RTOL, err.max(axis=1)


@pytest.mark.parametrize("flag", ["split", "surrogate"])
def test_sliced_currents_for_a_separate_update(torch_cuda, flag):
    """The sliced kernel's currents (SPLIT, SURROGATE) against the direct kernel's, 6 steps:
    the sums differ in order only (1e-6 of the current's terms, at most 0.1 uA/cm^2 here, over
    dt = 0.05: 1e-7 mV a step; the learned rates pass BF16 thresholds that such a difference
    can cross, one BF16 unit of a rate, 0.4 %, in a step that moves a gate by less than 0.01)."""
    n, k = 3000, 80
    rp, col = _uneven_graph(n, k, 57)
    w = np.full(len(col), inputs.junction_weight(0.04, k), np.float32)
    S0 = ion.ion_default_state(n)
    S0[0] = (S0[0] + inputs.vdend_jitter(n, 57)).astype(np.float32)
    kw = dict(flags=ion.FLAG_KAHAN | ion.FLAG_SPLIT)
    if flag == "surrogate":
        rng = np.random.default_rng(3)
        p = {"w1": rng.normal(0, 1, (64, 2)), "b1": rng.normal(0, 1, 64), "w2": rng.normal(0, .12, (64, 64)),
             "b2": rng.normal(0, .1, 64), "w3": rng.normal(0, .05, (24, 64)), "b3": np.zeros(24)}
        kw = dict(flags=ion.FLAG_KAHAN | ion.FLAG_SURROGATE,
                  surrogate=ion.weights_from_dict(p, in_shift=(-25.0, 1.5), in_scale=(1 / 75.0, 0.67)))
    out = []
    for staging in (1, 2):
        with ion.Simulation(n, ion.CSR, row_ptr=rp, col=col, w=w, init_state=S0, tune=dict(csr_staging=staging), **kw) as sim:
            assert ion.ion_csr_layout(sim.h)["staged"] == staging - 1
            sim.step(6)
            out.append(sim.state())
    assert np.isfinite(out[0]).all()
    tol = 1e-4 if flag == "split" else 5e-3
    assert np.abs(out[0][:4] - out[1][:4]).max() <= tol
