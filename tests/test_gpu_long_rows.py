"""Networks in which a few cells have far more partners than the rest: their rows get more lanes,
so that a step does not last as long as one lane pair needs for the longest row."""
import time

import numpy as np
import pytest

from paper_1612_01501_gb300 import inputs
from paper_1612_01501_gb300 import ion

from helpers import STEP_RTOL
from test_gpu_parity import _one_step_case, _sgj_one_step, torch_cuda  # noqa: F401

pytestmark = pytest.mark.gpu


def hub_graph(n, k, hubs, length, seed=5):
    """A random symmetric graph of mean degree k in which `hubs` cells have `length` partners."""
    rp, col = inputs.random_symmetric_csr(n, k, seed)
    rng = np.random.default_rng(seed)
    rows = np.repeat(np.arange(n), np.diff(rp)).astype(np.int64)
    key = [rows * n + col]
    for h in range(hubs):
        a = (h * (n // hubs) + n // (2 * hubs)) % n
        p = rng.choice(n, length, replace=False).astype(np.int64)
        p = p[p != a]
        key += [a * n + p, p * n + a]
    key = np.unique(np.concatenate(key))
    row_ptr = np.zeros(n + 1, np.int64)
    np.cumsum(np.bincount(key // n, minlength=n), out=row_ptr[1:])
    return row_ptr.astype(np.int32), (key % n).astype(np.int32)


def _weights(col, kind):
    w = np.full(len(col), 0.0005, np.float32)
    if kind == "random":
        w = (w * inputs.uniform(inputs.stream_seed(len(col), "long_rows"), len(col), 0.5, 1.5)).astype(np.float32)
    return w


# staging 2: the sliced layout with one chunk, two buffers, rows with every count of lanes up to
# a warp (lengths 40 to n - 1); 1: the direct kernel
@pytest.mark.parametrize("staging", [1, 2])
@pytest.mark.parametrize("n,k,hubs,length", [(300, 3, 1, 299), (2000, 6, 3, 200), (2000, 6, 40, 60), (5000, 20, 2, 4000),
                                             (60000, 12, 5, 3000), (3000, 80, 30, 900)])
@pytest.mark.parametrize("weights", ["uniform", "random"])
def test_long_rows_one_step(torch_cuda, O, n, k, hubs, length, weights, staging):
    rp, col = hub_graph(n, k, hubs, length)
    err = _one_step_case(O, "csr", n, O.CSR, rp=rp, col=col, w=_weights(col, weights), warm=3,
                         tune=dict(csr_staging=staging))
    assert err.max() <= STEP_RTOL, err.max(axis=1)


@pytest.mark.parametrize("staging", [1, 2])
def test_long_rows_linear_junctions(torch_cuda, O, staging):
    rp, col = hub_graph(4000, 10, 4, 2500)
    err = _sgj_one_step(O, 4000, O.CSR, rp=rp, col=col, w=_weights(col, "random"), tune=dict(csr_staging=staging))
    assert err.max() <= STEP_RTOL, err.max(axis=1)


def _us_per_step(h, steps=200):
    ion.ion_step(h, steps)
    ion.ion_sync(h)
    best = 1e9
    for _ in range(5):
        t = time.perf_counter()
        ion.ion_step(h, steps)
        ion.ion_sync(h)
        best = min(best, (time.perf_counter() - t) / steps * 1e6)
    return best


# (cells, mean degree, staging asked, hubs, their length, most times the step of the same network
# without hubs): with the lanes of a mean row the steps took 31, 13 and 18 times as long
@pytest.mark.parametrize("n,k,staging,hubs,length,most", [(65536, 100, 2, 8, 30000, 12), (65536, 10, 1, 8, 3000, 8)])
def test_long_rows_do_not_hold_a_step(torch_cuda, n, k, staging, hubs, length, most):
    us = []
    for rp, col in (inputs.random_symmetric_csr(n, k, 5), hub_graph(n, k, hubs, length)):
        h = ion.ion_create(n, ion.CSR, row_ptr=rp, col=col, w=np.full(len(col), 1e-5, np.float32),
                           tune=dict(csr_staging=staging))
        try:
            us.append(_us_per_step(h))
        finally:
            ion.ion_destroy(h)
    assert us[1] <= most * us[0], us


# the rule between the two kernels without staging: 16-bit rows of 56 or more edges in networks of
# more than 40 000 cells take 16-byte loads
@pytest.mark.parametrize("n,k", [(40000, 60), (40001, 60), (40001, 52), (65536, 64), (65535, 130)])
@pytest.mark.parametrize("weights,linear", [("uniform", False), ("random", False), ("uniform", True), ("random", True)])
def test_unstaged_16_bit_rows_one_step(torch_cuda, O, n, k, weights, linear):
    rp, col = inputs.random_symmetric_csr(n, k, 3)
    w, tune = _weights(col, weights), dict(csr_staging=1)
    if linear:
        err = _sgj_one_step(O, n, O.CSR, rp=rp, col=col, w=w, tune=tune)
    else:
        err = _one_step_case(O, "csr", n, O.CSR, rp=rp, col=col, w=w, warm=2, tune=tune)
    assert err.max() <= STEP_RTOL, err.max(axis=1)


# both sides of the line between gathering and staging (the figures are beside the rule); short
# rows of 40 000 to 50 000 cells gather although staging gains 3 to 5 %
@pytest.mark.parametrize("n,k,staged", [(2000, 200, 0), (10000, 24, 0), (30000, 10, 0), (20000, 24, 0), (40000, 10, 0), (50000, 10, 0),
                                        (20000, 40, 1), (65536, 10, 0), (65536, 24, 1), (100000, 24, 1), (300000, 10, 0)])
def test_default_staging(torch_cuda, n, k, staged):
    rp, col = inputs.random_symmetric_csr(n, k, 3)
    with ion.Simulation(n, ion.CSR, row_ptr=rp, col=col, w=np.full(len(col), 0.001, np.float32)) as sim:
        assert ion.ion_csr_layout(sim.h)["staged"] == staged
