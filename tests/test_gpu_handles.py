"""Several live handles: what the setup of one sets on a kernel (its shared-memory limit) holds
for the others; and a tuned batch steps in every form."""
import numpy as np
import pytest

from paper_1612_01501_gb300 import inputs
from paper_1612_01501_gb300 import ion

from test_gpu_parity import torch_cuda  # noqa: F401

pytestmark = pytest.mark.gpu


def _dense_nets(sizes):
    return [dict(n=n, kind=ion.DENSE_UNIFORM, g=inputs.junction_weight(0.04, n)) for n in sizes]


def _csr(n, k, **kw):
    rp, col = inputs.random_symmetric_csr(n, k, 5)
    return dict(n=n, kind=ion.CSR, row_ptr=rp, col=col, w=np.full(len(col), 2e-3, np.float32), **kw)


def _sim(n, kind, **kw):
    return ion.ion_create(n, kind, **kw), n


CASES = {
    # the same launch shape, hence the same kernel, for both sizes
    "dense": (lambda n: _sim(n, ion.DENSE_UNIFORM, g=1e-4, tune=dict(dense_rows_per_warp=4, dense_warps=8, dense_col_splits=1)),
              9000, 64),
    "persistent": (lambda n: _sim(n, ion.DENSE_UNIFORM, g=1e-4, flags=ion.FLAG_KAHAN | ion.FLAG_PERSISTENT,
                                  tune=dict(dense_rows_per_warp=4, dense_warps=16, dense_col_splits=1)), 9000, 300),
    "chunked": (lambda n: _sim(**_csr(n, 20, flags=ion.FLAG_KAHAN | ion.FLAG_CSR_AS_GIVEN, tune=dict(csr_staging=2))),
                40000, 500),
    "batch": (lambda n: (ion.ion_create_batch(_dense_nets([n, n]) + [_csr(n, 20)]), 3 * n), 4096, 40),
    "batch_persistent": (lambda n: (ion.ion_create_batch(_dense_nets([n, n]) + [_csr(n, 20)],
                                                         flags=ion.FLAG_KAHAN | ion.FLAG_PERSISTENT), 3 * n), 4096, 40),
}


@pytest.mark.parametrize("case", CASES)
def test_a_smaller_handle_leaves_a_larger_one_working(torch_cuda, case):
    make, large, small = CASES[case]
    a, n = make(large)
    b, m = make(small)
    try:
        ion.ion_step(a, 3)
        ion.ion_step(b, 3)
        got = ion.ion_read_state(a, n)
        assert np.isfinite(ion.ion_read_state(b, m)).all()
    finally:
        ion.ion_destroy(a)
        ion.ion_destroy(b)
    c, _ = make(large)
    try:
        ion.ion_step(c, 3)
        assert np.array_equal(got, ion.ion_read_state(c, n))
    finally:
        ion.ion_destroy(c)


def test_tuned_persistent_batch_steps_with_dense_input(torch_cuda):
    """A dense input takes the per-step launches, whose tiles follow the tuned rows per warp."""
    sizes = [1792] * 12
    n = sum(sizes)
    drive = np.random.default_rng(1).uniform(0, 4, (3, n)).astype(np.float32)
    out = []
    for flags in (ion.FLAG_KAHAN, ion.FLAG_KAHAN | ion.FLAG_PERSISTENT):
        h = ion.ion_create_batch(_dense_nets(sizes), flags=flags)
        try:
            if flags & ion.FLAG_PERSISTENT:
                ion.ion_autotune(h, 4)
            ion.ion_step(h, 3, dense=drive)
            out.append(ion.ion_read_state(h, n))
        finally:
            ion.ion_destroy(h)
    assert np.isfinite(out[1]).all()
    assert np.abs(out[0][:3] - out[1][:3]).max() <= 1e-3   # rows per warp move the sums' order only
