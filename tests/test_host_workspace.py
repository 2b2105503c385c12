"""Workspace sizes follow the rows of the call (CPU: the size functions launch nothing)."""
import ctypes as C

import pytest

from paper_2410_01657_gb300 import _build
from paper_2410_01657_gb300 import binding as B


@pytest.fixture(scope="module", autouse=True)
def built():
    _build.build()
    B.load()


def _sizes(dims, rows):
    S = B.gnn_mlp()
    S.n_lin = len(dims) - 1
    for k, d in enumerate(dims):
        S.dims[k] = d
    for k in range(S.n_lin):
        S.W[k] = S.b[k] = 256   # (not read)
    S.gamma = S.beta = 256
    f, b = C.c_size_t(), C.c_size_t()
    B.call("gnn_mlp_workspace_size", C.byref(S), rows, C.byref(f), C.byref(b))
    return f.value, b.value


@pytest.mark.parametrize("dims", [[4, 128, 128, 128, 128], [64, 64, 64], [128, 16, 128]])
def test_row_mlp_backward_partials(dims):
    # Activations, two gradient buffers and dY, 4 bytes each, and one set of partial gradients per 64 rows
    grads = sum(dims[k] * dims[k + 1] + dims[k + 1] for k in range(len(dims) - 1)) + 2 * dims[-1]
    for rows in (1, 10, 64, 65, 1000, 100000):
        acts = rows * (sum(dims[1:]) + 3 * max(dims)) * 4
        ctas = min((rows + 63) // 64, 160)
        assert _sizes(dims, rows)[1] <= acts + ctas * grads * 4 + 64 * 1024
    assert _sizes(dims, 10)[1] <= _sizes(dims, 1000)[1] <= _sizes(dims, 100000)[1]
