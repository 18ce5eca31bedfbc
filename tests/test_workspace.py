"""Sizes of the caller-owned buffers (host only)."""
import ctypes

import numpy as np
import pytest

from workloads.heavyhex import LATTICES, heavy_hex


def _bytes(name, copies, D):
    from paper_2309_15642_gb300 import _abi, _build
    _build.build()
    lib = _abi.load()
    n, edges = heavy_hex(*LATTICES[name])
    edges = np.ascontiguousarray(edges, dtype=np.int32)
    graphs = (_abi.GraphC * copies)()
    for g in graphs:
        g.n_qubits, g.n_edges = n, len(edges)
        g.edges = edges.ctypes.data_as(ctypes.POINTER(ctypes.c_int32))
        g.colour = None
    h, s, w = ctypes.c_void_p(), ctypes.c_size_t(), ctypes.c_size_t()
    assert lib.gpeps_create(ctypes.cast(graphs, ctypes.c_void_p), copies, D, _abi.GPEPS_C128, None,
                            ctypes.byref(h)) == 0
    assert lib.gpeps_query_workspace(h, ctypes.byref(s), ctypes.byref(w)) == 0
    lib.gpeps_destroy(h)
    return s.value, w.value


@pytest.mark.parametrize("D,copies", [(128, 2), (96, 6), (64, 39), (32, 340), (17, 1800)])
def test_complex128_batches_that_filled_the_card_still_fit(D, copies):
    """Batches of 1121 qubits whose tensors and Gram partials, one set per colour class, are as much
    as 284208 MiB hold, have to be accepted by the card with the kicked rows kept as well."""
    assert sum(_bytes(1121, copies, D)) <= 284208 << 20


@pytest.mark.parametrize("D,copies,work", [(65, 2, 2 * 7.98e9), (96, 2, 2 * 35.7e9), (128, 2, 2 * 110.5e9)])
def test_kicked_rows_take_the_room_of_the_lower_triangles(D, copies, work):
    """Beyond D = 64 the rows and the upper triangles of the partials are no larger than the full
    partials alone were."""
    assert _bytes(1121, copies, D)[1] <= work
