"""Matrices whose column order changed after scipy looked at it: the caller's
cached flag is not taken for the order, and results carry none."""
import ctypes as C

import numpy as np
import scipy.sparse as sp

from paper_2407_09848_gb300 import amgps


def _matrix():
    return sp.csr_matrix(np.array([[4.0, 0, 1, 2], [0, 5, 3, 0], [1, 3, 6, 0], [2, 0, 0, 7]]))


def test_a_stale_flag_is_not_trusted():
    A = _matrix()
    assert A.has_sorted_indices  # cached from here on
    A.indices[:3] = A.indices[:3][::-1].copy()
    A.data[:3] = A.data[:3][::-1].copy()
    got = amgps._sorted_csr(A)
    for i in range(4):
        assert np.all(np.diff(got.indices[got.indptr[i]:got.indptr[i + 1]]) > 0)
    assert np.array_equal(got.toarray(), _matrix().toarray())
    assert A.indices[0] == 3     # the caller's arrays stay as they are


def test_results_can_be_renumbered_in_place():
    A = _matrix()
    libc = C.CDLL(None)
    libc.malloc.restype, libc.malloc.argtypes = C.c_void_p, [C.c_size_t]
    buf = amgps.CSRBuf(4, 4, A.nnz)

    def put(a, dtype, ctype):
        a = np.ascontiguousarray(a, dtype=dtype)
        p = libc.malloc(a.nbytes)
        C.memmove(p, a.ctypes.data, a.nbytes)
        return C.cast(p, C.POINTER(ctype))
    buf.rowptr = put(A.indptr, np.int32, C.c_int32)
    buf.col = put(A.indices, np.int32, C.c_int32)
    buf.val = put(A.data, np.float64, C.c_double)
    R = amgps._from_buf(buf)
    perm = np.array([2, 0, 3, 1], dtype=np.int32)
    R.indices[:] = perm[R.indices]
    R.sort_indices()             # nothing to do if the result claims to be sorted
    assert all(np.all(np.diff(R.indices[R.indptr[i]:R.indptr[i + 1]]) > 0) for i in range(4))
    dense = np.zeros((4, 4))
    dense[:, perm] = _matrix().toarray()
    assert np.array_equal(R.toarray(), dense)
