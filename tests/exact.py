"""Small dense problems in extended precision (numpy's longdouble), to measure errors against:
LDL^T, x and N^-1 of a dense N, and problems made from a dense matrix."""
import dataclasses

import numpy as np
import scipy.sparse as sp

from spigen import random_spd

LD = np.longdouble


def dense(pb, values=None):
    a = sp.csc_matrix((pb.values if values is None else values, pb.rowind, pb.colptr), shape=(pb.n, pb.n)).toarray()
    return a + np.tril(a, -1).T


def problem(a, pattern=None):
    """The problem of the dense symmetric matrix a (its nonzeros, or all of `pattern`)."""
    n = len(a)
    low = sp.csc_matrix(np.tril(np.ones((n, n)) if pattern is None else pattern))
    low.sort_indices()
    col = np.repeat(np.arange(n), np.diff(low.indptr))
    return dataclasses.replace(random_spd(n, 0.0, n, dominance=1.0), colptr=low.indptr.astype(np.int64),
                               rowind=low.indices.astype(np.int32), values=np.ascontiguousarray(a[low.indices, col]))


def ldl(a):
    a = a.astype(LD)
    n = len(a)
    L, d = np.eye(n, dtype=LD), np.zeros(n, LD)
    for c in range(n):
        d[c] = a[c, c]
        L[c + 1:, c] = a[c + 1:, c] / d[c]
        a[c + 1:, c + 1:] -= np.outer(L[c + 1:, c], a[c + 1:, c])
    return L, d


def inverse(a):
    """N^-1 in extended precision."""
    L, d = ldl(a)
    Z = np.eye(len(d), dtype=LD)
    for c in range(len(d)):
        Z[c + 1:] -= np.outer(L[c + 1:, c], Z[c])
    return Z.T @ (Z / d[:, None])


def backward_error(a, x, b):
    """||b - N x|| / (||N|| ||x|| + ||b||), the residual in extended precision."""
    r = b.astype(LD) - a.astype(LD) @ x.astype(LD)
    return float(np.linalg.norm(r.astype(float)) / (np.linalg.norm(a, 2) * np.linalg.norm(x) + np.linalg.norm(b)))
