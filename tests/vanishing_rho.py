"""A system on which (r^, r) of BiCGStab vanishes exactly after the first iteration
while r does not: 3x3 blocks [[1, 1, -1], [1, 2, 0], [1, 0, 4]], b = e1 in each, so
that alpha = 1 and the first entries of s, t and r are zero in exact small integers
(with a power of two of blocks, in any order of the sums)."""
import numpy as np


def blocks(m, pad=0):
    """m blocks (a power of two) and `pad` rows of the identity with b = 0."""
    n = 3 * m + pad
    k = 3 * np.arange(m)[:, None]
    cols = np.concatenate([(k + np.array([0, 1, 2, 0, 1, 0, 2])).ravel(), 3 * m + np.arange(pad)])
    vals = np.concatenate([np.tile([1.0, 1, -1, 1, 2, 1, 4], m), np.ones(pad)]).astype(np.complex128)
    lens = np.concatenate([np.tile([3, 2, 2], m), np.ones(pad, np.int64)])
    rowptr = np.concatenate([[0], np.cumsum(lens)])
    b = np.zeros(n, np.complex128)
    b[0:3 * m:3] = 1.0
    return rowptr.astype(np.int32), cols.astype(np.int32), vals, b
