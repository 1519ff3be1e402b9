"""The Jacobi SVD over its size range, through compression: the truncation of
a state with prescribed sector sizes is its SVD at every bond.

Reference: the dense SVD of every bond in numpy, on the same state.  Tolerance:
the singular values of both sides carry a few n 2^-53 of the largest; the
1-RDM and the discarded weight of the truncated state follow within 1e-9 for
the gaps of a random spectrum (n <= 100, gaps of 1e-4 and more: 1e-14 / 1e-4
with a margin of 10)."""
import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def td():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1902_08489_gb300 as mod
    mod.lib()
    return mod


def _right_canonical(C):
    C = list(C)
    for i in range(len(C) - 1, 0, -1):
        Q, R = np.linalg.qr(C[i].reshape(C[i].shape[0], -1).conj().T)
        C[i] = Q.conj().T.reshape(-1, 4, C[i].shape[2])
        C[i - 1] = np.tensordot(C[i - 1], R.conj().T, axes=1)
    return C


def _compress(C, D):
    C, lost = _right_canonical(C), 0.0
    for i in range(len(C) - 1):
        a, _, b = C[i].shape
        U, s, V = np.linalg.svd(C[i].reshape(4 * a, b), full_matrices=False)
        k = min(D, int((s > 1e-12 * s[0]).sum()))
        lost += (s[k:] ** 2).sum() / (s ** 2).sum()
        C[i] = U[:, :k].reshape(a, 4, k)
        C[i + 1] = np.tensordot(s[:k, None] * V[:k], C[i + 1], axes=1)
    return C, lost


def _overlap(B, A):
    E = np.ones((1, 1), dtype=np.complex128)
    for x, y in zip(B, A):
        E = np.tensordot(x.conj(), np.tensordot(E, y, axes=1), axes=([0, 1], [0, 1]))
    return E[0, 0]


@pytest.mark.parametrize("L,n,D,scale", [(2, 2, 4, 1.0), (4, 4, 17, 1e-130), (6, 5, 64, 1e130),
                                         (8, 8, 200, 1.0), (10, 10, 700, 1.0), (10, 10, 1000, 1.0)])
def test_compression_is_the_dense_svd(td, L, n, D, scale):
    A, q = synth.random_mps(L, n, n % 2, D, seed=5)
    A[0] = A[0] * scale
    keep = max(2, max(len(x) for x in q) * 2 // 3)
    ctx = td.Context("fp64")
    psi = td.mps_import(ctx, A, q)
    lost = td.compress(ctx, psi, keep, 0.0)
    ref, lost_ref = _compress([a / (scale if i == 0 else 1.0) for i, a in enumerate(A)], keep)
    got = psi.export()[0]
    got[0] = got[0] / scale
    nn = _overlap(ref, ref).real
    assert abs(lost - lost_ref) <= 1e-9
    assert abs(_overlap(got, got).real - nn) <= 1e-9 * nn
    assert abs(_overlap(ref, got) - nn) <= 1e-9 * nn
    ctx.close()
