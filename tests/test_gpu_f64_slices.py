"""The FP64 block GEMM where its operands are cut into slices: edges of its
tiles above the small-launch line, and data whose scales meet badly.

Chains of three sites whose inner bonds hold one charge sector (two on the
second bond in the segmented cases), so that the middle site's products are
(d1 x k1)(k1 x d2) and (e2 x d1)(d1 x d2).

Tolerance: a sum of K products in FP64 is within K 2^-53 of the sum of their
absolute values (first order), the slices within the same; the overlap chains
two such sums per site: 12 max(K) 2^-53 of the overlap of the absolute values."""
import numpy as np
import pytest

import synth
from synth.states import SITE_CHARGE

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def td():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1902_08489_gb300 as mod
    mod.lib()
    return mod


def _chain(rng, d1, d2, d2b=0):
    """Charges (0,0) - (1,1) - {(1,1) x d2b, (2,0) x d2} - (2,0)."""
    labels = [np.array(q, dtype=np.int64) for q in
              ([(0, 0)], [(1, 1)] * d1, [(1, 1)] * d2b + [(2, 0)] * d2, [(2, 0)])]
    dims = [len(q) for q in labels]
    tensors = []
    for i in range(3):
        A = np.zeros((dims[i], 4, dims[i + 1]), dtype=np.complex128)
        for s, q in enumerate(SITE_CHARGE):
            on = (labels[i][:, None, :] + np.array(q) == labels[i + 1][None]).all(axis=2)
            A[:, s] = on * (rng.standard_normal(on.shape) + 1j * rng.standard_normal(on.shape))
        tensors.append(A)
    return tensors, labels


def _overlap(B, A):
    E = np.ones((1, 1), dtype=np.complex128)
    for x, y in zip(B, A):
        E = np.einsum("xsq,xsp->qp", x.conj(), np.tensordot(E, y, axes=1), optimize=True)
    return E[0, 0]


def _check(td, B, A, labels_b, labels_a):
    ctx = td.Context("fp64")
    got = td.overlap(ctx, td.mps_import(ctx, B, labels_b), td.mps_import(ctx, A, labels_a))
    ctx.close()
    ref = _overlap(B, A)
    scale = _overlap([np.abs(x) for x in B], [np.abs(x) for x in A]).real
    tol = 12 * max(max(x.shape) for x in A + B) * 2.0 ** -53
    assert abs(got - ref) <= tol * scale
    return got, ref, tol


@pytest.mark.parametrize("d1,k1,d2,e2,d2b", [
    (63, 31, 25, 40, 0), (64, 32, 48, 33, 0), (65, 33, 49, 64, 0), (32, 17, 97, 65, 0),
    (40, 24, 193, 48, 0), (33, 64, 24, 63, 0), (130, 129, 128, 127, 0),
    (33, 1500, 40, 48, 0), (33, 1500, 7, 24, 40), (70, 32, 50, 60, 31), (48, 90, 1, 64, 90)])
def test_overlap_at_tile_edges(td, d1, k1, d2, e2, d2b):
    rng = np.random.default_rng([d1, k1, d2, e2, d2b])
    B, qb = _chain(rng, d1, e2, d2b // 2)
    A, qa = _chain(rng, k1, d2, d2b)
    _check(td, B, A, qb, qa)


@pytest.mark.parametrize("s", [10, 30, 300])
@pytest.mark.parametrize("d1,k1,d2,e2", [(64, 32, 48, 33), (65, 100, 97, 64)])
def test_overlap_in_an_unbalanced_gauge(td, d1, k1, d2, e2, s):
    """A_i X, X^-1 A_(i+1) with X = diag(2^g), |g| <= s on both inner bonds: every
    product of the contraction is the same, only how it is shared out differs."""
    rng = np.random.default_rng([d1, k1, s])
    B, qb = _chain(rng, d1, e2)
    A, qa = _chain(rng, k1, d2)
    ref = _overlap(B, A)
    scale = _overlap([np.abs(x) for x in B], [np.abs(x) for x in A]).real
    for i in (0, 1):
        x = 2.0 ** rng.integers(-s, s + 1, size=A[i].shape[2])
        A[i], A[i + 1] = A[i] * x, A[i + 1] / x[:, None, None]
    got, again, tol = _check(td, B, A, qb, qa)
    assert again == ref
    assert abs(got - ref) <= tol * scale


def test_imaginary_part_of_nearly_real_data(td):
    """<a|b + i 2^-40 c> with real tensors: the imaginary part has its own relative
    accuracy, as FP64 sums of its products have."""
    rng = np.random.default_rng(6)
    eps = 2.0 ** -40
    B, qb = _chain(rng, 64, 40)
    A, qa = _chain(rng, 48, 65)
    B, A = [x.real + 0j for x in B], [x.real + 0j for x in A]
    C = A[1] * rng.standard_normal(A[1].shape)
    ctx = td.Context("fp64")
    got = td.overlap(ctx, td.mps_import(ctx, B, qb),
                     td.mps_import(ctx, [A[0], A[1] + 1j * eps * C, A[2]], qa))
    ctx.close()
    ref = eps * _overlap(B, [A[0], C, A[2]]).real
    scale = eps * _overlap([abs(x) for x in B], [abs(A[0]), abs(C), abs(A[2])]).real
    assert abs(got.imag - ref) <= 12 * 65 * 2.0 ** -53 * scale


def test_gradient_in_an_unbalanced_gauge(td):
    """Element by element: the gradient of A_i X and X^-1 A_(i+1) is that of the plain
    tensors times X^-1 and X.  Both are rounded sums over environments of K <= 400
    products per step and L = 10 steps, 4000 2^-53 of the sum of absolute values,
    for which the largest element times 100 stands: 1e-10 with a margin of 2."""
    L, n = 10, 10
    I = synth.make_integrals(L, seed=3)
    A, q = synth.random_mps(L, n, 0, 200, seed=4)
    rng = np.random.default_rng(8)
    X = [2.0 ** rng.integers(-15, 16, size=len(x)) for x in q]
    X[0][:] = X[L][:] = 1.0
    U = [a * X[i + 1] / X[i][:, None, None] for i, a in enumerate(A)]
    ctx = td.Context("fp64")
    mpo = td.build_mpo(ctx, I.h, I.eri, n_elec=n)
    e0, g0, _ = td.energy_gradient(ctx, mpo, td.mps_import(ctx, A, q))
    e1, g1, _ = td.energy_gradient(ctx, mpo, td.mps_import(ctx, U, q))
    assert abs(e1 - e0) <= 1e-11 * abs(e0)
    g0, g1 = g0.export()[0], g1.export()[0]
    for i in range(L):
        back = g1[i] * X[i + 1] / X[i][:, None, None]
        assert np.abs(back - g0[i]).max() <= 1e-10 * np.abs(g0[i]).max()
    ctx.close()
