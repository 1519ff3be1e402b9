"""The Gram-Schmidt QR far from unit scale: a one-term, one-site fit of a state
that lies in its own manifold returns the state, also where the norms square
to the edge of the FP64 range and one direction is 1e-10 of another one.

Tolerances as at unit scale: Q^H Q - 1 within 1e-13, the overlap within 1e-12
(12 sites at a few n 2^-53 each); an overlap of 1e-294 itself is a multiple of
2^-1074, 5e-30 of it."""
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


@pytest.mark.parametrize("scale", [1e-147, 1e-130, 1.0, 1e130, 1e147])
@pytest.mark.parametrize("L,n,D", [(6, 5, 33), (8, 8, 130), (10, 9, 400)])
def test_one_term_fit_far_from_unit_scale(td, L, n, D, scale):
    A, q = synth.random_mps(L, n, n % 2, D, seed=12)
    k = L // 2
    same = np.flatnonzero((q[k] == q[k][len(q[k]) // 2]).all(axis=1))
    A[k][same[1]] = A[k][same[0]] + 1e-10 * A[k][same[1]]
    for i, a in enumerate(A):
        A[i] = a / np.linalg.norm(a) * (scale if i == 0 else np.sqrt(a.shape[2]))
    ctx = td.Context("fp64")
    ctx.set_schedule(0, 1)
    psi = td.mps_import(ctx, A, q)
    out = td.mps_sum(ctx, [1.0], [psi], D, 0.0)
    nn = td.overlap(ctx, psi, psi).real
    assert np.isfinite(nn) and nn > 0
    assert all(np.isfinite(T).all() for T in out.export()[0])
    assert abs(td.overlap(ctx, psi, out) - nn) <= 1e-12 * nn
    assert abs(td.overlap(ctx, out, out).real - nn) <= 1e-12 * nn
    for T in out.export()[0][1:]:
        M = T.reshape(T.shape[0], -1)
        assert np.abs(M @ M.conj().T - np.eye(len(M))).max() <= 1e-13
    ctx.close()
