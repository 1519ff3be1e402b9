"""The Gram-Schmidt QR over its shapes: one matrix per CTA, per cluster in
shared memory and in global memory.  A one-term, one-site fit of a state that
lies in its own manifold returns the state, with right-orthonormal sites.

Tolerances: Gram-Schmidt with re-orthogonalisation leaves Q^H Q - 1 at a small
multiple of sqrt(n) 2^-53 (n <= 200: 1e-13 with a margin of 50); every site
adds a few n 2^-53 to the overlap (12 sites: below 1e-12)."""
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


@pytest.mark.parametrize("L,n,D", [(2, 1, 2), (4, 3, 9), (6, 5, 33), (8, 8, 130), (10, 9, 400),
                                   (12, 12, 2000)])
def test_one_term_fit_is_the_state_in_right_gauge(td, L, n, D):
    A, q = synth.random_mps(L, n, n % 2, D, seed=11)
    ctx = td.Context("fp64")
    ctx.set_schedule(0, 1)
    psi = td.mps_import(ctx, A, q)
    out = td.mps_sum(ctx, [1.0], [psi], D, 0.0)
    nn = td.overlap(ctx, psi, psi).real
    assert abs(td.overlap(ctx, psi, out) - nn) <= 1e-12 * nn
    assert abs(td.overlap(ctx, out, out).real - nn) <= 1e-12 * nn
    for T in out.export()[0][1:]:
        M = T.reshape(T.shape[0], -1)
        assert np.abs(M @ M.conj().T - np.eye(len(M))).max() <= 1e-13
    ctx.close()
