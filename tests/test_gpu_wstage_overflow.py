"""The MPO stage on complex FP32 data where a channel has overflowed: outputs
that do not depend on it are those of the FP64 operator.

One element of one site tensor is out of FP32 range (1e60) in the split-TF32
operator, and 1e200 in the FP64 one, so that its square overflows there too.
Entries of the FP64 result that stayed finite and small do not contain the
square, nor a single factor of the element.  Tolerance: split TF32 keeps products
to 2^-21 and sums of at most 1000 of them to 1e-5 of the largest entry in the
worst case; 1e-4 with a margin of 10."""
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


def _apply(td, prec, h, n, T, A, q):
    L = len(A)
    ctx = td.Context(prec)
    mpo = td.build_mpo(ctx, h, np.zeros((L,) * 4), n_elec=n)
    psi, x, y = (td.mps_import(ctx, t, q) for t in (T, A, A))
    out = []
    for site in range(L):
        op = td.local_hamiltonian(ctx, mpo, psi, site)
        op.apply(x, y)
        out.append(y.export()[0][site])
        op.free()
    ctx.close()
    return out


@pytest.mark.parametrize("seed", range(6))
def test_outputs_that_do_not_depend_on_an_overflow(td, seed):
    L, n, D = 7, 3, 8
    rng = np.random.default_rng(seed)
    h = rng.standard_normal((L, L)) * (rng.random((L, L)) < 0.35)
    A, q = synth.random_mps(L, n, n % 2, D, seed=seed)
    for i in range(L - 1):
        at = rng.permutation(np.argwhere(A[i] != 0))[0]
        def big(v):
            T = [a.copy() for a in A]
            T[i][tuple(at)] *= v
            return T
        ref = _apply(td, "fp64", h + h.T, n, big(1e200), A, q)
        got = _apply(td, "tf32x3", h + h.T, n, big(1e60), A, q)
        for r, g in zip(ref, got):
            ok = np.isfinite(r) & (np.abs(r) < 1e20)
            if ok.any():
                assert np.abs(r - g)[ok].max() <= 1e-4 * np.abs(r[ok]).max()
