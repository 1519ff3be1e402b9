"""The FP64 block GEMM at the edges of its tiles: overlaps of three-site MPS
whose two inner bonds each hold one charge sector, so that the middle site's
products have the shapes (d1 x k1)(k1 x d2) and (e2 x d1)(d1 x d2) exactly.

Tolerance: with u = 2^-53, a sum of K products in any order is within K u of
the sum of their absolute values (first order), and the overlap chains two
such sums per site: fewer than 6 max(K) <= 1000 roundings, i.e. 1.2e-13 of the
overlap of the absolute values.  The sliced operands add less than 2^-60 of
the largest row and column elements, far below that."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def td():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1902_08489_gb300 as mod
    mod.lib()
    return mod


def _mps(rng, d1, d2, spread):
    """Charges (0,0) - (1,1) - (2,0) - (2,0): one sector per bond."""
    q = [(0, 0), (1, 1), (2, 0), (2, 0)]
    dims = [1, d1, d2, 1]
    labels = [np.array([q[k]] * dims[k], dtype=np.int64) for k in range(4)]
    tensors = []
    for i, s in enumerate((1, 2, 0)):
        a, b = dims[i], dims[i + 1]
        A = np.zeros((a, 4, b), dtype=np.complex128)
        v = rng.standard_normal((a, b)) + 1j * rng.standard_normal((a, b))
        A[:, s] = v * 2.0 ** rng.integers(-spread, spread + 1, size=(a, 1))
        tensors.append(A)
    return tensors, labels


def _overlap(B, A):
    E = np.ones((1, 1), dtype=np.complex128)
    for x, y in zip(B, A):
        E = np.einsum("xsp,xy,ysq->pq", x.conj(), E, y, optimize=True)
    return E[0, 0]


@pytest.mark.parametrize("spread", [0, 30])
@pytest.mark.parametrize("d1,k1,d2,e2", [
    (1, 1, 1, 1), (7, 3, 5, 2), (15, 31, 23, 17), (16, 32, 24, 16), (17, 33, 25, 3),
    (33, 8, 4, 64), (64, 9, 96, 65), (65, 40, 97, 48), (3, 130, 50, 129), (128, 100, 193, 161)])
def test_overlap_at_tile_edges(td, d1, k1, d2, e2, spread):
    rng = np.random.default_rng([d1, k1, d2, e2, spread])
    B, qb = _mps(rng, d1, e2, spread)
    A, qa = _mps(rng, k1, d2, spread)
    ctx = td.Context("fp64")
    got = td.overlap(ctx, td.mps_import(ctx, B, qb), td.mps_import(ctx, A, qa))
    ref = _overlap(B, A)
    scale = _overlap([np.abs(x) for x in B], [np.abs(x) for x in A]).real
    assert abs(got - ref) <= 1.2e-13 * scale
    ctx.close()
