"""FP32 mode products on the CUDA cores at the edges of their tiles: rows padded
to eight, blocks of 128 rows and 64 fibres, contractions around the 16-entry
chunk, fibres and rows in aligned groups of four and not, both orientations,
launches of few blocks (4 x 8 outputs per thread) and of many (8 x 8).

Bound: a mode product rounds its two FP32 operands and n FMAs, each by at most
2^-24, so each mode adds (n + 2) 2^-24 of the product of absolute values, and
the modes' sum 2^-24 more to second order."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dims", [(2, 3, 5), (7, 9, 8), (16, 15, 17), (100, 12, 20), (128, 33, 4), (129, 64, 6),
                                  (250, 31, 3), (36, 100, 200)])
@pytest.mark.parametrize("transpose", [False, True])
def test_tucker_f32_at_tile_edges(dims, transpose):
    from paper_2310_07551_gb300 import ds
    rng = np.random.default_rng(sum(dims))
    X = rng.standard_normal(dims[::-1])
    Ls = [rng.standard_normal((n, n)) for n in dims]
    got = ds.tucker(torch.from_numpy(X).cuda(), [torch.from_numpy(L).cuda() for L in Ls], transpose=transpose,
                    precision="f32").cpu().numpy()
    ref, mag = X, np.abs(X)
    for mu, L in enumerate(Ls):
        M = L.T if transpose else L
        ref = np.moveaxis(np.tensordot(M, ref, (1, 2 - mu)), 0, 2 - mu)
        mag = np.moveaxis(np.tensordot(np.abs(M), mag, (1, 2 - mu)), 0, 2 - mu)
    assert np.all(np.abs(got - ref) <= 2.0**-24 * sum(n + 3 for n in dims) * mag)
