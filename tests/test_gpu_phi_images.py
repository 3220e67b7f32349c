"""Matrices stored as images of their shared-memory tiles (csrc/tc.cu): sizes around
the 32-entry K chunk, the 128-row block and the 256-row padding, both tile widths,
along the first mode (rows of the matrix are the tile's rows) and a strided one.

Bound per output, mag the Tucker operator of the absolute values: each mode drops
products below 2^-24 and rounds its operands and its result to 2^-24 (at most four
such terms), and its FP32 accumulation truncates after each of 6 ceil(n / 16)
instructions by at most 2^-23 of a partial sum no larger than mag."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dims", [(8, 33), (136, 31), (128, 129), (264, 127), (256, 257), (40, 8, 64), (24, 160, 33)])
@pytest.mark.parametrize("precision", ["bf16x6", "bf16x6c", "f16x10"])
@pytest.mark.parametrize("transpose", [False, True])
def test_tucker_at_image_edges(dims, precision, transpose):
    from paper_2310_07551_gb300 import ds
    rng = np.random.default_rng(sum(dims))
    X = rng.uniform(-1, 1, dims[::-1])
    Ls = [rng.uniform(-1, 1, (n, n)) for n in dims]
    got = ds.tucker(torch.from_numpy(X).cuda(), [torch.from_numpy(L).cuda() for L in Ls], transpose=transpose,
                    precision=precision).cpu().numpy()
    ref, mag, tol = X, np.abs(X), 0.0
    for mu, L in enumerate(Ls):
        ax = len(dims) - 1 - mu
        M = L.T if transpose else L
        ref = np.moveaxis(np.tensordot(M, ref, (1, ax)), 0, ax)
        mag = np.moveaxis(np.tensordot(np.abs(M), mag, (1, ax)), 0, ax)
        tol += (6 * -(-dims[mu] // 16) + 4) * 2.0**-23
    assert np.all(np.abs(got - ref) <= tol * mag), float((np.abs(got - ref) / mag).max() / tol)
