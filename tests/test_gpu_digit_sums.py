"""FP64 contractions of integers by digits (csrc/mm64.cu) whose sums cancel to small
numbers of either sign: every product and sum is an integer below 2^53 and the result
is exact, as an FP64 FMA chain has it."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("bits", [8, 16, 21])
@pytest.mark.parametrize("n,dims", [(64, (8, 8, 8)), (130, (11, 11)), (300, (11, 11))])
def test_cancelling_integer_sums_are_exact(bits, n, dims):
    from paper_2310_07551_gb300 import ds
    rng = np.random.default_rng(bits + n)
    rows, h = int(np.prod(dims)), n // 2
    x, l = rng.integers(-2**bits, 2**bits + 1, (rows, h)), rng.integers(-2**bits, 2**bits + 1, (n, h))
    # the second half of each sum takes the first away, but for small differences
    X = np.concatenate([x, x + rng.integers(-1, 2, x.shape)], 1)
    L = np.concatenate([l, -l + (rng.integers(0, 40, l.shape) == 0)], 1)
    L[0], L[1] = np.r_[l[0], -l[0]], 0
    X[:, h:][:16] = x[:16]
    T = torch.from_numpy(X.astype(np.float64).reshape(dims[::-1] + (n,))).cuda()
    Ls = [torch.from_numpy(M.astype(np.float64)).cuda() for M in (L, *(np.eye(m) for m in dims))]
    want = X @ L.T
    assert (want < 0).any() and (want > 0).any() and (want == 0).any() and np.abs(want).max() < 2**53
    assert np.array_equal(ds.tucker(T, Ls).cpu().numpy().reshape(rows, n), want.astype(np.float64))
