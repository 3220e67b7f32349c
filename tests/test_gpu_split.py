"""The split of an FP64 tensor into three BF16 parts (integer arithmetic, with
the FP64 form at the ends of the range) through the split-BF16 Tucker operator
with identity matrices, whose products and sums are exact: a value of 24
significant bits comes back unchanged, any other within the parts' 2^-24."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu


def through(X):
    from paper_2310_07551_gb300 import ds
    n2, n1 = X.shape
    eyes = [torch.eye(n, dtype=torch.float64, device="cuda") for n in (n1, n2)]
    return ds.tucker(torch.from_numpy(X).cuda(), eyes, precision="bf16x6").cpu().numpy()


@pytest.mark.parametrize("exponent", [-40, 0, 1, 60, 100])
def test_24_bit_values_are_exact(exponent):
    rng = np.random.default_rng(1)
    m = rng.integers(2**23, 2**24, (24, 64)).astype(np.float64) * 2.0**-23
    # every part at its rounding ties: bits 8 and 16 set and nothing below
    m[0, :4] = 1 + 2.0**-8, 1 + 3 * 2.0**-8, 1 + 2.0**-16, 1 + 2.0**-7 + 2.0**-16
    m[0, 4:8] = 2 - 2.0**-23, 1.0, 1 + 2.0**-23, 2 - 2.0**-8
    # one nonzero entry per row and column: the identities' zero products stay zero
    X = m * rng.choice([-1.0, 1.0], m.shape) * 2.0**exponent
    assert np.array_equal(through(X), X)


def test_other_values_within_the_parts():
    rng = np.random.default_rng(2)
    X = rng.standard_normal((24, 64)) * 2.0 ** rng.integers(-30, 30, (24, 64)).astype(np.float64)
    assert np.all(np.abs(through(X) - X) <= 2.0**-23 * np.abs(X))


def test_ends_of_the_range():
    X = np.zeros((24, 64))
    X[0, 0], X[1, 1], X[2, 2] = 2.0**-70, -(2.0**-126), 2.0**120
    got = through(X)
    assert np.array_equal(got, X)
    X[3, 3] = np.nan
    assert np.isnan(through(X)[3, 3])
