"""The FP64 stencil (csrc/f64.cu) on tridiagonal matrices of every kind of row, against
long double: diffusion (outer bands as heavy as the diagonal), advection (central
differences, no diagonal to speak of), reaction (a diagonal alone), mixed directions.

Bound: a row's terms are rounded once each and added in a chain, 2 d + 1 roundings, and
a difference form adds as much again of |lo| |u| + |up| |u|, at most twice |di| |u|:
3 (2 d + 2) 2^-53 of the product of absolute values."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu


def tridiagonal(rng, n, kind):
    A = np.zeros((n, n))
    i = np.arange(n)
    if kind == "diffusion":
        A[i, i], A[i[1:], i[1:] - 1], A[i[:-1], i[:-1] + 1] = -2.0, 1.0, 1.0
        return A * rng.uniform(50, 100)
    if kind == "advection":
        w = rng.uniform(1e5, 1e6, n)
        A[i[1:], i[1:] - 1], A[i[:-1], i[:-1] + 1] = -w[1:], w[:-1]
        A[i, i] = rng.uniform(-1, 1, n) * 1e-3
        return A
    if kind == "reaction":
        A[i, i] = rng.standard_normal(n)
        return A
    A[i, i], A[i[1:], i[1:] - 1], A[i[:-1], i[:-1] + 1] = rng.standard_normal(n), rng.standard_normal(n - 1), rng.standard_normal(n - 1)
    return A


@pytest.mark.parametrize("kinds", [("diffusion", "diffusion"), ("advection", "advection"), ("diffusion", "advection"),
                                   ("random", "reaction"), ("advection", "diffusion", "random")])
def test_kronsum_of_spiky_states(kinds):
    from paper_2310_07551_gb300 import ds
    rng = np.random.default_rng(len("".join(kinds)))
    dims = (40, 36, 9)[:len(kinds)]
    As = [[tridiagonal(rng, n, k) for n, k in zip(dims, kinds)] for _ in range(2)]
    ps = ds.PhiSet(dims, As, 1e-9)
    # large values between small ones, in every direction
    where = sum(np.indices(dims[::-1])) % 2
    X = rng.standard_normal(dims[::-1]) * np.where(where, 1.0, 1e-9)
    for c in range(2):
        got = ps.kronsum(c, torch.from_numpy(X).cuda()).cpu().numpy()
        want, mag = 0.0, 0.0
        for mu, A in enumerate(As[c]):
            ax = len(dims) - 1 - mu
            apply = lambda M, T: np.moveaxis(np.tensordot(M.astype(np.longdouble), T, (1, ax)), 0, ax)
            want, mag = want + apply(A, X), mag + apply(np.abs(A), np.abs(X))
        assert np.all(np.abs(got - want) <= 3 * (2 * len(dims) + 2) * 2.0**-53 * mag), c


def test_constant_states_stay_exactly_constant():
    from paper_2310_07551_gb300 import ds, inputs
    dims = (41, 37)
    ps = ds.PhiSet(dims, [[dl * inputs.fd_neumann(n, 0.0, 1.0) for n in dims] for dl in (1.0, 10.0)], 1e-4)
    X = torch.full(dims[::-1], 0.737281918273, dtype=torch.float64, device="cuda")
    assert not ps.kronsum(0, X).any() and not ps.kronsum(1, X).any()
