"""FP64 contractions whose entries span many decades (csrc/mm64.cu): an output that is
small against the largest entries of its fibres is as accurate as an FP64 FMA chain
makes it, entry by entry, where its digits alone would lose it.

Bound per output y = sum_k x_k l_k, S = sum_k |x_k| |l_k|.  An FMA chain of n entries is
within n 2^-53 S, one rounding more for a term's weight.  The digit sum is one rounding
(2^-53 |y|) and, per entry and in units of the fibres' 2^(ex + el), 2^-59.2 for the
dropped digit products (7 pairs of at most 2^14 at 2^-76), at most 2^-58.6 for what the
last classes lose and 2^-62 for the operands' own: below n 2^-57.7; it is kept only where
S is at least 2^-8 of that unit, so within n 2^-49.7 S."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu

LD = np.longdouble


@pytest.fixture(scope="module")
def ds():
    from paper_2310_07551_gb300 import ds as _ds
    _ds.lib()
    return _ds


def mode(X, mu, M):
    ax = X.ndim - 1 - mu
    return np.moveaxis(np.tensordot(M, X, (1, ax)), 0, ax)


@pytest.mark.parametrize("dims", [(64, 8, 8, 8), (130, 70, 33), (300, 41)])
@pytest.mark.parametrize("span", [30, 290])
def test_identity_matrices_give_the_tensor_back(ds, dims, span):
    rng = np.random.default_rng(span + dims[0])
    X = rng.standard_normal(dims[::-1]) * 10.0 ** rng.uniform(-span, 0, dims[::-1])
    Xd = torch.from_numpy(X).cuda()
    eyes = [torch.eye(n, dtype=torch.float64, device="cuda") for n in dims]
    for transpose in (False, True):
        assert torch.equal(ds.tucker(Xd, eyes, transpose=transpose), Xd)
        assert torch.equal(ds.tucker_static(Xd, eyes, transpose=transpose), Xd)


def graded(rng, rows, n, kind):
    k, r = np.arange(n), np.arange(rows)[:, None]
    sign = rng.choice([-1.0, 1.0], (rows, n)) * rng.uniform(0.5, 1, (rows, n))
    if kind == "peak":          # each row around its own place
        return sign * np.exp(-((k - r * n / rows) / (0.03 * n + 1)) ** 2)
    if kind == "front":         # the same tail in every row
        return sign * np.exp(-np.maximum(k - n / 3, 0) * 60.0 / n)
    if kind == "random":        # any entry of any size
        return sign * 10.0 ** rng.uniform(-40, 0, (rows, n))
    if kind == "sparse":        # mostly zeros
        return sign * (rng.uniform(size=(rows, n)) < 0.05) * 10.0 ** rng.uniform(-20, 0, (rows, n))
    return sign                 # one size


@pytest.mark.parametrize("n,dims", [(64, (8, 8, 8)), (65, (9, 7, 10)), (129, (11, 11)), (257, (11, 11)), (520, (11, 11))])
@pytest.mark.parametrize("kx,kl", [("peak", "peak"), ("front", "peak"), ("random", "random"), ("sparse", "peak"),
                                   ("flat", "random"), ("peak", "flat"), ("sparse", "sparse")])
def test_products_of_graded_operands(ds, n, dims, kx, kl):
    rng = np.random.default_rng(n)
    rows = int(np.prod(dims))
    X, L = graded(rng, rows, n, kx), graded(rng, n, n, kl)
    T = torch.from_numpy(X.reshape(dims[::-1] + (n,))).cuda()
    eyes = [torch.eye(m, dtype=torch.float64, device="cuda") for m in dims]
    got = ds.tucker(T, [torch.from_numpy(L).cuda()] + eyes).cpu().numpy().reshape(rows, n)
    y = X.astype(LD) @ L.T.astype(LD)
    S = np.abs(X).astype(LD) @ np.abs(L.T).astype(LD)
    tol = 2.0**-53 * np.abs(y) + n * 2.0**-49.7 * S + LD(2.0) ** -1074
    assert np.all(np.abs(got - y) <= tol), float((np.abs(got - y) / tol).max())


def test_phi_matrices_far_from_the_diagonal(ds):
    """entry by entry against the oracle's phi-matrices of the same algorithm"""
    from oracle import oracle as O
    from paper_2310_07551_gb300 import inputs
    dims, tau = (96, 80), 2e-5
    As = [[dl * inputs.fd_neumann(n, 0.0, 1.0) for n in dims] for dl in (1.0, 10.0)]
    ps, ref = ds.PhiSet(dims, As, tau), O.phi_set_blocks(dims, O.phi_set(dims, As, tau))
    for c in range(2):
        for slot in range(5):
            for i in range(2):
                for mu in range(2):
                    got, want = ps.get(c, slot, i, mu), ref[c][slot][i][mu]
                    # products of entries of one sign: some 40 in a row, each within the bound above
                    assert np.all(np.abs(got - want) <= 40 * 96 * 2.0**-49.7 * np.abs(want) + 1e-290), (c, slot, i, mu)


def test_step_of_a_localised_state(ds):
    """one linear step, both terms of each sum in one contraction, tails down to 1e-60"""
    from paper_2310_07551_gb300 import inputs
    dims, tau = (96, 80), 2e-5
    As = [[dl * inputs.fd_neumann(n, 0.0, 1.0) for n in dims] for dl in (1.0, 10.0)]
    ps = ds.PhiSet(dims, As, tau)
    x, y = (np.linspace(-1, 1, n) for n in dims)
    U = np.stack([np.exp(-140 * (y[:, None] + 0.3 * c) ** 2 - 140 * x[None, :] ** 2) for c in range(2)])
    plan = ds.Plan(ps, "linear", (0.0, 0.0, 0.0), precision="f64")
    V = torch.from_numpy(U.copy()).cuda()
    plan.step(V)
    plan.sync(V, check_state=True)
    got = V.cpu().numpy()
    for c in range(2):
        u = U[c].astype(LD)
        F = sum(mode(u, mu, As[c][mu].astype(LD)) for mu in range(2))
        Fm = sum(mode(np.abs(u), mu, np.abs(As[c][mu]).astype(LD)) for mu in range(2))
        want, mag = u.copy(), np.abs(u)
        for i, eta in enumerate((-1.25, 9.0)):
            Ps = [ps.get(c, 3, i, mu).astype(LD) for mu in range(2)]
            want = want + tau * eta * mode(mode(F, 0, Ps[0]), 1, Ps[1])
            mag = mag + tau * abs(eta) * mode(mode(Fm, 0, np.abs(Ps[0])), 1, np.abs(Ps[1]))
        assert np.all(np.abs(got[c] - want) <= (96 + 2 * 80) * 2.0**-49.7 * mag), c


@pytest.mark.parametrize("kx,kl", [("peak", "peak"), ("random", "random"), ("sparse", "peak")])
def test_row_blocks_change_no_bit(ds, kx, kl):
    """the static entry point's smaller scratch cuts the tensor's rows into blocks, so
    that other numbers of outputs go to the FMA chains at a time"""
    rng = np.random.default_rng(7)
    dims = (520, 44, 43)
    X = graded(rng, 44 * 43, 520, kx).reshape(43, 44, 520)
    Ls = [torch.from_numpy(graded(rng, n, n, kl)).cuda() for n in dims]
    Xd = torch.from_numpy(X).cuda()
    assert torch.equal(ds.tucker_static(Xd, Ls), ds.tucker(Xd, Ls))
