"""FP64 mode products on the tensor cores (exact products of 8-bit digits,
csrc/mm64.cu) against long double, at the edges of their tiles: contractions
around the 32-entry slab and the 256-entry drain, row counts around the
128-row tile, column counts around the tile widths, both orientations.

The other modes of the tested Tucker operators are identities of at most 11
rows, which run as FP64 FMA chains and are exact.

Bound per output y_ri = sum_k x_rk l_ik: one rounding to FP64 (2^-53 |y|) plus
what the digits drop.  Each operand entry is rounded to a multiple of 2^-62 of
its fibre's power-of-two ceiling (at most twice the fibre's largest entry M), an
error of at most 2^-62 M; the dropped digit products and the rounding of the
last kept classes weigh less than 2^-57 M_x M_l per entry.  Together below
2^-53 |y| + n 2^-56 M_x M_l."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ds():
    from paper_2310_07551_gb300 import ds as _ds
    _ds.lib()
    return _ds


def first_mode(ds, X, L, dims, transpose=False):
    """X (rows, n) as a tensor of sizes (n, *dims), rows = prod dims; identities after mode 1"""
    T = torch.from_numpy(X.reshape(tuple(reversed(dims)) + (X.shape[1],))).cuda()
    eyes = [torch.eye(m, dtype=torch.float64, device="cuda") for m in dims]
    got = ds.tucker(T, [torch.from_numpy(L).cuda()] + eyes, transpose=transpose)
    return got.cpu().numpy().reshape(X.shape)


def check(got, X, L):
    y = X.astype(np.longdouble) @ L.T.astype(np.longdouble)
    n = X.shape[1]
    tol = 2.0**-53 * np.abs(y) + n * 2.0**-56 * np.outer(np.abs(X).max(1), np.abs(L).max(1))
    assert np.all(np.abs(got - y) <= tol), float(np.nanmax(np.abs(got - y) / tol))


def identities(ref):
    """the three 8 x 8 identity modes on FP64 results: infinities spread as NaN (0 x inf)"""
    ref = ref.reshape(8, 8, 8, -1)
    with np.errstate(all="ignore"):
        for ax in range(3):
            ref = np.moveaxis((np.eye(8)[:, :, None, None, None] * np.moveaxis(ref, ax, 0)[None]).sum(1), 0, ax)
    return ref.reshape(512, -1)


@pytest.mark.parametrize("n,dims", [(36, (11, 11, 11)), (63, (11, 10, 8)), (64, (8, 8, 8)), (65, (9, 7, 10)),
                                    (129, (11, 11)), (255, (8, 8, 2)), (256, (11, 6, 2)), (257, (11, 11)),
                                    (288, (8, 8, 2)), (520, (11, 11))])
@pytest.mark.parametrize("transpose", [False, True])
def test_first_mode_at_tile_edges(ds, n, dims, transpose):
    rng = np.random.default_rng(n)
    rows = int(np.prod(dims))
    # entries over six decades, every row of both operands at its own scale
    X, L = (rng.standard_normal((m, n)) * 10.0 ** rng.uniform(-3, 3, (m, n)) * 10.0 ** rng.integers(-40, 40, (m, 1))
            for m in (rows, n))
    check(first_mode(ds, X, L.T.copy() if transpose else L, dims, transpose), X, L)


@pytest.mark.parametrize("value", [2.0**-8, 0.737281918273, 1.0 - 2.0**-53])
def test_constant_operands_fill_the_accumulators(ds, value):
    """equal entries: every digit product of a class has the same sign"""
    X, L = np.full((512, 256), value), np.full((256, 256), value)
    check(first_mode(ds, X, L, (8, 8, 8)), X, L)


@pytest.mark.parametrize("dims", [(40, 96, 37), (130, 70, 33), (16, 300, 50)])
def test_strided_modes(ds, dims):
    """modes 2 and 3 (fibre index contiguous, slices crossing row tiles)"""
    rng = np.random.default_rng(sum(dims))
    X = rng.uniform(-1, 1, dims[::-1])
    Ls = [rng.uniform(-1, 1, (n, n)) for n in dims]
    got = ds.tucker(torch.from_numpy(X).cuda(), [torch.from_numpy(L).cuda() for L in Ls]).cpu().numpy()
    ref, mag = X.astype(np.longdouble), np.abs(X)
    for mu, L in enumerate(Ls):
        ax = 2 - mu
        ref = np.moveaxis(np.tensordot(L.astype(np.longdouble), ref, (1, ax)), 0, ax)
        mag = np.moveaxis(np.tensordot(np.abs(L), mag, (1, ax)), 0, ax)
    # one rounding per mode and the digits' loss, each of results no larger than mag
    assert np.all(np.abs(got - ref) <= 4 * 2.0**-53 * mag)


@pytest.mark.parametrize("scale", [2.0**1015, 2.0**-1020, 2.0**-1060])
def test_ends_of_the_exponent_range(ds, scale):
    """huge, nearly subnormal and subnormal rows; zero rows; overflow to inf"""
    rng = np.random.default_rng(3)
    X, L = rng.uniform(-1, 1, (512, 64)) * scale, rng.uniform(0.25, 1, (64, 64))
    X[2] = 0.0
    L[10] *= 2.0**20
    got = first_mode(ds, X, L, (8, 8, 8))
    y = X.astype(np.longdouble) @ L.T.astype(np.longdouble)
    with np.errstate(over="ignore"):
        ref = identities(y.astype(np.float64))
    fin, inf = np.isfinite(ref), np.isinf(ref)
    assert np.array_equal(np.isnan(got), np.isnan(ref)) and np.array_equal(np.isinf(got), inf)
    assert np.array_equal(got[inf] > 0, ref[inf] > 0)
    tol = 2.0**-53 * np.abs(y) + 64 * 2.0**-56 * np.outer(np.abs(X).max(1), np.abs(L).max(1)) + 2.0**-1074
    assert np.all(np.abs(np.where(fin, got, 0) - np.where(fin, y, 0)) <= np.where(fin, tol, 0))


@pytest.mark.parametrize("special", [[np.nan], [np.inf], [-np.inf], [np.inf, -np.inf]])
@pytest.mark.parametrize("where", ["tensor", "matrix"])
def test_non_finite_entries(ds, special, where):
    """NaN and infinities come out as an FP64 FMA chain has them"""
    rng = np.random.default_rng(4)
    X, L = rng.uniform(-1, 1, (512, 64)), rng.uniform(0.25, 1, (64, 64))
    L[9, 7] = X[:64, 7] = 0.0    # 0 x inf
    (X if where == "tensor" else L)[100 % 64, 7:7 + len(special)] = special
    got = first_mode(ds, X, L, (8, 8, 8))
    with np.errstate(all="ignore"):
        ref = identities((X[:, None, :] * L[None, :, :]).sum(2))
    assert np.array_equal(np.isnan(got), np.isnan(ref))
    inf = np.isinf(ref)
    assert np.array_equal(np.isinf(got), inf) and np.array_equal(got[inf] > 0, ref[inf] > 0)
    fin = np.isfinite(ref)
    assert np.allclose(got[fin], ref[fin], rtol=0, atol=64 * 2.0**-52)


@pytest.mark.parametrize("n,mode", [(470, 0), (513, 0), (470, 2), (513, 2)])
def test_long_tensors(ds, n, mode):
    """tensors whose digit images have eight entries per thread (shorter ones have
    four), contracted along the first mode and along a strided one; a sample of rows"""
    rng = np.random.default_rng(n + mode)
    X, L = (rng.standard_normal((m, n)) * 10.0 ** rng.uniform(-3, 3, (m, n)) * 10.0 ** rng.integers(-40, 40, (m, 1))
            for m in (11**3, n))
    T = np.moveaxis(X.reshape(11, 11, 11, n), 3, 3 - mode)
    Ls = [torch.from_numpy(L if mu == mode else np.eye(11)).cuda() for mu in range(4)]
    got = ds.tucker(torch.from_numpy(T.copy()).cuda(), Ls).cpu().numpy()
    got = np.moveaxis(got, 3 - mode, 3).reshape(11**3, n)
    r = np.r_[0:16, 120:130, 1000:1010, 1315:1331]
    check(got[r], X[r], L)
