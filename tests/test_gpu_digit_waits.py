"""FP64 calls whose digit products give up a wait (csrc/mm64.cu): the test hook
DS_WAIT_LIMIT_CYCLES lets every wait for a tile's MMAs run out, and the outputs
behind it are FP64 FMA chains.  No call fails, no result is NaN, and calls made
afterwards are not affected.  No fault and no hang: the waits that give up are
ordinary bounded waits, and copies and MMAs in flight are waited for in full.

Bounds: an FMA chain of n entries is within n 2^-53 of the product of absolute
values; a Tucker operator's modes add up."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu

LIMIT = "200"   # cycles; one slab's MMAs take over a thousand
P = (0.1, 2.0, -0.1)


@pytest.mark.parametrize("dims", [(64, 8, 8, 8), (130, 70, 33)])
@pytest.mark.parametrize("static", [False, True])
def test_tucker_is_right_and_the_next_calls_are_clean(monkeypatch, dims, static):
    from paper_2310_07551_gb300 import ds
    rng = np.random.default_rng(sum(dims))
    X = rng.uniform(-1, 1, dims[::-1])
    Ls = [rng.uniform(-1, 1, (n, n)) for n in dims]
    Xd, Ld = torch.from_numpy(X).cuda(), [torch.from_numpy(L).cuda() for L in Ls]
    tucker = ds.tucker_static if static else ds.tucker
    before = tucker(Xd, Ld)
    monkeypatch.setenv("DS_WAIT_LIMIT_CYCLES", LIMIT)
    short = tucker(Xd, Ld)
    torch.cuda.synchronize()
    monkeypatch.delenv("DS_WAIT_LIMIT_CYCLES")
    ref, mag = X.astype(np.longdouble), np.abs(X)
    for mu, L in enumerate(Ls):
        ax = len(dims) - 1 - mu
        ref = np.moveaxis(np.tensordot(L.astype(np.longdouble), ref, (1, ax)), 0, ax)
        mag = np.moveaxis(np.tensordot(np.abs(L), mag, (1, ax)), 0, ax)
    assert np.all(np.abs(short.cpu().numpy() - ref) <= sum(dims) * 2.0**-53 * mag)
    assert not torch.equal(short, before)          # the waits did give up
    assert torch.equal(tucker(Xd, Ld), before)


def test_phi_setup_and_plan(monkeypatch):
    from paper_2310_07551_gb300 import ds, inputs
    dims = (72, 40, 24)
    Ds = [inputs.fd_neumann(n, -1.0, 1.0) for n in dims]
    As = [[dl * D for D in Ds] for dl in (1.0, 42.1887)]
    U0 = torch.from_numpy(inputs.initial_state("fhn", dims, seed=4)).cuda()

    def run():
        ps = ds.PhiSet(dims, As, 1e-3)
        plan = ds.Plan(ps, "fhn", P, "f64")
        U = U0.clone()
        plan.integrate(U, 2)
        plan.sync(U, check_state=True)
        return ps.get(1, 4, 0, 0), U.cpu().numpy()

    phi, ref = run()
    monkeypatch.setenv("DS_WAIT_LIMIT_CYCLES", LIMIT)
    phi_short, got = run()
    monkeypatch.delenv("DS_WAIT_LIMIT_CYCLES")
    # some 40 products in a row, each within 72 2^-53 of values below one
    assert np.abs(phi_short - phi).max() <= 40 * 72 * 2.0**-53
    assert np.abs(got - ref).max() <= 1e-12 * np.abs(ref).max()
    again = run()
    assert np.array_equal(again[0], phi) and np.array_equal(again[1], ref)
