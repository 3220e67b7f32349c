"""Plans where device memory is short: what the library's memory pool keeps between
calls is given back before an allocation is refused, and FP64 and FP32 plans run with
less workspace (one sum at a time, term by term, products on the FP64 pipe) to the
same results.  The rest of the device's memory is held by a torch allocation."""
import contextlib

import numpy as np
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu

MIB = 1 << 20
P = (0.1, 2.0, -0.1)


@contextlib.contextmanager
def only(mib, pool=False):
    """Leaves about that much device memory free; pool: beside what the library's pool
    keeps, else that is driven out too."""
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    block = lambda m: torch.empty(m * MIB, dtype=torch.uint8, device="cuda")
    held = [block(torch.cuda.mem_get_info()[0] // MIB - mib)]
    if not pool:
        with contextlib.suppress(torch.cuda.OutOfMemoryError):
            while True:
                held.append(block(16))
        del held[1:1 + mib // 16]
        torch.cuda.empty_cache()
    try:
        yield
    finally:
        torch.cuda.synchronize()
        del held
        torch.cuda.empty_cache()


def problem(dims):
    from paper_2310_07551_gb300 import ds, inputs
    As = [[dl * inputs.fd_neumann(n, -1.0, 1.0) for n in dims] for dl in (1.0, 42.1887)]
    return ds.PhiSet(dims, As, 1e-3), torch.from_numpy(inputs.initial_state("fhn", dims, seed=3)).cuda()


def fill_pool():
    """a large FP64 Tucker operator: some 500 MiB stay in the pool"""
    from paper_2310_07551_gb300 import ds
    X = torch.rand(64, 512, 512, dtype=torch.float64, device="cuda")
    ds.tucker(X, [torch.eye(n, dtype=torch.float64, device="cuda") for n in (512, 512, 64)])
    torch.cuda.synchronize()


@pytest.mark.parametrize("precision", ["bf16x6", "f16x13"])
def test_the_pool_gives_way_to_plans(precision):
    from paper_2310_07551_gb300 import ds
    ps, U = problem((128, 128, 64))
    fill_pool()
    with only(160, pool=True):   # the plan needs some 300 to 400 MiB
        plan = ds.Plan(ps, "fhn", P, precision=precision)
        plan.integrate(U, 1)
        plan.sync(U, check_state=True)
        plan.close()


@pytest.mark.parametrize("precision", ["f64", "f32"])
def test_plans_in_little_memory_give_the_same(precision):
    """10 tensors of N points where an ordinary plan takes 48"""
    from paper_2310_07551_gb300 import ds
    ps, U0 = problem((128, 128, 64))
    N = U0.numel() // 2
    ordinary = ds.Plan(ps, "fhn", P, precision=precision)
    ref = ordinary.integrate(U0.clone(), 2).cpu().numpy()
    ordinary.close()
    U = U0.clone()
    size = 8 if precision == "f64" else 4
    with only(11 * N * size // MIB + 24):
        plan = ds.Plan(ps, "fhn", P, precision=precision)
        got = plan.integrate(U, 2).cpu().numpy()
        plan.sync(U, check_state=True)
        plan.close()
    # as many roundings, in another order: some 60 modes of 128 entries a step
    tol = 2 * 60 * 128 * (2.0**-53 if precision == "f64" else 2.0**-24)
    assert np.abs(got - ref).max() <= tol * np.abs(ref).max()


@pytest.mark.parametrize("dims", [(128, 128, 64), (512, 1024)])
def test_adjoint_in_little_memory_gives_the_same(dims):
    """24 tensors of N points with the gradient in the diffusion scalings, which
    ordinarily takes its own workspace"""
    from paper_2310_07551_gb300 import ds, inputs
    ps, U = problem(dims)
    N = U.numel() // 2
    plan = ds.Plan(ps, "fhn", P, precision="f64")
    lam = torch.from_numpy(inputs.initial_state("fhn", dims, seed=4)).cuda()
    zeros = lambda n: torch.zeros(n, dtype=torch.float64, device="cuda")
    dp, dscale = zeros(3), zeros(2)
    ref = plan.step_backward(U, lam, dp, dscale).clone()
    plan.close()
    tight, dp2, dscale2 = ds.Plan(ps, "fhn", P, precision="f64"), zeros(3), zeros(2)
    with only((24 if len(dims) == 3 else 23) * N * 8 // MIB + 32):
        got = tight.step_backward(U, lam, dp2, dscale2)
        torch.cuda.synchronize()
    tight.close()
    # some 100 modes of up to 1024 entries; the scalings' gradients are sums of terms of
    # both signs over the grid
    assert (got - ref).abs().max() <= 1e-11 * ref.abs().max()
    assert torch.allclose(dp2, dp, rtol=1e-9, atol=0) and torch.allclose(dscale2, dscale, rtol=1e-8, atol=0)
