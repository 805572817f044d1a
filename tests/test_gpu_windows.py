"""The numeric pass's ways to hold a column's sums, at the sizes where they can
go wrong, against each other (the sums are exact, so every way gives the same
bits) and against the FP64 oracle."""
import pytest

from paper_2002_10083_gb300 import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_2002_10083_gb300 import mcl
    c = mcl.Context(0)
    yield c
    c.close()


def _dev(A):
    from paper_2002_10083_gb300 import mcl
    return mcl.DeviceCSC.from_host(A)


@pytest.mark.parametrize("k", [-50, -20, 30, 50])
def test_scaled_input_gives_the_same_iteration(ctx, k):
    """A scaled by 2^k (k = -50: fixed-point scales beyond the integer
    conversion's range; 50: large sums) scales every product exactly, so with
    theta = 0 and r = 1 the renormalised iteration keeps its bits."""
    from paper_2002_10083_gb300 import mcl
    A = synth.random_sparse(1200, 0.02, seed=5, w="lognormal").with_val32()
    prm = mcl.Params(threshold=0.0, select_k=60, recover_pct=0.9, inflation=1.0)
    ref, ch_ref = ctx.expand(_dev(A), prm)
    out, ch = ctx.expand(_dev(synth.CSC(A.n, A.colptr, A.rowidx, A.val * 2.0 ** k)), prm)
    assert torch.equal(out.colptr, ref.colptr) and torch.equal(out.rowidx, ref.rowidx)
    assert torch.equal(out.val.view(torch.int32), ref.val.view(torch.int32)) and ch == ch_ref


def _random(n, d, seed, zeros=False):
    """About d entries per column at random rows; with zeros, a third of the values are 0 or
    so small that their products are truncated to 0 (they still are entries of A A)."""
    g = torch.Generator().manual_seed(seed)
    key = torch.unique(torch.randint(n * n, (n * d,), generator=g))
    col, row = key // n, key % n
    val = torch.exp(torch.randn(key.numel(), generator=g))
    if zeros:
        u = torch.rand(key.numel(), generator=g)
        val = torch.where(u < 0.2, torch.zeros(()), torch.where(u < 0.35, torch.tensor(1e-30), val))
    colptr = torch.zeros(n + 1, dtype=torch.int64)
    colptr[1:] = torch.cumsum(torch.bincount(col, minlength=n), 0)
    from paper_2002_10083_gb300 import mcl
    return mcl.DeviceCSC(n, colptr.cuda(), row.int().cuda(), val.cuda())


# rows of a direct window: 10,240; one window, its edges, several; products per source and
# window on both sides of the bucket rule; a candidate buffer smaller and larger than a column
@pytest.mark.parametrize("n,d,K,theta,zeros,budget", [
    (2049, 40, 50, 1e-3, False, 32 << 30), (10240, 60, 300, 1e-4, False, 32 << 30),
    (10241, 60, 1100, 1e-4, True, 32 << 30), (20481, 80, 4096, 0.0, True, 32 << 30),
    (31000, 100, 1100, 1e-4, False, 0), (4500, 700, 1100, 1e-5, True, 32 << 30),
    (12000, 500, 64, 0.0, False, 32 << 30)])
def test_direct_windows_equal_hashed_ones(ctx, n, d, K, theta, zeros, budget):
    from paper_2002_10083_gb300 import mcl
    A = _random(n, d, seed=n + d, zeros=zeros)
    prm = mcl.Params(threshold=theta, select_k=K, recover_pct=0.9, inflation=2.0)
    try:
        ctx.set_option(mcl.OPT_BUCKET_BUDGET, budget)
        out, ch = ctx.expand(A, prm)
        nnz_b = ctx.stats()["nnz_b"]
        ctx.set_option(mcl.OPT_CONF_MASK, 1)
        ref, ch_ref = ctx.expand(A, prm)
    finally:
        ctx.set_option(mcl.OPT_CONF_MASK, 3)
        ctx.set_option(mcl.OPT_BUCKET_BUDGET, 32 << 30)
    assert nnz_b == ctx.stats()["nnz_b"] and ch == ch_ref
    assert torch.equal(out.colptr, ref.colptr) and torch.equal(out.rowidx, ref.rowidx)
    assert torch.equal(out.val.view(torch.int32), ref.val.view(torch.int32))
