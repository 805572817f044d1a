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
