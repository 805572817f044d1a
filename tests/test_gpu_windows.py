"""The numeric pass's ways to hold a column's sums, at the sizes where they can
go wrong, against each other (the sums are exact, so every way gives the same
bits) and against the FP64 oracle."""
import numpy as np
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


# several passes of sums per window, 64-bit global atomics (more than eight passes: 80k entries),
# the edges of the bitmaps, several bitmap windows; merges of 2 to 4 and a last merge of leftovers
@pytest.mark.parametrize("n,d,ns", [(12000, 130, 4), (32768, 300, 2), (32769, 20, 2), (45000, 250, 2), (100000, 400, 2), (140000, 20, 3), (600000, 5, 2), (33, 5, 7)])
def test_split_shapes_equal_one_pass(ctx, n, d, ns):
    from paper_2002_10083_gb300 import mcl
    A = _random(n, d, seed=n, zeros=n < 20000)
    prm = mcl.Params(threshold=1e-4, select_k=200, recover_pct=0.9, inflation=2.0)
    ref, ch_ref = ctx.expand(A, prm)
    out, ch, _ = ctx.expand_split(A, prm, ns)
    assert ch == ch_ref and torch.equal(out.colptr, ref.colptr) and torch.equal(out.rowidx, ref.rowidx)
    assert torch.equal(out.val.view(torch.int32), ref.val.view(torch.int32))


# both CTA sizes, more sources than one batch lists, several bitmap windows
@pytest.mark.parametrize("n,d", [(1, 1), (100, 7), (4500, 700), (17000, 20), (30000, 60), (600000, 5)])
def test_symbolic_shapes(ctx, n, d):
    import scipy.sparse as sp
    A = _random(n, d, seed=3 * n + d)
    P = sp.csc_matrix((torch.ones(A.nnz).numpy(), A.rowidx.cpu().numpy(), A.colptr.cpu().numpy()), shape=(n, n))
    B = P @ P
    flops, nnz = ctx.symbolic(A)
    assert (nnz.cpu().numpy() == B.indptr[1:] - B.indptr[:-1]).all()
    assert (flops.cpu().numpy() == np.asarray(B.sum(axis=0)).ravel()).all()


@pytest.mark.parametrize("n", [1, 31, 33, 64, 65, 5000])
def test_mlp_sample_counts(ctx, n):
    """Forward: a sample's outputs do not depend on the samples beside it.  Backward: against
    FP64; sums of n FP32 gradients, each a few hundred roundings (2^-24) of terms near its size."""
    from paper_2002_10083_gb300 import estimator, mcl
    w_bits, norm, _, _ = estimator.load()
    w = torch.as_tensor(w_bits.astype("int16")).cuda()
    norm = torch.from_numpy(norm).cuda()
    g = torch.Generator(device="cuda").manual_seed(n)
    feats = (norm[:16] + norm[16:] * torch.randn(5000, 16, generator=g, device="cuda")).contiguous()
    t = torch.randn(n, 2, generator=g, device="cuda")
    y = ctx.mlp_forward(feats[:n].contiguous(), w, norm)
    assert torch.equal(y, ctx.mlp_forward(feats, w, norm)[:n])
    grad, loss = torch.zeros(mcl.MLP_NPARAM, device="cuda"), torch.zeros(1, dtype=torch.float64, device="cuda")
    ctx.mlp_backward(feats[:n].contiguous(), t, w, norm, 1.0 / n, grad, loss)
    p = w.view(torch.bfloat16).double().requires_grad_()
    z = (feats[:n].double() - norm[:16].double()) / norm[16:].double()
    h = torch.relu(z @ p[:1024].view(64, 16).t() + p[1024:1088])
    h = torch.relu(h @ p[1088:5184].view(64, 64).t() + p[5184:5248])
    total = (h @ p[5248:5376].view(2, 64).t() + p[5376:] - t.double()).square().sum()
    (total / n).backward()
    assert abs(float(loss) / float(total.detach()) - 1) < 1e-5
    assert float((grad.double() - p.grad).abs().max()) < 1e-4 * float(p.grad.abs().max())


# columns whose candidates are ranked by counting (up to 128 keys) and by radix selects, with the
# cut at the threshold, at K, at the mass and at nothing
@pytest.mark.parametrize("K,theta,p", [(1000, 1e-3, 0.9), (40, 0.0, 0.5), (40, 5e-3, 0.99), (1000, 0.05, 1.0),
                                       (127, 0.0, 0.0), (128, 1e-4, 0.95), (5, 1.0, 0.3)])
def test_few_candidates(ctx, K, theta, p):
    from tests.test_gpu_expand import _check, _prm
    A = synth.random_sparse(700, 0.016, seed=21, w="lognormal")
    _check(ctx, A, _prm(theta=theta, K=K, p=p))


def test_bunched_rows_are_sorted(ctx):
    """Kept rows in a few places of a wide span: more keys per bucket of the row sort than it
    orders, and the radix passes take over."""
    import scipy.sparse as sp
    from tests.test_gpu_expand import _check, _prm
    n, m = 60000, 900
    rng = np.random.default_rng(4)
    B = sp.random(m, m, 0.2, random_state=5, format="coo")
    row, col = np.concatenate([B.row, [n - 1] * m]), np.concatenate([B.col, np.arange(m)])
    M = sp.csc_matrix((rng.uniform(0.1, 1, len(row)), (row, col)), shape=(n, n)) + sp.identity(n, format="csc")
    M.sort_indices()
    A = synth.CSC(n, M.indptr.astype(np.int64), M.indices.astype(np.int32), M.data)
    _check(ctx, A, _prm(K=600, theta=1e-5), cols=np.arange(0, m, 7).astype(np.int32))


# every graph that one CTA plans, and the first that it does not
@pytest.mark.parametrize("n", [1, 1023, 1025, 16384, 16385])
def test_small_plan_sizes(ctx, n):
    from paper_2002_10083_gb300 import mcl
    A = _random(n, 12, seed=n)
    prm = mcl.Params(threshold=1e-4, select_k=30, recover_pct=0.9, inflation=2.0)
    out, ch = ctx.expand(A, prm)
    st = ctx.stats()
    try:
        ctx.set_option(mcl.OPT_PHASE_BUDGET, 1 << 34)  # the steps kernel by kernel
        ref, ch_ref = ctx.expand(A, prm)
    finally:
        ctx.set_option(mcl.OPT_PHASE_BUDGET, 0)
    assert ch == ch_ref and torch.equal(out.colptr, ref.colptr) and torch.equal(out.rowidx, ref.rowidx)
    assert torch.equal(out.val.view(torch.int32), ref.val.view(torch.int32))
    assert all(st[k] == ctx.stats()[k] for k in ("flops", "nnz_b", "nnz_out", "estimator_misses"))


@pytest.fixture(scope="module")
def sparse_spans(ctx):
    """Columns of about 27,000 products in spans of 160,000 rows: too sparse for a sum per row,
    17 windows or more in every table of the large configuration.  With the exact iteration."""
    from paper_2002_10083_gb300 import mcl
    A = _random(160_000, 140, seed=17)
    flops, _ = ctx.symbolic(A)
    assert int(flops.max()) * 4 < 0.95 * A.n
    prm = mcl.Params(threshold=1e-5, select_k=300, recover_pct=0.9, inflation=2.0)
    return A, prm, ctx.expand(A, prm), ctx.stats()["nnz_b"]


# estimates that are right, short, and so short that a window's redone quarter overflows too
@pytest.mark.parametrize("scale", [1000, 100, 10])
@pytest.mark.parametrize("table,plan", [(0, 0), (0, 300), (1, 0), (1, 3000), (2, 0), (2, 1024)])
def test_table_shapes_and_overflowing_windows(ctx, sparse_spans, table, plan, scale):
    from paper_2002_10083_gb300 import mcl
    A, prm, (ref, ch_ref), nnz_b = sparse_spans
    opts = {mcl.OPT_CONF_MASK: (2, 3), mcl.OPT_TABLE: (table, 0), mcl.OPT_PLAN: (plan, 0),
            mcl.OPT_EST_SCALE: (scale, 1000)}
    try:
        for o, (v, _) in opts.items():
            ctx.set_option(o, v)
        for _ in range(5):
            out, ch = ctx.expand(A, prm)
            st = ctx.stats()
            assert st["nnz_b"] == nnz_b and ch == ch_ref
            assert scale == 1000 or st["range_splits"] > A.n * (0.5 if scale == 100 else 1.5)
            assert torch.equal(out.colptr, ref.colptr) and torch.equal(out.rowidx, ref.rowidx)
            assert torch.equal(out.val.view(torch.int32), ref.val.view(torch.int32))
    finally:
        for o, (_, v) in opts.items():
            ctx.set_option(o, v)


# columns of many windows without product buckets: no bucket space, space for some columns only
# (8 MB: about 1,700 products each), the small configuration alone; estimates right and short
@pytest.mark.parametrize("budget,mask,scale", [(0, 3, 1000), (0, 3, 50), (8 << 20, 3, 1000), (8 << 20, 2, 30),
                                               (32 << 30, 1, 1000), (0, 1, 20)])
@pytest.mark.parametrize("n,d", [(300, 3), (9000, 2), (40000, 30), (60000, 41), (90000, 130)])
def test_walked_sources_equal_buckets(ctx, n, d, budget, mask, scale):
    from paper_2002_10083_gb300 import mcl
    A = _random(n, d, seed=n + 3 * d, zeros=d == 41)
    prm = mcl.Params(threshold=1e-4, select_k=150, recover_pct=0.9, inflation=2.0)
    ref, ch_ref = ctx.expand(A, prm)
    nnz_b = ctx.stats()["nnz_b"]
    opts = {mcl.OPT_BUCKET_BUDGET: (budget, 32 << 30), mcl.OPT_CONF_MASK: (mask, 3), mcl.OPT_EST_SCALE: (scale, 1000)}
    try:
        for o, (v, _) in opts.items():
            ctx.set_option(o, v)
        out, ch = ctx.expand(A, prm)
        assert ctx.stats()["nnz_b"] == nnz_b
    finally:
        for o, (_, v) in opts.items():
            ctx.set_option(o, v)
    assert ch == ch_ref and torch.equal(out.colptr, ref.colptr) and torch.equal(out.rowidx, ref.rowidx)
    assert torch.equal(out.val.view(torch.int32), ref.val.view(torch.int32))


# columns on both sides of the rule that reads a bit before it is set (16 products per row of the
# window, counted in units of 128), several windows of batches on both sides of it, and graphs on both sides of the small CTAs' line
@pytest.mark.parametrize("n,d", [(1500, 12), (1500, 150), (1500, 900), (16384, 30), (16385, 30), (17000, 700), (530000, 3)])
def test_symbolic_dense_columns(ctx, n, d):
    test_symbolic_shapes(ctx, n, d)


def _graph(n, col, row):
    from paper_2002_10083_gb300 import mcl
    key = torch.unique(col * n + row)
    col, row = key // n, key % n
    colptr = torch.zeros(n + 1, dtype=torch.int64)
    colptr[1:] = torch.cumsum(torch.bincount(col, minlength=n), 0)
    return mcl.DeviceCSC(n, colptr.cuda(), row.int().cuda(), torch.ones(key.numel(), device="cuda"))


# long paths in both directions and in random order, bands, trees, rows shared by all columns, empty
# columns; sizes on both sides of the rules that link every entry at once
@pytest.mark.parametrize("n", [1, 7, 12288, 12289, 70000, 1200000])
@pytest.mark.parametrize("kind", ["up", "down", "perm", "band", "tree", "pairs", "one row", "one column", "blocks"])
def test_components_of_long_and_shallow_graphs(ctx, n, kind):
    import scipy.sparse as sp
    from scipy.sparse.csgraph import connected_components
    v, g = torch.arange(n), torch.Generator().manual_seed(n)
    perm = torch.randperm(n, generator=g)
    col, row = {"up": (v, (v + 1) % n), "down": (v, (v - 1) % n), "perm": (perm, perm.roll(1)),
                "band": (v.repeat(5), torch.cat([(v + o).clamp(0, n - 1) for o in range(-2, 3)])),
                "tree": (v, (torch.rand(n, generator=g) * v).long()), "pairs": (v, (v ^ 1).clamp(max=n - 1)),
                "one row": (v[::3], v[::3] * 0 + n // 2), "one column": (v[::3] * 0 + n // 2, v[::3]),
                "blocks": (v.repeat(4), torch.cat([v // 97 * 97 + (v * m) % 97 for m in (0, 5, 11, 13)]).clamp(max=n - 1))}[kind]
    A = _graph(n, col, row)
    label = ctx.components(A).cpu().numpy()
    S = sp.csc_matrix((np.ones(A.nnz), A.rowidx.cpu().numpy(), A.colptr.cpu().numpy()), shape=(n, n))
    k, ref = connected_components(S, directed=False)
    first = np.full(k, n, np.int64)
    np.minimum.at(first, ref, np.arange(n))
    assert (label == first[ref]).all()


def _near_ties():
    """FP32 numbers (u, w) with u / (u + w) within 2^-45 of the middle of two FP32 numbers: for odd
    s < 2^24 and small odd d, u = (s t - d) / 2^25 with t = d / s mod 2^25, so u / s = (t - d / s) / 2^25."""
    rng = np.random.default_rng(11)
    out = []
    for s in rng.integers(1 << 22, 1 << 23, 4000) * 2 + 1:
        for d in (-3, -1, 1, 3):
            t = d * pow(int(s), -1, 1 << 25) % (1 << 25)
            if t >= 1 << 24 and t & 1:
                u = (int(s) * t - d) >> 25
                out.append((u, int(s) - u))
    return np.array(out, np.float64)


def test_normalised_values_are_fp64_quotients(ctx):
    """v / sum in FP64, rounded once to FP32, where that is hardest: near the middle of two FP32
    numbers (sums of whole numbers are exact in any order)."""
    from paper_2002_10083_gb300 import mcl
    uw = _near_ties()
    m = len(uw)
    assert m > 1000
    want = torch.from_numpy((uw / uw.sum(1, keepdims=True)).astype(np.float32).ravel())
    val = torch.from_numpy(uw.astype(np.float32).ravel()).cuda()
    M = mcl.DeviceCSC(m, torch.arange(m + 1).cuda() * 2, torch.tensor([0, 1]).int().repeat(m).cuda(), val.clone())
    ctx.inflate_normalize(M, 1.0)
    assert torch.equal(M.val.cpu().view(torch.int32), want.view(torch.int32))
    # columns 2 .. m + 1 hold the pairs; column m + 2 + i of A A is column 2 + i
    n = 2 * m + 2
    colptr = torch.cat([torch.arange(3), 2 + 2 * torch.arange(1, m + 1), 2 + 2 * m + torch.arange(1, m + 1)])
    row = torch.cat([torch.tensor([0, 1]), torch.tensor([0, 1]).repeat(m), 2 + torch.arange(m)])
    one = torch.ones(1, device="cuda")
    A = mcl.DeviceCSC(n, colptr.cuda(), row.int().cuda(), torch.cat([one.repeat(2), val, one.repeat(m)]))
    out, _ = ctx.expand(A, mcl.Params(threshold=0.0, select_k=8, recover_pct=0.9, inflation=1.0))
    assert int(out.colptr[n]) == 2 + 4 * m
    assert torch.equal(out.val[2 + 2 * m:].cpu().view(torch.int32), want.view(torch.int32))
    # results and sums at the ends of FP32's range
    for scale in (1e-37, 1e-32, 1e-20, 1e20, 1e30):
        v = torch.tensor([1.0, 3.0, 7e-7, 1e-12, 3e-25]) * scale
        M = mcl.DeviceCSC(5, torch.tensor([0, 5, 5, 5, 5, 5]).cuda(), torch.arange(5).int().cuda(), v.cuda())
        ctx.inflate_normalize(M, 1.0)
        d = v.double()
        assert torch.equal(M.val.cpu(), (d / d.sum()).float())


def test_bins_used_counts_the_mask(ctx):
    from paper_2002_10083_gb300 import mcl
    prm = mcl.Params(threshold=1e-4, select_k=50, recover_pct=0.9, inflation=2.0)
    try:
        for A in (_random(500, 5, seed=1), _random(9000, 60, seed=2)):
            for mask, bins in ((1, 1), (2, 1), (3, 2)):
                ctx.set_option(mcl.OPT_CONF_MASK, mask)
                ctx.expand(A, prm)
                assert ctx.stats()["bins_used"] == bins
    finally:
        ctx.set_option(mcl.OPT_CONF_MASK, 3)


# columns of no entry, of one, and of more side by side
@pytest.mark.parametrize("n", [40, 20000, 600000])
def test_symbolic_columns_of_one_entry(ctx, n):
    v, g = torch.arange(n), torch.Generator().manual_seed(n)
    A = _graph(n, torch.cat([v[v % 5 > 0], v[v % 3 > 0]]),
               torch.randint(n, (int((v % 5 > 0).sum() + (v % 3 > 0).sum()),), generator=g))
    import scipy.sparse as sp
    P = sp.csc_matrix((np.ones(A.nnz), A.rowidx.cpu().numpy(), A.colptr.cpu().numpy()), shape=(n, n))
    B = P @ P
    flops, nnz = ctx.symbolic(A)
    assert (nnz.cpu().numpy() == np.diff(B.indptr)).all()
    assert (flops.cpu().numpy() == np.asarray(B.sum(axis=0)).ravel()).all()


# sparse columns over bitmaps whose words are not a multiple of four, or of four per thread
@pytest.mark.parametrize("n,d,ns", [(33, 3, 2), (97, 4, 3), (32767, 4, 2), (65600, 4, 2), (131073, 5, 3), (524289, 3, 2), (1000003, 3, 2)])
def test_split_of_sparse_columns(ctx, n, d, ns):
    test_split_shapes_equal_one_pass(ctx, n, d, ns)


# columns of one window on both sides of the rules by which lanes search their products' sources (256
# sources, 4,096 products), against the split form, whose kernel has no such rule
@pytest.mark.parametrize("n,d", [(900, 64), (500, 66), (700, 252), (1500, 258), (3000, 40)])
def test_searched_and_walked_products(ctx, n, d):
    from paper_2002_10083_gb300 import mcl
    A = _random(n, d, seed=n + d, zeros=True)
    prm = mcl.Params(threshold=1e-4, select_k=120, recover_pct=0.9, inflation=2.0)
    out, ch = ctx.expand(A, prm)
    ref, ch_ref, _ = ctx.expand_split(A, prm, 2)
    assert ch == ch_ref and torch.equal(out.colptr, ref.colptr) and torch.equal(out.rowidx, ref.rowidx)
    assert torch.equal(out.val.view(torch.int32), ref.val.view(torch.int32))
