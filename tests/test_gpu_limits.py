"""Inputs at the limits of what the kernels' rules and bounds cover: squares
below binary32's range, data on which a rule's fast path decides little."""
import numpy as np
import pytest

import oracle
from paper_2407_12208_gb300 import workloads
from gpu_util import RTOL_MD, check_assign

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def ctx():
    import paper_2407_12208_gb300 as pkg
    from paper_2407_12208_gb300 import build
    build.build()
    c = pkg.Context(0)
    yield c
    c.close()


def _dev(a, offset=0):
    """a on the GPU, `offset` floats past an allocation's start."""
    buf = torch.empty(a.size + offset, dtype=torch.float32, device="cuda")
    t = buf[offset:].view(a.shape)
    t.copy_(torch.from_numpy(np.ascontiguousarray(a)))
    return t


def _subnormal_squares(n, d, k, s):
    """Rows (s, 0, 0, ..): centre 0 is off by two squares of 0.49 of binary32's least number (each
    rounds to 0), the last centre by one of 0.51 (rounds to 1): the last is nearer, but its fp32
    distance is the larger.  The others lie far away."""
    least = 2.0 ** -149
    X = np.zeros((n, d), np.float32)
    X[:, 0] = s
    C = np.ones((k, d), np.float32)
    C[0] = C[-1] = X[0]
    C[0, 1:3] = np.float32(np.sqrt(0.49 * least))
    C[-1, 1] = np.float32(np.sqrt(0.51 * least))
    return X, C


# every path that decides labels from fp32 direct values: the small-d, tiled and listed-row kernels
# (low formats: rows near zero have no usable norms and go there), the refinement in one launch, in
# a flat pair list and by the whole warp
@pytest.mark.parametrize("low,n,d,k,s", [("fp32", 70, 3, 2, 0.0), ("fp32", 70, 8, 40, 1.0), ("fp32", 70, 9, 3, 0.0),
                                         ("fp32", 130, 130, 100, 1.0), ("fp32", 4100, 3, 4000, 1.0), ("bf16", 70, 20, 5, 0.0),
                                         ("e4m3", 70, 300, 5, 0.0), ("bf16", 70, 20, 5, 2.0 ** -49),
                                         ("fp16", 570, 21, 500, 0.0), ("bf16", 270000, 128, 5, 2.0 ** -49)])
def test_squares_below_the_range(ctx, low, n, d, k, s):
    import paper_2407_12208_gb300 as pkg
    X, C = _subnormal_squares(n, d, k, s)
    lab, _, _ = ctx.assign(_dev(X), _dev(C), pkg.params(low))
    assert oracle.assign(X[:1], C)[0][0] == k - 1
    assert (lab == k - 1).all()


def test_squares_below_the_range_grouped(ctx):
    import paper_2407_12208_gb300 as pkg
    X, C = _subnormal_squares(50, 4, 6, 0.0)
    (out,) = ctx.lloyd_run_batch([(_dev(X), _dev(C))], pkg.params("fp32", max_iter=0))
    assert (out[1] == 5).all()


def _smallest_workspace(ctx, run, ws):
    """Bytes of the smallest workspace that `run` accepts, to 256."""
    import paper_2407_12208_gb300 as pkg
    lo, hi = 0, ws.numel()  # refused at lo, accepted at hi
    while hi - lo > 256:
        mid = (lo + hi) // 2
        try:
            run(ws[:mid])
            hi = mid
        except pkg.KmError:
            lo = mid
    return hi


# the serving engine takes a job, and two side by side, when the arena holds what they need: the
# buffers of the centred screen (n k d >= 2^30) are no part of that
def test_admission_without_optional_buffers(ctx):
    import time
    import paper_2407_12208_gb300 as pkg
    n, d, k = 17000, 64, 1000
    X, C = workloads.cancellation(n, d, k, seed=6)
    Xd, Cd, p = _dev(X), _dev(C), pkg.params("bf16", max_iter=2)
    need = _smallest_workspace(ctx, lambda ws: ctx.lloyd_run(Xd, Cd, p, ws=ws), ctx.workspace(n, d, k, p))
    want = ctx.lloyd_run(Xd, Cd, p)
    job = need + 4 * (n + 2 * k * d) + 2048  # labels, centres and their rounding to 256
    s = pkg.Context(0, arena_bytes=2 * job + 1024)
    try:
        ids = [s.submit(Xd, Cd, p) for _ in range(2)]
        for i in ids:  # both run although neither result is released
            t0 = time.time()
            while (r := s.poll(i)) is None:
                assert time.time() - t0 < 60, "not admitted"
                time.sleep(0.002)
            assert r["status"] == pkg._binding.KM_OK
            assert torch.equal(pkg.device_array(r["labels"], (n,), "<i4"), want[1])
            assert torch.equal(pkg.device_array(r["C"], (k, d), "<f4"), want[0])
    finally:
        s.close()


# the flat pair list (n d > 2^25, d > 64) and the centred screen's buffers share a span: rows
# decided by the one, by the other and by neither in the same call and the same run, with and
# without room for the larger of the two
def test_workspace_of_the_largest_step(ctx):
    import paper_2407_12208_gb300 as pkg
    n, d = 10 ** 6, 128
    screen = n * (2 * d + 16) + n * 4 * (48 + 16)   # X in bf16, statistics, lists and per-row words
    tail = n * (2 * d + 16 + 4)                      # the larger of the two sets
    assert ctx.workspace_size(n, d, 1024, pkg.params("bf16")) < screen + tail + (8 << 20)


@pytest.mark.parametrize("call", ["assign", "run", "host"])
def test_shared_scratch_span(ctx, call):
    import paper_2407_12208_gb300 as pkg
    n, d, k = 270001, 128, 40
    X, C = workloads.gaussian_mixture(n, d, k, seed=8)
    far, near = workloads.cancellation(90000, d, 20, seed=9)
    C[:20] = near  # a third of the rows: lists that overflow
    X[::3][:90000] = far
    C[39] = C[38]
    p = pkg.params("bf16", max_iter=3)
    Xd, Cd = _dev(X), _dev(C)
    if call == "host":
        got = ctx.lloyd_step_host(torch.from_numpy(X), torch.from_numpy(C), p)
        want = ctx.lloyd_step(Xd, Cd, p)
        assert torch.equal(got[0], want[0].cpu()) and torch.equal(got[2], want[2].cpu()) and got[4] == want[4]
        return
    f = (lambda ws: ctx.assign(Xd, Cd, p, ws=ws)[:2]) if call == "assign" else (lambda ws: ctx.lloyd_run(Xd, Cd, p, ws=ws)[:3])
    ws = ctx.workspace(n, d, k, p)
    hi = _smallest_workspace(ctx, f, ws)
    assert hi < ws.numel() - n * 100
    a, b = f(ws), f(ws[:hi])
    assert all(np.array_equal(torch.as_tensor(u).cpu().numpy(), torch.as_tensor(v).cpu().numpy()) for u, v in zip(a, b))
    if call == "assign":
        check_assign(a[0].cpu().numpy()[:3000], a[1].cpu().numpy()[:3000], X[:3000], C, oracle, RTOL_MD)


def _sums(X, lab, k, bits, n):
    """Integer sums of the rounded fixed-point values."""
    import math
    amax = float(np.array([bits], dtype=np.uint32).view(np.float32)[0])
    S = 60 - (n - 1).bit_length() - (math.frexp(amax)[1] - 1)
    v = torch.round(X.double() * 2.0 ** (S // 2) * 2.0 ** (S - S // 2)).long()
    return torch.zeros(k, X.shape[1], dtype=torch.int64, device="cuda").index_add_(0, lab.long(), v)


def _labels(kind, n, k, r):
    u = r.integers(0, k, size=n)
    return {"spread": u, "sorted": np.sort(u), "one": np.full(n, k - 1), "two": np.where(r.random(n) < 0.5, 0, k - 1),
            "most": np.where(r.random(n) < 0.9, k // 2, u), "runs": (np.arange(n) // 11) % k}[kind].astype(np.int32)


# centre sums in one launch: blocks of 16 to 128 rows ordered by label and their slices (runs of one
# label that end in, cross and fill slices, in the last block's few rows too), the shared sums with
# several rows of a label added up first, and the bucketed sums' long segments, on both sides of
# the dispatch's lines
@pytest.mark.parametrize("kind", ["spread", "sorted", "one", "two", "most", "runs"])
@pytest.mark.parametrize("n,d,k,offset", [(1, 9, 1, 0), (15, 20, 3, 0), (17, 33, 5, 1), (2447, 70, 164, 0), (19457, 24, 37, 0),
                                          (19585, 64, 40, 1), (3000, 257, 9, 0), (1500, 512, 30, 0), (5000, 3, 700, 0),
                                          (100003, 10, 100, 0), (100003, 20, 500, 0), (20001, 16, 128, 1), (20001, 16, 129, 0),
                                          (30000, 130, 31, 0), (33001, 127, 20, 0), (70001, 64, 12, 0), (9000, 250, 26000, 0)])
def test_sums_of_any_labels(ctx, n, d, k, offset, kind):
    r = np.random.default_rng(n + d + k)
    X = _dev(r.normal(size=(n, d)).astype(np.float32), offset)
    lab = torch.from_numpy(_labels(kind, n, k, r)).cuda()
    bits = ctx.absmax(X)
    sums, counts = ctx.update_partial(X, lab, k, bits, n)
    assert torch.equal(counts, torch.bincount(lab.long(), minlength=k))
    assert torch.equal(sums, _sums(X, lab, k, bits, n))


# and none of them takes much longer when most rows have one label (atomics on one address take
# turns: up to 20 times as long, were they left to)
@pytest.mark.parametrize("n,d,k", [(16384, 64, 300), (65536, 16, 1024), (8192, 128, 128), (100000, 10, 100), (100000, 20, 500),
                                   (200000, 10, 1000), (20000, 10, 1000)])
def test_sums_time_of_any_labels(ctx, n, d, k):
    import paper_2407_12208_gb300 as pkg
    r = np.random.default_rng(n)
    X, p, times = _dev(r.normal(size=(n, d)).astype(np.float32)), pkg.params("fp32", empty="keep"), {}
    for kind in ("spread", "one", "two", "most"):
        lab = torch.from_numpy(_labels(kind, n, k, r)).cuda()
        best = float("inf")
        for _ in range(8):
            a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            a.record()
            for _ in range(20):
                ctx.update_centroids(X, lab, X[:k], p, want_shift=False)
            b.record()
            b.synchronize()
            best = min(best, a.elapsed_time(b) / 20)
        times[kind] = best
    assert max(times.values()) < 1.8 * times["spread"], times


def _small(kind, n, d, k, r):
    X = r.random(size=(n, d)).astype(np.float32)
    C = X[r.permutation(n)[:k]].copy()
    if kind == "outlier":      # one centre far away: the window of every row is wide
        C[k // 2] = 1e4
    elif kind == "rows":       # a few rows far away
        X[::100] *= np.float32(1e4)
    elif kind == "grey":       # few distinct values, ties everywhere
        X = np.round(X * 16) / np.float32(16)
        C = X[:k].copy()
    elif kind == "blocks":     # warps whose rows all need more than the window, among others that do not
        C[: k // 2] = C[0] + np.float32(1e-4) * r.random(size=(k // 2, d)).astype(np.float32)
        X[: n // 2] = C[0]
        X[n // 4 : n // 4 + 3] = C[k - 1]
    return X.astype(np.float32), C.astype(np.float32)


# small d: rows that the window test leaves open, by the warp, by the direct pass and in the steps
# after it, and its near-ties; one and two dimensions, which take the direct pass throughout
@pytest.mark.parametrize("offset", [0, 1])
@pytest.mark.parametrize("kind", ["uniform", "outlier", "rows", "grey", "blocks"])
@pytest.mark.parametrize("n,d,k", [(2, 1, 1), (64, 1, 9), (9000, 1, 300), (9001, 1, 8192), (30000, 2, 700), (5000, 2, 4096),
                                   (129, 3, 8), (40001, 3, 16), (9000, 3, 2730), (30000, 5, 17), (20000, 8, 1024),
                                   (5000, 1, 32), (5000, 2, 33), (5001, 3, 128), (5001, 6, 129), (70, 8, 70), (700, 4, 700),
                                   (9300, 1, 9100), (30000, 2, 25000), (4000, 4, 3600), (9728, 8, 1100), (9729, 8, 1100),
                                   (2000, 7, 1300), (9729, 8, 1920), (9729, 8, 1936)])
def test_small_d_open_rows(ctx, n, d, k, kind, offset):
    import paper_2407_12208_gb300 as pkg
    k = min(k, n)
    X, C = _small(kind, n, d, k, np.random.default_rng(n + d + k))
    lab, md, _ = ctx.assign(_dev(X, offset), _dev(C, offset), pkg.params("fp32"))
    lab, md = lab.cpu().numpy(), md.cpu().numpy()
    m = min(n, 1 + (1 << 23) // (k * d))  # (the rows that the oracle is asked about: evenly spread)
    at = np.unique(np.linspace(0, n - 1, m).astype(np.int64))
    check_assign(lab[at], md[at], X[at], C, oracle, RTOL_MD)
    _, first, inverse = np.unique(C, axis=0, return_index=True, return_inverse=True)
    assert np.array_equal(first[inverse.ravel()][lab], lab)  # the lowest index of identical centres


def _time(f):
    best = float("inf")
    for _ in range(6):
        a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        a.record()
        for _ in range(10):
            f()
        b.record()
        b.synchronize()
        best = min(best, a.elapsed_time(b) / 10)
    return best


# and it costs little when the window decides little: many centres on a line (64 times the centres
# of the other), one centre far away
@pytest.mark.parametrize("d,k,kind,than,most", [(1, 1024, "uniform", (1, 16, "uniform"), 20), (2, 1024, "uniform", (2, 16, "uniform"), 22),
                                                (8, 1024, "outlier", (8, 1024, "uniform"), 1.8),
                                                (8, 64, "outlier", (8, 64, "uniform"), 1.8)])
def test_small_d_time(ctx, d, k, kind, than, most):
    r, n, times = np.random.default_rng(d), 1000000, []
    lab = torch.empty(n, dtype=torch.int32, device="cuda")
    md = torch.empty(n, dtype=torch.float64, device="cuda")
    for dd, kk, kind in ((d, k, kind), than):
        X, C = (_dev(a) for a in _small(kind, n, dd, kk, r))
        times.append(_time(lambda: ctx.assign_static(X, C, lab, md)))
    assert times[0] < most * times[1], times


# rows and centres that are no numbers or infinite: the other rows' results are not touched, their
# own labels are valid
@pytest.mark.parametrize("low,n,d,k", [("fp32", 3000, 1, 40), ("fp32", 3000, 5, 40), ("fp32", 3000, 20, 70), ("fp32", 3000, 130, 9),
                                       ("bf16", 3000, 32, 40), ("fp16", 3001, 33, 300), ("e4m3", 3000, 200, 40),
                                       ("e4m3", 900, 300, 40), ("bf16", 20000, 64, 1000), ("bf16", 270000, 128, 40)])
@pytest.mark.parametrize("centre", [False, True])
def test_not_numbers(ctx, low, n, d, k, centre):
    import paper_2407_12208_gb300 as pkg
    X, C = workloads.gaussian_mixture(n, d, k, seed=n + d)
    bad = np.arange(5, n, 97)
    for i, v in enumerate((np.nan, np.inf, -np.inf, 3e38)):
        X[bad[i::4], i % d] = np.float32(v)
    X[bad[::8]] = np.float32(np.nan)
    if centre:
        C[k // 2] = np.float32(np.nan)
        C[k // 3, 0] = np.float32(np.inf)
    lab, md, _ = ctx.assign(_dev(X), _dev(C), pkg.params(low))
    lab, md = lab.cpu().numpy(), md.cpu().numpy()
    assert lab.min() >= 0 and lab.max() < k
    good = np.setdiff1d(np.arange(n), bad)[:: max(1, n // 6000)]
    fin = np.isfinite(C).all(1)
    want = np.nonzero(fin)[0][oracle.assign(X[good], C[fin])[0]]
    assert np.array_equal(lab[good], want)
    np.testing.assert_allclose(md[good], oracle.dist_labelled(X[good], C, want), rtol=RTOL_MD)


# few coordinates against more centres than 32 KB hold, and rows of 9 to 31 coordinates against a
# few centres: the time per row and centre stays near that of fewer centres and of more coordinates
@pytest.mark.parametrize("d,k,than,most", [(1, 10000, (1, 5000), 3), (2, 5000, (2, 2500), 3), (4, 2100, (4, 1050), 3),
                                           (9, 10, (32, 10), 1.0), (12, 8, (32, 8), 0.5)])
def test_few_coordinates_time(ctx, d, k, than, most):
    n, times = 500000, []
    lab = torch.empty(n, dtype=torch.int32, device="cuda")
    md = torch.empty(n, dtype=torch.float64, device="cuda")
    for dd, kk in ((d, k), than):
        X = torch.rand(n, dd, generator=torch.Generator(device="cuda").manual_seed(dd), device="cuda")
        C = X[:kk].clone()
        times.append(_time(lambda: ctx.assign_static(X, C, lab, md)))
    assert times[0] < most * times[1], times


# ties: rows between equal centres, a few and all of a block's, by the warp (eight at a time; a centre
# or a coordinate per lane, four, two or one binary64 sums together, more candidates than it lists at
# once) and by the block
@pytest.mark.parametrize("every", [1, 13, 40])
@pytest.mark.parametrize("n,d,k,copies", [(365, 128, 20, 2), (200, 9, 17, 2), (333, 31, 70, 2), (333, 32, 70, 35), (300, 64, 66, 33),
                                          (129, 217, 64, 2), (131, 218, 130, 3), (257, 256, 128, 64), (5000, 20, 300, 4),
                                          (40000, 16, 65, 5), (300, 12, 200, 200)])
def test_ties(ctx, n, d, k, copies, every):
    import paper_2407_12208_gb300 as pkg
    r = np.random.default_rng(n + d + k)
    base = r.random(size=(k // copies, d)).astype(np.float32)
    C = np.concatenate([np.tile(base, (copies, 1)), 9 + r.random(size=(k - k // copies * copies, d))]).astype(np.float32)
    X = (9 + r.random(size=(n, d))).astype(np.float32)  # nearest to one of the last, or tied as well
    X[::every] = r.random(size=X[::every].shape)
    lab, md, _ = ctx.assign(_dev(X), _dev(C), pkg.params("fp32"))
    lab, md = lab.cpu().numpy(), md.cpu().numpy()
    olab, od1, _ = oracle.assign(X, C)
    _, first, inverse = np.unique(C, axis=0, return_index=True, return_inverse=True)
    assert np.array_equal(first[inverse.ravel()][lab], lab)
    far = np.abs(lab - olab) > 0  # (ties between different rows of base: within rounding)
    assert far.mean() < 0.01
    np.testing.assert_allclose(md, oracle.dist_labelled(X, C, lab), rtol=RTOL_MD)
    np.testing.assert_allclose(md, od1, rtol=1e-6)


# small-d centre sums: chunks of 32 rows and more per warp, eight warps folded together, in the last
# block too; steps of one label, a few, many in runs and in no order
@pytest.mark.parametrize("kind", ["spread", "sorted", "one", "two", "most", "runs"])
@pytest.mark.parametrize("n,d,k,offset", [(257, 1, 1, 0), (600, 8, 3, 0), (8191, 3, 7, 1), (77825, 5, 16, 0), (311301, 2, 256, 0),
                                          (311299, 8, 64, 1), (2600000, 4, 100, 0)])
def test_small_d_sums_of_any_labels(ctx, n, d, k, offset, kind):
    r = np.random.default_rng(n + d + k)
    X = torch.randn(n + offset, d, generator=torch.Generator(device="cuda").manual_seed(n), device="cuda").view(-1)[offset : offset + n * d].view(n, d)
    lab = torch.from_numpy(_labels(kind, n, k, r)).cuda()
    bits = ctx.absmax(X)
    sums, counts = ctx.update_partial(X, lab, k, bits, n)
    assert torch.equal(counts, torch.bincount(lab.long(), minlength=k))
    assert torch.equal(sums, _sums(X, lab, k, bits, n))


# and their time does not grow when no two neighbours share a label (folds of few rows each on the same
# few addresses took four times as long as the rows)
@pytest.mark.parametrize("n,d,k", [(409360, 5, 19), (1000000, 2, 256)])
def test_small_d_sums_time(ctx, n, d, k):
    import paper_2407_12208_gb300 as pkg
    p, times = pkg.params("fp32", empty="keep"), []
    X = torch.rand(n, d, generator=torch.Generator(device="cuda").manual_seed(1), device="cuda")
    for kind in ("spread", "sorted"):
        lab = torch.from_numpy(_labels(kind, n, k, np.random.default_rng(3))).cuda()
        times.append(_time(lambda: ctx.update_centroids(X, lab, X[:k], p, want_shift=False)))
    assert times[0] < 1.8 * times[1], times


# ties in the refinement's one launch: the warp's binary64 products in the candidates' own shared memory
# and past it, any width and alignment, odd and many candidates
@pytest.mark.parametrize("low,n,d,k,copies", [("fp16", 500, 64, 30, 2), ("bf16", 300, 95, 60, 3), ("fp16", 300, 96, 60, 2),
                                              ("bf16", 300, 97, 60, 3), ("fp16", 300, 100, 90, 18), ("bf16", 129, 256, 40, 20),
                                              ("bf16", 5000, 33, 40, 3), ("e4m3", 5000, 64, 20, 4)])
def test_ties_in_the_refinement(ctx, low, n, d, k, copies):
    import paper_2407_12208_gb300 as pkg
    r = np.random.default_rng(n + d + k)
    base = 8 * r.integers(0, 2, size=(k // copies, d)) + r.random(size=(k // copies, d))
    C = np.tile(base, (copies, 1)).astype(np.float32)
    X = (C[r.integers(0, len(C), n)] + 0.1 * r.random(size=(n, d))).astype(np.float32)
    lab, md, _ = ctx.assign(_dev(X), _dev(C), pkg.params(low))
    lab, md = lab.cpu().numpy(), md.cpu().numpy()
    assert np.array_equal(lab, oracle.assign(X, C)[0])
    np.testing.assert_allclose(md, oracle.dist_labelled(X, C, lab), rtol=RTOL_MD)


# a block of tied rows takes its warps, not its turns
def test_ties_time(ctx):
    times = []
    for copies in (1, 2):
        X = torch.rand(365, 128, generator=torch.Generator(device="cuda").manual_seed(1), device="cuda")
        C = X[: 20 // copies].repeat(copies, 1).contiguous()
        lab = torch.empty(365, dtype=torch.int32, device="cuda")
        md = torch.empty(365, dtype=torch.float64, device="cuda")
        times.append(_time(lambda: ctx.assign_static(X, C, lab, md)))
    assert times[1] < times[0] + 0.12, times
