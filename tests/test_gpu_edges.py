"""Kernels and dispatch rules at the sizes where they can go wrong: edges of
tiles, remainders, unaligned rows, many ties, the smallest inputs.  Labels
against the oracle's, min_dist at its binary64 tolerance."""
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


def _assign(ctx, X, C, low, offset=0, **kw):
    import paper_2407_12208_gb300 as pkg
    lab, md, nf = ctx.assign(_dev(X, offset), _dev(C, offset), pkg.params(low, **kw))
    return lab.cpu().numpy(), md.cpu().numpy(), nf


# the tiled direct kernel: 64-coordinate chunks, 64-centre tiles, 32 / 64 / 128 rows per block,
# one, two or four floats per load
@pytest.mark.parametrize("offset", [0, 1, 2])
@pytest.mark.parametrize("n,d,k", [(1, 9, 1), (33, 13, 7), (127, 50, 63), (129, 64, 64), (300, 65, 65), (257, 66, 129),
                                   (700, 128, 100), (321, 130, 64), (200, 148, 33), (200, 152, 33), (333, 255, 70),
                                   (500, 256, 128), (20000, 20, 300), (40001, 12, 40), (5000, 8, 1500)])
def test_direct_tiled_edges(ctx, n, d, k, offset):
    X, C = workloads.gaussian_mixture(n, d, k, seed=n + d)
    lab, md, _ = _assign(ctx, X, C, "fp32", offset)
    check_assign(lab, md, X, C, oracle, RTOL_MD)


# rows left open: ties between duplicated centres go to the lowest index, whether the open
# centres fit the block's list or not, and whether the fp32 values fit shared memory or not
@pytest.mark.parametrize("copies,d,k", [(2, 20, 40), (64, 33, 128), (65, 33, 130), (200, 16, 400), (3, 12, 60000)])
def test_open_rows_take_the_lowest_index(ctx, copies, d, k):
    r = np.random.Generator(np.random.PCG64(k))
    base = r.normal(size=(k // copies, d)).astype(np.float32)
    C = np.tile(base, (copies, 1))  # centre j = base[j % (k // copies)]
    X = np.concatenate([base[:37] + r.normal(0, 1e-3, size=(len(base[:37]), d)).astype(np.float32), C])[: max(k, 200)]
    X = X.astype(np.float32)
    lab, md, _ = _assign(ctx, X, C, "fp32")
    assert lab.max() < len(base)
    olab, od1, _ = oracle.assign(X[:64], C)
    assert np.array_equal(lab[:64], olab)
    np.testing.assert_allclose(md[:64], od1, rtol=RTOL_MD, atol=1e-30)


# rows that the plain screen cannot decide go through the centred screen (from 2^30
# pair-coordinates on): far from the origin, past fp16's range, 8 bits on close distances
@pytest.mark.parametrize("offset", [0, 1])
@pytest.mark.parametrize("low,kind,n,d,k", [("bf16", "cancellation", 20011, 53, 1024), ("bf16", "cancellation", 16500, 128, 513),
                                            ("fp16", "cancellation", 17000, 256, 250), ("fp16", "huge", 17001, 64, 1000),
                                            ("e4m3", "uniform", 17000, 64, 1024), ("e4m3", "uniform", 16999, 250, 255),
                                            ("bf16", "copies3", 17001, 128, 510), ("bf16", "copies20", 17001, 128, 500),
                                            ("bf16", "copies64", 17001, 128, 512), ("bf16", "copies3", 60001, 9, 2001)])
def test_centred_screen(ctx, low, kind, n, d, k, offset):
    if kind == "uniform":
        X, C = workloads.uniform_pairs(n, d, k, seed=5)
    elif kind == "huge":
        X, C = workloads.gaussian_mixture(n, d, k, seed=5)
        X, C = X * np.float32(1e5), C * np.float32(1e5)
    else:
        X, C = workloads.cancellation(n, d, k, seed=5)
        if kind.startswith("copies"):  # ties: two candidates to more than a list holds
            c = int(kind[6:])
            C = np.tile(C[: k // c], (c, 1))
    lab, md, _ = _assign(ctx, X, C, low, offset)
    assert ctx.stats()["overflow_rows"] > n // 2
    check_assign(lab, md, X, C, oracle, RTOL_MD)
    if kind.startswith("copies"):
        assert lab.max() < len(C) // int(kind[6:])


def test_smallest_accepted_workspace(ctx):
    """A workspace without room for the centred screen is still accepted."""
    import paper_2407_12208_gb300 as pkg
    X, C = workloads.cancellation(17000, 64, 1000, seed=6)
    Xd, Cd, p = _dev(X), _dev(C), pkg.params("bf16")
    ws = ctx.workspace(17000, 64, 1000, p)
    lo, hi = 0, ws.numel()  # refused at lo, accepted at hi
    while hi - lo > 256:
        mid = (lo + hi) // 2
        try:
            ctx.assign(Xd, Cd, p, ws=ws[:mid])
            hi = mid
        except pkg.KmError:
            lo = mid
    full = ctx.assign(Xd, Cd, p)
    small = ctx.assign(Xd, Cd, p, ws=ws[:hi])
    assert hi < ws.numel() - 17000 * 64 * 2
    assert torch.equal(full[0], small[0]) and torch.equal(full[1], small[1]) and full[2] == small[2]


# the two forms of the refinement (n d > 2^25 and d > 64: the flat pair list) at ragged shapes,
# with near-ties, single candidates and rows of more than 12 candidates
@pytest.mark.parametrize("low", ["bf16", "fp16"])
@pytest.mark.parametrize("n,d,k,scale", [(31, 24, 9, 1.0), (33, 100, 33, 1.0), (5003, 30, 70, 1.0), (4001, 130, 257, 0.02),
                                         (9000, 8, 64, 0.01), (525000, 65, 40, 1.0), (263000, 128, 66, 0.02)])
def test_refine_forms(ctx, low, n, d, k, scale):
    X, C = workloads.uniform_pairs(n, d, k, seed=n)
    X, C = 1 + np.float32(scale) * X, 1 + np.float32(scale) * C  # (scale << 1: wide bounds, many candidates)
    C[k // 2 :] = C[: k - k // 2]  # near-ties of identical centres
    lab, md, _ = _assign(ctx, X, C, low)
    _, first, inverse = np.unique(C, axis=0, return_index=True, return_inverse=True)
    assert np.array_equal(first[inverse.ravel()][lab], lab)  # the lowest index of identical centres
    m = min(n, 20000)
    check_assign(lab[:m], md[:m], X[:m], C, oracle, RTOL_MD)
    check_assign(lab[-200:], md[-200:], X[-200:], C, oracle, RTOL_MD)


# rows of unaligned or odd length quantise with the statistics of a full warp's tree (eight
# lanes standing for 32): equal to the aligned form's up to the fp32 sums' own rounding
@pytest.mark.parametrize("low", ["bf16", "fp16", "e4m3"])
@pytest.mark.parametrize("d", [1, 7, 8, 9, 31, 32, 33, 40, 57, 63, 64, 65])
def test_quantise_short_rows(ctx, low, d):
    if low == "e4m3" and d < 16:
        pytest.skip("E4M3 takes d >= 16")
    r = np.random.Generator(np.random.PCG64(d))
    X = r.normal(size=(1003, d)).astype(np.float32) * np.exp2(r.integers(-8, 8, size=(1003, 1))).astype(np.float32)
    X[5] = 0
    q, st, sc = (t.cpu().numpy() for t in ctx.quantize(_dev(X, 1), low))
    x = X.astype(np.float64)
    esz = 1 if low == "e4m3" else 2
    dt = {"bf16": torch.bfloat16, "fp16": torch.float16, "e4m3": torch.float8_e4m3fn}[low]
    xq = torch.from_numpy(q).view(dt).double().numpy()[:, :d] * sc[:, None]
    assert q.shape[1] // esz >= d and not q[:, d * esz :].any()
    infl = 1 + 2.0 ** -12
    for got, want in ((st[:, 0], (x * x).sum(1)), (st[:, 1], infl * np.linalg.norm(x, axis=1)),
                      (st[:, 2], infl * np.linalg.norm(xq, axis=1)), (st[:, 3], infl * np.linalg.norm(xq - x, axis=1))):
        np.testing.assert_allclose(got, want, rtol=(d + 4) * 2.0 ** -24)


# the deterministic sum: a warp or a block per part, parts of no, one and many rows
@pytest.mark.parametrize("n", [1, 2, 1023, 1024, 1025, 300000, 1024 * 1024, 1024 * 1024 + 1, 1500007])
def test_sse_sum(ctx, n):
    import paper_2407_12208_gb300 as pkg
    r = np.random.Generator(np.random.PCG64(n))
    X = _dev(r.normal(size=(n, 3)).astype(np.float32))
    _, md, _ = ctx.assign(X, X[:1].clone(), pkg.params("fp32"))
    sse = ctx.stats()["sse"]
    np.testing.assert_allclose(sse, md.sum().item(), rtol=n * 2.0 ** -53 + 1e-15)
    ctx.assign(X, X[:1].clone(), pkg.params("fp32"))
    assert ctx.stats()["sse"] == sse  # the same order whatever the launch


# empty clusters: the rows of largest min_dist in order, ties to the lowest index, when the
# radix selection can stop early (distinct distances) and when it cannot (ties at the threshold)
@pytest.mark.parametrize("ties", [False, True])
@pytest.mark.parametrize("n,e", [(300, 1), (5000, 7), (70000, 300)])
def test_farthest_rows_selection(ctx, ties, n, e):
    r = np.random.Generator(np.random.PCG64(n))
    md = r.random(n)
    if ties:
        md = np.floor(md * 4)
    rows, vals = ctx.farthest_rows(torch.from_numpy(md).cuda(), e)
    want = np.lexsort((np.arange(n), -md))[:e]
    assert np.array_equal(rows.cpu().numpy(), want)
    assert np.array_equal(vals.cpu().numpy(), md[want])


# seeding: chunks of 16 or 32 rows and their groups of eight, one and several lanes per row,
# unaligned rows, more rows than one chunk size covers
@pytest.mark.parametrize("n,d,offset", [(1, 3, 0), (33, 8, 0), (127, 9, 1), (129, 20, 0), (1025, 33, 1), (4099, 64, 0),
                                        (2047, 130, 0), (900, 260, 1), (240001, 2, 0), (235000, 12, 1)])
def test_seeding_chunks(ctx, n, d, offset):
    X, _ = workloads.blobs(n, d, 1, seed=n)
    k = min(n, 12)
    C, idx = ctx.seed_pp(_dev(X, offset), workloads.seed_uniforms(k, seed=d))
    oidx, margin = oracle.kmeanspp(X, workloads.seed_uniforms(k, seed=d), follow=idx)
    assert np.array_equal(idx[margin > 1e-9], oidx[margin > 1e-9])
    assert np.array_equal(C.cpu().numpy(), X[idx])


# the distance matrix: column ranges of few row blocks, 16-byte and single stores (k % 4),
# unstaged wide rows, flag masks that straddle words, and the binary64 fallback's values
# (bit for bit the rounded binary64 sums) from the queue and by the scan of D
@pytest.mark.parametrize("low,test,n,d,k,near", [("fp16", "tc", 130, 128, 129, 0.5), ("bf16", "tc", 300, 64, 300, 0.1),
                                                 ("bf16", "paper", 257, 128, 255, 0.0), ("bf16", "paper", 1200, 100, 1100, 0.3),
                                                 ("fp16", "tc", 5000, 37, 33, 0.9), ("fp16", "tc", 500, 200, 130, 0.5),
                                                 ("e4m3", "tc", 200, 128, 131, 0.5), ("bf16", "tc", 64, 9, 1, 1.0),
                                                 ("fp16", "tc", 20000, 16, 512, 0.02)])
def test_distance_matrix_edges(ctx, low, test, n, d, k, near):
    import paper_2407_12208_gb300 as pkg
    X, C = workloads.near_far(n, d, near, seed=n + k)
    C = C[:k].copy()
    C[0] = X[0]
    D, bits, nf = ctx.distances(_dev(X), _dev(C), pkg.params(low, test))
    D, bits = D.cpu().numpy(), bits.cpu().numpy().view(np.uint32)
    fl = np.unpackbits(bits.view(np.uint8), bitorder="little")[: n * k].reshape(n, k).astype(bool)
    assert fl.sum() == nf and fl[0, 0] and not (D < 0).any()
    want = oracle.dist_direct(X, C)
    assert np.array_equal(D[fl], want[fl].astype(np.float32))
    if low != "e4m3" and (~fl).any():  # Eq. (quantis-rel-bound-expand): unflagged pairs to 1 / (rho - 1)
        assert (np.abs(D[~fl] - want[~fl]) <= 0.26 * want[~fl]).all()


# the centre update at the edges of its dispatch (shared sums in one launch, buckets, global
# sums): counts and means against the oracle's within Lemma 4.4's fp32 store, kept, reseeded
# and shifted centres; the fused distances equal a separate assignment's bit for bit
@pytest.mark.parametrize("empty", ["keep", "farthest"])
@pytest.mark.parametrize("n,d,k,offset", [(1, 9, 1, 0), (100, 10, 7, 0), (5000, 16, 8, 0), (5000, 16, 8, 1), (131072, 16, 4, 0),
                                          (131073, 16, 4, 0), (3000, 130, 150, 1), (4000, 33, 250, 0), (2000, 129, 199, 0),
                                          (2000, 129, 201, 0), (1500, 8, 90, 0), (700, 256, 40, 0)])
def test_update_dispatch_edges(ctx, n, d, k, offset, empty):
    import paper_2407_12208_gb300 as pkg
    X, C = workloads.blobs(n, d, k, seed=n + k)
    if k > 4:
        C[1] += 1e3  # empty
    p = pkg.params("fp32", empty=empty)
    Xd, Cd = _dev(X, offset), _dev(C, offset)
    lab, md, Cn, counts, shift = ctx.lloyd_step(Xd, Cd, p)
    lab2, md2, _ = ctx.assign(Xd, Cd, p)
    assert torch.equal(lab, lab2) and torch.equal(md, md2)
    Cn2, counts2, shift2 = ctx.update_centroids(Xd, lab, Cd, p, min_dist=md)
    assert torch.equal(Cn, Cn2) and torch.equal(counts, counts2) and shift == shift2
    lab, md, Cn, counts = (t.cpu().numpy() for t in (lab, md, Cn, counts))
    cnt = np.bincount(lab, minlength=k)
    assert np.array_equal(counts, cnt)
    want = C.astype(np.float64)
    for j in np.nonzero(cnt)[0]:
        want[j] = X[lab == j].astype(np.float64).mean(0)
    if empty == "farthest":
        far = np.lexsort((np.arange(n), -md))
        for r, j in enumerate(np.nonzero(cnt == 0)[0]):
            want[j] = X[far[r]]
    np.testing.assert_allclose(Cn, want, rtol=2.0 ** -23, atol=np.abs(X).max() * 2.0 ** -30)
    np.testing.assert_allclose(shift, np.linalg.norm(Cn.astype(np.float64) - C, axis=1).max(), rtol=1e-12)


# small d: the window test on centred data (two rows per lane, steps of 64, chunks of eight
# centres), staged and unaligned rows, listed rows (low formats whose lists overflow), ties,
# data far from the origin and below binary32's normal squares
@pytest.mark.parametrize("offset", [0, 1])
@pytest.mark.parametrize("kind", ["mixture", "cancellation", "copies", "tiny"])
@pytest.mark.parametrize("n,d,k", [(1, 1, 1), (63, 2, 9), (64, 3, 8), (65, 4, 16), (1000, 5, 17), (4097, 6, 33), (777, 7, 100),
                                   (5000, 8, 1024), (3000, 2, 3000)])
def test_small_d_edges(ctx, n, d, k, kind, offset):
    if kind == "cancellation":
        X, C = workloads.cancellation(n, d, k, seed=n)
    else:
        X, C = workloads.gaussian_mixture(n, d, k, seed=n)
        if kind == "copies":
            C[k // 2 :] = C[: k - k // 2].copy()
        if kind == "tiny":
            X, C = X * np.float32(1e-19), C * np.float32(1e-19)
    for low in ("fp32", "bf16") if kind == "cancellation" else ("fp32",):
        lab, md, _ = _assign(ctx, X, C, low, offset)
        olab, od1, od2 = oracle.assign(X, C)
        sure = (od2 - od1) > 1e-6 * od2
        assert np.array_equal(lab[sure], olab[sure])
        first = np.unique(C, axis=0, return_index=True, return_inverse=True)
        assert np.array_equal(first[1][first[2].ravel()][lab], lab)
        if kind != "tiny":  # (there the double-float squares underflow, as they always did)
            np.testing.assert_allclose(md, oracle.dist_labelled(X, C, lab), rtol=RTOL_MD, atol=1e-30)


# small-d centre sums: whole steps of one label, few labels, many labels; two and three parts
# per value (2^22 rows and more), also at the ends of the float range, where the fixed-point
# scale leaves it: sums equal to integer sums of the rounded values
@pytest.mark.parametrize("scale", [1.0, 1e30, 1e-36])
@pytest.mark.parametrize("n,d,k", [(31, 3, 2), (40000, 5, 16), (100001, 8, 64), (4194304 + 77, 2, 7), (4194304 + 77, 5, 16)])
def test_small_d_sums_parts(ctx, n, d, k, scale):
    import math
    import paper_2407_12208_gb300 as pkg
    g = torch.Generator(device="cuda").manual_seed(n + d)
    X = (torch.randn(n, d, generator=g, device="cuda") * scale).contiguous()
    i = torch.arange(n, device="cuda")
    lab = torch.where(i % 3000 < 1800, (i // 700) % k, torch.where(i % 3000 < 2400, (i // 5) % k, (i * 7919) % k)).int()
    bits = ctx.absmax(X)
    sums, counts = ctx.update_partial(X, lab, k, bits, n)
    assert torch.equal(counts, torch.bincount(lab.long(), minlength=k))
    amax = float(np.array([bits], dtype=np.uint32).view(np.float32)[0])
    S = 60 - (n - 1).bit_length() - (math.frexp(amax)[1] - 1)
    v = torch.round(X.double() * 2.0 ** (S // 2) * 2.0 ** (S - S // 2)).long()  # (ties to even, as the kernel's additions)
    want = torch.zeros(k, d, dtype=torch.int64, device="cuda").index_add_(0, lab.long(), v)
    assert torch.equal(sums, want)


# the screen's epilogue groups: row blocks of 1, 2, 3, 4 and 7 column tiles, several per CTA, so
# that groups pass by row blocks without a tile for them; every variant of the epilogue gives
# the same flags and labels
@pytest.mark.parametrize("low", ["bf16", "e4m3"])
@pytest.mark.parametrize("k", [1, 128, 129, 256, 300, 385, 512, 800])
def test_screen_groups(ctx, low, k):
    import paper_2407_12208_gb300 as pkg
    n, d = 152 * 128 * 3 + 5, 24
    X, C = workloads.gaussian_mixture(n, d, k, seed=k)
    Xd, Cd = _dev(X), _dev(C)
    ref = torch.empty(n, dtype=torch.int64, device="cuda")
    for s in range(0, n, 8192):
        ref[s : s + 8192] = ((Xd[s : s + 8192, None, :].double() - Cd[None].double()) ** 2).sum(2).argmin(1)
    flags = set()
    try:
        for variant in ("full", "half", "c32"):
            ctx.set_screen_variant(n, d, k, low, variant)
            lab, _, nf = ctx.assign(Xd, Cd, pkg.params(low))
            assert torch.equal(lab.long(), ref)
            flags.add(int(nf))
    finally:
        ctx.set_screen_variant(n, d, k, low, "auto")
    assert len(flags) == 1


# quantisation, a thread per row (d <= 16, from 38,912 rows on) and several rows per eight lanes
# (d <= 64 aligned, from 77,825 rows on), on both sides of the lines and past the end of a round
@pytest.mark.parametrize("low", ["fp16", "bf16", "e4m3"])
@pytest.mark.parametrize("n,d,offset", [(38911, 10, 0), (38912, 10, 0), (38913, 16, 0), (77824, 32, 0), (77825, 32, 0),
                                        (155651, 24, 0), (311299, 20, 0), (90001, 64, 0), (160003, 40, 0), (60001, 12, 1),
                                        (60001, 3, 0), (60001, 1, 0), (60002, 4, 0), (60003, 8, 2), (60005, 15, 0),
                                        (50000, 16, 1)])
def test_quantise_rows_per_thread(ctx, low, n, d, offset):
    if low == "e4m3" and d < 16:
        pytest.skip("E4M3 takes d >= 16")
    k = 30
    X, C = workloads.gaussian_mixture(n, d, k, seed=n + d)
    lab, md, nf = _assign(ctx, X, C, low, offset)
    check_assign(lab, md, X, C, oracle, RTOL_MD)
    # the first rows by themselves, in the form for few rows: the same statistics, so the same flags
    _, _, nf1 = _assign(ctx, X[:30000], C, low, offset)
    _, _, nf2 = _assign(ctx, X[30000:], C, low, offset)
    assert nf == nf1 + nf2


# centre sums of few rows straight in L2 (n <= 64 k, n d <= 2^20), on both sides of the lines, and
# the bucketed sums' short segments: equal to integer sums of the rounded values, also when all
# rows have one label
@pytest.mark.parametrize("one_label", [False, True])
@pytest.mark.parametrize("n,d,k,offset", [(1, 1, 1, 0), (64, 33, 1, 0), (65, 33, 1, 0), (6400, 70, 100, 0), (6401, 70, 100, 1),
                                          (16384, 64, 300, 0), (16385, 64, 300, 0), (3000, 3, 200, 0), (2000, 512, 64, 0),
                                          (2000, 513, 64, 0), (20000, 130, 90, 0), (37638, 128, 44, 0), (2371, 256, 164, 2)])
def test_sums_of_few_rows(ctx, n, d, k, offset, one_label):
    import math
    import paper_2407_12208_gb300 as pkg
    r = np.random.default_rng(n + d)
    X = _dev(r.normal(size=(n, d)).astype(np.float32), offset)
    lab = torch.from_numpy((np.full(n, k - 1) if one_label else r.integers(0, k, size=n)).astype(np.int32)).cuda()
    bits = ctx.absmax(X)
    sums, counts = ctx.update_partial(X, lab, k, bits, n)
    assert torch.equal(counts, torch.bincount(lab.long(), minlength=k))
    amax = float(np.array([bits], dtype=np.uint32).view(np.float32)[0])
    S = 60 - (n - 1).bit_length() - (math.frexp(amax)[1] - 1)
    v = torch.round(X.double() * 2.0 ** (S // 2) * 2.0 ** (S - S // 2)).long()
    assert torch.equal(sums, torch.zeros(k, d, dtype=torch.int64, device="cuda").index_add_(0, lab.long(), v))


# refinement, four, eight and 32 rows per warp: near-ties and many candidates on both sides of the lines
@pytest.mark.parametrize("n", [130, 131, 133, 19456, 19457, 38912, 38913])
@pytest.mark.parametrize("d", [16, 70])
def test_refine_rows_per_warp(ctx, n, d):
    r = np.random.default_rng(n + d)
    C = r.uniform(size=(90, d)).astype(np.float32)
    C = np.concatenate([C, C[:40] + np.float32(1e-7)]).astype(np.float32)  # near-ties
    X = r.uniform(size=(n, d)).astype(np.float32)
    lab, md, _ = _assign(ctx, X, C, "bf16")
    check_assign(lab, md, X, C, oracle, RTOL_MD)


# rows of more than twelve candidates: none, a few per warp (decided in the first pass) and many
# (listed), among rows of one candidate, with and without a centred screen after
@pytest.mark.parametrize("every", [0, 40, 9, 6, 2])
@pytest.mark.parametrize("n,d,k", [(20000, 24, 300), (60000, 40, 600), (6000, 16, 200)])
def test_rows_of_many_candidates(ctx, n, d, k, every):
    r = np.random.default_rng(n + every)
    C = (20 * r.normal(size=(k, d))).astype(np.float32)
    C[: 40] = C[0] + (0.02 * r.normal(size=(40, d))).astype(np.float32)  # forty centres close together
    at = r.integers(40, k, size=n)
    if every:
        at[::every] = r.integers(0, 40, size=len(at[::every]))
    X = (C[at] + 0.05 * r.normal(size=(n, d))).astype(np.float32)
    lab, md, _ = _assign(ctx, X, C, "bf16")
    check_assign(lab, md, X, C, oracle, RTOL_MD)
