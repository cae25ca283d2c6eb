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
