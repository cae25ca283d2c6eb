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
