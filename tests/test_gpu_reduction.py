"""Block and grid sums of inner products (warp_sum adds in integer arithmetic): <p, A p> with a
diagonal A against an exactly rounded sum, over the exponent range, with cancellation, and with
infinities and NaN."""
import math

import numpy as np
import pytest
import torch

from paper_1410_4054_gb300 import pk

pytestmark = pytest.mark.gpu

EPS = 2.0 ** -53


def dot(p, d):
    n = len(p)
    A = pk.CSRMatrix(np.arange(n + 1, dtype=np.int32), np.arange(n, dtype=np.int32), d)
    pt = torch.from_numpy(p).cuda()
    q, out = torch.empty_like(pt), torch.empty(1, dtype=torch.float64, device="cuda")
    pk.spmv_dot(A, pt, q, out)
    got = out.item()
    A.close()
    return got, p, q.cpu().numpy()


def inputs(kind, n, rng):
    p = rng.uniform(-1, 1, n)
    d = rng.uniform(0.5, 2, n)
    if kind == "cancel":
        p = np.abs(p) + 0.1
        d = np.where(np.arange(n) % 2 == 0, 1.0, -1.0) * d
    elif kind == "wide":
        p = p * 2.0 ** rng.integers(-60, 60, n)
    elif kind == "one_large":
        p = p * 1e-9
        p[n // 2] = 3.0
    elif kind == "huge":
        p, d = p * 1e150, d * 1e5
    elif kind == "tiny":
        p, d = p * 1e-153, d * 1e-4
    elif kind == "zeros":
        p[:] = 0.0
    elif kind == "few":
        p[rng.random(n) < 0.99] = 0.0
    return p, d


@pytest.mark.parametrize("kind", ["plain", "cancel", "wide", "one_large", "huge", "tiny", "zeros", "few"])
@pytest.mark.parametrize("n", [1, 31, 33, 257, 4096, 300_001])
def test_dot_is_as_exact_as_a_tree_of_fp64_sums(kind, n):
    """Every product is rounded into its thread's sum (fma, ceil(n / (grid 256)) of them), then at
    most two warp stages and two grid stages follow: bound each by one rounding of the sum of
    absolute values, plus underflow."""
    p, d = inputs(kind, n, np.random.default_rng(n))
    got, p, q = dot(p, d)
    # (the large terms are added scaled by 2^-64, which is exact, as their sum may overflow)
    s = 2.0 ** -64 if kind == "huge" else 1.0
    want = math.fsum((p * s * q).tolist()) / s
    mass = math.fsum(np.abs(p * s * q).tolist()) / s
    if math.isinf(want):
        assert got == want
        return
    per_thread = -(-n // 256) if n <= 256 * 1000 else 2
    assert abs(got - want) <= (min(per_thread, 4) + 6) * EPS * mass + n * 2.0 ** -1074


@pytest.mark.parametrize("bad", [np.inf, -np.inf, np.nan, "both"])
def test_dot_keeps_infinities_and_nan(bad):
    rng = np.random.default_rng(5)
    p, d = rng.uniform(0.5, 1, 5000), np.ones(5000)
    if bad == "both":
        d[7], d[4000] = np.inf, -np.inf
    else:
        d[77] = bad
    got, _, _ = dot(p, d)
    if bad in (np.inf, -np.inf):
        assert got == bad
    else:
        assert math.isnan(got)
