"""The subtree kernel of the splitter where its selection changes path, bit for bit against the oracle: bins
that hold more rows than a list takes (far outliers, repeated values, infinite variances), subsets of fewer rows
than a full sample, subtrees of exactly and just above the largest size, one wave of CTAs or several;
split coordinates beyond those that are kept coordinate-major, and infinite coordinates."""
import numpy as np
import pytest
import torch

from oracle import clusterattn_oracle as orc
from paper_2608_26965_b200 import binding

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


def _coordinates(kind, heads, n, d, seed):
    r = np.random.default_rng(seed)
    Y = r.standard_normal((heads, n, d)).astype(np.float32)
    if kind == "outliers":
        Y *= np.where(r.random((heads, n, 1)) < 0.01, 1e4, 1.0).astype(np.float32)
    elif kind == "repeated":
        Y[r.random((heads, n)) < 0.9] = 0.0
    elif kind == "two values":
        Y = np.where(Y > 0.3, np.float32(2.0), np.float32(-1.0))
    elif kind == "huge":
        Y[:, 5::7] *= np.float32(1e25)
        Y[:, 3::4] *= np.float32(1e-30)
    return Y


@pytest.mark.parametrize("kind,heads,n,d,c", [
    ("normal", 1, 4096, 64, 128), ("normal", 1, 4097, 128, 128), ("normal", 40, 4096, 128, 128),
    ("normal", 90, 515, 64, 16), ("normal", 2, 513, 128, 16),
    ("outliers", 1, 4096, 128, 256), ("outliers", 80, 1030, 64, 64), ("outliers", 40, 2000, 128, 64),
    ("repeated", 2, 4095, 64, 128), ("repeated", 80, 700, 128, 32),
    ("two values", 1, 4096, 64, 128), ("huge", 1, 2049, 64, 64), ("huge", 80, 600, 128, 64),
    # subtrees of at most 512 rows, of 1,024, and one row more; 512 threads and 256
    ("normal", 1, 513, 128, 64), ("normal", 24, 1536, 64, 64), ("outliers", 25, 1537, 128, 64), ("normal", 148, 1024, 64, 128),
    ("repeated", 149, 1024, 128, 64), ("two values", 75, 2049, 64, 256),
])
def test_subtrees_match_the_oracle(kind, heads, n, d, c):
    Y = _coordinates(kind, heads, n, d, n + d)
    p = binding.make_problem(1, heads, n, n, d, "bf16", c, c, 1, flags=binding.CA_Y_IN)
    plan = binding.Plan(p, DEV)
    X = torch.zeros((1, heads, n, d), dtype=torch.bfloat16, device=DEV)
    Yd = torch.from_numpy(Y[None]).to(DEV)
    plan.cluster_qk(X, X, X, Yq=Yd, Yk=Yd)
    torch.cuda.synchronize()
    assert all(v == 0 for v in plan.last_status().values())
    for h in sorted({0, heads // 2, heads - 1}):
        ref = orc.recursive_split_f32(Y[h], c)
        assert np.array_equal(plan.perm_q[0, h].cpu().numpy(), ref), f"queries, head {h}"
        assert np.array_equal(plan.perm_k[0, h].cpu().numpy(), ref), f"keys, head {h}"


@pytest.mark.parametrize("heads,n,d,c", [(2, 3000, 64, 16), (40, 6000, 128, 32), (1, 20000, 64, 16)])
def test_split_coordinates_beyond_the_coordinate_major_ones(heads, n, d, c):
    """Isotropic rows: small subsets split along any of the d coordinates."""
    g = torch.Generator(device=DEV)
    g.manual_seed(n)
    X = torch.randn((3, 1, heads, n, d), generator=g, device=DEV).to(torch.bfloat16)
    plan = binding.Plan(binding.make_problem(1, heads, n, n, d, "bf16", c, c, 1), DEV)
    Yq = torch.empty((1, heads, n, d), device=DEV)
    Yk = torch.empty((1, heads, n, d), device=DEV)
    plan.cluster_qk(X[0], X[1], X[2], Yq=Yq, Yk=Yk)
    torch.cuda.synchronize()
    assert all(v == 0 for v in plan.last_status().values())
    for h in sorted({0, heads - 1}):
        assert np.array_equal(plan.perm_q[0, h].cpu().numpy(), orc.recursive_split_f32(Yq[0, h].cpu().numpy(), c))
        assert np.array_equal(plan.perm_k[0, h].cpu().numpy(), orc.recursive_split_f32(Yk[0, h].cpu().numpy(), c))


@pytest.mark.parametrize("kind,heads,n,d,c", [
    ("normal", 1, 4097, 64, 64), ("normal", 20, 8193, 128, 128), ("normal", 2, 65537, 64, 128),
    ("normal", 1, 140000, 64, 128),                       # slices of more than 8,192 rows
    ("outliers", 2, 30000, 64, 128), ("repeated", 2, 30000, 64, 128), ("repeated", 1, 4200, 128, 128),
    ("two values", 1, 70000, 64, 256), ("two values", 40, 4500, 64, 128),
    ("normal", 1, 200003, 64, 256), ("repeated", 1, 200003, 64, 256),   # slices beyond shared memory
])
def test_levels_of_large_sets_match_the_oracle(kind, heads, n, d, c):
    """The same through the per-level kernel: one CTA per set up to eight, thresholds from a bin, from
    the digits, and among equal keys whose positions lie in several CTAs."""
    test_subtrees_match_the_oracle(kind, heads, n, d, c)


def _choose_among_numbers(sub):
    """The float32 choice with a variance that is not a number below every other."""
    _, var = orc.choose_coordinate_f32(sub)
    return int(np.argmax(np.where(np.isnan(var), np.float32(-1.0), var))), var


@pytest.mark.parametrize("heads,n,d,c,columns", [
    (2, 4096, 64, 64, [0, 5, 18, 40]), (2, 1500, 128, 16, [1, 2, 64, 127]), (40, 2000, 128, 64, [0, 8, 31, 90]),
    (1, 30000, 64, 128, [3, 16, 33, 63]), (1, 20000, 128, 64, [0, 1, 70]), (2, 5000, 64, 32, range(64)),
])
@pytest.mark.filterwarnings("ignore:invalid value")
def test_coordinates_with_infinities(heads, n, d, c, columns):
    """Infinite coordinates give variances that are not numbers, beside ones that are: those columns are not
    chosen (the first column where no variance is a number), whichever lanes hold them."""
    r = np.random.default_rng(n + d)
    Y = (r.standard_normal((heads, n, d)) * r.uniform(0.5, 2.0, d)).astype(np.float32)
    for t in columns:
        rows = r.random((heads, n)) < 0.2
        Y[:, :, t][rows] = np.where(r.random(int(rows.sum())) < 0.5, np.inf, -np.inf)
    p = binding.make_problem(1, heads, n, n, d, "bf16", c, c, 1, flags=binding.CA_Y_IN)
    plan = binding.Plan(p, DEV)
    X = torch.zeros((1, heads, n, d), dtype=torch.bfloat16, device=DEV)
    Yd = torch.from_numpy(Y[None]).to(DEV)
    plan.cluster_qk(X, X, X, Yq=Yd, Yk=Yd)
    torch.cuda.synchronize()
    assert all(v == 0 for v in plan.last_status().values())
    for h in sorted({0, heads - 1}):
        ref = orc.recursive_split(Y[h], c, choose=_choose_among_numbers)
        assert np.array_equal(plan.perm_q[0, h].cpu().numpy(), ref), f"queries, head {h}"
        assert np.array_equal(plan.perm_k[0, h].cpu().numpy(), ref), f"keys, head {h}"
