"""The factors of rank-deficient metrics: which pivots drop out."""
import numpy as np
import pytest
import torch

from paper_2608_26965_b200 import binding, build

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


@pytest.fixture(scope="module", autouse=True)
def _lib():
    build.build()
    binding.load_library()


def _rows(r, n, d, at, direction, largest):
    """n rows +-a * direction on the coordinates `at`, zero elsewhere, of mean zero.  a is a power of two, so that its
    products with any factor are exact and those of opposite sign cancel."""
    X = np.zeros((n, d), np.float32)
    a = 2.0 ** r.integers(0, largest + 1, n // 2)
    X[:, at] = np.concatenate([a, -a])[:, None] * np.array(direction)
    return X[r.permutation(n)]


@pytest.mark.parametrize("dtype", ["fp32", "bf16"])
@pytest.mark.parametrize("d", [64, 128])
def test_one_dominant_direction_leaves_one_column(d, dtype):
    """Keys along (1, 1, 1) and queries along (1, -1, 0) of three coordinates: both metrics are of rank one, and each maps
    the other side's rows to zero, exactly.  The second pivot is zero or what rounding leaves of the first (its sign
    depends on the head's numbers); a factor that keeps it makes unit vectors of the queries' representations, which are
    normalised, and splits by them.  The three coordinates, those of the largest diagonal entries, stand all along the diagonal."""
    r = np.random.default_rng(7 + d)
    at = [(i, (i + 2) % d, (i + 4) % d) for i in range(0, d, 1 if d == 64 else 2)] + [(1, 3, 5)] * 24
    H, n_q, n_k = len(at), 130, 262
    Q = np.stack([_rows(r, n_q, d, list(x), (1, -1, 0), h % 4) for h, x in enumerate(at)])
    K = np.stack([_rows(r, n_k, d, list(x), (1, 1, 1), h % 3) for h, x in enumerate(at)])
    dt = torch.bfloat16 if dtype == "bf16" else torch.float32
    Q, K = (torch.from_numpy(x[None]).to(dt).to(DEV) for x in (Q, K))
    plan = binding.Plan(binding.make_problem(1, H, n_q, n_k, d, dtype, 16, 16, 2), DEV, keep_y=True)
    for _ in range(2):
        plan.cluster_qk(Q, K, K)
        torch.cuda.synchronize()
        assert all(v == 0 for v in plan.last_status().values())
        for Y, perm, n in ((plan.Yq, plan.perm_q, n_q), (plan.Yk, plan.perm_k, n_k)):
            wrong = [at[h] for h in range(H) if bool((Y[0, h] != 0).any())]
            assert not wrong, wrong
            assert torch.equal(perm, torch.arange(n, dtype=torch.int32, device=DEV).expand(1, H, n))
