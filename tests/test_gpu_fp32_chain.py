"""The chain of float32 storage from Q and K to the clusters at a size where rows lie close to split thresholds
(5,003 rows, d = 128), against the oracle's own chain in float64: coordinates column by column, and the split tree
down to its leaves.  A clustering is discrete, so a rounding moves a row that lies at a threshold; every
set at which the two trees part has to be of that kind, and such sets have to be rare."""
import numpy as np
import pytest
import torch

from oracle import clusterattn_oracle as orc
from paper_2608_26965_b200 import binding, inputs
from tests import decisions

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


def _grouped_rows(w, seed):
    """Rows of `components` groups per head, anisotropic inside a group: 15 leading components, all separated."""
    r = np.random.default_rng(seed)
    d, G = w.head_dim, w.components
    out = [np.empty((w.heads, n, d), np.float32) for n in (w.n_q, w.n_k)]
    for h in range(w.heads):
        means = r.standard_normal((G, d))
        means *= 3.0 * d ** 0.25 / np.linalg.norm(means, axis=1, keepdims=True)
        spread = 10.0 ** r.uniform(-0.5, 0.5, (G, d))
        spread *= 0.5 / np.sqrt((spread ** 2).mean(axis=1, keepdims=True))
        for x in out:
            g = r.integers(0, G, x.shape[1])
            x[h] = means[g] + r.standard_normal((x.shape[1], d)) * spread[g]
    return out


def test_clusters_of_float32_storage_follow_the_float64_chain():
    w = inputs.WORKLOADS["tiny"].scaled(heads=4, head_dim=128, n_q=5003, n_k=5003, cluster=128, keep=5, components=16)
    plan = binding.Plan(binding.problem_from_workload(w), DEV, keep_y=True)
    parted, sides = 0, 0
    for seed in (1, 2, 3):
        Q, K = _grouped_rows(w, seed)
        q, k = (torch.from_numpy(x[None]).to(DEV) for x in (Q, K))
        plan.cluster_qk(q, k, k)
        torch.cuda.synchronize()
        assert all(v == 0 for v in plan.last_status().values())
        for h in range(w.heads):
            label = f"float32 chain, inputs {seed}, head {h}"
            Y = [y[0, h].cpu().numpy() for y in (plan.Yq, plan.Yk)]
            perm = [p[0, h].cpu().numpy() for p in (plan.perm_q, plan.perm_k)]
            for y, p in zip(Y, perm):
                assert np.array_equal(p, orc.recursive_split_f32(y, w.cluster))
            if h == 0:
                decisions.check_coordinates(label, w, Q[h], K[h], Y[0], Y[1], perm[0], perm[1])
            for side, y, y_orc in zip(("queries", "keys"), Y, orc.split_coordinates(Q[h], K[h])):
                a = decisions.split_partings(y, y_orc, w.cluster)
                sides += 1
                parted += bool(a)
                for x in a:
                    print(label, side, x)
                    if x["t_dev"] != x["t_orc"]:        # each variance off by the error of its coordinate, and rounded
                        assert x["gap"] <= 1e-4
                    else:                               # the row and the threshold each move by at most the difference
                        assert x["distance"] <= 2 * x["key_difference"] + 1e-12
                        assert x["key_difference"] <= 2e-3
    # Of 12,000 sides of such inputs 53 part from the float64 chain (0.4 %; with an eigensolver of another order of
    # operations 106): of 24 sides more than two do by chance once in 6,000 runs.
    assert parted <= 2, f"{parted} of {sides} sides"
