"""Inputs whose covariance is not a number (infinities, NaN, values whose sums leave float32): the principal
components of that matrix are lost, every index stays in range, and the other matrices or heads of the call come out as without it."""
import numpy as np
import pytest
import torch

from paper_2608_26965_b200 import binding

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


@pytest.mark.parametrize("d", [64, 128])
def test_matrices_that_are_not_numbers(d):
    r = np.random.default_rng(d)
    X = r.standard_normal((12, 300, d)) * r.uniform(0.1, 2.0, d)
    clean = np.einsum("hni,hnj->hij", X, X) / 300
    A = np.concatenate([clean, clean])
    A[0] = np.nan
    A[2, 5, 9] = A[2, 9, 5] = np.nan
    A[4, d // 2, d // 2] = np.inf
    A[6, 3] = A[6, :, 3] = -np.inf
    A[8] *= 1e38                                         # products overflow
    A[10, d - 1, d - 1] = np.nan
    bad = [0, 2, 4, 6, 8, 10]
    W, ev = binding.debug_eigh(torch.from_numpy(A).to(DEV))
    W0, ev0 = binding.debug_eigh(torch.from_numpy(clean).to(DEV))
    torch.cuda.synchronize()
    good = [i for i in range(24) if i not in bad]
    assert torch.equal(W[good], torch.cat([W0, W0])[good]) and torch.equal(ev[good], torch.cat([ev0, ev0])[good])


@pytest.mark.parametrize("dtype,d", [("fp32", 64), ("bf16", 64), ("fp32", 128), ("bf16", 128)])
@pytest.mark.parametrize("value", [float("nan"), float("inf"), 1e25])
def test_heads_with_rows_that_are_not_numbers(dtype, d, value):
    n, c, heads = 1500, 64, 6
    g = torch.Generator(device=DEV)
    g.manual_seed(d)
    X = torch.randn((3, 1, heads, n, d), generator=g, device=DEV).to(torch.float32 if dtype == "fp32" else torch.bfloat16)
    plan = binding.Plan(binding.make_problem(1, heads, n, n, d, dtype, c, c, 4), DEV)
    O = plan.forward(*X).clone()
    clean = plan.perm_q.clone(), plan.perm_k.clone()
    B = X.clone()
    B[0, 0, 1, 700, 3] = value                           # a query of head 1, a key of head 2, both in head 4
    B[1, 0, 2, :, 7] = value
    B[0, 0, 4, ::3] = value
    B[1, 0, 4, 11] = value
    O_bad = plan.forward(*B)
    torch.cuda.synchronize()
    assert all(v == 0 for v in plan.last_status().values())
    rows = torch.arange(n, device=DEV, dtype=torch.int32).expand(heads, n)
    for perm, before in zip((plan.perm_q[0], plan.perm_k[0]), clean):
        assert torch.equal(perm.sort(dim=1).values, rows)
        assert torch.equal(perm[[0, 3, 5]], before[0, [0, 3, 5]])
    assert torch.equal(O_bad[0, [0, 3, 5]], O[0, [0, 3, 5]])
