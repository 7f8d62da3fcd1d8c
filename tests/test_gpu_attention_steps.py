"""The tensor-core attention kernel at the edges of its walk over tiles and steps: tiles of one to four
steps (fewer than its softmax groups, and one more), several tiles per CTA, lists without a key, key
clusters of every size against query clusters of every size, short last clusters.  Compared with the
library's fp32 kernel on the same clustering."""
import pytest
import torch

from paper_2608_26965_b200 import binding

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


def _clustering(heads, n_q, n_k, d, c_q, c_k, seed):
    g = torch.Generator(device=DEV)
    g.manual_seed(seed)
    n_qc, n_kc = -(-n_q // c_q), -(-n_k // c_k)

    def padded(n, c, gain):
        x = torch.zeros((1, heads, -(-n // c) * c, d), device=DEV)
        x[:, :, :n] = gain * torch.randn((1, heads, n, d), generator=g, device=DEV)
        return x.to(torch.bfloat16)

    Qp, Kp, Vp = padded(n_q, c_q, 1.5), padded(n_k, c_k, 1.5), padded(n_k, c_k, 1.0)
    size = (n_k - torch.arange(n_kc, device=DEV) * c_k).clamp(max=c_k)
    mean = lambda x: x.float().reshape(1, heads, n_kc, c_k, d).sum(3) / size[:, None]
    count = size.int().expand(1, heads, n_kc).contiguous()
    perm = torch.stack([torch.randperm(n_q, generator=g, device=DEV) for _ in range(heads)]).int()[None].contiguous()
    lists = torch.rand((1, heads, n_qc, n_kc), generator=g, device=DEV).argsort(-1).int()
    return Qp, Kp, Vp, mean(Kp).contiguous(), mean(Vp).contiguous(), count, perm, lists


@pytest.mark.parametrize("d,c_q,c_k,heads,n_q,n_k,compensate", [
    (64, 64, 64, 7, 64 * 60 - 1, 64 * 9 - 63, True),      # three tiles per CTA, 64-row query clusters
    (64, 128, 128, 7, 128 * 60 - 5, 128 * 7 - 100, False),
    (64, 128, 16, 2, 300, 16 * 70 - 3, True),             # eight boxes per step, a partial centroid step
    (128, 64, 128, 3, 64 * 5, 128 * 6, False),            # the lower half of a tile sees keys 64-127 only
    (128, 64, 256, 2, 500, 256 * 3 - 200, True),
    (128, 256, 32, 5, 256 * 17 - 130, 32 * 20 - 31, True),  # two tiles per query cluster, the last one partly empty
])
def test_tiles_of_few_steps_and_many_tiles(d, c_q, c_k, heads, n_q, n_k, compensate):
    Qp, Kp, Vp, ck, cv, count, perm, lists = _clustering(heads, n_q, n_k, d, c_q, c_k, d + c_q + c_k)
    n_qc, n_kc = lists.shape[2:]
    # list lengths 0 .. 4 and the whole row, side by side
    keep = torch.arange(heads * n_qc, device=DEV).remainder(6).reshape(1, heads, n_qc)
    keep = torch.where(keep == 5, n_kc, keep).clamp(max=n_kc).int().contiguous()
    rows = torch.arange(n_kc, device=DEV)
    idx = torch.where(rows < keep[..., None], lists, n_kc + 1).sort(-1).values
    idx = torch.where(rows < keep[..., None], idx, -1).int().contiguous()
    out = []
    for flags in (0, binding.CA_ATTN_FP32):
        p = binding.make_problem(1, heads, n_q, n_k, d, "bf16", c_q, c_k, 1, compensate, flags=flags)
        plan = binding.Plan(p, DEV)
        O, lse = plan.cluster_attention_fwd_ragged(idx, keep, Qp, Kp, Vp, ck, cv, count, perm)
        torch.cuda.synchronize()
        assert plan.last_status()["attn"] == 0
        out.append((O.float(), lse))
        if flags == 0:
            assert plan.recomputed_clusters() == 0
    (O, lse), (o_ref, lse_ref) = out
    empty = torch.isneginf(lse_ref)
    assert torch.equal(torch.isneginf(lse), empty)
    assert (O[empty] == 0).all()
    # probabilities and value centroids are bf16 on one side (2^-9 each), results on both
    assert (O - o_ref).norm() <= 1e-2 * o_ref.norm()
    assert (O - o_ref).abs().max() <= 5e-2
    assert (lse - lse_ref)[~empty].abs().max() <= 2e-3
