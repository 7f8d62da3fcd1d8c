"""The tensor-core attention kernel at the edges of its walk over tiles and steps: tiles of one to four
steps (fewer than its softmax groups, and one more), several tiles per CTA, lists without a key, key
clusters of every size against query clusters of every size, short last clusters.  Compared with the
library's fp32 kernel on the same clustering, which itself is compared with float64 sums at each of its tile widths."""
import ctypes

import pytest
import torch

from oracle import clusterattn_oracle as orc
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


@pytest.mark.parametrize("dtype", ["fp32", "bf16"])
@pytest.mark.parametrize("d,c_q,c_k,heads,n_q,n_k,compensate", [
    (64, 16, 32, 3, 16 * 9 - 5, 32 * 6 - 7, True), (128, 16, 16, 2, 16 * 5, 16 * 20 - 3, False),      # tiles of 16 rows
    (128, 16, 256, 1, 33, 700, True),
    (64, 32, 64, 2, 32 * 4 - 31, 64 * 5, True), (128, 32, 32, 1, 100, 32 * 9 - 1, False),             # of 32
    (64, 256, 64, 1, 300, 64 * 4 - 9, True),
    (128, 64, 128, 5, 64 * 30 - 3, 128 * 3 - 60, True), (64, 128, 32, 3, 128 * 26, 32 * 8, False),    # of 64: from 148 tiles on
    # fp32 storage: tiles of 8 and 16 rows while there is an SM for each, then 32, with 64 keys and 32
    (64, 64, 64, 2, 64 * 9 - 5, 64 * 5 - 9, True), (64, 64, 128, 2, 64 * 10 - 9, 128 * 4 - 77, False), (128, 64, 64, 2, 64 * 10 - 9, 64 * 6 - 1, True),
    (64, 128, 64, 3, 128 * 7 - 5, 64 * 6 - 9, True), (128, 128, 256, 2, 128 * 10, 256 * 3 - 100, True),
    (128, 128, 64, 5, 128 * 16 - 3, 64 * 5 - 7, True),
    # ... 16 rows and 32 keys where there are many CTAs; 32 rows by way of registers
    (64, 16, 32, 5, 16 * 60 - 3, 32 * 5 - 9, True), (64, 64, 32, 3, 64 * 30 - 1, 32 * 5 - 3, True), (128, 64, 32, 3, 64 * 30 - 1, 32 * 4, False),
])
def test_fp32_kernel_against_float64(d, c_q, c_k, heads, n_q, n_k, compensate, dtype):
    Qp, Kp, Vp, ck, cv, count, perm, lists = _clustering(heads, n_q, n_k, d, c_q, c_k, d + c_q + c_k + n_q)
    if dtype == "fp32":
        Qp, Kp, Vp = Qp.float(), Kp.float(), Vp.float()
    n_qc, n_kc = lists.shape[2:]
    keep = torch.arange(heads * n_qc, device=DEV).remainder(5).reshape(1, heads, n_qc).clamp(max=n_kc).int().contiguous()
    rows = torch.arange(n_kc, device=DEV)
    idx = torch.where(rows < keep[..., None], lists, n_kc + 1).sort(-1).values
    idx = torch.where(rows < keep[..., None], idx, -1).int().contiguous()
    plan = binding.Plan(binding.make_problem(1, heads, n_q, n_k, d, dtype, c_q, c_k, 1, compensate, flags=binding.CA_ATTN_FP32), DEV)
    O, lse = plan.cluster_attention_fwd_ragged(idx, keep, Qp, Kp, Vp, ck, cv, count, perm)
    torch.cuda.synchronize()
    assert plan.last_status()["attn"] == 0
    # every key and every centroid as columns, masked per query cluster
    kept = torch.zeros((heads, n_qc, n_kc + 2), dtype=torch.bool, device=DEV).scatter_(2, torch.where(idx[0] < 0, n_kc, idx[0]).long(), True)
    kept = kept[:, :, :n_kc]
    pos = torch.arange(n_kc * c_k, device=DEV)
    member = kept[:, :, pos // c_k] & (pos < n_k)
    cluster = torch.arange(n_qc * c_q, device=DEV) // c_q
    scale = 1.0 / d ** 0.5
    x = torch.cat([Qp[0].double() @ Kp[0].double().mT, Qp[0].double() @ ck[0].double().mT], dim=2) * scale
    x[:, :, n_kc * c_k:] += count[0, :, None].double().log()
    live = torch.cat([member[:, cluster], ~kept[:, cluster] & compensate], dim=2)
    x = x.masked_fill(~live, -torch.inf)
    want_lse = x.logsumexp(2)[:, :n_q]
    w = (x - x.logsumexp(2, keepdim=True)).exp().nan_to_num(0.0)
    want = (w @ torch.cat([Vp[0], cv[0]], dim=1).double())[:, :n_q]
    back = perm[0].long()
    got, got_lse = O[0].double().gather(1, back[..., None].expand(-1, -1, d)), lse[0].double().gather(1, back)
    empty = torch.isneginf(want_lse)
    assert torch.equal(torch.isneginf(got_lse), empty) and bool((got[empty] == 0).all())
    # float32 sums of up to d products and of all columns; results rounded to 2^-9 in bf16 storage
    assert (got - want).norm() <= (1e-5 if dtype == "fp32" else 4e-3) * want.norm()
    assert (got_lse - want_lse)[~empty].abs().max() <= 2e-5


@pytest.mark.parametrize("n_kc,c_q", [(2 ** 20 + 37, 16), (1_640_000, 64)])
def test_fp32_kernel_with_very_many_key_clusters(n_kc, c_q):
    """More key clusters than the bitmap of the selected ones covers at a time, with selected ones at the edges of its windows."""
    d, c_k, n_q = 64, 16, 61
    g = torch.Generator(device=DEV)
    g.manual_seed(c_q)
    n_qc = -(-n_q // c_q)
    Qp = torch.zeros((n_qc * c_q, d), dtype=torch.bfloat16, device=DEV)
    Qp[:n_q] = torch.randn((n_q, d), generator=g, device=DEV).to(torch.bfloat16)
    Kp, Vp = (torch.randn((n_kc * c_k, d), generator=g, device=DEV, dtype=torch.bfloat16) for _ in range(2))
    ck, cv = (torch.randn((n_kc, d), generator=g, device=DEV) for _ in range(2))
    count = torch.full((n_kc,), c_k, dtype=torch.int32, device=DEV)
    picked = [0, 31, 2 ** 20 - 1, 2 ** 20, 2 ** 20 + 32, n_kc - 1]
    idx = torch.tensor(picked, dtype=torch.int32, device=DEV).expand(n_qc, -1).contiguous()
    perm = torch.randperm(n_q, generator=g, device=DEV).int()
    O = torch.empty((n_q, d), dtype=torch.bfloat16, device=DEV)
    lse = torch.empty((n_q,), device=DEV)
    ws = torch.zeros((256,), dtype=torch.uint8, device=DEV)
    p = binding.make_problem(1, 1, n_q, n_kc * c_k, d, "bf16", c_q, c_k, len(picked), True)
    rc = binding.load_library().cluster_attention_fwd(
        ctypes.byref(p), *[ctypes.c_void_p(t.data_ptr()) for t in (Qp, Kp, Vp, ck, cv, count, idx, perm, O, lse, ws)], 256, None)
    assert rc == binding.CA_OK
    torch.cuda.synchronize()
    assert binding.load_library().ca_last_status(ctypes.c_void_p(ws.data_ptr())) == 0
    q = Qp[:n_q].double()
    rows = (idx[0].long()[:, None] * c_k + torch.arange(c_k, device=DEV)).flatten()
    cen = (q @ ck.double().mT) / d ** 0.5 + count.double().log()
    cen[:, idx[0].long()] = -torch.inf
    x = torch.cat([(q @ Kp[rows].double().mT) / d ** 0.5, cen], dim=1)
    want_lse = x.logsumexp(1)
    want = (x - want_lse[:, None]).exp() @ torch.cat([Vp[rows].double(), cv.double()])
    got, got_lse = O.double()[perm.long()], lse.double()[perm.long()]
    # results rounded to 2^-9; float32 sums of up to 1.6 million terms, 32 at a time
    assert (got - want).norm() <= 4e-3 * want.norm()
    assert (got_lse - want_lse).abs().max() <= 1e-3


@pytest.mark.parametrize("compensate", [False, True])
@pytest.mark.parametrize("d,c_q,c_k,keep", [(64, 64, 64, 3), (128, 64, 128, 2), (128, 64, 256, 1), (64, 64, 16, 9),
                                            (64, 128, 64, 4), (128, 256, 128, 3)])
def test_values_with_infinities(d, c_q, c_k, keep, compensate):
    """An infinite value makes the outputs that attend to it infinite (NaN where both signs meet), and those that do
    not stay as they are: as from the fp32 kernel."""
    heads, n_q, n_k = 2, c_q * 5 - 3, c_k * 12 - 5
    Qp, Kp, Vp, ck, cv, count, perm, lists = _clustering(heads, n_q, n_k, d, c_q, c_k, d + c_q + c_k)
    n_kc = lists.shape[3]
    idx = lists[..., :keep].sort(-1).values.contiguous()
    Vp[0, 0, 3 * c_k + 5, 7] = torch.inf                 # in clusters 3 and 8 of head 0
    Vp[0, 0, 8 * c_k + c_k - 1, 7] = -torch.inf
    Vp[0, 0, 8 * c_k, d - 1] = -torch.inf
    out = []
    for flags in (0, binding.CA_ATTN_FP32):
        plan = binding.Plan(binding.make_problem(1, heads, n_q, n_k, d, "bf16", c_q, c_k, keep, compensate, flags=flags), DEV)
        out.append(plan.cluster_attention_fwd(Qp, Kp, Vp, ck, cv, count, idx, perm)[0].float())
        torch.cuda.synchronize()
        assert plan.last_status()["attn"] == 0
    (O, want) = out
    assert bool(torch.isinf(want).any()) and bool(torch.isfinite(want[0, 1]).all())
    for mask in (torch.isnan, torch.isposinf, torch.isneginf):
        assert torch.equal(mask(O), mask(want)), mask.__name__
    fine = torch.isfinite(want)
    assert (O - want)[fine].norm() <= 1e-2 * want[fine].norm()


@pytest.mark.parametrize("compensate", [False, True])
@pytest.mark.parametrize("heads", [9, 2])
@pytest.mark.parametrize("d,c_k,infinite", [(64, 64, False), (64, 16, False), (128, 32, False), (128, 64, False), (64, 128, False), (128, 256, False),
                                            (64, 64, True), (128, 128, True)])
def test_pairs_of_64_row_query_clusters(d, c_k, infinite, compensate, heads):
    """More 64-row query clusters than SMs go two to a tile, with the key clusters of both lists taken once: lists that
    share everything, something and nothing, of the same and of very different lengths, empty ones, in any order, with a
    cluster twice, an odd number of clusters per head.  Fewer stand in both halves of a tile, each with half of the keys."""
    n_qc, n_kc = 35, 45
    n_q, n_k = 64 * n_qc - 17, c_k * n_kc - 5
    Qp, Kp, Vp, ck, cv, count, perm, lists = _clustering(heads, n_q, n_k, d, 64, c_k, d + c_k)
    if infinite:
        Vp[0, :, 3 * c_k + 5, 7] = torch.inf
        Vp[0, :, 8 * c_k, d - 1] = -torch.inf
    even = lists[:, :, ::2].repeat_interleave(2, dim=2)[:, :, :n_qc]      # both clusters of a pair have one order
    kind = torch.arange(heads * n_qc, device=DEV).reshape(1, heads, n_qc) // 2 % 5
    keep = torch.tensor([9, 14, 5, 9, 0], device=DEV)[kind] + torch.arange(n_qc, device=DEV) % 2 * torch.tensor([0, 3, 0, 20, 4], device=DEV)[kind]
    idx = torch.where((kind % 5 == 2)[..., None], lists, even)      # kind 2: unrelated lists
    idx = torch.where(((kind == 3) & (torch.arange(n_qc, device=DEV) % 2 == 1))[..., None], even.roll(-4, -1), idx)     # kind 3: shifted
    idx[:, 1::3, 3, 0] = idx[:, 1::3, 3, 1]                               # a cluster twice
    keep[:, 1::3, 3] = 37                                                 # (and others behind it in the list's second 32)
    idx, keep = idx.int().contiguous(), keep.int().contiguous()
    out = []
    for flags in (0, binding.CA_ATTN_FP32):
        plan = binding.Plan(binding.make_problem(1, heads, n_q, n_k, d, "bf16", 64, c_k, 1, compensate, flags=flags), DEV)
        O, lse = plan.cluster_attention_fwd_ragged(idx, keep, Qp, Kp, Vp, ck, cv, count, perm)
        torch.cuda.synchronize()
        assert plan.last_status()["attn"] == 0
        out.append((O.float(), lse))
        if flags == 0 and not infinite:
            assert plan.recomputed_clusters() == 0
    (O, lse), (want, want_lse) = out
    for mask in (torch.isnan, torch.isposinf, torch.isneginf):
        assert torch.equal(mask(O), mask(want)), mask.__name__
    fine, live = torch.isfinite(want), ~torch.isneginf(want_lse)
    assert torch.equal(torch.isneginf(lse), ~live)
    # probabilities and value centroids are bf16 on one side (2^-9 each), results on both
    assert (O - want)[fine].norm() <= 1e-2 * want[fine].norm()
    assert (O - want)[fine].abs().max() <= 5e-2
    assert (lse - want_lse)[live].abs().max() <= 2e-3


@pytest.mark.parametrize("heads,n_qc", [(4, 73), (2, 3)])                 # two clusters to a tile, and one
def test_an_infinite_value_of_negligible_probability(heads, n_qc):
    """A key 100 below the row's largest logit: exp(-100) is not zero in float32 but is where subnormal numbers are flushed,
    and 0 x inf is NaN.  64-row query clusters whose outputs are not numbers are recomputed, also where both lists of a
    tile are the same."""
    d, n_kc, n_q = 64, 5, 64 * n_qc - 7
    Qp, Kp, Vp, ck, cv, count, perm, _ = _clustering(heads, n_q, 64 * n_kc, d, 64, 64, n_qc)
    Qp, Kp = 0.1 * Qp, 0.1 * Kp
    Qp[:, :, :n_q, 0] = 10.0
    Kp[:, :, 5, 0] = -80.0
    Vp[:, :, 5, 7] = torch.inf
    idx = torch.tensor([0, 3], dtype=torch.int32, device=DEV).expand(1, heads, n_qc, 2).contiguous()
    plan = binding.Plan(binding.make_problem(1, heads, n_q, 64 * n_kc, d, "bf16", 64, 64, 2, False), DEV)
    O = plan.cluster_attention_fwd(Qp, Kp, Vp, ck, cv, count, idx, perm)[0]
    torch.cuda.synchronize()
    assert plan.last_status()["attn"] == 0 and plan.recomputed_clusters() == heads * n_qc
    assert bool(torch.isposinf(O[..., 7]).all()) and int(torch.isinf(O).sum()) == heads * n_q


@pytest.mark.parametrize("c_k,compensate", [(64, True), (64, False), (128, True), (256, True)])
def test_quantised_pairs_of_64_row_query_clusters(c_k, compensate):
    """Quantised Q K^T with two 64-row query clusters to a tile: the scales go with the rows of either cluster and with the
    runs of 64 keys of shared, split and one-sided steps.  Rows, key clusters and centroids of very different size, and
    ones that are zero."""
    d, heads, n_qc, n_kc = 128, 9, 35, 45
    n_q, n_k = 64 * n_qc - 17, c_k * n_kc - 5
    Qp, Kp, Vp, _, cv, count, perm, lists = _clustering(heads, n_q, n_k, d, 64, c_k, c_k)
    g = torch.Generator(device=DEV)
    g.manual_seed(c_k)
    gain = lambda n: (2.0 * torch.rand((1, heads, n, 1), generator=g, device=DEV) - 1.0).exp()
    Qp = (Qp * gain(64 * n_qc)).bfloat16()
    Kp = (Kp * gain(n_kc).repeat_interleave(c_k, dim=2)).bfloat16()
    Qp[:, :, 70] = 0
    Kp[:, :, 4 * c_k:5 * c_k] = 0
    ck = (Kp.float().reshape(1, heads, n_kc, c_k, d).sum(3) / count[..., None]).contiguous()
    kind = torch.arange(heads * n_qc, device=DEV).reshape(1, heads, n_qc) // 2 % 4
    odd = torch.arange(n_qc, device=DEV) % 2
    keep = torch.tensor([9, 14, 5, 3], device=DEV)[kind] + odd * torch.tensor([0, 3, 0, 20], device=DEV)[kind]
    even = lists[:, :, ::2].repeat_interleave(2, dim=2)[:, :, :n_qc]
    idx = torch.where((kind == 2)[..., None], lists, even)                # the same lists, longer ones, unrelated ones
    idx, keep = idx.int().contiguous(), keep.int().contiguous()
    plan = binding.Plan(binding.make_problem(1, heads, n_q, n_k, d, "bf16", 64, c_k, 1, compensate, flags=binding.CA_ATTN_FP8_QK), DEV)
    O, lse = plan.cluster_attention_fwd_ragged(idx, keep, Qp, Kp, Vp, ck, cv, count, perm)
    torch.cuda.synchronize()
    assert plan.last_status()["attn"] == 0 and plan.recomputed_clusters() == 0
    pos, row = torch.arange(n_k, device=DEV), torch.arange(n_q, device=DEV)
    for h in (0, 4, 8):
        host = lambda t, n: t[0, h, :n].float().cpu().numpy()
        Qd, Kd, cd = (torch.from_numpy(a).to(DEV) for a in orc.quantize_qk(host(Qp, n_q), host(Kp, n_k), range(n_k), c_k, host(ck, n_kc)))
        kept = torch.zeros((n_qc, n_kc), dtype=torch.bool, device=DEV)
        kept.scatter_(1, idx[0, h].long(), torch.arange(n_kc, device=DEV) < keep[0, h, :, None])
        x = torch.cat([Qd @ Kd.T, Qd @ cd.T + count[0, h].double().log() * d ** 0.5], dim=1) / d ** 0.5
        x = x.masked_fill(~torch.cat([kept[:, pos // c_k], ~kept & compensate], dim=1)[row // 64], -torch.inf)
        want_lse = x.logsumexp(1)
        want = (x - want_lse[:, None]).exp() @ torch.cat([Vp[0, h, :n_k], cv[0, h]]).double()
        got, got_lse = O[0, h].double()[perm[0, h].long()], lse[0, h].double()[perm[0, h].long()]
        # the codes and their products are the same on both sides; probabilities, value centroids and results are bf16
        assert (got - want).norm() <= 1e-2 * want.norm() and (got - want).abs().max() <= 5e-2
        assert (got_lse - want_lse).abs().max() <= 2e-3
