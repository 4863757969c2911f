"""The fp32 scoring kernels at the sizes where they can go wrong: key tiles of 128 (64 at head_dim 256) and their remainders,
every height of the row tile and its remainders, requests of different lengths in one launch, both element types, and both
routes: exponentials kept (chunks of heads), and the product done twice (no room; a head too long to be kept; the entry
point with fixed scratch).

Bound: a logit is a sum of d products in fp32, off by at most d 2^-24 of sum_t |q_t k_t| scale, about 0.64 sqrt(d) for normal
q and k; half as much again for the fluctuation of that sum, and twice (the row's normaliser is as far off). The exponentials
and the sums over at most 1024 rows add 2^-19."""
import numpy as np
import pytest
import torch

from paper_2604_06694_b200 import workloads as wl
from helpers import oracle_scores, rel_err, to_dev

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def B():
    from paper_2604_06694_b200 import build as akv_build
    akv_build.build()
    from paper_2604_06694_b200 import binding
    return binding


def _bound(d):
    return 2 * 1.5 * d * 2.0 ** -24 * 0.64 * np.sqrt(d) + 2.0 ** -19


def _check(w, g):
    assert np.isfinite(g).all()
    off = 0
    for r in range(len(w.spec.seq_lens)):
        o, _ = oracle_scores(w, r)
        gr = g[off:off + o.size].reshape(o.shape)
        off += o.size
        for l in range(o.shape[0]):
            for h in range(o.shape[1]):
                assert rel_err(gr[l, h], o[l, h]) <= _bound(w.spec.head_dim), (r, l, h)
    assert off == g.size


# (window, query heads per KV head): W * G = 1, 15, 16, 63, 64, 65, 112, 113, 128, 129, 224, 225, 1024
ROWS = [(1, 1), (5, 3), (16, 1), (9, 7), (32, 2), (13, 5), (16, 7), (113, 1), (32, 4), (43, 3), (32, 7), (45, 5), (128, 8)]


@pytest.mark.parametrize("W,G", ROWS)
@pytest.mark.parametrize("d", [64, 128, 256])
def test_score_f32_rows(B, W, G, d):
    lens = [W + 1, W + 63, W + 64, 65, 128, 129, 300]      # a tile less, full and one key more; several
    lens = [max(W + 1, L) for L in lens]
    w = wl.generate(wl.WorkloadSpec("fma", "f32", 1, 2 * G, 2, d, lens, [0.8] * len(lens), 0, window=W), seed=W * G + d)
    prob = B.Problem.from_workload(w)
    ctx = B.Context(prob)
    scores = torch.full((B.audiokv_scores_len(prob),), float("nan"), device="cuda")
    B.audiokv_score(ctx, prob, to_dev(w, w.q), to_dev(w, w.k), scores)
    torch.cuda.synchronize()
    assert ctx.last_score_path() == "fma" and ctx.last_device_status() == 0
    _check(w, scores.cpu().numpy())


def test_score_f32_chunks_of_heads(B):
    """Forty heads of 3.4 MB of exponentials and statistics each go through at once where the workspace has room for them, in
    chunks of seven and one of five where it has room for seven, and with the product done twice where it has none. What
    is kept does not depend on the chunks to the last bit."""
    w = wl.generate(wl.WorkloadSpec("fma", "f32", 10, 28, 4, 64, [3700], [0.8], 0, window=32), seed=4)
    prob = B.Problem.from_workload(w)
    head = 29 * 224 * (128 * 4 + 8)                 # 29 tiles of 128 keys, 224 rows
    need = B.audiokv_workspace_bytes(prob) - 40 * head
    q, k = to_dev(w, w.q), to_dev(w, w.k)
    S, tb = torch.from_numpy(w.head_scores).cuda(), [int(x) for x in w.total_budget]
    results = []
    for heads, launches in ((40, 3), (7, 18), (0, 3)):
        ctx = B.Context(prob, workspace_bytes=need + heads * head)
        scores = torch.full((B.audiokv_scores_len(prob),), float("nan"), device="cuda")
        for _ in range(2):                          # the first call brings the plan
            before = ctx.launch_count()
            B.audiokv_score(ctx, prob, q, k, scores)
        assert ctx.launch_count() - before == launches
        kept = [torch.zeros((tb[0], 64), device="cuda"), torch.zeros((tb[0], 64), device="cuda"),
                *(torch.zeros(n, dtype=torch.int32, device="cuda") for n in (tb[0], 40, 41))]
        B.audiokv_evict(ctx, prob, q, k, k, S, tb, *kept)  # scoring beside the allocation
        torch.cuda.synchronize()
        assert ctx.last_device_status() == 0
        _check(w, scores.cpu().numpy())
        results.append((scores, kept[2]))
    assert torch.equal(results[0][0], results[1][0]) and torch.equal(results[0][1], results[1][1])
    with pytest.raises(B.AudioKVError) as e:
        B.audiokv_score(B.Context(prob, workspace_bytes=need - 256), prob, q, k, scores)
    assert e.value.status == B.AUDIOKV_EWORKSPACE


def test_profile_lists_every_kernel_of_a_long_pass(B):
    """Chunks of three heads make some 42 launches of the scoring alone; the profile ends with the gather."""
    w = wl.generate(wl.WorkloadSpec("fma", "f32", 10, 28, 4, 64, [3700], [0.8], 0, window=32), seed=4)
    prob = B.Problem.from_workload(w)
    head = 29 * 224 * (128 * 4 + 8)
    ctx = B.Context(prob, workspace_bytes=B.audiokv_workspace_bytes(prob) - 37 * head)
    q, k, tb = to_dev(w, w.q), to_dev(w, w.k), [int(x) for x in w.total_budget]
    out = [torch.zeros((tb[0], 64), device="cuda"), torch.zeros((tb[0], 64), device="cuda"),
           *(torch.zeros(n, dtype=torch.int32, device="cuda") for n in (tb[0], 40, 41))]
    ctx.profile_enable(True)
    for _ in range(2):                              # the first call brings the plan
        before = ctx.launch_count()
        B.audiokv_evict(ctx, prob, q, k, k, torch.from_numpy(w.head_scores).cuda(), tb, *out)
    prof = ctx.profile_read()
    assert len(prof) == ctx.launch_count() - before > 40
    assert prof[0][0] == "allocate" and prof[-1][0] == "gather" and all(ms >= 0 for _, ms in prof)


def test_score_f32_head_too_long_to_keep(B):
    """W * G = 1024 and 33000 keys: 135 MB of exponentials for one head, so the product is done twice."""
    w = wl.generate(wl.WorkloadSpec("fma", "f32", 1, 8, 1, 64, [33000], [0.8], 0, window=128), seed=6)
    prob = B.Problem.from_workload(w)
    ctx = B.Context(prob)
    scores = torch.full((B.audiokv_scores_len(prob),), float("nan"), device="cuda")
    B.audiokv_score(ctx, prob, to_dev(w, w.q), to_dev(w, w.k), scores)
    torch.cuda.synchronize()
    _check(w, scores.cpu().numpy())


@pytest.mark.parametrize("dtype,W,G,d", [("f32", 32, 7, 128), ("bf16", 32, 7, 128), ("bf16", 9, 7, 64), ("bf16", 33, 4, 256)])
def test_score_noalloc_tiles(B, dtype, W, G, d):
    w = wl.generate(wl.WorkloadSpec("fma", dtype, 2, 2 * G, 2, d, [W + 1, 511, 512, 513, 1100], [0.8] * 5, 0, window=W), seed=9)
    prob = B.Problem.from_workload(w)
    scores = torch.full((B.audiokv_scores_len(prob),), float("nan"), device="cuda")
    B.audiokv_score_noalloc(prob, to_dev(w, w.q), to_dev(w, w.k), scores)
    torch.cuda.synchronize()
    _check(w, scores.cpu().numpy())
