"""The gather that runs beside the smoothing, head by head: the pass must leave what its steps leave when they are called one by
one (their gather runs behind the selection), bit for bit, several times in a row on one context. Shapes: one head and
more heads than blocks, units of rows that are full, short by one and over by one, heads that keep their window alone or
everything, rows of 8 to 64 chunks, pages, ragged requests."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def B():
    from paper_2604_06694_b200 import build as akv_build
    akv_build.build()
    from paper_2604_06694_b200 import binding
    return binding


CASES = [  # layers, KV heads, head_dim, type, window, lengths, kept share, page
    (1, 1, 256, "bf16", 16, [90001], 0.6, 0),
    (150, 1, 64, "bf16", 8, [1531], 64 / 1531, 0),     # units of 64 rows
    (150, 1, 64, "bf16", 8, [1531], 65.5 / 1531, 0),   # one more
    (40, 4, 64, "bf16", 8, [97], 0.3, 0),
    (75, 2, 128, "bf16", 8, [40], 0.0, 0),             # the windows alone
    (38, 4, 128, "bf16", 16, [200], 1.0, 0),           # everything
    (25, 2, 256, "bf16", 16, [33, 3001, 1444], 0.37, 0),
    (20, 4, 256, "f32", 8, [1999], 0.5, 0),
    (30, 4, 64, "f32", 8, [131, 64], 0.25, 0),
    (40, 2, 128, "bf16", 16, [1407, 2050], 0.4, 16),
    (4, 2, 128, "bf16", 16, [1407, 2050], 0.4, 16),    # small: behind the selection
]


@pytest.mark.parametrize("layers,hkv,d,dtype,W,lens,share,page", CASES)
def test_pass_equals_its_steps(B, layers, hkv, d, dtype, W, lens, share, page):
    gen = torch.Generator(device="cuda").manual_seed(layers * 1000 + lens[0])
    dt = torch.float32 if dtype == "f32" else torch.bfloat16
    G, heads = 2, layers * hkv
    hq = G * hkv
    q = (3.0 * torch.randn((len(lens), layers, W, hq, d), generator=gen, device="cuda")).to(dt)
    more = {}
    if page:
        per = [-(-L // page) for L in lens]
        n_pages = sum(per)
        order = torch.randperm(n_pages, generator=gen, device="cuda").to(torch.int32)
        table = torch.full((len(lens), max(per)), -1, dtype=torch.int32, device="cuda")
        for r, n in enumerate(per):
            table[r, :n] = order[sum(per[:r]):sum(per[:r + 1])]
        rows = n_pages * page
        more = dict(page_size=page, n_pages=n_pages, page_table=table)
    else:
        rows = sum(lens)
        more = dict(kv_req_offset=[sum(lens[:r]) * d for r in range(len(lens))])
    k, v = (torch.randn((layers, hkv, rows, d), generator=gen, device="cuda").to(dt) for _ in range(2))
    prob = B.Problem(B.AUDIOKV_F32 if dtype == "f32" else B.AUDIOKV_BF16, layers, hq, hkv, d, lens, W,
                     (layers * W * hq * d, W * hq * d, hq * d, d), (hkv * rows * d, d, rows * d), **more)
    budget = [B.audiokv_budget_from_ratio(share, heads, L, W) for L in lens]
    S = torch.from_numpy(np.random.default_rng(1).beta(0.5, 2.0, size=(len(lens), heads)).astype(np.float32)).cuda()
    ctx, TH, total = B.Context(prob), prob.total_heads, sum(budget)

    def outputs():
        return [torch.full((total, d), 7.0, dtype=dt, device="cuda") for _ in range(2)] + [
            torch.full((n,), -1, dtype=torch.int32, device="cuda") for n in (total, TH, TH + 1)]

    ko, vo, kept, bud, cu = want = outputs()
    scores = torch.empty(B.audiokv_scores_len(prob), device="cuda")
    smoothed = torch.empty_like(scores)
    B.audiokv_score(ctx, prob, q, k, scores)
    B.audiokv_smooth(ctx, prob, scores, smoothed)
    B.audiokv_allocate(ctx, prob, S, budget, bud, cu)
    B.audiokv_select_gather(ctx, prob, smoothed, bud, cu, k, v, ko, vo, kept)
    for _ in range(3):
        got = outputs()
        B.audiokv_evict(ctx, prob, q, k, v, S, budget, *got)
        torch.cuda.synchronize()
        assert ctx.last_device_status() == 0
        for a, b in zip(got, want):
            assert torch.equal(a.view(torch.int16 if a.dtype == torch.bfloat16 else torch.int32),
                               b.view(torch.int16 if b.dtype == torch.bfloat16 else torch.int32))
