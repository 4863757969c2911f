"""The head-score kernel at the row shapes where its paths part ways: rows shorter than a warp's worth of 16-byte pieces,
remainders before and after them, long rows, top_k around the limit of a warp's list and far above it, rows of so many
equal values that the list overflows, and more rows than one turn of the grid. Counts are whole numbers: they equal
the oracle's."""
import numpy as np
import pytest
import torch

import oracle

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def B():
    from paper_2604_06694_b200 import build as akv_build
    akv_build.build()
    from paper_2604_06694_b200 import binding
    return binding


@pytest.mark.parametrize("lens,K", [((1, 2, 31, 65), 1), ((66, 127, 128, 129, 133), 64), ((1025, 1026, 1027), 65),
                                    ((8191, 8192, 8193, 9001), 24), ((20011, 16384), 8), ((5000,), 63),
                                    ((2049, 31, 300, 33), 32), ((259, 4100), 33), ((8190, 1003), 1000)])
@pytest.mark.parametrize("kind", ["softmax", "steps"])
def test_hit_score_row_shapes(B, lens, K, kind):
    rng = np.random.default_rng(sum(lens) + K)
    H, width = 7, max(lens) + 1                     # an odd stride in places: rows start off the 16-byte grid
    attn = np.zeros((len(lens), H, width), dtype=np.float32)
    span = np.zeros((len(lens), 2), dtype=np.int32)
    for t, L in enumerate(lens):
        x = rng.standard_normal((H, L))
        if kind == "steps":                         # a handful of distinct values: ties decide by index
            x = np.round(x)
        attn[t, :, :L] = np.exp(x) / L
        span[t] = (L // 4, min(L - 1, L // 4 + 40))
    row_len = np.array(lens, dtype=np.int32)
    prob = B.Problem(B.AUDIOKV_BF16, 1, 4, 4, 64, [64], 8, (0, 0, 0, 0), (0, 64, 0))
    ctx = B.Context(prob)
    counts = torch.full((H,), -1, dtype=torch.int32, device="cuda")
    s = torch.full((H,), float("nan"), device="cuda")
    B.audiokv_hit_score(ctx, torch.from_numpy(attn).cuda(), torch.from_numpy(row_len).cuda(),
                        torch.from_numpy(span).cuda(), K, counts, s)
    torch.cuda.synchronize()
    want_s, want = oracle.hit_score(attn, row_len, span, K)
    assert np.array_equal(counts.cpu().numpy(), want)
    assert np.array_equal(s.cpu().numpy(), want_s.astype(np.float32))
    assert ctx.last_device_status() == 0


@pytest.mark.parametrize("K", [24, 65])
def test_hit_score_nan(B, K):
    """A NaN ranks above every number (below with its sign bit set), whichever way its row takes: among the 16-byte pieces
    or the single values before and after them, inside the span or pushing a number of the span out of the K largest."""
    rng = np.random.default_rng(K)
    L, places = 1003, (0, 2, 500, 1000, 1002)
    attn = np.exp(rng.standard_normal((1, 2 * len(places) + 1, L))).astype(np.float32)
    for i, j in enumerate(places):
        attn[0, 2 * i, j] = np.nan
        attn[0, 2 * i + 1, j] = -np.float32(np.nan)
    attn[0, -1, 100:140] = np.nan                   # more of them than the smaller K
    bits = attn.view(np.uint32)
    key = np.where(bits >> 31, ~bits, bits | 0x80000000).astype(np.uint32)
    for span in ((0, 120), (495, 510), (900, 1002)):
        order = np.argsort(-key[0].astype(np.int64), axis=1, kind="stable")[:, :K]
        want = ((order >= span[0]) & (order <= span[1])).sum(axis=1)
        ctx = B.Context(B.Problem(B.AUDIOKV_BF16, 1, 4, 4, 64, [64], 8, (0, 0, 0, 0), (0, 64, 0)))
        H = attn.shape[1]
        counts, s = torch.full((H,), -1, dtype=torch.int32, device="cuda"), torch.zeros(H, device="cuda")
        B.audiokv_hit_score(ctx, torch.from_numpy(attn).cuda(), torch.tensor([L], dtype=torch.int32, device="cuda"),
                            torch.tensor([span], dtype=torch.int32, device="cuda"), K, counts, s)
        torch.cuda.synchronize()
        assert np.array_equal(counts.cpu().numpy(), want)


@pytest.mark.parametrize("K", [8, 33])
def test_hit_score_many_short_rows(B, K):
    """100000 rows of 47 values are more than every block takes in one turn; a third of them are constant and left to the block."""
    rng = np.random.default_rng(K)
    T, H, L = 100, 1000, 47
    attn = rng.random((T, H, L), dtype=np.float32)
    attn[:, ::3] = 0.5
    row_len = np.full(T, L, dtype=np.int32)
    span = np.stack([np.arange(T) % 30, np.arange(T) % 30 + 12], axis=1).astype(np.int32)
    ctx = B.Context(B.Problem(B.AUDIOKV_BF16, 1, 4, 4, 64, [64], 8, (0, 0, 0, 0), (0, 64, 0)))
    counts, s = torch.full((H,), -1, dtype=torch.int32, device="cuda"), torch.zeros(H, device="cuda")
    B.audiokv_hit_score(ctx, torch.from_numpy(attn).cuda(), torch.from_numpy(row_len).cuda(),
                        torch.from_numpy(span).cuda(), K, counts, s)
    torch.cuda.synchronize()
    assert np.array_equal(counts.cpu().numpy(), oracle.hit_score(attn, row_len, span, K)[1])
