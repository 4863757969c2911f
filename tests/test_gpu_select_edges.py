"""The selection inside the pass at the sizes where it can go wrong: word and warp remainders, both ways the work buffer holds
its keys (pairs for even lengths, singles for odd ones), a buffer on chip and in global memory, and keys that defeat the
first histogram: all equal, two values, a tight cluster under a far outlier. With alpha = 0 the smoothed scores are the
scores, so the kept tokens have to equal the oracle's selection from audiokv_score's output exactly, ties included."""
import numpy as np
import pytest
import torch

import oracle

pytestmark = pytest.mark.gpu
W = 8


@pytest.fixture(scope="module")
def B():
    from paper_2604_06694_b200 import build as akv_build
    akv_build.build()
    from paper_2604_06694_b200 import binding
    return binding


def _keys(kind, L, rng):
    k = rng.standard_normal((L, 64)).astype(np.float32) * 0.3
    if kind == "equal":
        k[:] = k[0]
    elif kind == "two":
        k[:] = k[rng.integers(0, 2, size=L)]
    elif kind == "cluster":
        k *= 1e-4
        k[L // 2] = 8.0
    return torch.from_numpy(k).to(torch.bfloat16).cuda()


@pytest.mark.parametrize("P", [1, 2, 31, 33, 64, 1023, 2049, 8160, 8161, 40001, 60000])
@pytest.mark.parametrize("kind", ["random", "equal", "two", "cluster"])
def test_selection_edges(B, P, kind):
    rng = np.random.default_rng(P)
    L = P + W
    k, q = _keys(kind, L, rng), torch.from_numpy(rng.standard_normal((W, 64)).astype(np.float32)).to(torch.bfloat16).cuda()
    prob = B.Problem(B.AUDIOKV_BF16, 1, 1, 1, 64, [L], W, (W * 64, W * 64, 64, 64), (L * 64, 64, L * 64), alpha=0.0)
    ctx = B.Context(prob)
    scores = torch.empty(P, device="cuda")
    B.audiokv_score(ctx, prob, q, k, scores)
    for keep in sorted({0, 1, P // 3, P // 2, P - 1, P}):
        total = W + keep
        ko, vo = (torch.zeros((total, 64), dtype=torch.bfloat16, device="cuda") for _ in range(2))
        kept = torch.full((total,), -1, dtype=torch.int32, device="cuda")
        bud, cu = (torch.zeros(n, dtype=torch.int32, device="cuda") for n in (1, 2))
        B.audiokv_evict(ctx, prob, q, k, k, torch.ones(1, device="cuda"), [total], ko, vo, kept, bud, cu)
        torch.cuda.synchronize()
        assert ctx.last_device_status() == 0
        want = np.concatenate([oracle.select(scores.cpu().numpy().astype(np.float64), keep), np.arange(P, L)])
        assert np.array_equal(kept.cpu().numpy(), want), (P, kind, keep)
