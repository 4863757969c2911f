"""Smoothing of ragged batches: a head's result must not depend on which heads its block had before it."""
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def B():
    from paper_2604_06694_b200 import build as akv_build
    akv_build.build()
    from paper_2604_06694_b200 import binding
    return binding


def _problem(B, heads, prefixes, **kw):
    W, d = 32, 64
    lens = [P + W for P in prefixes]
    return B.Problem(B.AUDIOKV_BF16, heads, 1, 1, d, lens, W, (heads * W * d, W * d, d, d),
                     (sum(lens) * d, d, sum(lens) * d), **kw)


def _smooth(B, prob, x):
    ctx = B.Context(prob)
    y, ks = torch.full_like(x, float("nan")), torch.full((prob.total_heads,), -1, dtype=torch.int32, device="cuda")
    B.audiokv_smooth(ctx, prob, x, y, ks)
    torch.cuda.synchronize()
    assert ctx.last_device_status() == 0
    return y, ks


@pytest.mark.parametrize("outer,inner", [(3604, 2703), (820, 882)])
def test_roots_of_one_plan_survive_the_heads_of_another(B, outer, inner):
    """Pairs of lengths of equal estimated cost, so that their requests are smoothed in the order they come in. With many more
    heads than blocks, a block meets a head of the first length that needs a transform, heads of the second that the first
    bins settle (their work buffer runs over the place of the first length's roots of unity), and the first length again."""
    heads, gen = 112, torch.Generator(device="cuda")
    gen.manual_seed(outer)
    parts = [1 + 0.05 * torch.randn((heads, inner), generator=gen, device="cuda") for _ in range(8)]
    for at in (0, len(parts) + 1):
        parts.insert(at, torch.exp(3 * torch.randn((heads, outer), generator=gen, device="cuda")))
    y, ks = _smooth(B, _problem(B, heads, [p.shape[1] for p in parts]), torch.cat([p.reshape(-1) for p in parts]))
    at = 0
    for r, p in enumerate(parts):
        alone, ks_alone = _smooth(B, _problem(B, heads, [p.shape[1]]), p.reshape(-1).contiguous())
        assert bool((ks_alone > 11).all() if p.shape[1] == outer else (ks_alone == 0).all())
        assert torch.equal(ks[r * heads:(r + 1) * heads], ks_alone)
        assert torch.equal(y[at:at + p.numel()], alone), f"request {r}"
        at += p.numel()
