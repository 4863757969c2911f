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


@pytest.mark.parametrize("mode", [0, 2])
@pytest.mark.parametrize("n", [1000, 3001, 8160, 8161, 40000])
def test_cutoff_close_to_all_of_the_energy(B, n, mode):
    """rho near 1 on spectra that fall off: many bins share what is left above the cut-off. It is found against the transform's
    own total, so it may be off only by bins that hold less than a thousandth of that rest: a bin of the transform is off by
    some 1e-7 of the root mean square of all of them, one near these cut-offs is 1e-2 to 1e-3 of it. (Against
    a total of another source, 1e-7 of the whole energy away, the rest would be off by a tenth.)"""
    heads, gen = 32, torch.Generator(device="cuda")
    gen.manual_seed(n)
    f = torch.fft.rfft(torch.randn((heads, n), generator=gen, device="cuda").double(), dim=1)
    x = torch.fft.irfft(f / (1 + (torch.arange(n // 2 + 1, device="cuda") / 20) ** 2), n=n, dim=1)
    x = (x - x.amin() + 0.1 * x.std()).float().contiguous()
    e = torch.fft.rfft(x.double(), dim=1).abs() ** 2
    if mode == B.AUDIOKV_SMOOTH_ENERGY_NO_MEAN:
        e[:, 0] = 0
    cum = torch.cumsum(e, 1)
    rest = torch.flip(torch.cumsum(torch.flip(e, [1]), 1), [1]) - e      # energy above bin k
    for rho in (0.999, 0.9999, 0.99999, 0.999999):
        prob = _problem(B, heads, [n], rho=rho, smooth_mode=mode)
        _, ks = _smooth(B, prob, x.reshape(-1))
        left = (1 - float(prob.p.rho)) * cum[:, -1:]
        k = ks.long()[:, None]
        assert (rest.gather(1, k) <= left * 1.001).all(), rho
        assert (rest.gather(1, k - 1) > left * 0.999).all(), rho


@pytest.mark.parametrize("n", [500, 1001, 1021, 2042])
def test_cutoff_at_rho_one(B, n):
    """All of the energy is reached at the last bin, or at once where there is none."""
    x = torch.rand((2, n), device="cuda")
    x[1] = 0
    y, ks = _smooth(B, _problem(B, 2, [n], rho=1.0), x.reshape(-1))
    assert ks.tolist() == [n // 2, 0] and bool((y[n:] == 0).all())


@pytest.mark.parametrize("n", [17, 19, 51, 76, 323, 646, 4 * 17 * 19, 17 ** 3, 2 * 19 ** 3, 34 * 2048, 38 * 2048])
def test_radix_17_and_19(B, n):
    """One pass or several of either radix, on chip and (the longest two) on the global buffer, against the filter in 64 bits."""
    gen = torch.Generator(device="cuda")
    gen.manual_seed(n)
    x = torch.exp(torch.randn((2, n), generator=gen, device="cuda"))
    prob = _problem(B, 2, [n], rho=0.9, alpha=1.0, transition_bins=2)
    y, ks = _smooth(B, prob, x.reshape(-1))
    f = torch.fft.rfft(x.double(), dim=1)
    e = torch.cumsum(f.abs() ** 2, 1)
    i, k = torch.arange(n // 2 + 1, device="cuda"), ks.long()[:, None]
    thr = float(prob.p.rho) * e[:, -1:]
    assert (e.gather(1, k) >= thr * (1 - 1e-6)).all() and (e.gather(1, (k - 1).clamp_min(0)) < thr * (1 + 1e-6)).all()
    band = 0.5 * (1 + torch.cos(torch.pi * (i - k) / 3))
    want = torch.fft.irfft(f * torch.where(i <= k, 1.0, torch.where(i <= k + 2, band, 0.0)), n=n, dim=1)
    # a transform is off by some sqrt(passes) roundings of the norm, two transforms by 1e-6
    assert float((y.view(2, n) - want).norm() / want.norm()) < 1e-6


@pytest.mark.parametrize("n,window", [(600, 1023), (2047, 1), (8160, 7), (50000, 1023), (50001, 255), (131040, 7)])
@pytest.mark.parametrize("mode", [3, 4])
def test_pooling_in_stretches(B, n, window, mode):
    """Sequences shorter than the window, on chip, and in several stretches, into another array and in place: the sum of a window
    in 32 bits is off by at most its length in roundings of it, a maximum by none."""
    gen = torch.Generator(device="cuda")
    gen.manual_seed(n)
    x = torch.rand((2, n), generator=gen, device="cuda")
    prob = _problem(B, 2, [n], smooth_mode=mode, pool_kernel=window, alpha=1.0)
    y, ks = _smooth(B, prob, x.reshape(-1))
    if mode == B.AUDIOKV_SMOOTH_AVG_POOL:
        want = torch.nn.functional.avg_pool1d(x.double()[:, None], window, 1, window // 2)[:, 0]
        assert float((y.view(2, n) - want).abs().max()) <= window * 2.0 ** -24
    else:
        want = torch.nn.functional.max_pool1d(torch.nn.functional.pad(x, (window // 2, window // 2))[:, None], window, 1)
        assert torch.equal(y.view(2, n), want[:, 0])     # the values are positive: zeros never win
    ctx = B.Context(prob)
    B.audiokv_smooth(ctx, prob, x, x)
    torch.cuda.synchronize()
    assert torch.equal(x.reshape(-1), y) and ks.tolist() == [0, 0]
