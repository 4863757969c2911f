"""The causal mask of the tensor-core scoring is decided per 64 keys: prefixes that end just before, at and behind a multiple of
64 or 128, windows inside one such stretch, across two and across three, and windows scored in several chunks, against the oracle."""
import numpy as np
import pytest
import torch

from paper_2604_06694_b200 import workloads as wl
from helpers import REL_TOL, oracle_scores, rel_err, to_dev

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def B():
    from paper_2604_06694_b200 import build as akv_build
    akv_build.build()
    from paper_2604_06694_b200 import binding
    return binding


@pytest.mark.parametrize("W,G", [(1, 4), (16, 4), (63, 2), (64, 2), (65, 2), (130, 1), (40, 8)])
def test_scores_around_multiples_of_64(B, W, G):
    prefixes = [p for m in (64, 128, 192, 256) for p in (m - W, m - 1, m, m + 1) if p > 0] + [1, 2]
    for at in range(0, len(prefixes), 6):
        lens = [p + W for p in prefixes[at:at + 6]]
        w = wl.generate(wl.WorkloadSpec("mask", "bf16", 1, 2 * G, 2, 64, lens, [0.8] * len(lens), 0, window=W), seed=W + at)
        prob = B.Problem.from_workload(w)
        ctx = B.Context(prob)
        scores = torch.full((B.audiokv_scores_len(prob),), float("nan"), device="cuda")
        B.audiokv_score(ctx, prob, to_dev(w, w.q), to_dev(w, w.k), scores)
        torch.cuda.synchronize()
        assert ctx.last_device_status() == 0 and ctx.last_score_path() == "tcgen05"
        got, pos = scores.cpu().numpy(), 0
        for r, L in enumerate(lens):
            want, _ = oracle_scores(w, r)
            for h in range(2):
                g = got[pos:pos + L - W]
                pos += L - W
                assert rel_err(g, np.asarray(want).reshape(2, -1)[h]) <= REL_TOL, (W, G, L, h)
