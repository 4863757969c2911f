"""New plans, on every way they travel to the device: in the arguments of one table kernel, of both, of kernels ahead of them, and
from pageable memory (8 to 2280 heads). One context takes a new length call after call with no wait in between, then on a
second stream, then inside a capture that follows the upload at once. Every result has to equal that of a context made
for the length, and that one the oracle's."""
import dataclasses

import numpy as np
import pytest
import torch

from paper_2604_06694_b200 import workloads as wl
from test_gpu_evict import B, check_against_oracle, run_evict  # noqa: F401 (B is the fixture)
from helpers import to_dev

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("layers,n_req", [(2, 1), (75, 1), (190, 1), (190, 3)])
def test_new_plans_back_to_back(B, layers, n_req):  # noqa: F811
    ws, probs, fresh, bufs = [], [], [], []
    for L in (170, 212, 171):            # prefixes of 162 = 2 3^4, 204 = 4 3 17 (packed), 163 (prime)
        spec = dataclasses.replace(wl.config(1), seq_lens=[L] * n_req, audio_frac=[0.9] * n_req, n_q_heads=4,
                                   head_dim=64, window=8)
        w = wl.generate(spec, seed=L, layers=layers)
        ws.append(w)
        probs.append(B.Problem.from_workload(w))
        fresh.append(run_evict(B, w))
        check_against_oracle(w, fresh[-1])
        bufs.append([to_dev(w, w.q), to_dev(w, w.k), to_dev(w, w.v), torch.from_numpy(w.head_scores).cuda()])
    ctx = B.Context(probs[0], workspace_bytes=max(B.audiokv_workspace_bytes(p) for p in probs))

    def call(i):
        rows, TH = int(ws[i].total_budget.sum()), probs[i].total_heads
        k_out = torch.zeros((rows, 64), dtype=torch.bfloat16, device="cuda")
        out = [k_out, torch.zeros_like(k_out), *(torch.zeros(n, dtype=torch.int32, device="cuda") for n in (rows, TH, TH + 1))]
        B.audiokv_evict(ctx, probs[i], *bufs[i], [int(x) for x in ws[i].total_budget], *out)
        return out

    def check(i, out):
        for a, name in zip(out, ("k_out", "v_out", "kept", "budgets", "cu")):
            got = a.cpu().view(torch.uint16).numpy() if a.dtype == torch.bfloat16 else a.cpu().numpy()
            assert np.array_equal(got, fresh[i][name]), (i, name)

    order = [0, 1, 2, 1, 0, 2, 0]
    outs = [call(i) for i in order]
    torch.cuda.synchronize()
    assert ctx.last_device_status() == 0
    for i, out in zip(order, outs):
        check(i, out)

    side = torch.cuda.Stream()
    call(1)                              # the upload, on the default stream
    side.wait_stream(torch.cuda.current_stream())
    with torch.cuda.stream(side):
        again = call(1)
        call(2)                          # an upload on this one
    graph = torch.cuda.CUDAGraph()
    held = torch.cuda.Stream()
    with torch.cuda.graph(graph, stream=held):
        captured = call(2)
    torch.cuda.synchronize()
    check(1, again)
    graph.replay()
    torch.cuda.synchronize()
    assert ctx.last_device_status() == 0
    check(2, captured)
