"""Calls under a caller's stream capture: captured once (after a first direct call), replayed on new inputs in the same
buffers, and compared with direct calls on them."""
import numpy as np
import pytest

from synth import hyps, kb as K, programs as P
from tests.gpu_util import H, device_kb

pytestmark = pytest.mark.gpu


def _captured(torch, call):
    call()
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        call()
    return g


@pytest.mark.parametrize("rows", [200, 5000])
def test_ranking_under_capture(rows):
    import torch
    from paper_2412_00802_gb300 import surrogate as sg
    s = sg.Surrogate(sg.init_params(5))
    r = np.random.default_rng(rows)
    draw = lambda: (r.integers(0, 50, (rows, 4)).astype(np.int32), (0.25 * r.poisson(0.3, (rows, 512))).astype(np.float32))
    counts = torch.zeros((rows, 4), dtype=torch.int32, device="cuda")
    X = torch.zeros((rows, 512), dtype=torch.bfloat16, device="cuda")
    scores, Y = torch.zeros((2, rows, 2), device="cuda")
    best, likely = torch.zeros((2, rows // 20), dtype=torch.int32, device="cuda")
    ws = torch.empty(H.hedl_select_workspace_size(rows), dtype=torch.uint8, device="cuda")
    mws = s._workspace(rows)

    def call():
        H.hedl_scores_from_counts(counts, scores)
        H.hedl_select_top(scores, best.numel(), best, ws)
        H.hedl_mlp_forward(s.mlp, X, Y, mws)
        H.hedl_select_top(Y, likely.numel(), likely, ws)
    out = (scores, best, Y, likely)
    g = _captured(torch, call)
    for _ in range(2):
        c, x = draw()
        counts.copy_(torch.from_numpy(c))
        X.copy_(torch.from_numpy(x))
        for o in out:
            o.zero_()
        g.replay()
        torch.cuda.synchronize()
        got = [o.clone() for o in out]
        call()
        torch.cuda.synchronize()
        assert all(torch.equal(a, b) for a, b in zip(got, out))
    H.hedl_mlp_status(s.mlp)


def test_evaluation_under_capture():
    """A concept's small plan travels as a kernel's argument, a batch's larger one as a copy."""
    import torch
    kb = K.generate(K.CONFIGS["small"])
    dkb = device_kb(kb)
    one = P.compile_text("(and (some r1 (min 2 r2- A1)) (all r0 (or A0 (ge p1 3))))")
    progs, offs = P.pack_batch(hyps.small_hyps(kb, 3, 20))
    plan = H.hedl_plan_batch(dkb.handle, progs, offs, H.HEDL_NO_GRAPH)
    sizes = [H.hedl_workspace_size(dkb.handle, one, np.array([0, len(one)], np.uint32)),
             H.hedl_plan_info_get(plan)["workspace_bytes"]]
    wa, wb = (torch.empty(n, dtype=torch.uint8, device="cuda") for n in sizes)
    bits = torch.zeros(H.hedl_row_words(kb.n), dtype=torch.int32, device="cuda")
    counts = torch.zeros((len(offs) - 1, 4), dtype=torch.int32, device="cuda")

    def call():
        H.hedl_eval_concept(dkb.handle, one, bits, wa)
        H.hedl_plan_execute(dkb.handle, plan, counts, None, wb)
    call()
    H.hedl_sync_status(dkb.handle)
    want = [bits.clone(), counts.clone()]
    g = _captured(torch, call)
    for _ in range(2):
        bits.fill_(-1)
        counts.fill_(-1)
        g.replay()
        torch.cuda.synchronize()
        assert torch.equal(bits, want[0]) and torch.equal(counts, want[1])
    H.hedl_sync_status(dkb.handle)
