"""New examples after a scoring call's graph was captured: the next call counts against the new ones."""
import numpy as np
import pytest

import oracle
from synth import hyps, kb as K, programs as P
from tests.gpu_util import H, device_kb

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("call", ["plan", "replay", "one_shot"])
def test_examples_set_between_scoring_calls(call):
    import torch
    kb = K.generate(K.CONFIGS["small"])
    dkb = device_kb(kb)
    progs, offs = P.pack_batch(hyps.small_hyps(kb, 3, 20))
    plan = H.hedl_plan_batch(dkb.handle, progs, offs)
    ws = torch.empty(max(H.hedl_plan_info_get(plan)["workspace_bytes"], H.hedl_workspace_size(dkb.handle, progs, offs)),
                     dtype=torch.uint8, device="cuda")
    counts = torch.zeros((len(offs) - 1, 4), dtype=torch.int32, device="cuda")

    def score():
        counts.fill_(-1)
        if call == "one_shot":
            H.hedl_score_batch(dkb.handle, progs, offs, counts, ws)
        else:
            (H.hedl_plan_replay if call == "replay" and ran else H.hedl_plan_execute)(dkb.handle, plan, counts, None, ws)
        H.hedl_sync_status(dkb.handle)
        return counts.cpu().numpy().astype(np.int64)

    _, sets, _ = oracle.eval_batch(oracle.from_synth(kb), progs, offs, keep_sets=True)
    sets = sets.astype(np.int64)
    r, keep, ran = np.random.default_rng(5), [], False
    for share in (0.1, 0.4, 0.02):          # every set of bitsets stays allocated
        u = r.random(kb.n)
        member = [(u < share).astype(np.int64), (u > 1.0 - share / 2).astype(np.int64)]
        bits = [torch.from_numpy(K.pack_bits(m, kb.wp).view(np.int32)).to("cuda") for m in member]
        keep.append(bits)
        H.hedl_examples_set(dkb.handle, *bits)
        want = np.stack([sets @ member[0], sets @ member[1], (1 - sets) @ member[0], (1 - sets) @ member[1]], 1)
        for _ in range(3):                  # direct, captured, replayed
            assert np.array_equal(score(), want), share
            ran = True
