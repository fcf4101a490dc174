"""Launches that begin while the one before them still runs (programmatic dependent launch): CTA pairs followed by single CTAs and
the other way round, step after step without a wait, give what the launches give one by one."""
import pytest
import torch

from paper_2407_08296_b200 import binding as B
from paper_2407_08296_b200.synth_device import build_stack

pytestmark = pytest.mark.gpu

STEPS = 60


def _run(base, pair_mode, wait, workspace_bytes=None):
    items = [{"G": it["G"], "P": it["P"], "W": it["W"].clone(), "M": it["M"]._base.clone()[:, :it["M"].shape[1]] if it["M"]._base is not None
              else it["M"].clone(), "V": it["V"]._base.clone()[:, :it["V"].shape[1]] if it["V"]._base is not None else it["V"].clone(),
              "seed": it["seed"]} for it in base]
    B.debug_set_pair_mode(pair_mode)
    try:
        plan = B.StepPlan(items, workspace_bytes=workspace_bytes)
    finally:
        B.debug_set_pair_mode(B.DEFAULT_PAIR_MODE)
    for t in range(1, STEPS + 1):
        plan.step(B.Hyper(step=t))
        if wait:
            torch.cuda.synchronize()
    torch.cuda.synchronize()
    assert int(plan.status.item()) == 0
    plan.close()
    return items


# Five LLaMA-130M layers are one chunk whose projection runs in pairs (310 tiles, ranks of whole 256s) and whose
# back-projection does not (1080 tiles), both short enough to overlap the launch before them; a workspace of a few matrices makes several such
# chunks a step; mode 3 has both in pairs.
@pytest.mark.parametrize("pair_mode,matrices", [(6, None), (6, 12), (3, None), (1, 12)])
def test_steps_behind_one_another_equal_steps_one_by_one(pair_mode, matrices):
    _, base = build_stack("llama130m", torch.device("cuda", 0), seed=7, layers=5)
    ws = None if matrices is None else matrices * B.workspace_bytes(B.QG_OP_PROJECT_STEP, 2048, 768, 256)
    got, want = _run(base, pair_mode, False, ws), _run(base, 0, True)
    for a, b in zip(got, want):
        assert torch.equal(a["W"].codes, b["W"].codes)
        assert torch.equal(a["W"].scales, b["W"].scales) and torch.equal(a["W"].zeros, b["W"].zeros)
        assert torch.equal(a["M"], b["M"]) and torch.equal(a["V"], b["V"])
