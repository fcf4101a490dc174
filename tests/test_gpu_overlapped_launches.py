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


def _matrices(count, m, n, r):
    gen = torch.Generator(device="cuda")
    gen.manual_seed(11)
    items = []
    for k in range(count):
        G = B.zeros_matrix(m, n, torch.bfloat16)
        G.copy_(1e-3 * torch.randn(m, n, device="cuda", generator=gen))
        w, p = B.zeros_matrix(m, n, torch.float32), B.zeros_matrix(m, r, torch.float32)
        w.copy_(0.02 * torch.randn(m, n, device="cuda", generator=gen))
        p.copy_(torch.randn(m, r, device="cuda", generator=gen) / m ** 0.5)
        items.append({"G": G, "P": B.quantize_int4(p), "W": B.quantize_int8(w), "M": B.zeros_matrix(r, n, torch.float32),
                      "V": B.zeros_matrix(r, n, torch.float32), "seed": k})
    return items


# Twelve matrices of 768 x 2048 at rank 512 are one chunk whose projection runs in pairs (384 tiles, a rank of whole 256s) and whose
# back-projection does not (576 tiles), both short enough to overlap the launch before them (five tiles a CTA); a workspace of a few
# of them makes chunks of single CTAs only; mode 3 has both in pairs, mode 1 the back-projection.
@pytest.mark.parametrize("pair_mode,at_once", [(6, 12), (6, 4), (3, 12), (1, 4)])
def test_steps_behind_one_another_equal_steps_one_by_one(pair_mode, at_once):
    base = _matrices(12, 768, 2048, 512)
    ws = (at_once + 1) * B.workspace_bytes(B.QG_OP_PROJECT_STEP, 768, 2048, 512)
    got, want = _run(base, pair_mode, False, ws), _run(base, 0, True)
    for a, b in zip(got, want):
        assert torch.equal(a["W"].codes, b["W"].codes)
        assert torch.equal(a["W"].scales, b["W"].scales) and torch.equal(a["W"].zeros, b["W"].zeros)
        assert torch.equal(a["M"], b["M"]) and torch.equal(a["V"], b["V"])


def test_a_stack_stepped_without_waiting_equals_steps_one_by_one():
    _, base = build_stack("llama130m", torch.device("cuda", 0), seed=7, layers=5)
    got, want = _run(base, 6, False), _run(base, 0, True)
    for a, b in zip(got, want):
        assert torch.equal(a["W"].codes, b["W"].codes) and torch.equal(a["W"].scales, b["W"].scales)
        assert torch.equal(a["M"], b["M"]) and torch.equal(a["V"], b["V"])
