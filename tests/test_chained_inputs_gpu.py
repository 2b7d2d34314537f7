"""Inputs written by a kernel that lets its dependents start before it has finished: the advance of the history
(asd_commit) writes the draft tokens, the LM head's product the logits, each right ahead of the call that reads
them, in the same buffers at every step, captured in one graph so that the launches chain. Integer-valued hidden
states and weights make the logits exact, so every output must equal the oracle's."""
import numpy as np
import pytest
import torch

from oracle import oracle
from paper_2608_03447_gb300 import inputs

pytestmark = pytest.mark.gpu

STEPS = 6
KEYS = ("accepted_len", "committed", "recovery", "row_argmax", "status")


def _steps(B, K, H, V):
    """Per step: hidden states, drafts, and the oracle's logits; one weight. Some hidden rows are zero, so that
    whole rows of logits tie at zero and the maximum's sign is looked up in the logits."""
    base = inputs.gen_lmhead_exact(B, K, H, V, 8100, "cuda")
    steps = []
    for i in range(STEPS):
        inp = inputs.gen_lmhead_exact(B, K, H, V, 8100 + i, "cuda")
        hidden = inp.hidden.clone()
        hidden[i::5] = 0
        z = oracle.lmhead_logits_matmul(hidden.cpu(), base.weight.cpu()).astype(np.float32)
        draft = np.where(np.random.default_rng(i).random((B, K)) < 0.7,
                         z.reshape(B, K + 1, V)[:, :K].argmax(2), inp.draft.cpu().numpy()).astype(np.int32)
        steps.append((hidden, torch.from_numpy(draft).cuda(), z))
    return base.weight, steps


@pytest.mark.parametrize("entry", ["lmhead_verify", "lmhead_partials", "verify", "verify_small", "verify_tma"])
def test_producers_that_finish_late(asd, entry):
    B, K, H, V = 12, 6, 64, 5000
    weight, steps = _steps(B, K, H, V)
    hidden = torch.empty_like(steps[0][0])
    logits = torch.empty(B * (K + 1), V, device="cuda")
    drafts = torch.zeros(B, K, dtype=torch.int32, device="cuda")     # a history of K tokens: one step's drafts
    accepted = torch.full((B,), K - 1, dtype=torch.int32, device="cuda")
    written = [torch.cat([x, torch.zeros(B, 1, dtype=torch.int32, device="cuda")], 1).contiguous() for _, x, _ in steps]
    lengths = [torch.zeros(B, dtype=torch.int32, device="cuda") for _ in steps]
    outs = [asd.alloc_outputs(B, K) for _ in steps]
    parts = torch.zeros(1, B * (K + 1), 6, dtype=torch.int32, device="cuda")
    ledger = asd.make_ledger(B, 8.0)
    lm_ws = asd.lmhead_workspace(B, K, V, H, torch.device("cuda"))
    ws = asd.Workspace(B, K, V, asd.F32)

    def run():
        for (h, _, _), tokens, length, out in zip(steps, written, lengths, outs):
            hidden.copy_(h)
            asd.commit(accepted, tokens, 1, tokens=drafts, token_len=length)
            if entry == "lmhead_verify":
                asd.lmhead_verify(hidden, weight, drafts, ledger, 1.0, 2, workspace=lm_ws, out=out)
            elif entry == "lmhead_partials":
                asd.lmhead_partials(hidden, weight, drafts, 0, V, workspace=lm_ws, out=parts[0])
                asd.shard_combine(parts, drafts, ledger, 1.0, 2, V, out=out)
            else:
                asd.lmhead_logits(hidden, weight, out=logits)
                asd.verify(logits.view(B, K + 1, V), drafts, ledger, 1.0, 2, workspace=ws, out=out)

    def check(what):
        led = np.array([[8.0, 0.0]] * B, np.float32)
        for i, ((_, x, z), out) in enumerate(zip(steps, outs)):
            o = oracle.verify(z.reshape(B, K + 1, V), x.cpu().numpy(), led, 1.0, 2)
            led = o["ledger"]
            for key in KEYS:
                assert np.array_equal(out[key].cpu().numpy(), o[key]), f"{what} step {i}: {key}"
            # as values: where a whole row is zero the products' signs are the tensor cores' own
            assert np.array_equal(out["row_regret"].cpu().numpy(), o["row_regret"]), f"{what} step {i}: row_regret"
        assert np.array_equal(ledger.cpu().numpy().view(np.uint32), led.view(np.uint32)), f"{what}: ledger"

    try:
        asd.set_launch_options(path={"verify_small": "small", "verify_tma": "tma"}.get(entry, "stream"))
        torch.cuda.synchronize()
        side = torch.cuda.Stream()
        with torch.cuda.stream(side):
            run()
        torch.cuda.synchronize()
        check("eager")
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph, stream=side):
            run()
        for length in lengths:
            length.zero_()
        ledger.copy_(torch.tensor([[8.0, 0.0]] * B))
        graph.replay()
        torch.cuda.synchronize()
        check("graph")
    finally:
        asd.reset_launch_options()
