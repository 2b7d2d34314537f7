"""asd_commit (advance along the emitted sequence, Sec. 3.3) against the oracle, over a decode loop and over captured
rounds."""
import numpy as np
import pytest
import torch

from oracle import oracle
from paper_2608_03447_gb300 import inputs

pytestmark = pytest.mark.gpu


def test_decode_loop_history_and_cache_lengths(asd):
    """12 rounds: verify, then commit; histories and KV lengths equal the oracle's, overflow included."""
    B, K, V, max_tokens = 16, 8, 3000, 40
    led = asd.make_ledger(B, 4.0)
    led_o = np.array([[4.0, 0.0]] * B, np.float32)
    tokens = torch.full((B, max_tokens), -1, dtype=torch.int32, device="cuda")
    token_len = torch.zeros(B, dtype=torch.int32, device="cuda")
    kv_len = torch.arange(B, dtype=torch.int32, device="cuda") * 3
    status = torch.zeros(B, dtype=torch.int32, device="cuda")
    o_tok = tokens.cpu().numpy()
    o_tl = token_len.cpu().numpy()
    o_kv = kv_len.cpu().numpy()
    overflowed = np.zeros(B, bool)
    for rnd in range(12):
        blk = inputs.gen_block(B, K, V, torch.float32, 81_000 + rnd, "cuda")
        out = asd.verify(blk.logits, blk.draft, led, 1.0, 2)
        asd.commit(out["accepted_len"], out["committed"], 1, kv_len, tokens, token_len, status)
        v = oracle.verify(blk.logits.cpu(), blk.draft.cpu().numpy(), led_o, 1.0, 2)
        led_o = v["ledger"]
        c = oracle.commit(v["accepted_len"], v["committed"], 1, o_kv, o_tok, o_tl)
        o_tok, o_tl, o_kv = c["tokens"], c["token_len"], c["kv_len"]
        torch.cuda.synchronize()
        assert np.array_equal(status.cpu().numpy(), c["status"]), f"round {rnd}: status"
        assert np.array_equal(token_len.cpu().numpy(), o_tl), f"round {rnd}: token_len"
        assert np.array_equal(kv_len.cpu().numpy(), o_kv), f"round {rnd}: kv_len"
        assert np.array_equal(tokens.cpu().numpy(), o_tok), f"round {rnd}: history"
        overflowed |= c["status"] == asd.STATUS_OVERFLOW
    assert overflowed.any(), "the loop should reach the history's capacity"


def test_commit_without_history(asd):
    a = torch.tensor([0, 3, 8], dtype=torch.int32, device="cuda")
    committed = torch.zeros(3, 9, dtype=torch.int32, device="cuda")
    kv = torch.tensor([10, 20, 30], dtype=torch.int32, device="cuda")
    asd.commit(a, committed, 0, kv_len=kv)
    torch.cuda.synchronize()
    assert kv.tolist() == [10, 23, 38]


@pytest.mark.parametrize("B,K,V,dtype", [
    (32, 8, 40000, torch.bfloat16),    # 80 KB rows, 23 MB: the TMA pipeline when resident, else the streaming kernel
    (24, 4, 12000, torch.float32),     # the streaming kernel
    (2, 4, 32000, torch.bfloat16),     # a cluster per request
    (40, 5, 700, torch.float32),       # a CTA per request
])
@pytest.mark.parametrize("resident", [True, False])
def test_captured_rounds(asd, B, K, V, dtype, resident):
    """Rounds of verify, opportunity counts and commit captured one behind the other, each over logits of its own
    and all over the same output, ledger and history buffers: the launches chain, and with resident inputs a
    round's logits stream while the rounds before it finish. What every round emitted is in the history."""
    rounds, max_tokens = 10, 10 * (K + 1)
    blocks = [inputs.gen_block(B, K, V, dtype, 82_000 + i, "cuda") for i in range(rounds)]
    ws = asd.Workspace(B, K, V, asd.BF16 if dtype == torch.bfloat16 else asd.F32)
    out = asd.alloc_outputs(B, K)
    ledger = asd.make_ledger(B, 6.0)
    counts = torch.zeros(5, dtype=torch.int64, device="cuda")
    tokens = torch.full((B, max_tokens), -1, dtype=torch.int32, device="cuda")
    token_len = torch.zeros(B, dtype=torch.int32, device="cuda")
    kv_len = torch.zeros(B, dtype=torch.int32, device="cuda")
    taus, ps = (0.5, 2.0), (1, 2)

    led = np.array([[6.0, 0.0]] * B, np.float32)
    o_tok, o_tl, o_kv = tokens.cpu().numpy(), token_len.cpu().numpy(), kv_len.cpu().numpy()
    o_counts = np.zeros(5, np.int64)
    for b in blocks:
        o = oracle.verify(b.logits.cpu(), b.draft.cpu().numpy(), led, 1.0, 2)
        led = o["ledger"]
        num, den = oracle.opportunity(o["row_argmax"], b.draft.cpu().numpy(), o["row_regret"], taus, ps,
                                      status=o["status"])
        o_counts += np.append(num.reshape(-1), den)
        c = oracle.commit(o["accepted_len"], o["committed"], 1, o_kv, o_tok, o_tl)
        o_tok, o_tl, o_kv = c["tokens"], c["token_len"], c["kv_len"]

    def run():
        for b in blocks:
            asd.verify(b.logits, b.draft, ledger, 1.0, 2, workspace=ws, out=out, resident=resident)
            asd.opportunity(out["row_argmax"], b.draft, out["row_regret"], taus, ps, status=out["status"],
                            counts=counts)
            asd.commit(out["accepted_len"], out["committed"], 1, kv_len, tokens, token_len)

    def reset():
        ledger.copy_(torch.tensor([[6.0, 0.0]] * B))
        counts.zero_()
        tokens.fill_(-1)
        token_len.zero_()
        kv_len.zero_()
        torch.cuda.synchronize()

    def check(what):
        torch.cuda.synchronize()
        assert np.array_equal(token_len.cpu().numpy(), o_tl), f"{what}: token_len"
        assert np.array_equal(tokens.cpu().numpy(), o_tok), f"{what}: history"
        assert np.array_equal(kv_len.cpu().numpy(), o_kv), f"{what}: kv_len"
        assert np.array_equal(counts.cpu().numpy(), o_counts), f"{what}: counts"
        assert np.array_equal(ledger.cpu().numpy().view(np.uint32), led.view(np.uint32)), f"{what}: ledger"
        for key in ("accepted_len", "committed", "recovery", "row_argmax", "status"):
            assert np.array_equal(out[key].cpu().numpy(), o[key]), f"{what}: {key} of the last round"
        assert ws.error() == 0

    side = torch.cuda.Stream()
    torch.cuda.synchronize()
    with torch.cuda.stream(side):
        run()
    check("eager")
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=side):
        run()
    for rep in range(3):
        reset()
        graph.replay()
        check(f"replay {rep}")
