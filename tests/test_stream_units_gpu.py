"""The row stages that cut rows into units, at the sizes where the cut can go wrong: one vector either side of
a unit, units of one to eight loads per lane, rows shorter than a vector, starts off the 16-byte and the
128-byte grid, rows whose maximum sits at a unit's edge or is tied across units, rows of -inf, infinities, the
lowest finite value and subnormal maxima; requests on both sides of each cluster size; several blocks per call.
Every output bit for bit the oracle's (comparisons and one fp32 subtraction decide all of them)."""
import math

import numpy as np
import pytest
import torch

from oracle import oracle

pytestmark = pytest.mark.gpu

VEC = {torch.bfloat16: 8, torch.float32: 4}


def _equal(got, want, what):
    for k in ("status", "accepted_len", "recovery", "committed", "row_argmax"):
        assert np.array_equal(got[k].cpu().numpy(), want[k]), f"{what}: {k}"
    g, o = got["row_regret"].cpu().numpy(), want["row_regret"]
    assert ((g.view(np.uint32) == o.view(np.uint32)) | (np.isnan(g) & np.isnan(o))).all(), f"{what}: row_regret"


@pytest.mark.parametrize("fused", [False, True])
@pytest.mark.parametrize("dtype", [torch.bfloat16, torch.float32])
@pytest.mark.parametrize("vectors", [0, 1, 31, 32, 33, 127, 128, 129, 255, 256, 257, 511, 513, 2049])
def test_unit_edges(asd, dtype, vectors, fused):
    vn = VEC[dtype]
    rng = np.random.default_rng(vectors)
    for extra, rows_mb in ((0, 0), (1, 0), (vn - 1, 12)):  # 12 MB of rows: eight loads per lane
        V = vectors * vn + extra
        if V < 1:
            continue
        K = 3
        B = max(3, (rows_mb << 20) // ((K + 1) * V * (16 // vn)))
        if B * (K + 1) > 6000:
            continue  # the longer rows cover this
        off = int(rng.integers(0, 64))
        flat = torch.randn(off + B * (K + 1) * V, device="cuda").mul_(3.0).to(dtype)
        z = flat[off:].view(B, K + 1, V)
        tops = [0, V - 1, min(V - 1, 32 * vn), min(V - 1, 256 * vn - 1), min(V - 1, 256 * vn)]
        for i, at in enumerate(tops[: K + 1]):
            z[0, i, at] = 40.0
        z[1, 0] = -math.inf                                  # no finite value: index 0
        z[1, 1, [V - 1, V // 2]] = 50.0                      # a tie: the lower index
        z[1, 2, V // 3] = math.inf
        z[1, 3] = torch.finfo(dtype).min
        z[2, 0] = -1.0
        z[2, 0, V // 2] = 1e-39                              # subnormal maxima
        z[2, 1] = -1e-39
        draft = torch.randint(0, V, (B, K), dtype=torch.int32, device="cuda")
        draft[:, 0] = z[:, 0].argmax(1)                      # the tops among the drafts, so longer prefixes occur
        ledger = asd.make_ledger(B, 8.0)
        try:
            asd.set_launch_options(path="stream", fused_select=fused)
            out = asd.verify(z, draft, ledger, 1.0, 2)
            torch.cuda.synchronize()
        finally:
            asd.reset_launch_options()
        want = oracle.verify(z.cpu(), draft.cpu().numpy(), np.array([[8.0, 0.0]] * B, np.float32), 1.0, 2)
        _equal(out, want, f"V={V} off={off} {dtype}")
        assert np.array_equal(ledger.cpu().numpy().view(np.uint32), want["ledger"].view(np.uint32))


@pytest.mark.parametrize("dtype", [torch.bfloat16, torch.float32])
@pytest.mark.parametrize("per", [64, 96, 128, 160, 192, 224])
@pytest.mark.parametrize("units", [1, 2, 3])
def test_units_of_several_loads(asd, per, units, dtype):
    """Inputs whose size gives units of `per` vectors (sixteen warps an SM share them), in rows one vector either
    side of a whole number of them."""
    vn, K = VEC[dtype], 3
    warps = 16 * torch.cuda.get_device_properties(0).multi_processor_count
    for vectors in (per * units - 1, per * units, per * units + 1, per * units - 7, per * units - 8):
        B = max(3, int(warps * (per - 16) / vectors) // (K + 1))
        share = -(-B * (K + 1) * vectors // warps)
        assert -(-share // 32) * 32 == per
        V = vectors * vn + vectors % vn
        off = vectors % 61
        flat = torch.randn(off + B * (K + 1) * V, device="cuda").mul_(3.0).to(dtype)
        z = flat[off:].view(B, K + 1, V)
        for i in range(min(B, 40)):
            edge = (i % (units + 1)) * per * vn
            at = [edge - 8 * vn, edge - 1, edge, edge + vn]
            for j in range(K + 1):
                z[i, j, min(max(at[j], 0), V - 1)] = 40.0
        z[2, 1, [0, V - 1]] = 50.0
        draft = torch.randint(0, V, (B, K), dtype=torch.int32, device="cuda")
        draft[:, 0] = z[:, 0].argmax(1)
        ledger = asd.make_ledger(B, 8.0)
        try:
            asd.set_launch_options(path="stream")
            out = asd.verify(z, draft, ledger, 1.0, 2)
            torch.cuda.synchronize()
        finally:
            asd.reset_launch_options()
        want = oracle.verify(z.cpu(), draft.cpu().numpy(), np.array([[8.0, 0.0]] * B, np.float32), 1.0, 2)
        _equal(out, want, f"per={per} V={V} off={off} {dtype}")
        assert np.array_equal(ledger.cpu().numpy().view(np.uint32), want["ledger"].view(np.uint32))


@pytest.mark.parametrize("row_kb, B", [(64, 21), (64, 22), (64, 113), (64, 152), (64, 153),
                                       (112, 63), (112, 153)])
@pytest.mark.parametrize("short", [0, 2])
@pytest.mark.parametrize("resident", [False, True])
def test_both_sides_of_the_dispatch(asd, row_kb, B, short, resident):
    """Rows, their number and their bytes on both sides of the lines between the two kernels for resident
    inputs (64 KB up to 456 rows, else 112 KB; 1 MB up to 64 rows, else 21.5 MB)."""
    V, K = (row_kb * 1024 - short) // 2, 2
    z = torch.randn(B, K + 1, V, device="cuda").mul_(3.0).to(torch.bfloat16)
    draft = z[:, :K].argmax(2).to(torch.int32).contiguous()
    draft[:, 1] = torch.randint(0, V, (B,), dtype=torch.int32, device="cuda")
    ledger = asd.make_ledger(B, 8.0)
    torch.cuda.synchronize()
    out = asd.verify(z, draft, ledger, math.inf, 2, resident=resident)
    torch.cuda.synchronize()
    want = oracle.verify(z.cpu(), draft.cpu().numpy(), np.array([[8.0, 0.0]] * B, np.float32), math.inf, 2)
    _equal(out, want, f"V={V} B={B}")


@pytest.mark.parametrize("resident", [False, True])
@pytest.mark.parametrize("K", [0, 8, 31])
@pytest.mark.parametrize("ctas", [1, 2, 4, 8])
def test_request_clusters(asd, ctas, K, resident):
    """Requests that just fill, and just do not fill, one round of loads of a cluster of each size; a NaN in
    one request flags that request only, whichever CTA of its cluster meets it."""
    limit = ctas * 65536 - 4096
    for dtype, size in ((torch.bfloat16, 2), (torch.float32, 4)):
        for V in (limit // size // (K + 1), limit // size // (K + 1) + 1):
            B = 5
            off = (V + K) % 8
            flat = torch.randn(off + B * (K + 1) * V, device="cuda").mul_(3.0).to(dtype)
            z = flat[off:].view(B, K + 1, V)
            for j in range(K + 1):
                z[0, j, (j * V) // (K + 1)] = 40.0
                z[1, j, V - 1 - j] = 40.0
            z[2, K, V - 1] = math.nan
            z[3, 0, 0] = math.nan
            draft = torch.randint(0, V, (B, K), dtype=torch.int32, device="cuda")
            if K:
                draft[:2] = z[:2, :K].float().argmax(2).to(torch.int32)
            ledger = asd.make_ledger(B, 8.0)
            torch.cuda.synchronize()
            try:
                asd.set_launch_options(path="small")
                out = asd.verify(z, draft, ledger, 1.0, 2, resident=resident)
                torch.cuda.synchronize()
            finally:
                asd.reset_launch_options()
            want = oracle.verify(z.cpu(), draft.cpu().numpy(), np.array([[8.0, 0.0]] * B, np.float32), 1.0, 2)
            assert np.array_equal(out["status"].cpu().numpy(), want["status"])
            clean = want["status"] == 0
            assert clean.tolist() == [True, True, False, False, True]
            got = {k: v[torch.from_numpy(clean).cuda()] for k, v in out.items()}
            _equal(got, {k: v[clean] for k, v in want.items() if k != "ledger"}, f"V={V} off={off} {dtype}")
            assert np.array_equal(ledger.cpu().numpy().view(np.uint32), want["ledger"].view(np.uint32))


@pytest.mark.parametrize("resident", [False, True])
@pytest.mark.parametrize("dtype", [torch.bfloat16, torch.float32])
@pytest.mark.parametrize("K,V,B", [(0, 1, 1672), (0, 17, 1673), (1, 9, 1064), (4, 100, 456), (4, 100, 457),
                                   (8, 255, 304), (8, 257, 305), (13, 5, 152), (14, 5, 152), (15, 5, 153),
                                   (31, 2, 152), (31, 33, 153), (0, 263, 200), (0, 520, 200), (2, 1100, 150)])
def test_tiny_requests(asd, K, V, B, dtype, resident):
    """Requests whose CTA has two to sixteen warps, with units of a load per lane and of more, as many as fit the
    GPU at once and one more; tied tops, a top at either end of a row, a NaN in one request."""
    vn = VEC[dtype]
    off = (V + B) % vn
    flat = torch.randn(off + B * (K + 1) * V, device="cuda").mul_(3.0).to(dtype)
    z = flat[off:].view(B, K + 1, V)
    z[0, :, 0] = 40.0
    z[1, :, V - 1] = 40.0
    z[2, :, V // 2:] = 40.0
    z[3] = -math.inf
    z[4, K, V // 3] = math.nan
    draft = torch.randint(0, V, (B, K), dtype=torch.int32, device="cuda")
    half = (K + 1) // 2
    draft[:, :half] = z[:, :half].float().nan_to_num(0.0, 9e9, -9e9).argmax(2).to(torch.int32)
    ledger = asd.make_ledger(B, 8.0)
    torch.cuda.synchronize()
    out = asd.verify(z, draft, ledger, 1.0, 2, resident=resident)
    torch.cuda.synchronize()
    want = oracle.verify(z.cpu(), draft.cpu().numpy(), np.array([[8.0, 0.0]] * B, np.float32), 1.0, 2)
    assert np.array_equal(out["status"].cpu().numpy(), want["status"])
    clean = want["status"] == 0
    assert clean.sum() == B - 1
    got = {k: v[torch.from_numpy(clean).cuda()] for k, v in out.items()}
    _equal(got, {k: v[clean] for k, v in want.items() if k != "ledger"}, f"K={K} V={V} B={B} {dtype}")
    assert np.array_equal(ledger.cpu().numpy().view(np.uint32), want["ledger"].view(np.uint32))


@pytest.mark.parametrize("nblk", [2, 7, 8, 9, 17])
def test_blocks_around_the_warps_of_a_selection(asd, nblk):
    """The ledger goes through fewer, as many and more blocks than the selection's CTA has warps; one block in
    the middle of a request has a NaN, an out-of-range draft sits in the last."""
    B, K, V = 5, 6, 4001
    z = torch.randn(nblk, B, K + 1, V, device="cuda").mul_(3.0).to(torch.bfloat16)
    draft = z[:, :, :K].float().argmax(3).to(torch.int32)
    near = torch.rand(nblk, B, K, device="cuda") < 0.4
    second = z[:, :, :K].float().topk(2, dim=3).indices[..., 1].to(torch.int32)
    draft = torch.where(near, second, draft).contiguous()
    z[nblk // 2, 1, 0, 7] = math.nan
    draft[nblk - 1, 2, 0] = V
    ledger = asd.make_ledger(B, 6.0)
    torch.cuda.synchronize()
    out = asd.verify_blocks(z, draft, ledger, 1.0, 3)
    torch.cuda.synchronize()
    want_ledger = np.array([[6.0, 0.0]] * B, np.float32)
    for i in range(nblk):
        want = oracle.verify(z[i].cpu(), draft[i].cpu().numpy(), want_ledger, 1.0, 3)
        want_ledger = want["ledger"]
        assert np.array_equal(out["status"][i].cpu().numpy(), want["status"])
        ok = torch.from_numpy((want["status"] & oracle.STATUS_NAN_LOGIT) == 0)
        _equal({k: v[i][ok.cuda()] for k, v in out.items()},
               {k: v[ok.numpy()] for k, v in want.items() if k != "ledger"}, f"block {i}")
    assert np.array_equal(ledger.cpu().numpy().view(np.uint32), want_ledger.view(np.uint32))
