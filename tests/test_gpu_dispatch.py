"""GPU tests of the kernel variants that a call's sizes choose between, at the sizes where each can go wrong
(edges of tiles and parts, remainders, the ends of a variant's range), against the CPU oracle."""
import numpy as np
import pytest
import torch

from bench import count_launches
from oracle import lvlm_oracle as O
from paper_2509_00419_b200 import binding as L
from paper_2509_00419_b200 import build as BU
from tests.util import assert_rows_close, assert_scores_close, f64, i32

pytestmark = pytest.mark.gpu


# decode attention cut into parts that a second launch adds: few heads with long caches, or more heads than clusters fit
@pytest.mark.parametrize("case", [        # B, H, Hkv, cap, append, acc_score
    (1, 1, 1, 512, True, True), (1, 3, 1, 1037, False, True), (1, 7, 1, 256, True, False), (2, 8, 1, 545, True, False),
    (1, 28, 4, 1536, True, False), (5, 8, 4, 511, True, True), (9, 24, 4, 223, True, True), (8, 16, 4, 224, False, False),
    (1, 2, 2, 7001, True, True), (9, 4, 4, 9300, True, True)])      # (the last: a CTA has several slices of the keys)
def test_decode_in_parts(case):
    B, H, Hkv, cap, append, with_acc = case
    r = np.random.default_rng(cap + H)
    bf = lambda *s: torch.from_numpy(r.normal(size=s).astype(np.float32)).to(torch.bfloat16)
    q, Kc, Vc, kn, vn = bf(B, H, 128), bf(B, Hkv, cap, 128), bf(B, Hkv, cap, 128), bf(B, Hkv, 128), bf(B, Hkv, 128)
    ln = r.integers(1, cap, size=(B, Hkv)).astype(np.int32)
    edges = [cap - 1, 0 if append else 1, 63, 64, 65, 16 * 4 * 3 - 1]       # one row short of a stage, a stage, one more
    ln.reshape(-1)[:len(edges)] = np.minimum(edges, cap - 1)[:ln.size]
    acc = r.random((B, Hkv, cap)).astype(np.float32) if with_acc else None
    want = O.decode_attn(f64(q), f64(Kc), f64(Vc), ln, k_new=f64(kn) if append else None,
                         v_new=f64(vn) if append else None, acc_score=acc)
    Kd, Vd, ld = Kc.cuda(), Vc.cuda(), torch.from_numpy(ln).cuda()
    ad = torch.from_numpy(acc).cuda() if with_acc else None
    flag = torch.zeros(1, dtype=torch.int32, device="cuda")
    out = L.decode_attn(q.cuda(), Kd, Vd, ld, k_new=kn.cuda() if append else None, v_new=vn.cuda() if append else None,
                        acc_score=ad, dev_status=flag, max_len=cap)
    torch.cuda.synchronize()
    assert flag.item() == 0
    assert_rows_close(f64(out), want["out"], what="attention output")
    assert np.array_equal(i32(ld), want["len"])
    if append:
        assert np.array_equal(f64(Kd), want["Kc"].astype(np.float64)) and np.array_equal(f64(Vd), want["Vc"].astype(np.float64))
    if with_acc:
        for b in range(B):
            for g in range(Hkv):
                m = want["len"][b, g]
                assert_scores_close(ad[b, g, :m].cpu().numpy(), want["acc_score"][b, g, :m], what="acc_score")
                assert np.array_equal(ad[b, g, m:].cpu().numpy(), acc[b, g, m:])


# the form follows the rows that the caller expects, not the capacity alone; rows beyond what was expected are attended to as well
@pytest.mark.parametrize("B,H,Hkv,cap,max_len,rows,acc,parts", [
    (1, 28, 4, 3072, None, 300, False, False), (1, 28, 4, 3072, 301, 300, False, False), (1, 28, 4, 3072, 2900, 2899, False, True),
    (1, 28, 4, 3072, 200, 3000, False, False), (1, 28, 4, 33000, None, 300, False, True), (1, 28, 4, 33000, 400, 9000, True, False),
    (1, 32, 8, 3056, None, 700, True, False), (1, 32, 8, 3072, None, 700, True, True), (9, 28, 4, 300, None, 290, False, True),
    (1, 28, 4, 2000, 5000, 1999, True, True)])
def test_decode_form(B, H, Hkv, cap, max_len, rows, acc, parts):
    g = torch.Generator(device="cuda").manual_seed(cap + rows)
    q, kn = (torch.randn(B, h, 128, generator=g, device="cuda").bfloat16() for h in (H, Hkv))
    Kc = torch.randn(B, Hkv, cap, 128, generator=g, device="cuda").bfloat16()
    ln = torch.full((B, Hkv), rows, dtype=torch.int32, device="cuda")
    accs, flag = torch.zeros(B, Hkv, cap, device="cuda") if acc else None, torch.zeros(1, dtype=torch.int32, device="cuda")

    def call():
        return L.decode_attn(q, Kc, Kc, ln, k_new=kn, v_new=kn, acc_score=accs, dev_status=flag, max_len=max_len)

    assert count_launches(call) == (2 if parts else 1)
    out = call()
    k = Kc[:, :, :rows + 1].double().repeat_interleave(H // Hkv, dim=1)
    assert flag.item() == 0 and ln.eq(rows + 1).all() and torch.equal(Kc[:, :, rows], kn)
    p = torch.softmax(torch.einsum("bhd,bhnd->bhn", q.double(), k) / 128 ** 0.5, dim=-1)
    assert_rows_close(f64(out), f64(torch.einsum("bhn,bhnd->bhd", p, k)), what="attention output")
    if acc:
        assert_scores_close(f64(accs[:, :, :rows + 1]), f64(p.view(B, Hkv, H // Hkv, -1).sum(dim=2)), what="acc_score")


def test_decode_without_room_for_parts():
    B, H, Hkv, cap = 1, 28, 4, 5000
    q, Kc = torch.randn(B, H, 128, device="cuda").bfloat16(), torch.randn(B, Hkv, cap, 128, device="cuda").bfloat16()
    ln = torch.full((B, Hkv), cap - 3, dtype=torch.int32, device="cuda")
    d, least = L.kv_dims(Kc, H=H), -(-B * H * cap * 4 // 256) * 256
    assert L.workspace_bytes(L.OP_DECODE_ATTN, d) > least
    outs, accs = [], []
    for n_ws in (L.workspace_bytes(L.OP_DECODE_ATTN, d), least):
        ws = torch.full((n_ws + 4096,), 0x77, dtype=torch.uint8, device="cuda")
        accs.append(torch.zeros(B, Hkv, cap, device="cuda"))
        outs.append(L.decode_attn(q, Kc, Kc, ln, acc_score=accs[-1], ws=ws[:n_ws]))
        assert ws[n_ws:].eq(0x77).all()
    with pytest.raises(L.LvlmError) as e:
        L.decode_attn(q, Kc, Kc, ln, ws=torch.empty(least - 256, dtype=torch.uint8, device="cuda"))
    assert e.value.code == L.ERR_WORKSPACE
    assert_rows_close(f64(outs[0]), f64(outs[1]), what="attention output")
    assert_scores_close(f64(accs[0]), f64(accs[1]), what="acc_score")


def test_decode_in_parts_bad_lengths_are_skipped():
    B, H, Hkv, cap = 1, 4, 4, 1100
    q, Kc = torch.randn(B, H, 128, device="cuda").to(torch.bfloat16), torch.randn(B, Hkv, cap, 128, device="cuda").to(torch.bfloat16)
    kn, flag = torch.randn(B, Hkv, 128, device="cuda").to(torch.bfloat16), torch.zeros(1, dtype=torch.int32, device="cuda")
    ln = torch.tensor([[cap + 1, -1, cap, 700]], dtype=torch.int32, device="cuda")
    acc = torch.zeros(B, Hkv, cap, device="cuda")
    K0 = Kc.clone()
    out = L.decode_attn(q, Kc, K0, ln, k_new=kn, v_new=kn, acc_score=acc, dev_status=flag, max_len=cap)
    assert flag.item() == L.DEV_BOUNDS and ln.tolist() == [[cap + 1, -1, cap, 701]]
    assert not out[0, :2].any() and not acc[0, :2].any()
    assert abs(acc[0, 2].sum().item() - 1) < 1e-4 and abs(acc[0, 3, :701].sum().item() - 1) < 1e-4 and not acc[0, 3, 701:].any()


# waits that run out (the test build fetches no stage): the call ends and says so, and the appended row and the length are what they
# are without a timeout, in all three forms (one CTA, a cluster, parts)
@pytest.mark.parametrize("B,H,Hkv,cap", [(40, 32, 8, 100), (1, 8, 2, 150), (1, 4, 4, 4200)])
def test_decode_timeout_keeps_the_appended_row(B, H, Hkv, cap):
    q, kn, vn = (torch.randn(B, h, 128, device="cuda").to(torch.bfloat16) for h in (H, Hkv, Hkv))
    Kc, Vc = torch.zeros(B, Hkv, cap, 128, device="cuda", dtype=torch.bfloat16), torch.zeros(B, Hkv, cap, 128, device="cuda", dtype=torch.bfloat16)
    ln = (torch.arange(B * Hkv, device="cuda", dtype=torch.int32) * 37 % 97).view(B, Hkv).contiguous()
    want, at = ln + 1, ln.long()[..., None, None].expand(B, Hkv, 1, 128)
    flag = torch.zeros(1, dtype=torch.int32, device="cuda")
    try:
        L.use_library(BU.build_test())
        L.lib().lvlm_debug_starve_decode(1)
        L.decode_attn(q, Kc, Vc, ln, k_new=kn, v_new=vn, dev_status=flag, max_len=cap)
        torch.cuda.synchronize()
        L.lib().lvlm_debug_starve_decode(0)
    finally:
        L.use_library(None)
    assert flag.item() == L.DEV_TIMEOUT and torch.equal(ln, want)
    for cache, row in ((Kc, kn), (Vc, vn)):
        assert torch.equal(cache.gather(2, at)[:, :, 0], row)
        assert (cache != 0).any(dim=3).sum(dim=2).eq(1).all()                  # and no other row


# scoring: few and many tiles (small and large shape of the kernel), heads of a group in one query tile or one each, windows
# whose rows lie several times in a tile, query tiles kept over key tiles or not, splits with remainders, own normalisers
@pytest.mark.parametrize("case", [        # B, H, Hkv, N, i0, n, T, causal, lse
    (1, 1, 1, 130, 0, 1, 1, True, False), (1, 2, 2, 700, 3, 640, 32, True, False), (2, 4, 4, 513, 0, 385, 33, True, True),
    (1, 8, 1, 400, 70, 250, 64, True, False), (1, 14, 2, 1155, 5, 1025, 65, False, False), (1, 28, 4, 3012, 1, 2880, 131, True, False),
    (3, 24, 4, 1300, 0, 1283, 17, True, True), (16, 8, 2, 1500, 0, 1409, 91, True, False), (8, 12, 4, 2100, 0, 2000, 100, True, True),
    (1, 14, 2, 16000, 7, 15900, 64, True, False),          # more than eight items to a query tile
    (1, 6, 2, 1200, 100, 1000, 1200, True, False), (2, 16, 8, 1409, 0, 1409, 1409, True, False), (1, 5, 1, 900, 0, 900, 900, False, True)])
def test_score_shapes(case):
    B, H, Hkv, N, i0, n, T, causal, own = case
    g = torch.Generator(device="cuda").manual_seed(N + H)
    Q = torch.randn(B, T, H, 128, generator=g, device="cuda").to(torch.bfloat16)
    K = torch.randn(B, Hkv, N, 128, generator=g, device="cuda").to(torch.bfloat16)
    k = K.double().repeat_interleave(H // Hkv, dim=1)
    logits = torch.einsum("bthd,bhnd->bhtn", Q.double(), k) / 128 ** 0.5
    if causal:
        hidden = torch.arange(N, device="cuda")[None] > torch.arange(N - T, N, device="cuda")[:, None]
        logits.masked_fill_(hidden, -torch.inf)
    lse = torch.logsumexp(logits, dim=-1)
    s_head = torch.exp(logits - lse[..., None])[..., i0:i0 + n].sum(dim=2)
    flag = torch.zeros(1, dtype=torch.int32, device="cuda")
    for _ in range(2):                     # the second call finds the workspace as the first one left it
        score, head = L.score_tokens(Q, K, N=N, i0=i0, n=n, q_lo=N - T, q_hi=N, causal=causal, want_head=True,
                                     lse=lse.float() if own else None, dev_status=flag)
    assert flag.item() == 0
    assert_scores_close(f64(score), f64(s_head.mean(dim=1)), what="score")
    assert_scores_close(f64(head), f64(s_head.view(B, Hkv, H // Hkv, n).sum(dim=2)), what="score_head")


# attention: pairs of heads, pairs of query tiles of the odd head, a lone last tile; the key tiles of one query tile split
# between the halves of a CTA (few tiles); one key tile, ragged ends, rows that see one key
@pytest.mark.parametrize("case", [        # B, H, Hkv, N, causal
    (1, 1, 1, 1, True), (1, 2, 2, 128, True), (1, 3, 1, 129, False), (1, 7, 1, 257, True), (2, 8, 2, 384, True),
    (1, 28, 4, 1025, True), (6, 12, 4, 900, True), (3, 9, 3, 1300, False), (1, 48, 8, 1409, True), (13, 8, 8, 515, True)])
def test_attention_shapes(case):
    B, H, Hkv, N, causal = case
    g = torch.Generator(device="cuda").manual_seed(N + H)
    Q = (3 * torch.randn(B, N, H, 128, generator=g, device="cuda")).to(torch.bfloat16)
    K = torch.randn(B, Hkv, N, 128, generator=g, device="cuda").to(torch.bfloat16)
    V = torch.randn(B, Hkv, N, 128, generator=g, device="cuda").to(torch.bfloat16)
    out, lse = torch.full_like(Q, 9.0), torch.empty(B, H, N, device="cuda")
    flag = torch.zeros(1, dtype=torch.int32, device="cuda")
    first = None
    for _ in range(4):
        L.prefill_attn(Q, K, V, N=N, causal=causal, out=out, lse=lse, dev_status=flag)
        first = out.clone() if first is None else first
        assert torch.equal(out, first)
    logits = torch.einsum("bthd,bhnd->bhtn", Q.double(), K.double().repeat_interleave(H // Hkv, dim=1)) / 128 ** 0.5
    if causal:
        logits.masked_fill_(torch.ones(N, N, dtype=torch.bool, device="cuda").triu(1), -torch.inf)
    want = torch.einsum("bhtn,bhnd->bthd", torch.softmax(logits, dim=-1), V.double().repeat_interleave(H // Hkv, dim=1))
    assert flag.item() == 0
    assert_rows_close(f64(out), f64(want), what="attention output")
    np.testing.assert_allclose(f64(lse), f64(torch.logsumexp(logits, dim=-1)), rtol=1e-5, atol=1e-5)   # fp32 sums


# the warpgroups' registers are shared out anew inside the kernel: launched with too few it would wait for ever, so it is not launched
def test_attention_refuses_too_few_registers():
    Q, K = torch.randn(1, 200, 2, 128, device="cuda").bfloat16(), torch.randn(1, 1, 200, 128, device="cuda").bfloat16()
    out, lse = torch.full_like(Q, 9.0), torch.empty(1, 2, 200, device="cuda")
    try:
        L.use_library(BU.build_test())
        L.lib().lvlm_debug_set_attn_regs(160)
        with pytest.raises(L.LvlmError) as e:
            L.prefill_attn(Q, K, K, N=200, out=out, lse=lse)
        torch.cuda.synchronize()
        assert e.value.code == L.ERR_CUDA and out.eq(9).all()
        L.lib().lvlm_debug_set_attn_regs(168)                # ... 3 x 168 = 104 + 2 x 200
        L.prefill_attn(Q, K, K, N=200, out=out, lse=lse)
        assert not out.eq(9).any()
    finally:
        L.lib().lvlm_debug_set_attn_regs(0)
        L.use_library(None)


# nearest-kept grouping: every dropped token to one kept token (one long segment), segments around a warp's 32 tokens, none
# at all for most; text rows that are the source of rows before them; runs over several CTAs of the plan's cluster
@pytest.mark.parametrize("case", [        # B, C, Hkv, i0, n, T, k, kept tokens that attract the dropped ones
    (1, 64, 1, 0, 40, 5, 7, 1), (2, 128, 2, 3, 300, 20, 33, 1), (1, 256, 1, 0, 700, 600, 20, 20), (1, 64, 2, 17, 4500, 31, 2500, 60),
    (3, 72, 1, 2, 2100, 300, 100, 3), (1, 64, 1, 0, 9000, 10, 1030, 1030),
    (1, 64, 1, 0, 8970, 3, 4500, 700)])    # (similarity: two groups of column tiles, an odd row tile, items cut in two behind whole ones)
def test_nearest_kept_groups(case):
    B, C, Hkv, i0, n, T, k, attract = case
    r = np.random.default_rng(n + k)
    N = i0 + n + T
    rank = np.stack([r.permutation(n) for _ in range(B)]).astype(np.int32)
    hidden = r.normal(size=(B, N, C)).astype(np.float32)
    for b in range(B):
        by_rank = np.argsort(rank[b])
        to = by_rank[:attract][r.integers(0, attract, size=n - k)]
        hidden[b, i0 + by_rank[k:]] = hidden[b, i0 + to] + 0.05 * hidden[b, i0 + by_rank[k:]]
    hid = torch.from_numpy(hidden).to(torch.bfloat16)
    K, V = (torch.from_numpy(r.normal(size=(B, Hkv, N, 128)).astype(np.float32)).to(torch.bfloat16) for _ in range(2))
    pos = np.tile(np.arange(N, dtype=np.int32), (B, 1))
    mass = (r.integers(1, 5, size=(B, N))).astype(np.float32)
    want = O.nearest_kept_merge(f64(hid), rank, i0, n, k, Kc=f64(K), Vc=f64(V), pos_ids=pos, mass=mass)
    Kd, Vd, pd, md = K.cuda(), V.cuda(), torch.from_numpy(pos).cuda(), torch.from_numpy(mass).cuda()
    flag = torch.zeros(1, dtype=torch.int32, device="cuda")
    out, new_len = L.merge_compact(hid.cuda(), torch.from_numpy(rank).cuda(), i0=i0, k=k, mode=L.W_NEAREST_KEPT, Kc=Kd, Vc=Vd,
                                   pos_ids=pd, mass=md, dev_status=flag)
    Nout = N - (n - k)
    assert flag.item() == 0 and new_len.tolist() == [Nout] * B
    assert_rows_close(f64(out), want["hidden"], what="hidden")
    assert_rows_close(f64(Kd)[:, :, :Nout], want["Kc"], what="K")
    assert_rows_close(f64(Vd)[:, :, :Nout], want["Vc"], what="V")
    assert np.array_equal(i32(pd)[:, :Nout], want["pos_ids"])
    np.testing.assert_allclose(md.cpu().numpy()[:, :Nout], want["mass"], rtol=1e-6)                 # small whole numbers


# cache compression, a CTA per head: scores that tie in one or a few values, keys that differ in one bit, in few bits or in
# all, entries that outweigh all others by 2^40, caches at the ends of a thread's 4 and 16 entries
@pytest.mark.parametrize("cap", [1, 31, 4096, 4097, 16384])
@pytest.mark.parametrize("kind", ["one_value", "two_neighbours", "four_values", "wide"])
def test_kv_threshold_search(cap, kind):
    r = np.random.default_rng(cap)
    acc = {"one_value": np.full((1, 3, cap), 0.3), "two_neighbours": 0.5 + (r.random((1, 3, cap)) < 0.5) * 2.0 ** -24,
           "four_values": r.integers(0, 4, size=(1, 3, cap)) * 0.125,
           "wide": 2.0 ** r.uniform(-24, 16, size=(1, 3, cap))}[kind].astype(np.float32)
    ln = np.array([[cap, max(1, cap - 5), (cap + 1) // 2]], np.int32)
    Kc = torch.from_numpy(r.normal(size=(1, 3, cap, 128)).astype(np.float32)).to(torch.bfloat16)
    for beta, budget in ((0.5, 0), (0.999, 0), (0.9, cap // 3), (1.0, max(1, cap // 2))):
        want = O.kv_compress(f64(Kc), f64(Kc), acc, ln, beta=beta, budget=budget or None)
        Kd, Vd, ad, ld = Kc.cuda(), Kc.cuda(), torch.from_numpy(acc).cuda(), torch.from_numpy(ln).cuda()
        flag = torch.zeros(1, dtype=torch.int32, device="cuda")
        L.kv_compress(Kd, Vd, ad, ld, beta=beta, budget=budget, dev_status=flag)
        assert flag.item() == 0 and np.array_equal(i32(ld), want["len"]), (beta, budget)
        for g in range(3):
            m = want["len"][0, g]
            assert np.array_equal(ad[0, g, :m].cpu().numpy(), want["acc_score"][0, g, :m]), (beta, budget, g)
            assert np.array_equal(f64(Kd)[0, g, :m], want["Kc"][0, g, :m].astype(np.float64)), (beta, budget, g)


# the same, scores whose sum in units of 2^-24 needs up to 63 bits, or more: whole multiples of one power of two, so that a coarser
# unit counts them exactly as well; a CTA per head (few heads) and a warp per head
@pytest.mark.parametrize("heads,cap", [(2, 7), (3, 1000), (2, 4100), (592, 33)])
@pytest.mark.parametrize("exponent", [24, 29, 39, 90, 117])
def test_kv_threshold_of_huge_scores(heads, cap, exponent):
    r = np.random.default_rng(cap + exponent)
    acc = (r.integers(0, 1000, size=(1, heads, cap)) * 2.0 ** exponent).astype(np.float32)
    acc[0, 0] = 2.0 ** exponent                                          # all alike
    acc[0, 1, cap // 2] = np.inf
    ln = np.full((1, heads), cap, np.int32)
    Kc = torch.from_numpy(r.normal(size=(1, heads, cap, 128)).astype(np.float32)).to(torch.bfloat16)
    for beta in (0.5, 0.97):
        want = O.kv_compress(f64(Kc), f64(Kc), acc, ln, beta=beta)
        Kd, Vd, ad, ld = Kc.cuda(), Kc.cuda(), torch.from_numpy(acc).cuda(), torch.from_numpy(ln).cuda()
        flag = torch.zeros(1, dtype=torch.int32, device="cuda")
        L.kv_compress(Kd, Vd, ad, ld, beta=beta, dev_status=flag)
        assert flag.item() == L.DEV_NONFINITE and np.array_equal(i32(ld), want["len"]), beta
        for g in range(0, heads, max(1, heads // 16)):
            m = want["len"][0, g]
            assert np.array_equal(ad[0, g, :m].cpu().numpy(), want["acc_score"][0, g, :m]), (beta, g)
            assert np.array_equal(f64(Kd)[0, g, :m], want["Kc"][0, g, :m].astype(np.float64)), (beta, g)


# selection by bins: 1, 2, 4 and 8 slices, 1, 2 and 4 tokens a thread, last slices that are shorter; bins as deep as they may be
# and one key deeper, one bin for all but one key, one value
@pytest.mark.parametrize("B,n", [(1, 511), (1, 512), (1, 1023), (1, 1025), (1, 2049), (1, 14337), (2, 34817), (37, 3001), (140, 1100)])
@pytest.mark.parametrize("kind", ["random", "deep", "outlier", "one_value"])
def test_select_bins(B, n, kind):
    r = np.random.default_rng(n)
    s = {"random": r.random((B, n)), "deep": (np.arange(n) * 4 // (n + n % 2)) * 0.25 + np.zeros((B, 1)),
         "outlier": np.where(np.arange(n) == n // 2, 1e30, 1.0 + r.random((B, n)) * 1e-3), "one_value": np.full((B, n), -0.5)}[kind]
    s = s.astype(np.float32)
    if kind != "deep":
        s[0] = s[0, r.permutation(n)]
    flag = torch.zeros(1, dtype=torch.int32, device="cuda")
    rank, _, _ = L.select_topk(torch.from_numpy(s).cuda(), n // 3, want_kept=False, dev_status=flag)
    order = np.argsort(-s, axis=1, kind="stable")                # whole numbers: nothing to tolerate
    want = np.empty_like(order)
    np.put_along_axis(want, order, np.arange(n)[None].repeat(B, 0), axis=1)
    assert flag.item() == 0 and np.array_equal(i32(rank), want)


# the plan of a merge: 1 to 8 CTAs of 1 to 4 tokens a thread, more than one round (a lone wide batch keeps rows short), image spans
# that end inside a warp, text behind the image of less and more than one round of rows, the first and the last token on top
@pytest.mark.parametrize("case", [        # N, i0, n, k
    (40, 0, 33, 1), (1100, 3, 1025, 700), (3000, 0, 2049, 100), (9000, 7, 8193, 8000), (33500, 0, 32769, 20000),
    (70000, 5, 65530, 3), (100040, 3, 100000, 40000), (30000, 2, 300, 200), (13000, 1, 3000, 0),
    (6001, 0, 33, 1), (6100, 3, 1025, 700), (6300, 0, 2049, 100)])      # (the first three are merged in one launch, without a plan)
@pytest.mark.parametrize("order", ["random", "first", "last"])
def test_merge_plan_rounds(case, order):
    N, i0, n, k = case
    r = np.random.default_rng(N)
    rank = {"random": r.permutation(n), "first": np.arange(n), "last": np.arange(n)[::-1].copy()}[order].astype(np.int32)
    hid = torch.from_numpy(r.normal(size=(1, N, 8)).astype(np.float32)).to(torch.bfloat16)
    pos = r.integers(0, 1 << 30, size=(1, N)).astype(np.int32)
    pd, flag = torch.from_numpy(pos.copy()).cuda(), torch.zeros(1, dtype=torch.int32, device="cuda")
    out, new_len = L.merge_compact(hid.cuda(), torch.from_numpy(rank[None]).cuda(), i0=i0, k=k, pos_ids=pd, dev_status=flag)
    kept = i0 + np.flatnonzero(rank < k)
    src = np.concatenate([np.arange(i0), kept, [i0 + int(np.flatnonzero(rank == k)[0])], np.arange(i0 + n, N)])
    assert flag.item() == 0 and new_len.item() == src.size
    assert np.array_equal(i32(pd)[0, :src.size], pos[0, src])            # whole numbers and rows that move: nothing to tolerate
    stay = np.arange(src.size) != i0 + k
    assert np.array_equal(f64(out)[0, stay], f64(hid)[0, src[stay]])


# a rank that is no permutation is reported, and no map entry that nobody wrote is followed
@pytest.mark.parametrize("N", [2000, 6600])              # (rank weights: in one launch, in three)
@pytest.mark.parametrize("mode", [L.W_LINEAR_RANK, L.W_NEAREST_KEPT])
@pytest.mark.parametrize("value", [0, 299, -5, 1 << 30])
def test_merge_of_a_bad_rank(mode, value, N):
    i0, n, k, C = 7, N - 100, 300, 64
    hid = torch.randn(1, N, C, device="cuda").bfloat16()
    K, V = (torch.randn(1, 2, N, 128, device="cuda").bfloat16() for _ in range(2))
    K0, flag = K.clone(), torch.zeros(1, dtype=torch.int32, device="cuda")
    rank = torch.full((1, n), value, dtype=torch.int32, device="cuda")
    if value == 1 << 30:
        rank[0, :200] = torch.arange(200, device="cuda")              # too few kept tokens
    ws = torch.full((1 << 24,), 0x7F, dtype=torch.uint8, device="cuda")     # (map entries that nobody writes would point far away)
    L.merge_compact(hid, rank, i0=i0, k=k, mode=mode, Kc=K, Vc=V, ws=ws, dev_status=flag)
    torch.cuda.synchronize()
    assert flag.item() == L.DEV_BOUNDS
    assert torch.equal(K[:, :, :i0], K0[:, :, :i0])


# the merged rows, from few and from many partial sums of the passes over the rows (1 to 16 threads add up a column group), of
# narrow rows and of rows wider than a column group per thread
@pytest.mark.parametrize("case", [        # B, N, i0, n, C, Hkv, k
    (1, 1000, 2, 900, 64, 1, 300), (1, 2500, 0, 2450, 8192, 1, 1000), (1, 9600, 0, 9500, 1024, 2, 4000), (6, 2100, 5, 2000, 512, 3, 700),
    (1, 6100, 2, 6000, 64, 1, 300), (1, 4800, 0, 4750, 8192, 1, 1000), (8, 2400, 5, 2300, 512, 3, 700)])       # (in three launches)
@pytest.mark.parametrize("in_place", [False, True])
def test_merge_partial_sums(case, in_place):
    B, N, i0, n, C, Hkv, k = case
    r = np.random.default_rng(N)
    hid, Kc, Vc = (torch.from_numpy(r.normal(size=s).astype(np.float32)).to(torch.bfloat16)
                   for s in ((B, N, C), (B, Hkv, N, 128), (B, Hkv, N, 128)))
    rank = np.stack([r.permutation(n) for _ in range(B)]).astype(np.int32)
    want = O.merge_compact(f64(hid), rank, i0, n, k, Kc=f64(Kc), Vc=f64(Vc))
    Kd, Vd, flag = Kc.cuda(), Vc.cuda(), torch.zeros(1, dtype=torch.int32, device="cuda")
    out, _ = L.merge_compact(hid.cuda(), torch.from_numpy(rank).cuda(), i0=i0, k=k, Kc=Kd, Vc=Vd, in_place=in_place, dev_status=flag)
    assert flag.item() == 0
    Nout = L.merged_rows(N, n, k)
    # a unit in the last place of bf16 (2^-7) where the two sums round apart, and fp32 sums of up to 300 terms in a row, whose
    # weights add up to one: 300 x 2^-24 x the largest |x| (below 6) < 1.1e-4
    for got, w, what in ((out[:, None], want["hidden"][:, None], "hidden"), (Kd, want["Kc"], "K"), (Vd, want["Vc"], "V")):
        got, w = f64(got)[:, :, :Nout], w.astype(np.float64)[:, :, :Nout]
        assert_rows_close(got[:, :, i0 + k], w[:, :, i0 + k], rtol=2.0 ** -7, atol=1.1e-4, what=what)
        got[:, :, i0 + k] = w[:, :, i0 + k]
        assert np.array_equal(got, w), what


# every weight rule where the rows take three launches: weights that underflow, a queue of two, weights of the caller's own
@pytest.mark.parametrize("mode", [L.W_GEOMETRIC, L.W_UNIFORM, L.W_CUSTOM])
@pytest.mark.parametrize("k", [300, 5898])
def test_merge_weights_in_three_launches(mode, k):
    B, N, i0, n, C, Hkv = 1, 6100, 2, 5900, 72, 2
    r = np.random.default_rng(k)
    hid, Kc, Vc = (torch.from_numpy(r.normal(size=s).astype(np.float32)).to(torch.bfloat16)
                   for s in ((B, N, C), (B, Hkv, N, 128), (B, Hkv, N, 128)))
    rank, custom = r.permutation(n)[None].astype(np.int32), (r.random(n - k) + 0.1).astype(np.float32)
    want = O.merge_compact(f64(hid), rank, i0, n, k, Kc=f64(Kc), Vc=f64(Vc), custom=custom if mode == L.W_CUSTOM else None,
                           mode={L.W_GEOMETRIC: O.GEOMETRIC, L.W_UNIFORM: O.UNIFORM, L.W_CUSTOM: O.CUSTOM}[mode])
    hd, rd, Kd, Vd, flag = hid.cuda(), torch.from_numpy(rank).cuda(), Kc.cuda(), Vc.cuda(), torch.zeros(1, dtype=torch.int32, device="cuda")
    w = torch.from_numpy(custom).cuda() if mode == L.W_CUSTOM else None
    assert count_launches(lambda: L.merge_compact(hd, rd, i0=i0, k=k, mode=mode, Kc=Kd, Vc=Vd, w_custom=w)) == 3
    out, _ = L.merge_compact(hd, rd, i0=i0, k=k, mode=mode, Kc=Kd, Vc=Vd, w_custom=w, dev_status=flag)
    assert flag.item() == 0
    Nout = L.merged_rows(N, n, k)
    # a unit in the last place of bf16; fp32 sums of at most 129 rows of a chunk of K or V and 46 chunks (of the hidden states fewer), and
    # weights that add up to one and are off by some 40 roundings: 215 x 2^-24 x the largest |x| (below 6) < 8e-5
    for got, w, what in ((out[:, None], want["hidden"][:, None], "hidden"), (Kd, want["Kc"], "K"), (Vd, want["Vc"], "V")):
        got, w = f64(got)[:, :, :Nout], w.astype(np.float64)[:, :, :Nout]
        assert_rows_close(got[:, :, i0 + k], w[:, :, i0 + k], rtol=2.0 ** -7, atol=8e-5, what=what)
        got[:, :, i0 + k] = w[:, :, i0 + k]
        assert np.array_equal(got, w), what


# a merge in one launch: columns of 64, 128 and 256 bytes, last ones that are narrower, one to eight CTAs a column, runs that end
# inside the rows ahead of, in and behind the image; and one row more than it takes (three launches)
@pytest.mark.parametrize("case", [        # B, N, i0, n, C, Hkv, k, launches
    (1, 1, 0, 1, 8, 0, 0, None), (1, 40, 3, 33, 72, 1, 5, 1), (1, 257, 0, 255, 8, 2, 253, 1), (1, 3008, 0, 2880, 3584, 4, 300, 1),
    (3, 900, 60, 800, 200, 3, 0, 1), (1, 1300, 35, 1200, 6144, 8, 600, 1), (16, 264, 0, 200, 1024, 8, 60, 1), (16, 464, 1, 400, 1024, 8, 120, 1),
    (1, 2000, 1700, 290, 64, 2, 100, 1), (1, 6000, 5, 5990, 64, 1, 2999, 1), (1, 6001, 5, 5990, 64, 1, 2999, 3)])
@pytest.mark.parametrize("mode,in_place", [(L.W_LINEAR_RANK, False), (L.W_CUSTOM, True)])
def test_merge_in_one_launch(case, mode, in_place):
    B, N, i0, n, C, Hkv, k, launches = case
    r = np.random.default_rng(N + C)
    bf = lambda *s: torch.from_numpy(r.normal(size=s).astype(np.float32)).to(torch.bfloat16)
    hid, Kc, Vc = bf(B, N, C), bf(B, max(Hkv, 1), N + 3, 128), bf(B, max(Hkv, 1), N + 3, 128)
    rank = np.stack([r.permutation(n) for _ in range(B)]).astype(np.int32)
    custom = (r.random(n - k) + 0.1).astype(np.float32) if mode == L.W_CUSTOM else None
    pos = r.integers(0, 1 << 30, size=(B, N)).astype(np.int32)
    want = O.merge_compact(f64(hid), rank, i0, n, k, mode=O.CUSTOM if custom is not None else O.LINEAR_RANK, custom=custom,
                           Kc=f64(Kc)[:, :, :N], Vc=f64(Vc)[:, :, :N], pos_ids=pos)
    rd, flag = torch.from_numpy(rank).cuda(), torch.zeros(1, dtype=torch.int32, device="cuda")
    hd, Kd, Vd, pd = hid.cuda(), Kc.cuda(), Vc.cuda(), torch.from_numpy(pos).cuda()
    out, new_len, Nout = None if in_place else torch.empty(B, want["hidden"].shape[1], C, dtype=hid.dtype, device="cuda"), torch.empty(B, dtype=torch.int32, device="cuda"), L.merged_rows(N, n, k)
    ws = torch.empty(1 << 24, dtype=torch.uint8, device="cuda")

    def call():
        L.merge_compact(hd, rd, i0=i0, k=k, mode=mode, Kc=Kd if Hkv else None, Vc=Vd if Hkv else None, pos_ids=pd, in_place=in_place, out=out,
                        w_custom=None if custom is None else torch.from_numpy(custom).cuda(), new_len=new_len, ws=ws, dev_status=flag)

    call()
    assert flag.item() == 0 and new_len.tolist() == [Nout] * B
    got = [(hd if in_place else out)[:, None, :Nout]] + ([Kd[:, :, :Nout], Vd[:, :, :Nout]] if Hkv else [])
    for x, w, what in zip(got, (want["hidden"][:, None], want["Kc"], want["Vc"]), ("hidden", "K", "V")):
        x, w = f64(x), w.astype(np.float64)[:, :, :Nout]
        # a unit in the last place of bf16; fp32 sums of at most 49 rows in a row (no CTA has more than 3129), 3 + 8 + 8 more steps over
        # the threads, warps and CTAs, and weights off by some 40 roundings: 108 x 2^-24 x the largest |x| (below 6) < 4e-5
        if Nout < N:
            assert_rows_close(x[:, :, i0 + k], w[:, :, i0 + k], rtol=2.0 ** -7, atol=4e-5, what=what)
            x[:, :, i0 + k] = w[:, :, i0 + k]
        assert np.array_equal(x, w), what
    assert np.array_equal(i32(pd)[:, :Nout], want["pos_ids"][:, :Nout])
    if Hkv:
        assert torch.equal(Kd[:, :, N:].cpu(), Kc[:, :, N:]) and torch.equal(Vd[:, :, N:].cpu(), Vc[:, :, N:])
    if launches and custom is None:
        assert count_launches(call) == launches


# the merged row of the hidden states is the same bits without K and V and with any number of heads of them, on both sides of the limit
# of a merge in one launch and where column widths and cluster sizes change
@pytest.mark.parametrize("B,N,C", [(1, 640, 1024), (3, 689, 1024), (9, 502, 1024), (2, 5900, 1024), (3, 4500, 1024), (1, 3008, 3584), (2, 3400, 3584), (2, 3500, 3584),
                                   (2, 1107, 3584), (8, 407, 3584), (2, 4064, 3584), (16, 264, 4096), (1, 6500, 512)])
def test_hidden_merge_does_not_depend_on_kv(B, N, C):
    g = torch.Generator(device="cuda").manual_seed(N)
    n, k = N - 33, N // 5
    hid = torch.randn(B, N, C, generator=g, device="cuda").bfloat16()
    rank = torch.argsort(torch.rand(B, n, generator=g, device="cuda"), dim=1).int()
    want, _ = L.merge_compact(hid, rank, i0=1, k=k)
    for heads in (1, 2, 4, 8, 16):
        K = torch.randn(B, heads, N, 128, generator=g, device="cuda").bfloat16()
        got, _ = L.merge_compact(hid, rank, i0=1, k=k, Kc=K, Vc=K.clone())
        assert torch.equal(got, want), heads


def _scoring(case):
    """Inputs of a scoring call and its scores in 64 bits."""
    B, H, Hkv, N, i0, n, T, causal = case
    g = torch.Generator(device="cuda").manual_seed(N + H)
    Q = torch.randn(B, T, H, 128, generator=g, device="cuda").to(torch.bfloat16)
    K = torch.randn(B, Hkv, N, 128, generator=g, device="cuda").to(torch.bfloat16)
    heads = torch.empty(B, H, n, device="cuda", dtype=torch.float64)
    for b in range(B):
        logits = torch.einsum("thd,hnd->htn", Q[b].double(), K[b].double().repeat_interleave(H // Hkv, dim=0)) / 128 ** 0.5
        if causal:
            logits.masked_fill_(torch.arange(N, device="cuda")[None] > torch.arange(N - T, N, device="cuda")[:, None], -torch.inf)
        heads[b] = torch.softmax(logits, dim=-1)[..., i0:i0 + n].sum(dim=1)
    return Q, K, heads.mean(dim=1), heads.view(B, Hkv, H // Hkv, n).sum(dim=2)


def _check_scoring(case):
    """Runs the call and returns how many kernels it launches."""
    B, H, Hkv, N, i0, n, T, causal = case
    Q, K, want, want_head = _scoring(case)
    flag = torch.zeros(1, dtype=torch.int32, device="cuda")

    def call():
        return L.score_tokens(Q, K, N=N, i0=i0, n=n, q_lo=N - T, q_hi=N, causal=causal, want_head=True, dev_status=flag)

    for _ in range(2):                     # the second call finds the workspace as the first one left it
        score, head = call()
    assert flag.item() == 0
    for got, w in ((score, want), (head, want_head)):
        assert_scores_close(f64(got), f64(w), what="score")
        # an exponential is good to two units in the last place (2^-22), a logit and its normaliser to about one more together
        assert torch.linalg.vector_norm(got.double() - w) < 2.0 ** -21 * torch.linalg.vector_norm(w)
    return count_launches(call)


# scoring in one pass over Q K^T: one to four key tiles a CTA, one to eight CTAs a cluster; of the shapes with one or two tiles a CTA
# (where teams take turns) and of the others some with a query tile or two a cluster and some with up to 14, which use
# every barrier and buffer of the exchange again and again; runs that share a KV group, rows of a query tile that are not there
@pytest.mark.parametrize("case", [        # B, H, Hkv, N, i0, n, T, causal          key tiles a CTA x CTAs, query tiles a cluster
    (1, 1, 1, 2, 0, 1, 1, True), (1, 3, 3, 128, 1, 100, 27, True), (1, 8, 1, 129, 0, 64, 65, True),      # 1 x 1, 1 x 1, 1 x 2
    (30, 56, 7, 110, 0, 60, 50, True), (6, 56, 7, 355, 5, 300, 50, True), (1, 8, 1, 900, 0, 300, 600, True),           # 1 x 1: 6, 1 x 3: 4, 1 x 8: 3
    (24, 12, 2, 250, 9, 200, 41, True), (30, 42, 7, 505, 5, 400, 100, True), (6, 49, 7, 700, 0, 600, 100, True),       # 2 x 1, 2 x 2: 14, 2 x 3: 6
    (4, 64, 8, 1000, 0, 900, 100, True), (2, 7, 7, 2005, 5, 1700, 300, True),                                          # 2 x 4: 7, 2 x 8: 3
    (20, 56, 7, 350, 0, 300, 50, True), (2, 42, 7, 700, 0, 400, 300, True), (13, 4, 1, 2933, 0, 2900, 33, True),       # 3 x 1: 4, 3 x 2: 3, 3 x 8: 2
    (30, 56, 7, 500, 0, 400, 100, True), (20, 56, 7, 950, 0, 900, 50, True), (2, 24, 8, 2005, 5, 1700, 300, True),     # 4 x 1: 10, 4 x 2: 8, 4 x 4: 4
    (3, 64, 8, 2550, 0, 2500, 50, False), (5, 12, 3, 3496, 0, 3400, 96, True), (1, 28, 4, 4096, 0, 3968, 128, True)])  # 4 x 5: 4, 4 x 7: 3, 4 x 8: 2
def test_score_one_pass(case):
    assert _check_scoring(case) == 2


# sums of another CTA that never come (the test build keeps the first CTA of a cluster from sending): the call ends and says so, and
# the next one is as ever; with one, two and four key tiles a CTA
@pytest.mark.parametrize("case", [(1, 8, 1, 129, 0, 64, 65, True), (4, 64, 8, 1000, 0, 900, 100, True), (1, 28, 4, 4096, 0, 3968, 128, True)])
def test_score_one_pass_timeout(case):
    B, H, Hkv, N, i0, n, T, causal = case
    Q, K, want, _ = _scoring(case)
    try:
        L.use_library(BU.build_test())
        for starve in (1, 0):
            flag = torch.zeros(1, dtype=torch.int32, device="cuda")
            L.lib().lvlm_debug_starve_score(starve)
            score, _ = L.score_tokens(Q, K, N=N, i0=i0, n=n, q_lo=N - T, q_hi=N, causal=causal, dev_status=flag)
            torch.cuda.synchronize()
            assert flag.item() & L.DEV_TIMEOUT if starve else flag.item() == 0
    finally:
        L.lib().lvlm_debug_starve_score(0)
        L.use_library(None)
    assert_scores_close(f64(score), f64(want), what="score")


# scoring in two passes: one key more than a cluster holds, windows that begin among the scored keys, shapes where it is quicker; with
# few rows pass 1 has them two or four times in a query tile, on the small and on the large shape of the kernel
@pytest.mark.parametrize("case", [
    (1, 4, 2, 4097, 0, 3968, 129, True), (40, 16, 8, 700, 0, 600, 100, True), (30, 7, 7, 2100, 0, 2000, 100, True),
    (1, 2, 2, 700, 3, 690, 32, True), (1, 8, 2, 4300, 0, 4200, 1, True), (1, 14, 2, 5000, 0, 4900, 9, True),
    (1, 4, 4, 6000, 5, 5900, 33, False), (13, 4, 4, 4500, 3, 4400, 17, True), (20, 3, 3, 4200, 0, 4100, 33, True)])
def test_score_two_passes(case):
    assert _check_scoring(case) > 2


# cache compression with 4, 8 and 16 entries a thread, few heads and more heads than SMs, at the ends of the ranges of each
@pytest.mark.parametrize("heads,cap", [(148, 1025), (149, 1025), (148, 4096), (149, 2055), (149, 3584), (149, 3585), (149, 4097),
                                       (2, 4097), (2, 8191), (2, 8193)])
def test_kv_entries_a_thread(heads, cap):
    r = np.random.default_rng(heads + cap)
    acc = r.integers(0, 40, size=(1, heads, cap)).astype(np.float32) * 0.25
    ln = r.integers(1, cap + 1, size=(1, heads)).astype(np.int32)
    Kc = torch.from_numpy(r.normal(size=(1, heads, cap, 128)).astype(np.float32)).to(torch.bfloat16)
    for beta, budget in ((0.9, 0), (1.0, cap // 2)):
        want = O.kv_compress(f64(Kc), f64(Kc), acc, ln, beta=beta, budget=budget or None)
        Kd, Vd, ad, ld = Kc.cuda(), Kc.cuda(), torch.from_numpy(acc).cuda(), torch.from_numpy(ln).cuda()
        L.kv_compress(Kd, Vd, ad, ld, beta=beta, budget=budget)
        assert np.array_equal(i32(ld), want["len"]), (beta, budget)
        for g in range(0, heads, max(1, heads // 8)):
            m = want["len"][0, g]
            assert np.array_equal(ad[0, g, :m].cpu().numpy(), want["acc_score"][0, g, :m]), (beta, budget, g)
            assert np.array_equal(f64(Kd[0, g, :m]), want["Kc"][0, g, :m].astype(np.float64)), (beta, budget, g)
