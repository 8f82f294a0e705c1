"""GPU tests of the kernel variants that a call's sizes choose between, at the sizes where each can go wrong
(edges of tiles and parts, remainders, the ends of a variant's range), against the CPU oracle."""
import numpy as np
import pytest
import torch

from oracle import lvlm_oracle as O
from paper_2509_00419_b200 import binding as L
from tests.util import assert_rows_close, assert_scores_close, f64, i32

pytestmark = pytest.mark.gpu


# decode attention cut into parts that a second launch adds: few heads with long caches, or more heads than clusters fit
@pytest.mark.parametrize("case", [        # B, H, Hkv, cap, append, acc_score
    (1, 1, 1, 512, True, True), (1, 3, 1, 1037, False, True), (1, 7, 1, 256, True, False), (2, 8, 1, 545, True, False),
    (1, 28, 4, 1024, True, False), (5, 8, 4, 511, True, True), (9, 24, 4, 223, True, True), (8, 16, 4, 224, False, False),
    (1, 2, 2, 7001, True, True)])
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
                        acc_score=ad, dev_status=flag)
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


def test_decode_in_parts_bad_lengths_are_skipped():
    B, H, Hkv, cap = 1, 4, 4, 1100
    q, Kc = torch.randn(B, H, 128, device="cuda").to(torch.bfloat16), torch.randn(B, Hkv, cap, 128, device="cuda").to(torch.bfloat16)
    kn, flag = torch.randn(B, Hkv, 128, device="cuda").to(torch.bfloat16), torch.zeros(1, dtype=torch.int32, device="cuda")
    ln = torch.tensor([[cap + 1, -1, cap, 700]], dtype=torch.int32, device="cuda")
    acc = torch.zeros(B, Hkv, cap, device="cuda")
    K0 = Kc.clone()
    out = L.decode_attn(q, Kc, K0, ln, k_new=kn, v_new=kn, acc_score=acc, dev_status=flag)
    assert flag.item() == L.DEV_BOUNDS and ln.tolist() == [[cap + 1, -1, cap, 701]]
    assert not out[0, :2].any() and not acc[0, :2].any()
    assert abs(acc[0, 2].sum().item() - 1) < 1e-4 and abs(acc[0, 3, :701].sum().item() - 1) < 1e-4 and not acc[0, 3, 701:].any()
