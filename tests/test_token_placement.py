"""Placement of new K/V rows (GPU): the row search of the KV append, the fp8
append and the fused RoPE append at the edges of its five-level steps, with
empty rows, ragged chunks and token counts that do not fill a CTA."""
from __future__ import annotations

import numpy as np
import pytest
import torch

import workloads as W
from _gpu import to_fp8_blocks
from paper_2608_22167_gb300 import mcpu

pytestmark = pytest.mark.gpu


def _batch(B, seed):
    rng = np.random.Generator(np.random.PCG64(seed))
    L = rng.choice([0, 1, 1, 1, 3, 17], size=B)
    L[rng.integers(0, B)] = 5  # at least one token
    S = L + rng.integers(0, 40, size=B)
    qsl = np.concatenate([[0], np.cumsum(L)])
    pages = -(-S // 16)
    bt = np.full((B, max(1, int(pages.max()))), -1, np.int64)
    perm = rng.permutation(int(pages.sum()) + 3)
    at = 0
    for r in range(B):
        bt[r, : pages[r]] = perm[at : at + pages[r]]
        at += int(pages[r])
    row = np.repeat(np.arange(B), L)
    pos = np.concatenate([np.arange(s - n, s) for s, n in zip(S, L)])
    dst = bt[row, pos // 16] * 16 + pos % 16
    dev = lambda x: torch.from_numpy(np.ascontiguousarray(x, np.int32)).cuda()  # noqa: E731
    return dev(bt), dev(S), dev(qsl), torch.from_numpy(dst).cuda(), torch.from_numpy(pos).cuda(), len(perm)


@pytest.mark.parametrize("hkv", [1, 8, 20])
@pytest.mark.parametrize("B", [1, 2, 31, 32, 33, 64, 1023, 1025, 2048])
def test_every_token_lands_in_its_slot(B, hkv):
    bt, sl, qsl, dst, pos, P = _batch(B, B + hkv)
    T = dst.numel()
    k = torch.randn(T, hkv, 64, device="cuda").bfloat16()
    v = torch.randn(T, hkv, 64, device="cuda").bfloat16()
    st = torch.zeros(1, dtype=torch.int32, device="cuda")

    def placed(new):
        pool = torch.zeros(P * 16, hkv, 64, dtype=new.dtype, device="cuda")
        pool[dst] = new
        return pool.view(P, 16, hkv, 64).transpose(1, 2).contiguous()

    kc, vc = (torch.zeros(P, hkv, 16, 64, dtype=torch.bfloat16, device="cuda") for _ in range(2))
    mcpu.mcpu_kv_append(k, v, kc, vc, bt, sl, qsl, st)
    assert torch.equal(kc, placed(k)) and torch.equal(vc, placed(v))

    # the fp8 append over zeroed blocks: K and V codes and scales, whole blocks
    # (slots of no token stay zero)
    kv8 = torch.zeros(P, hkv, 2176, dtype=torch.uint8, device="cuda")
    mcpu.mcpu_kv_append_fp8(k, v, kv8, bt, sl, qsl, st)
    codes, scales = [], []
    for x in (k, v):
        a = x.float().abs().amax(-1, keepdim=True)
        top = torch.full_like(a, 448.0)
        codes.append(placed((x.float() * (top / a)).to(torch.float8_e4m3fn).view(torch.uint8)))
        pool = torch.zeros(P * 16, hkv, device="cuda")
        pool[dst] = (a / top)[..., 0]
        scales.append(pool.view(P, 16, hkv).transpose(1, 2))
    want = to_fp8_blocks(*(x.cpu().numpy() for x in codes + scales))
    assert np.array_equal(kv8.cpu().numpy(), want)

    # RoPE: q in place for a head count that leaves a partial step of eight
    # rows, cos/sin table both 16-byte aligned and not
    table = torch.from_numpy(W.rope_table(64)).cuda()
    shifted = torch.empty(table.numel() + 1, device="cuda")[1:].view_as(table).copy_(table)
    ref = []
    for x in (torch.randn(T, 2 * hkv, 64, device="cuda").bfloat16(), k):
        c, s = table[pos][:, None, :32].double(), table[pos][:, None, 32:].double()
        lo, hi = x[..., :32].double(), x[..., 32:].double()
        ref.append((x, torch.cat([lo * c - hi * s, hi * c + lo * s], -1)))
    for cs in (table, shifted):
        q = ref[0][0].clone()
        kc.zero_(), vc.zero_()
        mcpu.mcpu_rope_kv_append(q, k, v, kc, vc, bt, sl, qsl, cs, st)
        got_k = kc.transpose(1, 2).reshape(P * 16, hkv, 64)[dst]
        for got, want in ((q, ref[0][1]), (got_k, ref[1][1])):
            # one bf16 rounding of a value within fp32 error of the exact one
            assert ((got.double() - want).abs() <= want.abs() * 2.0**-8 + 1e-6).all()
        assert torch.equal(vc, placed(v))
    assert int(st) == 0
