"""Prefill attention over record layouts and sizes at the edges of its kernels, against 64-bit
attention over the dequantized coefficients (aatc_dequantize, itself checked bit for bit against
the oracle).  Tolerances: the acceptance bounds of harness.py (max-abs 1e-2, relative L2 1e-3)."""
import ctypes
import math

import numpy as np
import pytest
import torch

import harness as Hn

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


def random_plan(aatc, rng, n_kv, group, b_max, total):
    """A plan whose streams have random bases and random non-increasing widths of about `total` bits."""
    basis = np.stack([np.linalg.qr(rng.standard_normal((128, 128)))[0] for _ in range(2 * n_kv)])
    basis = basis.reshape(1, n_kv, 2, 128, 128).astype(np.float32)
    bits = np.zeros((1, n_kv, 2, 128), np.uint8)
    for i in np.ndindex(1, n_kv, 2):
        decay = rng.uniform(0.01, 0.06)
        w = np.exp(-decay * np.arange(128)) * rng.uniform(0.3, 1.0, 128)
        b = np.minimum(np.round(w / w.sum() * total[i[1] % len(total)]), b_max)
        b = np.sort(b)[::-1]
        b[32:] = np.minimum(b[32:], 8)               # device limit: only the first 32 channels above 8 bits
        bits[i] = b
    scales = (2.6 * np.arange(1, 129) ** -0.7 * np.ones((1, n_kv, 2, 1))).astype(np.float32)
    return aatc.Plan(aatc.dims(1, n_kv, n_kv * group, b_max=b_max), basis, bits, scales), basis, bits


def tokens(rng, basis, batch, n, n_kv):
    g = torch.Generator(DEV).manual_seed(int(rng.integers(1 << 30)))
    std = torch.arange(1, 129, device=DEV) ** -0.7
    out = []
    for kind in (0, 1):
        z = torch.randn((batch, n, n_kv, 128), generator=g, device=DEV) * std
        x = torch.einsum("bnhc,hdc->bnhd", z, torch.from_numpy(basis[0, :, kind]).to(DEV))
        out.append(x.to(torch.bfloat16).contiguous())
    return out


def reference(coef, basis, q, q_start, group):
    """64-bit causal attention; coef fp32 [batch][n][n_kv][2][128], q bf16 [batch][n_q][H_q][128]."""
    k = torch.einsum("bnhc,hdc->bnhd", coef[..., 0, :].double(), torch.from_numpy(basis[0, :, 0]).to(DEV).double())
    v = torch.einsum("bnhc,hdc->bnhd", coef[..., 1, :].double(), torch.from_numpy(basis[0, :, 1]).to(DEV).double())
    k, v = k.repeat_interleave(group, 2), v.repeat_interleave(group, 2)
    s = torch.einsum("bqhd,bnhd->bhqn", q.double(), k) / math.sqrt(128)
    pos = q_start + torch.arange(q.shape[1], device=DEV)
    s.masked_fill_(torch.arange(k.shape[1], device=DEV)[None, None, None] > pos[None, None, :, None], -math.inf)
    return torch.einsum("bhqn,bnhd->bqhd", torch.softmax(s, -1), v)


CASES = [
    # n_kv, group, b_max, bit totals of the heads, batch, n_ctx, n_q
    (1, 1, 8, (352,), 1, 1, 1),                      # one token, one row
    (2, 4, 8, (100, 352), 2, 127, 3),                # last tile short by one, few bits
    (3, 5, 8, (352, 611, 37), 1, 128, 128),          # odd widths, exactly one tile
    (1, 8, 8, (900,), 1, 129, 17),                   # a second tile of one token; widths up to 8
    (2, 3, 8, (255, 449), 3, 700, 43),               # digits moved out of the last D2 word
    (2, 2, 12, (600, 333), 1, 391, 65),              # channels above 8 bits
]


@pytest.mark.parametrize("n_kv,group,b_max,total,batch,n_ctx,n_q", CASES)
def test_prefill_record_layouts(aatc, n_kv, group, b_max, total, batch, n_ctx, n_q):
    rng = np.random.default_rng([n_ctx, n_q, b_max])
    plan, basis, bits = random_plan(aatc, rng, n_kv, group, b_max, total)
    if b_max > 8:
        assert bits.max() > 8
    k, v = tokens(rng, basis, batch, n_ctx, n_kv)
    cap = n_ctx + 130
    cache = plan.new_cache(batch, cap, DEV)
    cache.fill_(-1)                                   # whatever the cache held before
    aatc.encode(plan, 0, k, v, cache, 0, cap)
    q = torch.from_numpy(rng.standard_normal((batch, n_q, n_kv * group, 128))).to(DEV).to(torch.bfloat16)
    out = aatc.prefill_attention(plan, 0, q, n_ctx - n_q, cache, n_ctx, cap)
    coef = aatc.dequantize(plan, 0, cache, batch, 0, n_ctx, cap)
    ref = reference(coef, basis, q, n_ctx - n_q, group)
    Hn.check_decode(out.cpu().numpy().reshape(-1, 128), ref.cpu().numpy().reshape(-1, 128))
    assert plan.device_error() == 0


SPLITS = [
    # n_kv, group, batch, n_ctx, n_q: a split context (few row blocks, many tiles)
    (1, 1, 1, 1024, 1),                              # eight tiles, one row
    (1, 4, 1, 2049, 70),                             # splits of unequal lengths, a last tile of one token
    (2, 3, 2, 1500, 700),                            # causal ranges that end in different splits
    (1, 2, 1, 4200, 2500),                           # rows that end before the later splits begin
]


def test_prefill_workspace_room(aatc):
    """The workspace has room for partial rows only where a context of that many sequences can be split."""
    n_kv = 2
    plan, _, _ = random_plan(aatc, np.random.default_rng(3), n_kv, 1, 8, (352,))
    sms = torch.cuda.get_device_properties(DEV).multi_processor_count

    def extra(batch, n_ctx):
        n = ctypes.c_size_t()
        assert aatc.load().aatc_prefill_workspace_bytes(plan.handle, batch, n_ctx, ctypes.byref(n)) == 0
        return n.value - batch * n_kv * 2 * ((n_ctx + 127) // 128) * 128 * 128 * 2

    assert extra(1, 896) == 0                        # seven tiles: at most one split
    assert extra(1, 897) == 2 * sms * 128 * 130 * 4  # eight tiles: two splits
    assert extra(1, 8192) == 4 * sms * 128 * 130 * 4
    assert extra(sms, 8192) == 4 * sms * 128 * 130 * 4   # 2 sms row blocks at least, two splits: four rounds
    assert extra(sms + 1, 8192) == 0


@pytest.mark.parametrize("room", ["full", "codes only"])
@pytest.mark.parametrize("n_kv,group,batch,n_ctx,n_q", SPLITS)
def test_prefill_split_context(aatc, n_kv, group, batch, n_ctx, n_q, room):
    """The split context against 64 bits, and the same call with a workspace that holds the codes
    alone (accepted, not split)."""
    rng = np.random.default_rng([n_ctx, n_q])
    plan, basis, _ = random_plan(aatc, rng, n_kv, group, 8, (352,))
    k, v = tokens(rng, basis, batch, n_ctx, n_kv)
    cache = plan.new_cache(batch, n_ctx, DEV)
    aatc.encode(plan, 0, k, v, cache, 0, n_ctx)
    q = torch.from_numpy(rng.standard_normal((batch, n_q, n_kv * group, 128))).to(DEV).to(torch.bfloat16)
    codes = batch * n_kv * 2 * ((n_ctx + 127) // 128) * 128 * 128 * 2
    ws = None if room == "full" else torch.empty(codes // 4, device=DEV)
    out = aatc.prefill_attention(plan, 0, q, n_ctx - n_q, cache, n_ctx, n_ctx, workspace=ws)
    coef = aatc.dequantize(plan, 0, cache, batch, 0, n_ctx, n_ctx)
    ref = reference(coef, basis, q, n_ctx - n_q, group)
    Hn.check_decode(out.cpu().numpy().reshape(-1, 128), ref.cpu().numpy().reshape(-1, 128))
    assert plan.device_error() == 0
    if ws is not None:
        with pytest.raises(aatc.AatcError):
            aatc.prefill_attention(plan, 0, q, n_ctx - n_q, cache, n_ctx, n_ctx, workspace=ws[:-1])
