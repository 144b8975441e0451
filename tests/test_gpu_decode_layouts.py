"""Decode attention over record layouts at the edges of the fused kernel's choice (value records of
each instantiation, streams that differ within a layer, empty streams, widths above 8 bits) and of its
tiling, against 64-bit attention over the dequantized coefficients (aatc_dequantize, itself checked
bit for bit against the oracle).  Tolerances: the acceptance bounds of harness.py, and a relative L2
of 1e-4 (operands of ~22 bits, fp32 sums: 1e-5 and below was measured)."""
import math

import numpy as np
import pytest
import torch

import harness as Hn
from oracle import aatc_oracle as O
from test_gpu_prefill_layouts import random_plan, tokens

DEV = "cuda:0"


def attention(coef, basis, q, group, first=0):
    """64-bit attention of q bf16 [batch][H_q][128] over tokens [first, n) of coef [batch][n][n_kv][2][128]."""
    k = torch.einsum("bnhc,hdc->bnhd", coef[:, first:, :, 0].double(), torch.from_numpy(basis[0, :, 0]).to(DEV).double())
    v = torch.einsum("bnhc,hdc->bnhd", coef[:, first:, :, 1].double(), torch.from_numpy(basis[0, :, 1]).to(DEV).double())
    k, v = k.repeat_interleave(group, 2), v.repeat_interleave(group, 2)
    p = torch.softmax(torch.einsum("bhd,bnhd->bhn", q.double(), k) / math.sqrt(128), -1)
    return torch.einsum("bhn,bnhd->bhd", p, v)


CASES = [
    # n_kv, group, b_max, bit totals of the heads, batch, n_ctx, first; the kernels that many sequences take
    (2, 4, 8, (0, 352), 1, 1, 0, 2),                 # one token; a head whose streams hold no bits
    (2, 4, 8, (0,), 1, 300, 0, 2),                   # no bits in the whole layer
    (2, 7, 8, (0,), 1, 300, 0, 2),
    (8, 4, 8, (352, 200, 97, 288), 1, 127, 0, 2),    # differing streams, value records up to 8 + 3 words
    (3, 3, 8, (352, 420, 131), 2, 129, 5, 2),        # up to 10 + 3 words; the range starts inside a tile
    (2, 1, 8, (900, 611), 1, 1000, 0, 0),            # up to 21 + 3: no room for sixteen warps' entry sums
    (1, 8, 8, (352,), 3, 4097, 130, 2),              # eight query heads, key and value records that differ
    (2, 7, 8, (420, 255), 1, 700, 0, 2),             # seven, differing streams
    (2, 6, 8, (900, 700), 1, 300, 0, 2),             # six, value records up to 13 + 2 words
    (4, 4, 12, (352, 449, 300), 1, 515, 0, 2),       # channels above 8 bits
    (1, 4, 16, (500,), 2, 260, 0, 0),                # channels above 14 bits
]


def sequences_for(aatc, plan, first, n_ctx, form):
    """The fewest sequences whose decode takes the kernels `form` (aatc_selftest_decode_form)."""
    for batch in range(1, 1300):
        got, splits = aatc.selftest_decode_form(plan, 0, batch, first, n_ctx)
        assert splits >= 1
        if got == form:
            return batch
    raise AssertionError(f"no number of sequences takes form {form}")


@pytest.mark.gpu
@pytest.mark.parametrize("many", [False, True])
@pytest.mark.parametrize("n_kv,group,b_max,total,batch,n_ctx,first,form", CASES)
def test_decode_record_layouts(aatc, n_kv, group, b_max, total, batch, n_ctx, first, form, many):
    rng = np.random.default_rng([n_ctx, n_kv, b_max])
    plan, basis, bits = random_plan(aatc, rng, n_kv, group, b_max, total)
    if many:
        batch = sequences_for(aatc, plan, first, n_ctx, form) if form else 160
    assert aatc.selftest_decode_form(plan, 0, batch, first, n_ctx)[0] == (form if many else 0)
    k, v = tokens(rng, basis, batch, n_ctx, n_kv)
    cap = n_ctx + 70
    cache = plan.new_cache(batch, cap, DEV)
    cache.fill_(-1)                                   # whatever the cache held before
    aatc.encode(plan, 0, k, v, cache, 0, cap)
    q = torch.from_numpy(rng.standard_normal((batch, n_kv * group, 128))).to(DEV).to(torch.bfloat16)
    if first:
        out = aatc.decode_attention_sw(plan, 0, q, cache, first, n_ctx, cap)
    else:
        out = aatc.decode_attention(plan, 0, q, cache, n_ctx, cap)
    coef = aatc.dequantize(plan, 0, cache, batch, 0, n_ctx, cap)
    ref = attention(coef, basis, q, group, first)
    if not torch.any(ref):
        assert not torch.any(out)
        return
    _, rel = Hn.check_decode(out.cpu().numpy().reshape(-1, 128), ref.cpu().numpy().reshape(-1, 128))
    assert rel <= 1e-4, rel
    assert plan.device_error() == 0


def widths(*runs):
    """Widths of a stream from (width, channels) runs, zeros behind them."""
    w = np.concatenate([np.full(n, b) for b, n in runs])
    return np.concatenate([w, np.zeros(128 - len(w))]).astype(np.uint8)


def record_words(bits):
    """(D2, D1) words of the stream's records, by the oracle's layout."""
    d2, d1 = O.record_entries(bits.astype(np.int64))
    return len(d2) // 16, -(-len(d1) // 32)


# Value widths of the largest record that each bound of the mixed kernel holds, then of records beyond them.
BOUNDS = {
    (8, 3): widths((3, 80), (2, 48)),
    (17, 2): widths((7, 16), (5, 40), (4, 72)),
    (15, 3): widths((7, 10), (5, 70), (4, 22), (2, 26)),
    (13, 4): widths((5, 90), (3, 28)),
    (11, 5): widths((5, 52), (3, 76)),
    (24, 5): widths((8, 4), (7, 124)),
    (32, 0): widths((8, 128)),
    (32, 1): widths((9, 32), (8, 96)),
}


@pytest.mark.gpu
@pytest.mark.parametrize("values,group,n_ctx,form", [
    (((8, 3), (17, 2)), 4, 640, 2),
    (((15, 3), (13, 4)), 3, 641, 2),                 # a last tile of one token
    (((11, 5), (15, 3)), 1, 24600, 2),               # several tiles of each warp group
    (((8, 3), (17, 2)), 7, 896, 2),                  # five to eight query heads: their instantiations
    (((15, 3), (13, 4)), 5, 897, 2),
    (((11, 5), (17, 2)), 8, 24600, 2),
    (((24, 5), (32, 0)), 4, 640, 3),
    (((32, 1), (8, 3)), 2, 24601, 3),
    (((24, 5), (32, 0)), 5, 24600, 0),               # large records, more than four query heads
])
def test_decode_record_bounds(aatc, values, group, n_ctx, form):
    """Value records of each bound of the mixed kernel, and those of the large one."""
    rng = np.random.default_rng([n_ctx, group])
    value_bits = [BOUNDS[v] for v in values]
    assert [record_words(b) for b in value_bits] == list(values)
    bits = np.stack([np.stack([value_bits[1 - h], value_bits[h]]) for h in (0, 1)])[None]   # each other's as keys
    basis = np.stack([np.linalg.qr(rng.standard_normal((128, 128)))[0] for _ in range(4)])
    basis = basis.reshape(1, 2, 2, 128, 128).astype(np.float32)
    scales = (2.6 * np.arange(1, 129) ** -0.7 * np.ones((1, 2, 2, 1))).astype(np.float32)
    plan = aatc.Plan(aatc.dims(1, 2, 2 * group, b_max=int(bits.max())), basis, bits, scales)
    batch = sequences_for(aatc, plan, 0, n_ctx, form)
    k, v = tokens(rng, basis, batch, n_ctx, 2)
    cache = plan.new_cache(batch, n_ctx, DEV)
    cache.fill_(-1)                                   # whatever the cache held before
    aatc.encode(plan, 0, k, v, cache, 0, n_ctx)
    q = torch.from_numpy(rng.standard_normal((batch, 2 * group, 128))).to(DEV).to(torch.bfloat16)
    out = aatc.decode_attention(plan, 0, q, cache, n_ctx, n_ctx)
    coef = aatc.dequantize(plan, 0, cache, batch, 0, n_ctx, n_ctx)
    for b in range(batch):                            # (one at a time: 64-bit keys and values)
        ref = attention(coef[b:b + 1], basis, q[b:b + 1], group)
        _, rel = Hn.check_decode(out[b].cpu().numpy(), ref[0].cpu().numpy())
        assert rel <= 1e-4, (b, rel)
    assert plan.device_error() == 0


# Value widths whose moved digits (each two entries) belong to one channel, with that channel's entries;
# the last is of a record shape (9 + 2 words) that the fused kernel has an exact form for.
MANY_ENTRIES = [
    (widths((10, 1), (2, 63)), 9),
    (widths((12, 1), (3, 127)), 11),
    (widths((13, 1), (4, 10), (2, 117)), 12),
    (widths((14, 1), (2, 127)), 13),
    (widths((9, 3)), 9),
    (widths((14, 1), (4, 15), (3, 30), (2, 82)), 12),
]


def entries_of_widest(bits):
    d2, d1 = O.record_entries(bits.astype(np.int64))
    return max(np.bincount([c for c, _ in d2 + d1], minlength=128)) if bits.any() else 0


def test_channel_entries(aatc):
    """The entry count that decides which decode kernels may take a layer, against the oracle's layout over
    random widths up to 16 and at the widths above (host only)."""
    for bits, most in MANY_ENTRIES:
        assert aatc.selftest_channel_entries(bits) == entries_of_widest(bits) == most
    rng = np.random.default_rng(9)
    seen = set()
    for _ in range(2000):
        n = int(np.exp(rng.uniform(0, np.log(128.9))))
        wide = int(np.exp(rng.uniform(0, np.log(min(n, 32) + 0.9))))
        b = np.concatenate([rng.integers(1, 17, wide), rng.integers(1, 9, n - wide)])
        bits = np.zeros(128, np.uint8)
        bits[:n] = np.sort(np.minimum(b, rng.integers(1, 17)))[::-1]
        most = aatc.selftest_channel_entries(bits)
        assert most == entries_of_widest(bits)
        assert most <= max(bits.max(), 1)              # one entry a bit: every width up to 8 fits eight slots
        seen.add(most)
    assert max(seen) > 8
    with pytest.raises(aatc.AatcError):
        aatc.selftest_channel_entries(np.full(128, 17, np.uint8))


@pytest.mark.gpu
@pytest.mark.parametrize("n_ctx", [300, 49000])       # a few tiles; five an SM (152), where a mixed layer is fused
@pytest.mark.parametrize("bits,most", MANY_ENTRIES)
def test_decode_channels_of_many_entries(aatc, bits, most, n_ctx):
    """Value channels of more record entries than the fused kernels' eight slots."""
    rng = np.random.default_rng([n_ctx, most])
    n_kv, group = 2, 4
    basis = np.stack([np.linalg.qr(rng.standard_normal((128, 128)))[0] for _ in range(2 * n_kv)])
    basis = basis.reshape(1, n_kv, 2, 128, 128).astype(np.float32)
    scales = (2.6 * np.arange(1, 129) ** -0.7 * np.ones((1, n_kv, 2, 1))).astype(np.float32)
    plan = aatc.Plan(aatc.dims(1, n_kv, n_kv * group, b_max=14), basis, np.tile(bits, (1, n_kv, 2, 1)), scales)
    k, v = tokens(rng, basis, 1, n_ctx, n_kv)
    cache = plan.new_cache(1, n_ctx, DEV)
    aatc.encode(plan, 0, k, v, cache, 0, n_ctx)
    assert aatc.selftest_decode_form(plan, 0, 1, 0, n_ctx)[0] == 0
    q = torch.from_numpy(rng.standard_normal((1, n_kv * group, 128))).to(DEV).to(torch.bfloat16)
    out = aatc.decode_attention(plan, 0, q, cache, n_ctx, n_ctx)
    ref = attention(aatc.dequantize(plan, 0, cache, 1, 0, n_ctx, n_ctx), basis, q, group)
    _, rel = Hn.check_decode(out.cpu().numpy().reshape(-1, 128), ref.cpu().numpy().reshape(-1, 128))
    assert rel <= 1e-4, rel
    assert plan.device_error() == 0


@pytest.mark.gpu
@pytest.mark.parametrize("batch", [1, 2, 3, 5])       # 32 .. 160 query heads: each form of the merge
@pytest.mark.parametrize("n_full", [1, 3, 65, 139, 512, 1031])
def test_merge_of_uncompressed_tokens(aatc, batch, n_full):
    n_kv, group, n_ctx = 8, 4, 150
    rng = np.random.default_rng([batch, n_full])
    plan, basis, _ = random_plan(aatc, rng, n_kv, group, 8, (352, 288))
    k, v = tokens(rng, basis, batch, n_ctx + n_full, n_kv)
    cache = plan.new_cache(batch, n_ctx, DEV)
    aatc.encode(plan, 0, k[:, :n_ctx].contiguous(), v[:, :n_ctx].contiguous(), cache, 0, n_ctx)
    full = [torch.cat([x[:, n_ctx:], torch.full_like(x[:, :3], float("nan"))], 1).contiguous() for x in (k, v)]
    q = torch.from_numpy(2.0 * rng.standard_normal((batch, n_kv * group, 128))).to(DEV).to(torch.bfloat16)
    out = aatc.decode_attention_sw(plan, 0, q, cache, 0, n_ctx, n_ctx, full[0], full[1], n_full)
    coef = aatc.dequantize(plan, 0, cache, batch, 0, n_ctx, n_ctx).double()
    rows = [torch.cat([torch.einsum("bnhc,hdc->bnhd", coef[:, :, :, kind],
                                    torch.from_numpy(basis[0, :, kind]).to(DEV).double()),
                       x[:, n_ctx:].double()], 1).repeat_interleave(group, 2) for kind, x in enumerate((k, v))]
    p = torch.softmax(torch.einsum("bhd,bnhd->bhn", q.double(), rows[0]) / math.sqrt(128), -1)
    ref = torch.einsum("bhn,bnhd->bhd", p, rows[1])
    _, rel = Hn.check_decode(out.cpu().numpy().reshape(-1, 128), ref.cpu().numpy().reshape(-1, 128))
    assert rel <= 1e-4, rel
