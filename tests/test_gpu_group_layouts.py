"""Head-group decode at the edges of its kernel's tiling (one token, a last tile of one token, several
tiles of one split, each number of value tiles a warp holds, few query heads), against 64-bit attention
over the dequantized coefficients (aatc_dequantize, itself checked bit for bit against the oracle).
Tolerances: the acceptance bounds of harness.py, and a relative L2 of 1e-4 (operands of ~22 bits)."""
import math

import numpy as np
import pytest
import torch

import harness as Hn
from oracle import aatc_oracle as O

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


def value_tiles_per_warp(bits, g_h):
    """8-entry tiles of the widest value slice over the 16 / g_h warps of a slice (by the oracle's layout)."""
    slices = [bits[0, g, 1, s::g_h].astype(np.int64) for g in range(bits.shape[1]) for s in range(g_h)]
    tiles = max((sum(map(len, O.record_entries(b))) + 7) // 8 for b in slices)
    return -(-tiles // (16 // g_h))


@pytest.mark.parametrize("g_h,n_groups,group,total,batch,n_ctx,per_warp", [
    (4, 2, 4, 250, 1, 1, 6),                          # one token; six value tiles a warp
    (4, 1, 2, 352, 3, 129, 7),                        # seven; a second tile of one token; eight query rows
    (4, 1, 4, 520, 1, 40001, 8),                      # eight; three tiles of one split
    (4, 1, 4, 900, 1, 20001, 11),                     # eleven: the kernel for up to twelve
    (2, 2, 8, 352, 1, 127, 4),
    (2, 1, 1, 300, 2, 30000, 3),                      # two query rows, four tiles of one split
    (2, 3, 5, 900, 1, 700, 6),                        # six value tiles a warp
    (2, 1, 8, 2000, 1, 40000, 7),                     # seven: the kernel for up to twelve
])
def test_group_decode_layouts(aatc, g_h, n_groups, group, total, batch, n_ctx, per_warp):
    n, n_kv = 128 * g_h, n_groups * g_h
    rng = np.random.default_rng([n_ctx, g_h])
    basis = np.stack([np.linalg.qr(rng.standard_normal((n, n)))[0] for _ in range(2 * n_groups)])
    basis = basis.reshape(1, n_groups, 2, n, n).astype(np.float32)
    w = np.exp(-0.03 / g_h * np.arange(n)) * rng.uniform(0.3, 1.0, (1, n_groups, 2, n))
    bits = np.minimum(np.round(w / w.sum(-1, keepdims=True) * total * g_h), 8)
    bits = np.sort(bits, -1)[..., ::-1].astype(np.uint8)
    assert value_tiles_per_warp(bits, g_h) == per_warp
    scales = (2.6 * np.arange(1, n + 1) ** -0.5 * np.ones((1, n_groups, 2, 1))).astype(np.float32)
    plan = aatc.GroupPlan(aatc.dims(1, n_kv, n_kv * group), g_h, basis, bits, scales)
    g = torch.Generator(DEV).manual_seed(n_ctx)
    std = torch.arange(1, n + 1, device=DEV) ** -0.5
    dev_basis = torch.from_numpy(basis[0]).to(DEV)
    kv = []
    for kind in (0, 1):
        z = torch.randn((batch, n_ctx, n_groups, n), generator=g, device=DEV) * std
        x = torch.einsum("btgc,gdc->btgd", z, dev_basis[:, kind])
        kv.append(x.reshape(batch, n_ctx, n_kv, 128).to(torch.bfloat16).contiguous())
    cap = n_ctx + 70
    cache = plan.new_cache(batch, cap, DEV)
    cache.fill_(-1)                                   # whatever the cache held before
    aatc.encode(plan, 0, kv[0], kv[1], cache, 0, cap)
    q = torch.from_numpy(3.0 * rng.standard_normal((batch, n_kv * group, 128))).to(DEV).to(torch.bfloat16)
    out = aatc.decode_attention(plan, 0, q, cache, n_ctx, cap)
    coef = aatc.dequantize(plan, 0, cache, batch, 0, n_ctx, cap).double()
    # slice s holds the group's channels s, s + g_h, ...
    coef = coef.reshape(batch, n_ctx, n_groups, g_h, 2, 128).permute(0, 1, 2, 4, 5, 3).reshape(batch, n_ctx, n_groups, 2, n)
    rows = [torch.einsum("btgc,gdc->btgd", coef[:, :, :, kind], dev_basis[:, kind].double())
            .reshape(batch, n_ctx, n_kv, 128).repeat_interleave(group, 2) for kind in (0, 1)]
    p = torch.softmax(torch.einsum("bhd,bthd->bht", q.double(), rows[0]) / math.sqrt(128), -1)
    ref = torch.einsum("bht,bthd->bhd", p, rows[1])
    _, rel = Hn.check_decode(out.cpu().numpy().reshape(-1, 128), ref.cpu().numpy().reshape(-1, 128))
    assert rel <= 1e-4, rel
    assert plan.device_error() == 0
