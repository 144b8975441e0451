"""Encode over record layouts at the edges of the tensor-core packing's rule (streams without bits, top
bits and moved digits that straddle half-words, the longest record and the most digit blocks it takes,
and plans just past either, which keep the register packing) and of its tiling: codes, token scales and
padding bits against the oracle, under the stated rule for codes next to a threshold."""
import numpy as np
import pytest
import torch

import oracle_jobs
from oracle import aatc_oracle as O
from test_gpu_prefill_layouts import tokens

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


def decaying(rng, total):
    """Random non-increasing widths up to 8 of about `total` bits."""
    w = np.exp(-rng.uniform(0.01, 0.06) * np.arange(128)) * rng.uniform(0.3, 1.0, 128)
    return np.sort(np.minimum(np.round(w / w.sum() * total), 8))[::-1]


def flat(width, n=128):
    return np.where(np.arange(128) < n, width, 0)


def packs_on_tensor_cores(bits):
    """Whether a stream has a packing operand: digit blocks of 8 columns and half-words in sixteens share 128
    columns, the record has at most 24 words, no channel more than 8 bits."""
    blocks = sum(-(-int((bits >= 2 * k + 1).sum()) // 32) for k in range(4))
    words = O.stream_words(bits)
    return bits.max() <= 8 and words <= 24 and 8 * blocks + (2 * words + 15) // 16 * 16 <= 128


CASES = [
    # widths of the streams (key, value, key, ...), batch, n_tokens, start; whether they pack on the tensor cores
    ([0, 352], 1, 1, 0, True),                                 # one token; a stream without bits
    ([37, 352, 97, 131], 2, 127, 3, True),                     # short records
    ([352, 449, 255, 500, 400, 288], 1, 129, 250, True),       # differing records, a second tile of one token
    ([352, 449, 255, 611, 700, 288], 1, 129, 250, False),      # one with 11 blocks and 48 columns: register packing
    ([flat(1), flat(2), flat(3), flat(4)], 1, 128, 64, True),  # top bits alone, whole layers
    ([flat(1, 1), flat(3, 5), flat(8, 3), flat(7, 17)], 1, 300, 1, True), # a few channels, odd counts
    ([flat(6, 64) + flat(4) - flat(4, 64), 352], 1, 200, 0, True), # 10 blocks and 48 half-word columns, the longest record
    ([flat(7, 65), flat(7, 64)], 1, 200, 2, True),             # 12 blocks and 32 columns, the most blocks
    ([flat(6, 65) + flat(4) - flat(4, 65), 352], 1, 200, 0, False), # 11 and 48: register packing
    ([flat(8, 97), 352], 1, 200, 7, False),                    # 25 words: register packing
    ([352] * 16, 1, 128 * 81 - 5, 11, True),                   # several items of each group
]


@pytest.mark.parametrize("widths,batch,n_tokens,start,tensor_cores", CASES)
def test_encode_record_layouts(aatc, widths, batch, n_tokens, start, tensor_cores):
    n_kv = len(widths) // 2
    rng = np.random.default_rng([n_tokens, n_kv])
    bits = np.stack([decaying(rng, w) if isinstance(w, int) else w for w in widths])
    assert all(packs_on_tensor_cores(b) for b in bits) == tensor_cores
    bits = bits.reshape(1, n_kv, 2, 128).astype(np.uint8)
    basis = np.stack([np.linalg.qr(rng.standard_normal((128, 128)))[0] for _ in widths])
    basis = basis.reshape(1, n_kv, 2, 128, 128).astype(np.float32)
    scales = (2.6 * np.arange(1, 129) ** -0.7 * np.ones((1, n_kv, 2, 1))).astype(np.float32)
    plan = aatc.Plan(aatc.dims(1, n_kv, n_kv), basis, bits, scales)
    x = tokens(rng, basis, batch, n_tokens, n_kv)
    cap = start + n_tokens + 70
    cache = plan.new_cache(batch, cap, DEV)
    cache.fill_(-1)                                            # whatever the cache held before
    aatc.encode(plan, 0, x[0], x[1], cache, start, cap)
    assert plan.device_error() == 0
    image = cache.cpu().numpy().view(np.uint32)
    encode_basis = torch.from_numpy(basis).to(torch.bfloat16).float().numpy()
    pick = np.unique(np.concatenate([np.arange(min(n_tokens, 300)), np.arange(max(0, n_tokens - 200), n_tokens),
                                     rng.integers(0, n_tokens, 200)]))
    mismatch = codes = 0
    for b, h, kind in np.ndindex(batch, n_kv, 2):
        rec, alpha = O.cache_records(image, batch, n_kv, cap, plan.n_words, b, h, kind, start, n_tokens)
        if not bits[0, h, kind].any():
            assert not rec.any() and not alpha.any()
            continue
        stats, err = oracle_jobs.code_check(x[kind][b, :, h].float().cpu().numpy()[pick], rec[pick], alpha[pick],
                                            encode_basis[0, h, kind], bits[0, h, kind], scales[0, h, kind])
        assert err is None, f"{err} (sequence {b} head {h} kind {kind})"
        mismatch += stats["mismatch"]
        codes += stats["codes"]
        if start:                                              # the tokens before are left alone
            rec, alpha = O.cache_records(image, batch, n_kv, cap, plan.n_words, b, h, kind, 0, start)
            assert (rec == 0xFFFFFFFF).all()
    assert mismatch <= 1 + 1e-5 * codes
