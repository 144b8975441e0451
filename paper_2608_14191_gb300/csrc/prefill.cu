// Prefill attention over the packed cache: a chunk of new query tokens attends causally to the
// cached tokens (Def. sdpa for every query row; Algorithm 1's reconstruct / attend lines, computed
// in the transformed space as the decode does: q . (U h) = (U^T q) . h).
//
// Two or three launches per call:
//   codes    per (128-token tile, kv-head x K|V, sequence): the packed records -> the signed codes
//            code_c = u_c - 2^(b_c - 1) as f16 (exact: |code| <= 2048) in a workspace of 32 KB tiles,
//            [b][h][K|V][tile]: key rows are tokens, value rows channels, both K-major tensor-core
//            operands laid out with the 128-byte swizzle, so one plain bulk copy fetches a tile;
//   attn     per (128 query rows, kv-head, sequence), rows = (query token, head of the GQA group),
//            everything on the tensor cores (tcgen05): q' = (U_K^T q) f^K log2(e) / sqrt(128),
//            per 128-token tile S = alpha^K (q'_hi + q'_lo) . code^K, causal mask, lazily
//            rescaled softmax, P' = 2^(S - m) alpha^V (f16) and O += P' code^V, finally
//            out = U_V (f^V O / l).  Few row blocks over a long context are split over the context;
//   merge    then adds the splits' outputs, weighted by their l 2^m.
#include <cuda_bf16.h>
#include <cuda_fp16.h>

#include <algorithm>

#include "aatc_internal.h"
#include "ptx.cuh"

namespace aatc {
namespace {

constexpr float kPLog2e = 1.4426950408889634f;
constexpr float kPOpMax = 16384.0f; // q' rows scaled so the largest |value| is 2^14

struct PrefillArgs {
  const uint32_t* words;     // cache word region (this layer)
  const float* alpha;        // cache alpha region
  const __nv_bfloat16* q;    // [batch][n_q][H_q][128]
  float* out;                // [batch][n_q][H_q][128]
  __half* codes;             // workspace [batch][n_kv][2][tile]: 128 x 128 operands (swizzled)
  const unsigned char* proj; // plan: [S / 2][5] projection operands (aatc_prefill_operands_kernel)
  const float* f;            // plan: [S][128]
  const ChanEnc* enc;        // plan: [S][128] (offsets 2^(b-1))
  const StreamLayout* lay;   // plan: [S]
  int layer, n_kv, n_q_heads, group, q_start, n_q, n_ctx, n_ctx_pad, n_tiles, n_words;
  float* part;               // splits of the context: [split][batch][n_kv][row][128] outputs of the split alone
  float2* part_ml;           // and [split][batch][n_kv][row] (reference maximum, l)
  int n_split;
  int* err;
};

constexpr int kTAtom = 128 * 128;                  // one 128-row K-atom (64 16-bit values per row)
constexpr int kTOp = 2 * kTAtom;                   // one 128 x 128 16-bit operand (two K-atoms)

// byte offset of element (row, k) of a 128-row K-major operand with the 128-byte swizzle
__device__ __forceinline__ int sw128_off(int row, int k) {
  return (k >> 6) * kTAtom + (row >> 3) * 1024 + (row & 7) * 128 + ((((k & 63) >> 3) ^ (row & 7)) << 4) + (k & 7) * 2;
}

// Four base-4 digits (8 bits) -> the low two bits of four bytes; four single bits -> four bytes.
__device__ __forceinline__ uint32_t spread_digits(uint32_t x) {
  const uint32_t y = (x | (x << 12)) & 0x000F000Fu;
  return (y | (y << 6)) & 0x03030303u;
}
__device__ __forceinline__ uint32_t spread_bits(uint32_t x) { return (x * 0x00204081u) & 0x01010101u; }
__device__ __forceinline__ uint32_t low_mask(int n) { return n >= 32 ? 0xFFFFFFFFu : (1u << n) - 1u; }

// One CTA per (128-token tile, kv-head x K|V, sequence), thread = (token, 64 channels): the packed record -> the
// signed codes as one 32 KB tensor-core operand, written as a whole by a bulk copy.
// The record is read as the bit stream that the encode wrote (digit layers in channel order, then
// the odd widths' top bits, then the digits moved out of the last D2 word): 16 digits or up to 32
// bits per step, spread into the byte lanes of 16 registers (stored value u_c of the thread's channel c =
// byte c & 3 of U[c >> 2]; kWide: UH holds the high bytes of the first 32 channels), which the run
// bounds, uniform over the warp, guard.  code = u - 2^(b-1) as f16: below 9 bits the byte is put
// into the mantissa of 1024 + u, and (1024 + u) - (1024 + 2^(b-1)) is exact.
// Bound by the ALU pipe (72 % active, issue 75 %) next to the write of 256 B per token and stream: 8 heads x
// 30011 tokens at 2.75 bits take 38 us (3.3 TB/s written), a single tile 4.8 us.  With all 128 channels
// of a token in one thread 46 us and 6 us, with 32 in each of four 41 us and 4.3 us; reading each
// channel's entries through the plan's entry lists, one field at a time in dependent loads, 280 and 60 us.
constexpr int kCodesThreads = 2 * TILE;
template <bool kWide>
__global__ void __launch_bounds__(kCodesThreads) aatc_prefill_codes_kernel(const PrefillArgs a) {
  extern __shared__ __align__(128) unsigned char smc[];
  unsigned char* op = smc;                                        // the operand, swizzled
  uint32_t* rec = reinterpret_cast<uint32_t*>(smc + kTOp);        // [n_words + 1][128], token-planar
  __shared__ __align__(16) uint32_t off2[D / 2];                  // f16 pairs 1024 + 2^(b-1) of channels 2i, 2i + 1
  __shared__ float offw[32];                                      // 2^(b-1) of the first 32 channels (kWide)
  __shared__ StreamLayout ly;
  const int tile = blockIdx.x, hk = blockIdx.y, b = blockIdx.z, tid = threadIdx.x;
  const int t = tid & (TILE - 1), half = ptx::warp_uniform(tid >> 7), ch0 = 64 * half;   // token; the thread's first channel
  const int head = hk >> 1, kind = hk & 1;
  const size_t cs = (static_cast<size_t>(b) * a.n_kv + head) * 2 + kind;
  const int s = (a.layer * a.n_kv + head) * 2 + kind;
  const int nw = a.lay[s].words;
  ptx::grid_launch_dependents();               // the attention kernel waits for this grid before its first codes
  const uint32_t* tw = a.words + (cs * a.n_tiles + tile) * static_cast<size_t>(a.n_words) * TILE;
  if (tid < D / 2) {
    const __half2 o = __floats2half2_rn(1024.0f + a.enc[s * D + 2 * tid].off, 1024.0f + a.enc[s * D + 2 * tid + 1].off);
    off2[tid] = *reinterpret_cast<const uint32_t*>(&o);
  }
  if (kWide && tid < 32) offw[tid] = a.enc[s * D + tid].off;
  if (tid < static_cast<int>(sizeof(StreamLayout) / 4))
    reinterpret_cast<int*>(&ly)[tid] = reinterpret_cast<const int*>(a.lay + s)[tid];
  for (int w0 = half; w0 < nw; w0 += 16) {     // every other word of the record
    uint32_t x[8];
#pragma unroll
    for (int i = 0; i < 8; ++i) x[i] = w0 + 2 * i < nw ? tw[(w0 + 2 * i) * TILE + t] : 0u;
#pragma unroll
    for (int i = 0; i < 8; ++i)
      if (w0 + 2 * i < nw) rec[(w0 + 2 * i) * TILE + t] = x[i];
  }
  rec[nw * TILE + t] = 0u;                     // read (and masked) past the last word
  if (kind == 1) {
    // quad-interleaved: byte t & 3 of slots 4Q + (0, 2, 1, 3)[r] is quarter r of this token's word
    const uint32_t lo = (t & 3) | ((4 + (t & 3)) << 4);
    for (int w = half; w < nw; w += 2) {
      __syncwarp();
      const uint4 q = *reinterpret_cast<const uint4*>(rec + w * TILE + (t & ~3));
      __syncwarp();
      rec[w * TILE + t] = __byte_perm(__byte_perm(q.x, q.z, lo), __byte_perm(q.y, q.w, lo), 0x5410);
    }
  }
  __syncthreads();                             // the other half's words; off2, offw, ly
  auto get = [&](int p) {                      // the 32 record bits from bit p on (own column)
    const uint32_t* r = rec + (p >> 5) * TILE + t;
    return __funnelshift_r(r[0], r[TILE], p & 31);
  };
  uint32_t U[16], UH[8];
#pragma unroll
  for (int i = 0; i < 16; ++i) U[i] = 0u;
#pragma unroll
  for (int i = 0; i < 8; ++i) UH[i] = 0u;
  constexpr int kLayers = kWide ? 8 : 4;
  int pos = 2 * ly.n2, mpos = pos;             // D1 bits; the moved digits after them
#pragma unroll
  for (int k = 0; k < kLayers; ++k) mpos += ly.lodd[k] - ly.l2all[k];
  // the odd widths' top bits: channels [a, b) have width 2k + 1
#pragma unroll 1
  for (int k = kLayers - 1; k >= 0; --k) {
    const int ca = ly.l2all[k], cb = ly.lodd[k];
    if (ca >= cb) continue;
    const int sh = 2 * (k & 3);
    auto put = [&](int c32, uint32_t (&dst)[8]) {          // 32 channels
      const int lo = max(ca - c32, 0), n = min(cb - c32, 32) - lo;
      const uint32_t v = (get(pos + c32 + lo - ca) & low_mask(n)) << lo;
#pragma unroll
      for (int j = 0; j < 8; ++j) dst[j] |= spread_bits((v >> (4 * j)) & 15u) << sh;
    };
    if (kWide && k >= 4) {
      if (half == 0) put(0, UH);
    } else {
#pragma unroll
      for (int i = 0; i < 2; ++i)
        if (ca < ch0 + 32 * i + 32 && cb > ch0 + 32 * i) put(ch0 + 32 * i, *reinterpret_cast<uint32_t(*)[8]>(&U[8 * i]));
    }
    pos += cb - ca;
  }
  // digit layers: layer k has the digits of channels [0, l2all[k]), the first l2[k] of them in D2
  pos = 0;
#pragma unroll 1
  for (int k = 0; k < kLayers; ++k) {
    const int lk = ly.l2[k], la = ly.l2all[k];
    if (la == 0) break;
    const int sh = 2 * (k & 3);
    auto put = [&](int c16, uint32_t (&dst)[4]) {          // 16 channels
      const int nd = min(max(lk - c16, 0), 16), nm = min(la - c16, 16) - nd;
      uint32_t v = nd > 0 ? get(pos + 2 * c16) & low_mask(2 * nd) : 0u;
      if (nm > 0)                                          // at most 15 digits move in all
        v |= (get(mpos + 2 * (c16 + nd - lk)) & low_mask(2 * nm)) << (2 * nd);
#pragma unroll
      for (int j = 0; j < 4; ++j) dst[j] |= spread_digits((v >> (8 * j)) & 0xFFu) << sh;
    };
    if (kWide && k >= 4) {
#pragma unroll
      for (int c = 0; c < 2; ++c)
        if (half == 0 && 16 * c < la) put(16 * c, *reinterpret_cast<uint32_t(*)[4]>(&UH[4 * c]));
    } else {
#pragma unroll
      for (int c = 0; c < 4; ++c)
        if (ch0 + 16 * c < la) put(ch0 + 16 * c, *reinterpret_cast<uint32_t(*)[4]>(&U[4 * c]));
    }
    pos += 2 * lk;
    mpos += 2 * (la - lk);
  }
  // f16 codes into the operand: keys K = channel, row = token; values K = token, row = channel
#pragma unroll
  for (int g8 = 0; g8 < 8; ++g8) {                         // eight channels, from c8
    const int c8 = ch0 + 8 * g8;
    const uint4 o4 = *reinterpret_cast<const uint4*>(off2 + c8 / 2);
    const uint32_t ov[4] = {o4.x, o4.y, o4.z, o4.w};
    uint32_t h[4];
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const uint32_t u = U[2 * g8 + (j >> 1)];
      if (kWide && g8 < 4 && half == 0) {
        const uint32_t uh = UH[2 * g8 + (j >> 1)], i0 = 16 * (j & 1);
        const float u0 = static_cast<float>(((u >> i0) & 0xFFu) | (((uh >> i0) & 0xFFu) << 8));
        const float u1 = static_cast<float>(((u >> (i0 + 8)) & 0xFFu) | (((uh >> (i0 + 8)) & 0xFFu) << 8));
        const __half2 c2 = __floats2half2_rn(u0 - offw[8 * g8 + 2 * j], u1 - offw[8 * g8 + 2 * j + 1]);
        h[j] = *reinterpret_cast<const uint32_t*>(&c2);
      } else {
        const uint32_t m = __byte_perm(u, 0x64646464u, (j & 1) ? 0x4342 : 0x4140);   // 1024 + u, twice
        const __half2 c2 = __hsub2(*reinterpret_cast<const __half2*>(&m), *reinterpret_cast<const __half2*>(&ov[j]));
        h[j] = *reinterpret_cast<const uint32_t*>(&c2);
      }
    }
    if (kind == 0) {
      *reinterpret_cast<uint4*>(op + sw128_off(t, c8)) = make_uint4(h[0], h[1], h[2], h[3]);
    } else {
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        *reinterpret_cast<uint16_t*>(op + sw128_off(c8 + 2 * j, t)) = static_cast<uint16_t>(h[j]);
        *reinterpret_cast<uint16_t*>(op + sw128_off(c8 + 2 * j + 1, t)) = static_cast<uint16_t>(h[j] >> 16);
      }
    }
  }
  ptx::fence_proxy_async_smem();
  __syncthreads();
  if (tid == 0) {
    ptx::bulk_store(a.codes + (cs * (a.n_ctx_pad / TILE) + tile) * static_cast<size_t>(TILE * D), op, kTOp);
    ptx::bulk_store_drain();
  }
}

__device__ __forceinline__ float ex2(float x) {
  float r;
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
  return r;
}
__device__ __forceinline__ uint32_t pack_h2(float lo, float hi) {
  const __half2 h = __floats2half2_rn(lo, hi);
  return *reinterpret_cast<const uint32_t*>(&h);
}

// ---------------------------------------------------------------- tensor-core (tcgen05) attention
// Per CTA 128 query rows (= TMEM lanes) of one (kv-head, sequence).  Warps 0-15 do the softmax:
// warp w owns TMEM lanes 32 (w & 3) .. + 31 and column quarter w >> 2 of every 128-column TMEM
// block.  Warp 16 issues every tensor-core MMA, one thread of warp 17 every copy; the roles talk
// through mbarriers only.
//   prologue  q' = (q U_K) f^K log2(e) / sqrt(128) on the tensor cores: q (bf16, exact) against
//             U_K split into three bf16 parts (about 2^-25 relative), rows scaled to 2^14 and
//             split into f16 hi / lo operands kept in TMEM (the A operand of the score MMA, so
//             only the key tile is read from shared memory)
//   per 128-token tile (key and value tiles in rings of three):
//             S = q'_hi . code_K + q'_lo . code_K   tcgen05.mma M = N = 128, K = 128 into score
//             buffer t & 1, one tile ahead of the softmax;
//             softmax with the scores held in registers: x = S alpha^K (causal mask), the row
//             maximum over the four quarters through shared memory and one barrier, lazy reference
//             maximum (O rescaled only when a row's maximum grows by more than 2^8, so
//             P' = 2^(s - m) alpha^V stays inside f16);
//             P' as f16 pairs over the first half of the score buffer it came from: the A operand
//             of O += P' . code_V^T.  S(t + 2), which reuses the buffer, is issued behind PV(t) and
//             the MMAs run in issue order.
//   epilogue  out = (f^V O / l) U_V^T on the tensor cores, both operands split hi / lo in bf16.
// Bound by the softmax's latency: the tensor pipe needs ~1730 cycles a tile (24 MMAs of ~72), a tile
// takes ~2700 (4 x 8192 x 28 heads, a call: 2.42 ms, 3.35 before this split of the roles).
// Sixteen warps, four a scheduler, hide more of it than eight; halving the MMAs, dropping the
// exponentials or the copies changes nothing, dropping the reads of alpha saves a sixth (a column's
// alpha is one shared-memory word for every row).
constexpr int kTRows = 128;
constexpr int kTSoftmax = 512;                     // softmax threads (warps 0-15)
constexpr int kTThreads = kTSoftmax + 64;          // + the MMA warp and the copy warp
constexpr int kTMma = kTSoftmax;                   // first thread of the warp that issues MMAs
constexpr int kTCopy = kTSoftmax + 32;             // the thread that issues copies
constexpr float kLazyLog2 = 8.0f;
constexpr uint32_t kIdescTT = ptx::idesc_f16_f32(128, 128);
constexpr uint32_t kIdescBB = ptx::idesc_bf16_f32(128, 128);
constexpr int kTRing = 3;                          // key tiles, value tiles in flight
constexpr uint32_t kColS = 0;                      // two score buffers (0, 128), P' over their first 64
                                                   // columns; projection results (0)
constexpr uint32_t kColO = 256;                    // O accumulator
constexpr uint32_t kColQ = 384;                    // q' hi (384) and lo (448): A operands of the score MMA

struct PrefillTcSmem {
  alignas(1024) unsigned char kt[kTRing][kTOp];    // key codes: K-atoms = channels, rows = tokens
  alignas(1024) unsigned char vt[kTRing][kTOp];    // value codes: K-atoms = tokens 0-63 | 64-127, rows = channels
  alignas(16) float al[kTRing][2][TILE];           // alpha^K, alpha^V of the tiles in the value ring
  float xch[2][4][kTRows];                         // per-row partials of the column quarters (two slots)
  uint64_t bar_k[kTRing], bar_v[kTRing], bar_a[kTRing], kfree[kTRing], vfree[kTRing], bar_s[2], pready[2], ofree[2],
      bar_p, bar_u;
  uint32_t tmem;
  int abort_flag, never;
};
// kt and vt together hold the four projection operands (prologue, epilogue)
static_assert(offsetof(PrefillTcSmem, vt) == offsetof(PrefillTcSmem, kt) + kTRing * kTOp, "operand slots contiguous");

__device__ __forceinline__ uint32_t pack_bf2(__nv_bfloat16 lo, __nv_bfloat16 hi) {
  return static_cast<uint32_t>(__bfloat16_as_ushort(lo)) | (static_cast<uint32_t>(__bfloat16_as_ushort(hi)) << 16);
}

// 8 fp32 values -> `parts` bf16 parts (u = p0 + p1 + p2 up to the last part's rounding), each
// stored as one 16-byte granule at dst[i * kTOp]
__device__ __forceinline__ void store_split_bf16(unsigned char* dst, const float (&u)[8], int parts) {
  uint32_t w[3][4];
#pragma unroll
  for (int j = 0; j < 4; ++j) {
    float x0 = u[2 * j], x1 = u[2 * j + 1];
#pragma unroll
    for (int p = 0; p < 3; ++p) {
      const __nv_bfloat16 h0 = __float2bfloat16_rn(x0), h1 = __float2bfloat16_rn(x1);
      w[p][j] = pack_bf2(h0, h1);
      x0 -= __bfloat162float(h0);
      x1 -= __bfloat162float(h1);
    }
  }
#pragma unroll
  for (int p = 0; p < 3; ++p)
    if (p < parts) *reinterpret_cast<uint4*>(dst + p * kTOp) = make_uint4(w[p][0], w[p][1], w[p][2], w[p][3]);
}

// barriers among the softmax warps only, and among the four warps that share 32 rows
__device__ __forceinline__ void row_sync(int wq) { asm volatile("bar.sync %0, 128;" ::"r"(2 + wq) : "memory"); }
__device__ __forceinline__ void softmax_sync() { asm volatile("bar.sync 1, %0;" ::"n"(kTSoftmax) : "memory"); }

// Plan constants of the attention kernel, per (layer, kv-head) five 32 KB operands in the layout the
// tensor cores read: U_K^T (rows = channel, K = dim) in three bf16 parts, U_V (rows = dim, K =
// channel) in two.  Splitting them in every CTA took a third of the time a CTA spends outside its
// tiles.
__global__ void __launch_bounds__(256) aatc_prefill_operands_kernel(const float* u32, const float* u32t, unsigned char* proj) {
  const int sk = 2 * blockIdx.x, g = blockIdx.y * 256 + threadIdx.x;
  const int row = g >> 4, k8 = (g & 15) * 8;
  unsigned char* dst = proj + static_cast<size_t>(blockIdx.x) * 5 * kTOp + sw128_off(row, k8);
#pragma unroll
  for (int kind = 0; kind < 2; ++kind) {
    const float* src = (kind == 0 ? u32t + static_cast<size_t>(sk) * D * D : u32 + static_cast<size_t>(sk + 1) * D * D) +
                       row * D + k8;
    const float4 u0 = *reinterpret_cast<const float4*>(src), u1 = *reinterpret_cast<const float4*>(src + 4);
    const float u[8] = {u0.x, u0.y, u0.z, u0.w, u1.x, u1.y, u1.z, u1.w};
    store_split_bf16(dst + 3 * kind * kTOp, u, 3 - kind);
  }
}

__global__ void __launch_bounds__(kTThreads, 1)
    aatc_prefill_tc_kernel(const PrefillArgs a) {
  extern __shared__ unsigned char smraw[];
  PrefillTcSmem& sm =
      *reinterpret_cast<PrefillTcSmem*>((reinterpret_cast<uintptr_t>(smraw) + 1023) & ~uintptr_t(1023));
  // row blocks in reverse: the longest causal ranges start first, the shortest fill the tail
  const int split = blockIdx.x % a.n_split, rb = (gridDim.x - 1 - blockIdx.x) / a.n_split;
  const int head = blockIdx.y, b = blockIdx.z;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const bool softmax = tid < kTSoftmax;
  const int wu = ptx::warp_uniform(warp);
  const int G = a.group, n_rows = a.n_q * G;
  const int sk = (a.layer * a.n_kv + head) * 2, sv = sk + 1;
  const size_t csk = (static_cast<size_t>(b) * a.n_kv + head) * 2, csv = csk + 1;
  const int R0 = rb * kTRows;
  const int r_last = min(n_rows - 1, R0 + kTRows - 1) - R0;
  const int kv_end = min(a.n_ctx, a.q_start + (R0 + r_last) / G + 1);
  const int all_tiles = (kv_end + TILE - 1) / TILE;
  const int tile0 = static_cast<int>(static_cast<long>(all_tiles) * split / a.n_split);   // this split's tiles
  const int n_kv_tiles = static_cast<int>(static_cast<long>(all_tiles) * (split + 1) / a.n_split) - tile0;
  const int tok0 = tile0 * TILE, ctx_left = a.n_ctx - tok0;
  const int r = 32 * (warp & 3) + lane, quarter = (warp >> 2) & 3, qc = 32 * quarter;
  const uint32_t lane_base = static_cast<uint32_t>(32 * (warp & 3)) << 16;
  const int R = R0 + r;
  unsigned char* const pj = sm.kt[0];              // projection operand i at pj + i * kTOp
  const unsigned char* proj = a.proj + static_cast<size_t>(sk / 2) * 5 * kTOp;
  volatile int* abort_flag = &sm.abort_flag;
  auto wait = [&](uint64_t* bar, uint32_t parity) {
    if (!ptx::mbar_wait_bounded(bar, parity, abort_flag)) {
      sm.abort_flag = 1;
      atomicOr(a.err, 2);
    }
  };

  if (tid == kTMma) {
    for (int i = 0; i < kTRing; ++i) {
      ptx::mbar_init(&sm.bar_k[i], 1);
      ptx::mbar_init(&sm.bar_v[i], 1);
      ptx::mbar_init(&sm.bar_a[i], 1);               // alpha of the value slot's tile
      ptx::mbar_init(&sm.kfree[i], 1);               // the MMAs have read key slot i, value slot i
      ptx::mbar_init(&sm.vfree[i], 1);
    }
    for (int i = 0; i < 2; ++i) {
      ptx::mbar_init(&sm.bar_s[i], 1);               // S of tiles i, i + 2, ... computed
      ptx::mbar_init(&sm.pready[i], kTSoftmax / 32); // their P' written (one arrival per warp)
      ptx::mbar_init(&sm.ofree[i], 1);               // their PV done
    }
    ptx::mbar_init(&sm.bar_p, 1);
    ptx::mbar_init(&sm.bar_u, 1);
    sm.abort_flag = 0;
    sm.never = 0;
    ptx::fence_mbar_init();
    ptx::mbar_arrive_expect_tx(&sm.bar_u, 3 * kTOp);
    ptx::bulk_load(pj + kTOp, proj, 3 * kTOp, &sm.bar_u);
  }
  if (warp == 0) {
    ptx::tmem_alloc(&sm.tmem, 512);
    ptx::tmem_relinquish();
  }
  // ---- projection operands: q rows (bf16) in slot 0; U_K^T (rows = channel, K = dim) in three bf16
  // parts in slots 1-3, a bulk copy
  if (softmax) {
    for (int g = tid; g < kTRows * 16; g += kTSoftmax) {
      const int row = g >> 4, k8 = (g & 15) * 8, RR = R0 + row;
      uint4 v = make_uint4(0u, 0u, 0u, 0u);
      if (RR < n_rows) {
        const int qi = RR / G, qh = head * G + RR % G;
        v = *reinterpret_cast<const uint4*>(a.q + ((static_cast<size_t>(b) * a.n_q + qi) * a.n_q_heads + qh) * D +
                                            k8);
      }
      *reinterpret_cast<uint4*>(pj + sw128_off(row, k8)) = v;
    }
  }
  ptx::fence_proxy_async_smem();
  ptx::tc_fence_before();
  __syncthreads();
  ptx::tc_fence_after();
  const uint32_t tmem = sm.tmem;
  const uint32_t pj_a = ptx::smem_u32(pj);
  if (wu == kTMma / 32) {
    const uint32_t el = ptx::elect_one(), tm = ptx::warp_uniform(tmem);
    const uint64_t ad = ptx::sdesc_kmajor_sw128(pj_a);
    wait(&sm.bar_u, 0);
#pragma unroll
    for (int part = 0; part < 3; ++part)
#pragma unroll
      for (int kk = 0; kk < 8; ++kk) {
        const uint32_t off = (kk >> 2) * kTAtom + (kk & 3) * 32;
        ptx::umma_bf16_w(tm + kColS, ad + (off >> 4), ad + (((1 + part) * kTOp + off) >> 4), kIdescBB,
                         (part | kk) ? 1u : 0u, el);
      }
    ptx::umma_commit_w(&sm.bar_p, el);
  }
  // ---- q' rows scaled to 2^14, f16 hi / lo into the score operands
  float rsr = 1.0f;
  if (softmax) {
    wait(&sm.bar_p, 0);
    ptx::tc_fence_after();
    uint32_t q0[32];
    ptx::tmem_ld_32raw(tmem + lane_base + kColS + qc, q0);
    ptx::tmem_ld_wait();
    ptx::tmem_regs_ready(q0);
    const float sc = kPLog2e * 0.08838834764831845f;
    const float* fk = a.f + sk * D + qc;
    float x[32];
    float m = 0.0f;
#pragma unroll
    for (int i = 0; i < 32; ++i) {
      x[i] = __uint_as_float(q0[i]) * fk[i] * sc;
      m = fmaxf(m, fabsf(x[i]));
    }
    sm.xch[0][quarter][r] = m;
    softmax_sync();
    m = fmaxf(fmaxf(sm.xch[0][0][r], sm.xch[0][1][r]), fmaxf(sm.xch[0][2][r], sm.xch[0][3][r]));
    const float inv = m > 0.0f ? kPOpMax / m : 0.0f;
    rsr = m > 0.0f ? m / kPOpMax : 1.0f;             // > 0, so the mask's -inf survives the scaling
    // this thread's 32 channels as 16 f16 pairs of hi and of lo: TMEM columns kColQ + 16 quarter ..
    // (hi) and kColQ + 64 + 16 quarter .. (lo), row = lane
    uint32_t hw[16], lw[16];
#pragma unroll
    for (int j = 0; j < 16; ++j) {
      const float y0 = x[2 * j] * inv, y1 = x[2 * j + 1] * inv;
      const __half2 h = __floats2half2_rn(y0, y1);
      const float2 hf = __half22float2(h);
      hw[j] = *reinterpret_cast<const uint32_t*>(&h);
      lw[j] = pack_h2(y0 - hf.x, y1 - hf.y);
    }
    ptx::tmem_st16(tmem + lane_base + kColQ + 16 * quarter, hw);
    ptx::tmem_st16(tmem + lane_base + kColQ + 64 + 16 * quarter, lw);
    ptx::tmem_wait_st();
  }
  ptx::fence_proxy_async_smem();
  ptx::tc_fence_before();
  __syncthreads();                                        // q' complete; operand slots, score buffers free
  ptx::tc_fence_after();

  if (tid == kTCopy) {
    // ---- copies: a slot is refilled once the MMAs that read it are complete
    auto load = [&](int t, unsigned char* dst, const __half* src, uint64_t* bar, uint64_t* freed) {
      const int st = t % kTRing;
      if (t >= kTRing) wait(freed + st, (t / kTRing - 1) & 1);
      if (*abort_flag) return false;
      ptx::mbar_arrive_expect_tx(bar + st, kTOp);
      ptx::bulk_load(dst + st * kTOp, src + static_cast<size_t>(t) * TILE * D, kTOp, bar + st);
      return true;
    };
    ptx::grid_dependency_wait();                          // the codes (the only thread that reads them)
    const __half* ck = a.codes + (csk * a.n_ctx_pad + tok0) * D;    // tiles of this head's keys, values: 32 KB
    const __half* cv = a.codes + (csv * a.n_ctx_pad + tok0) * D;
    int nk = 0, nv = 0;                                   // tiles requested
    while (nv < n_kv_tiles) {
      if (!load(nk, sm.kt[0], ck, sm.bar_k, sm.kfree)) break;
      ++nk;
      if (!load(nv, sm.vt[0], cv, sm.bar_v, sm.vfree)) break;
      // alpha of the tile, into the slot of a tile whose PV is complete (so its softmax is too);
      // past the context it may hold any bits
      const int st = nv % kTRing;
      const size_t tok = static_cast<size_t>(tok0) + static_cast<size_t>(nv) * TILE;
      ptx::mbar_arrive_expect_tx(&sm.bar_a[st], 2 * TILE * 4);
      ptx::bulk_load(sm.al[st][0], a.alpha + csk * a.n_tiles * TILE + tok, TILE * 4, &sm.bar_a[st]);
      ptx::bulk_load(sm.al[st][1], a.alpha + csv * a.n_tiles * TILE + tok, TILE * 4, &sm.bar_a[st]);
      ++nv;
    }
    if (*abort_flag) {                                    // a wait gave up: let the copies in flight land (bounded)
      for (int t = max(0, nk - kTRing); t < nk; ++t)
        ptx::mbar_wait_bounded(&sm.bar_k[t % kTRing], (t / kTRing) & 1, &sm.never);
      for (int t = max(0, nv - kTRing); t < nv; ++t) {
        ptx::mbar_wait_bounded(&sm.bar_v[t % kTRing], (t / kTRing) & 1, &sm.never);
        ptx::mbar_wait_bounded(&sm.bar_a[t % kTRing], (t / kTRing) & 1, &sm.never);
      }
    }
  } else if (wu == kTMma / 32 && n_kv_tiles > 0) {
    // ---- MMAs, issued by the converged warp
    const uint32_t el = ptx::elect_one();
    const uint32_t tm = ptx::warp_uniform(tmem);
    const uint64_t kdesc = ptx::sdesc_kmajor_sw128(ptx::smem_u32(sm.kt[0]));
    const uint64_t vdesc = ptx::sdesc_kmajor_sw128(ptx::smem_u32(sm.vt[0]));
    auto issue_s = [&](int t) {                           // S = q'_hi . code_K + q'_lo . code_K, A from TMEM
      const int st = t % kTRing;
      wait(&sm.bar_k[st], (t / kTRing) & 1);
      const uint32_t ts = tm + kColS + 128 * (t & 1);
      const uint64_t kd = kdesc + static_cast<uint64_t>(st * (kTOp >> 4));
      ptx::tc_fence_after();
#pragma unroll
      for (int kk = 0; kk < 16; ++kk) {                   // hi, then lo
        const uint32_t off = ((kk >> 2) & 1) * kTAtom + (kk & 3) * 32;
        ptx::umma_f16_ta_w(ts, tm + kColQ + 8 * kk, kd + (off >> 4), kIdescTT, kk > 0 ? 1u : 0u, el);
      }
      ptx::umma_commit_w(&sm.bar_s[t & 1], el);
      ptx::umma_commit_w(&sm.kfree[st], el);
    };
    issue_s(0);
    if (n_kv_tiles > 1) issue_s(1);
    for (int t = 0; t < n_kv_tiles; ++t) {
      const int st = t % kTRing;
      wait(&sm.bar_v[st], (t / kTRing) & 1);
      wait(&sm.pready[t & 1], (t >> 1) & 1);
      ptx::tc_fence_after();
      const uint64_t vd = vdesc + static_cast<uint64_t>(st * (kTOp >> 4));
#pragma unroll
      for (int kk = 0; kk < 8; ++kk) {
        const uint32_t off = (kk >> 2) * kTAtom + (kk & 3) * 32;
        ptx::umma_f16_ta_w(tm + kColO, tm + kColS + 128 * (t & 1) + 8 * kk, vd + (off >> 4), kIdescTT,
                           (t > 0 || kk > 0) ? 1u : 0u, el);
      }
      ptx::umma_commit_w(&sm.ofree[t & 1], el);
      ptx::umma_commit_w(&sm.vfree[st], el);
      if (t + 2 < n_kv_tiles) issue_s(t + 2);
    }
  }
  if (wu == kTMma / 32) {
    // U_V (rows = dim, K = channel) hi / lo into slots 2 / 3, once the last PV (and with it every MMA
    // that reads the rings) is complete
    if (n_kv_tiles > 0) wait(&sm.ofree[(n_kv_tiles - 1) & 1], ((n_kv_tiles - 1) >> 1) & 1);
    if (lane == 0) {
      ptx::mbar_arrive_expect_tx(&sm.bar_u, 2 * kTOp);
      ptx::bulk_load(pj + 2 * kTOp, proj + 3 * kTOp, 2 * kTOp, &sm.bar_u);
    }
  }
  __syncwarp();                                           // the MMA and copy warps reconverge
  float m_row = -INFINITY, l_row = 0.0f;                  // of row r, over this split
  if (softmax) {
    // ---- softmax warps
    const int pos = R < n_rows ? a.q_start + R / G : -1;   // padding rows attend to nothing
    const int last = min(pos, a.n_ctx - 1) - tok0;        // last token this row attends to, from the split's first
    float m_used = -INFINITY;
    uint64_t l2 = ptx::f2_pack(0.0f, 0.0f);
    const uint64_t rs2 = ptx::f2_pack(rsr, rsr);
    for (int t = 0; t < n_kv_tiles; ++t) {
      const int buf = t & 1;
      const float* akt = sm.al[t % kTRing][0] + qc;
      const float* avt = sm.al[t % kTRing][1] + qc;
      wait(&sm.bar_a[t % kTRing], (t / kTRing) & 1);
      const uint32_t ts = tmem + lane_base + kColS + 128 * buf;
      wait(&sm.bar_s[buf], (t >> 1) & 1);
      ptx::tc_fence_after();
      // x = S alpha^K over this thread's 32 tokens (masked), partial row maximum
      uint32_t x[32];
      ptx::tmem_ld_32raw(ts + qc, x);
      const int lim = last - t * TILE - qc;                 // tokens i <= lim are attended
      const bool full = __all_sync(0xffffffffu, lim >= 31);
      ptx::tmem_ld_wait();
      ptx::tmem_regs_ready(x);
      float mt0 = -INFINITY, mt1 = -INFINITY;
#pragma unroll
      for (int i = 0; i < 32; i += 4) {
        const float4 al = *reinterpret_cast<const float4*>(akt + i);
        float y0, y1, y2, y3;
        ptx::f2_unpack(ptx::f2_mul(ptx::f2_pack(__uint_as_float(x[i]), __uint_as_float(x[i + 1])), ptx::f2_pack(al.x, al.y)),
                       y0, y1);
        ptx::f2_unpack(ptx::f2_mul(ptx::f2_pack(__uint_as_float(x[i + 2]), __uint_as_float(x[i + 3])),
                                   ptx::f2_pack(al.z, al.w)), y2, y3);
        mt0 = ptx::fmax3(mt0, y0, y1);
        mt1 = ptx::fmax3(mt1, y2, y3);
        x[i] = __float_as_uint(y0);
        x[i + 1] = __float_as_uint(y1);
        x[i + 2] = __float_as_uint(y2);
        x[i + 3] = __float_as_uint(y3);
      }
      if (!full) {
        mt0 = mt1 = -INFINITY;
#pragma unroll
        for (int i = 0; i < 32; ++i) {
          x[i] = i <= lim ? x[i] : 0xFF800000u;             // -inf
          mt0 = fmaxf(mt0, __uint_as_float(x[i]));
        }
      }
      // alpha^V past the context may hold any bits, and would meet p = 0 below
      // (the warps of a column quarter write the same zeros)
      if ((t + 1) * TILE > ctx_left) {
        if (t * TILE + qc + lane >= ctx_left) sm.al[t % kTRing][1][qc + lane] = 0.0f;
        __syncwarp();
      }
      sm.xch[buf][quarter][r] = fmaxf(mt0, mt1);
      ptx::tc_fence_before();
      row_sync(warp & 3);                                   // partial maxima exchanged; S(t) of these rows read out
      ptx::tc_fence_after();
      const float mt = fmaxf(ptx::fmax3(sm.xch[buf][0][r], sm.xch[buf][1][r], sm.xch[buf][2][r]), sm.xch[buf][3][r]) * rsr;
      const bool need = mt > m_used + kLazyLog2;
      if (__any_sync(0xffffffffu, need)) {
        const float c = need ? (m_used == -INFINITY ? 0.0f : ex2(m_used - mt)) : 1.0f;
        if (t > 0) {                                        // rescale this quarter of O once PV(t - 1) is done
          wait(&sm.ofree[buf ^ 1], ((t - 1) >> 1) & 1);
          ptx::tc_fence_after();
          uint32_t o[32];
          ptx::tmem_ld_32raw(tmem + lane_base + kColO + qc, o);
          ptx::tmem_ld_wait();
          ptx::tmem_regs_ready(o);
#pragma unroll
          for (int i = 0; i < 32; ++i) o[i] = __float_as_uint(__uint_as_float(o[i]) * c);
          ptx::tmem_st32(tmem + lane_base + kColO + qc, o);
        }
        l2 = ptx::f2_mul(l2, ptx::f2_pack(c, c));
        if (need) m_used = mt;
      }
      // P' = 2^(x rs - m) alpha^V as f16 pairs over the first half of the score buffer
      {
        const float msub = m_used == -INFINITY ? 0.0f : -m_used;
        const uint64_t ms2 = ptx::f2_pack(msub, msub);
        uint32_t pw[16];
#pragma unroll
        for (int i = 0; i < 32; i += 4) {
          const float4 al = *reinterpret_cast<const float4*>(avt + i);
          float e0, e1, e2, e3;
          ptx::f2_unpack(ptx::f2_fma(ptx::f2_pack(__uint_as_float(x[i]), __uint_as_float(x[i + 1])), rs2, ms2), e0, e1);
          ptx::f2_unpack(ptx::f2_fma(ptx::f2_pack(__uint_as_float(x[i + 2]), __uint_as_float(x[i + 3])), rs2, ms2), e2, e3);
          const uint64_t p01 = ptx::f2_pack(ex2(e0), ex2(e1)), p23 = ptx::f2_pack(ex2(e2), ex2(e3));
          l2 = ptx::f2_add(l2, ptx::f2_add(p01, p23));
          ptx::f2_unpack(ptx::f2_mul(p01, ptx::f2_pack(al.x, al.y)), e0, e1);
          ptx::f2_unpack(ptx::f2_mul(p23, ptx::f2_pack(al.z, al.w)), e2, e3);
          pw[i / 2] = pack_h2(e0, e1);
          pw[i / 2 + 1] = pack_h2(e2, e3);
        }
        ptx::tmem_st16(ts + 16 * quarter, pw);
      }
      ptx::tmem_wait_st();
      ptx::tc_fence_before();
      __syncwarp();
      if (lane == 0) ptx::mbar_arrive(&sm.pready[buf]);
    }
    if (n_kv_tiles > 0) wait(&sm.ofree[(n_kv_tiles - 1) & 1], ((n_kv_tiles - 1) >> 1) & 1);
    ptx::tc_fence_after();
    float l, lb;
    ptx::f2_unpack(l2, l, lb);
    softmax_sync();                                       // every warp is past its last maximum exchange
    sm.xch[0][quarter][r] = l + lb;
    softmax_sync();
    const float lt = (sm.xch[0][0][r] + sm.xch[0][1][r]) + (sm.xch[0][2][r] + sm.xch[0][3][r]);
    m_row = m_used;
    l_row = lt;
    // ---- o_hat = f^V O / l, hi / lo bf16 in slots 0 / 1
    {
      const float il = lt > 0.0f ? 1.0f / lt : 0.0f;
      uint32_t o0[32];
      ptx::tmem_ld_32raw(tmem + lane_base + kColO + qc, o0);
      ptx::tmem_ld_wait();
      ptx::tmem_regs_ready(o0);
      const float* fv = a.f + sv * D + qc;
#pragma unroll
      for (int g8 = 0; g8 < 4; ++g8) {
        float u[8];
#pragma unroll
        for (int j = 0; j < 8; ++j) {
          const int i = 8 * g8 + j;
          u[j] = lt > 0.0f ? __uint_as_float(o0[i]) * il * fv[i] : 0.0f;
        }
        store_split_bf16(pj + sw128_off(r, qc + 8 * g8), u, 2);
      }
    }
  }
  ptx::fence_proxy_async_smem();
  ptx::tc_fence_before();
  __syncthreads();
  ptx::tc_fence_after();
  // ---- out = o_hat U_V^T = hi.hi + hi.lo + lo.hi
  if (wu == kTMma / 32) {
    const uint32_t el = ptx::elect_one(), tm = ptx::warp_uniform(tmem);
    const uint64_t ad = ptx::sdesc_kmajor_sw128(pj_a);
    if (!ptx::mbar_wait_bounded(&sm.bar_u, 1, &sm.never)) atomicOr(a.err, 2);
#pragma unroll
    for (int pr = 0; pr < 3; ++pr) {
      const uint32_t as = pr == 2 ? 1u : 0u, bs = pr == 1 ? 3u : 2u;
#pragma unroll
      for (int kk = 0; kk < 8; ++kk) {
        const uint32_t off = (kk >> 2) * kTAtom + (kk & 3) * 32;
        ptx::umma_bf16_w(tm + kColS, ad + ((as * kTOp + off) >> 4), ad + ((bs * kTOp + off) >> 4), kIdescBB,
                         (pr | kk) ? 1u : 0u, el);
      }
    }
    ptx::umma_commit_w(&sm.bar_p, el);
  }
  if (softmax) {
    wait(&sm.bar_p, 1);
    ptx::tc_fence_after();
    uint32_t o0[32];
    ptx::tmem_ld_32raw(tmem + lane_base + kColS + qc, o0);
    ptx::tmem_ld_wait();
    ptx::tmem_regs_ready(o0);
    if (R < n_rows) {
      const int qi = R / G, qh2 = head * G + R % G;
      float* o = a.out + ((static_cast<size_t>(b) * a.n_q + qi) * a.n_q_heads + qh2) * D;
      if (a.n_split > 1) {
        const size_t prow = ((static_cast<size_t>(split) * gridDim.z + b) * a.n_kv + head) * n_rows + R;
        o = a.part + prow * D;
        if (quarter == 0) a.part_ml[prow] = make_float2(m_row, l_row);
      }
      float4* dst = reinterpret_cast<float4*>(o + qc);
#pragma unroll
      for (int i = 0; i < 8; ++i)
        dst[i] = make_float4(__uint_as_float(o0[4 * i]), __uint_as_float(o0[4 * i + 1]), __uint_as_float(o0[4 * i + 2]),
                             __uint_as_float(o0[4 * i + 3]));
    }
  }
  ptx::tc_fence_before();
  __syncthreads();
  if (warp == 0) {
    ptx::tc_fence_after();
    ptx::tmem_dealloc(tmem, 512);
  }
}

// One warp per query row: out = sum_s w_s out_s / sum_s w_s with w_s = l_s 2^(m_s - max m) over the
// splits of the context (a split's output is already divided by its l; no tokens: l = 0).
constexpr int kPMergeRows = 8;
__global__ void __launch_bounds__(32 * kPMergeRows) aatc_prefill_merge_kernel(const PrefillArgs a, int batch) {
  const int n_rows = a.n_q * a.group, lane = threadIdx.x & 31;
  const long row = static_cast<long>(blockIdx.x) * kPMergeRows + (threadIdx.x >> 5), all = static_cast<long>(batch) * a.n_kv * n_rows;
  if (row >= all) return;
  float M = -INFINITY;
  for (int s = 0; s < a.n_split; ++s) M = fmaxf(M, a.part_ml[s * all + row].x);
  float den = 0.0f;
  float4 o = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
#pragma unroll 4
  for (int s = 0; s < a.n_split; ++s) {
    const float2 ml = a.part_ml[s * all + row];
    const float4 v = *reinterpret_cast<const float4*>(a.part + (s * all + row) * D + 4 * lane);
    const float w = ml.y > 0.0f ? ml.y * ex2(ml.x - M) : 0.0f;
    den += w;
    o.x = fmaf(w, v.x, o.x);
    o.y = fmaf(w, v.y, o.y);
    o.z = fmaf(w, v.z, o.z);
    o.w = fmaf(w, v.w, o.w);
  }
  const float inv = den > 0.0f ? 1.0f / den : 0.0f;
  const int R = static_cast<int>(row % n_rows), head = static_cast<int>(row / n_rows % a.n_kv);
  const size_t b = static_cast<size_t>(row / n_rows / a.n_kv);
  *reinterpret_cast<float4*>(a.out + ((b * a.n_q + R / a.group) * a.n_q_heads + head * a.group + R % a.group) * D +
                             4 * lane) = make_float4(o.x * inv, o.y * inv, o.z * inv, o.w * inv);
}

// Splits of the context for a call whose row blocks leave SMs idle or a last wave nearly empty: the
// fewest rounds of one CTA per SM over (tiles of a split + the ~8 tiles' worth of time a CTA spends
// outside its tiles, and ~3 more for the merge), counted on the blocks' mean causal range.  At least
// four tiles a split.  333 queries x 4 heads over 30011 tokens on 8 kv-heads (88 row blocks on 152
// SMs), a call: 356 us unsplit, 259 in five splits; 78 queries over 60710 tokens (24 row blocks) 699 and
// 195 us.
constexpr int kPMaxSplits = 16, kPCtaTiles = 8, kPMergeTiles = 3;
int prefill_splits(long ctas, int mean_tiles, int num_sms, size_t room_rows) {
  int best = 1;
  long cost = (ctas + num_sms - 1) / num_sms * (mean_tiles + kPCtaTiles);
  for (int n = 2; n <= std::min(kPMaxSplits, mean_tiles / 4); ++n) {
    if (static_cast<size_t>(ctas) * n * kTRows > room_rows) break;
    const long c = (ctas * n + num_sms - 1) / num_sms * ((mean_tiles + n - 1) / n + kPCtaTiles) + kPMergeTiles;
    if (c < cost) {
      cost = c;
      best = n;
    }
  }
  return best;
}
constexpr size_t kPRowBytes = (D + 2) * sizeof(float);     // of one row's partial

}  // namespace

size_t prefill_operand_bytes(int n_layers, int n_kv) { return static_cast<size_t>(n_layers) * n_kv * 5 * kTOp; }

cudaError_t launch_prefill_operands(const Plan& plan, void* proj, cudaStream_t st) {
  aatc_prefill_operands_kernel<<<dim3(plan.n_streams / 2, D * 16 / 256), 256, 0, st>>>(
      plan.dev.u32, plan.dev.u32t, static_cast<unsigned char*>(proj));
  return cudaGetLastError();
}

size_t prefill_codes_bytes(int batch, int n_kv, int n_ctx) {
  const size_t pad = (static_cast<size_t>(n_ctx) + TILE - 1) / TILE * TILE;
  return static_cast<size_t>(batch) * n_kv * 2 * pad * D * sizeof(__half);
}
// The codes, then room for the partial rows of up to four rounds of split CTAs (none for contexts that are
// never split: too short, or of so many sequences that two splits of a row block each are past that).
size_t prefill_workspace(const Plan& plan, int batch, int n_ctx) {
  const int most = std::min(kPMaxSplits, (n_ctx + TILE - 1) / TILE / 4);
  const long ctas = most < 2 ? 0 : std::min(4L, static_cast<long>(most)) * plan.num_sms;
  const size_t rows = 2L * batch * plan.dims.n_kv_heads <= ctas ? static_cast<size_t>(ctas) * kTRows : 0;
  return prefill_codes_bytes(batch, plan.dims.n_kv_heads, n_ctx) + rows * kPRowBytes;
}

cudaError_t launch_prefill(const Plan& plan, int layer, const void* q, int q_start, int n_q, const void* cache,
                           int batch, int n_ctx, int max_tokens, float* out, void* ws, size_t ws_bytes,
                           cudaStream_t st) {
  const CacheGeom g = cache_geom(batch, plan.dims.n_kv_heads, max_tokens, plan.n_words);
  PrefillArgs a;
  a.words = static_cast<const uint32_t*>(cache);
  a.alpha = reinterpret_cast<const float*>(static_cast<const uint32_t*>(cache) + g.words_elems);
  a.q = static_cast<const __nv_bfloat16*>(q);
  a.out = out;
  a.codes = static_cast<__half*>(ws);
  a.proj = plan.dev.proj;
  a.f = plan.dev.f;
  a.enc = plan.dev.enc;
  a.lay = plan.dev.lay;
  a.layer = layer;
  a.n_kv = plan.dims.n_kv_heads;
  a.n_q_heads = plan.dims.n_q_heads;
  a.group = a.n_q_heads / a.n_kv;
  a.q_start = q_start;
  a.n_q = n_q;
  a.n_ctx = n_ctx;
  a.n_ctx_pad = (n_ctx + TILE - 1) / TILE * TILE;
  a.n_tiles = g.n_tiles;
  a.n_words = plan.n_words;
  a.err = plan.dev.err;
  if (plan.n_words > 32) return cudaErrorNotSupported;
  // one instantiation for plans with a channel wider than 8 bits (high bytes kept), one without
  auto* codes = plan.max_bits > 8 ? aatc_prefill_codes_kernel<true> : aatc_prefill_codes_kernel<false>;
  const size_t csm = kTOp + static_cast<size_t>(plan.n_words + 1) * TILE * 4;
  cudaError_t e = ensure_smem_optin(reinterpret_cast<const void*>(codes), csm);
  if (e != cudaSuccess) return e;
  codes<<<dim3(a.n_ctx_pad / TILE, a.n_kv * 2, batch), kCodesThreads, csm, st>>>(a);
  e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  const size_t smem = sizeof(PrefillTcSmem) + 1024;
  e = ensure_smem_optin(reinterpret_cast<const void*>(aatc_prefill_tc_kernel), smem);
  if (e != cudaSuccess) return e;
  const int n_rows = n_q * a.group, blocks = (n_rows + kTRows - 1) / kTRows;
  // splits of the context, as far as the workspace has room for their partial rows
  const size_t codes_bytes = prefill_codes_bytes(batch, a.n_kv, n_ctx);
  const size_t room = (ws_bytes - codes_bytes) / kPRowBytes;
  const int mean_tiles = (q_start + n_q / 2) / TILE + 1;
  a.n_split = prefill_splits(static_cast<long>(blocks) * a.n_kv * batch, mean_tiles, std::max(1, plan.num_sms), room);
  const size_t rows = static_cast<size_t>(a.n_split) * batch * a.n_kv * n_rows;
  a.part = reinterpret_cast<float*>(static_cast<char*>(ws) + codes_bytes);
  a.part_ml = reinterpret_cast<float2*>(a.part + rows * D);
  // Up to a CTA per SM a programmatic dependent of the codes kernel: its prologue (5 us) needs only q and
  // plan constants, which were complete when that one started.  Two tokens of two sequences, a call:
  // 17.2 -> 13.8 us.  Larger grids gain nothing by it (a chunk of 440 CTAs 258 us both ways) or lose (16
  // rounds of CTAs 2414 -> 2477 us).
  const dim3 grid(blocks * a.n_split, a.n_kv, batch);
  if (static_cast<long>(grid.x) * grid.y * grid.z <= plan.num_sms) {
    e = launch_pdl(aatc_prefill_tc_kernel, grid, dim3(kTThreads), smem, st, a);
  } else {
    aatc_prefill_tc_kernel<<<grid, kTThreads, smem, st>>>(a);
    e = cudaGetLastError();
  }
  if (e != cudaSuccess || a.n_split == 1) return e;
  const long all = static_cast<long>(batch) * a.n_kv * n_rows;
  aatc_prefill_merge_kernel<<<static_cast<unsigned>((all + kPMergeRows - 1) / kPMergeRows), 32 * kPMergeRows, 0, st>>>(
      a, batch);
  return cudaGetLastError();
}

}  // namespace aatc
