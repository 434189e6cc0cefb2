// Quantise-and-pack cache writer (App. C.4 quantiser; App. C.5 cache update:
// content- and RoPE-cache quantisation, integer packing and slot-mapped page
// insertion) for this library's block and for the paper's own page, and the
// plain BF16 writer for the comparison cache.
//
// A block of nine warps writes a few tokens: warp g quantises group g (64
// coordinates) of four or sixteen tokens, eight lanes per token with eight
// coordinates (16 bytes) each. A warp then reads four whole 128-byte lines and,
// where the tokens take consecutive slots (a prefill), writes their code rows
// and scales as contiguous runs; the bit width and the scale format are uniform
// in a warp. See quant_append_kernel for what bounds it.
#include <cuda_runtime.h>

#include "common.cuh"
#include "kernels.h"
#include "ptx.cuh"

namespace qmla {
namespace {

// Stored fp16 scale and integer zero point of one group (App. C.4 with the
// fp16 staging of include/qmla.h): s = RN_f16(RN_f32(max(d, 1e-8) / m)),
// clamped to [2^-24, 65504]; z = clip(rne(-x_min / s), 0, m).
__device__ __forceinline__ void group_scale(float xmin, float xmax, int m, float& s, float& z) {
  const float d = xmax - xmin;
  const float s32 = __fdiv_rn(fmaxf(d, 1e-8f), static_cast<float>(m));
  s = __half2float(__float2half_rn(s32));
  if (s == 0.0f) s = 5.9604644775390625e-08f;  // 2^-24, the smallest fp16 subnormal
  if (isinf(s)) s = 65504.0f;
  z = fminf(fmaxf(rintf(__fdiv_rn(-xmin, s)), 0.0f), static_cast<float>(m));
}

// Scales of the paper's page (App. C.4 with that format's staging): content
// s = RN_bf16(RN_f32(max(d, 1e-8) / 15)), RoPE s = RN_f32(max(d, 1e-8) / 15);
// z = clip(rne(-x_min / s), 0, 15) from an fp32 quotient. A bf16 scale and a
// bf16 input carry 8 significant bits each, so the fp32 quotients of the
// content path round to the same codes as exact arithmetic would.
__device__ __forceinline__ void paper_scale(float xmin, float xmax, bool content, float& s, float& z) {
  const float s32 = __fdiv_rn(fmaxf(xmax - xmin, 1e-8f), 15.0f);
  s = content ? __bfloat162float(__float2bfloat16_rn(s32)) : s32;
  z = fminf(fmaxf(rintf(__fdiv_rn(-xmin, s)), 0.0f), 15.0f);
}

__device__ __forceinline__ uint32_t quant_code(float x, float s, float z, float m) {
  // q = clip(rne(x / s + z), 0, m): z is added before rounding.
  return static_cast<uint32_t>(fminf(fmaxf(rintf(__fdiv_rn(x, s) + z), 0.0f), m));
}

// The codes clip(rne(x / s + z), 0, m) of eight bf16 values (four words of two),
// as four words with one code in each half, without a division per value: y =
// RN(1 / s), q = RN(x y) corrected once by its exact residual x - q s (P.
// Markstein, IBM J. Res. Dev. 34(1), 1990) is within 2^-22 relative of x / s and
// exact where x / s is representable. The codes need no more: s has at most 11
// and x 8 significant bits, so an x / s of magnitude 16 or less is a half-integer
// (representable) or at least 2^-12 away from one, and what lies outside is
// clipped. Adding 1.5 * 2^23 leaves the integer nearest to q + z (ties to even)
// in the low bits, for |q| <= 2^14 in the low 16 as a signed number, and a NaN as
// -1, which is clipped to 0.
__device__ __forceinline__ void codes8(const uint32_t (&w)[4], float s, float y, float z, uint32_t m, uint32_t (&c)[4]) {
  const uint64_t yy = f32x2(y, y), ns = f32x2(-s, -s), zz = f32x2(z, z), magic = f32x2(12582912.0f, 12582912.0f);
#pragma unroll
  for (int e = 0; e < 4; ++e) {
    const uint64_t x = f32x2(__uint_as_float(w[e] << 16), __uint_as_float(w[e] & 0xFFFF0000u));
    uint64_t q = mul2(x, yy);
    q = fma2(fma2(q, ns, x), yy, q);
    q = add2(add2(q, zz), magic);
    c[e] = __vimin_s16x2_relu(__byte_perm(static_cast<uint32_t>(q), static_cast<uint32_t>(q >> 32), 0x5410),
                              m | (m << 16));
  }
}

// Looks up and validates the destination of token i: its block id, or -1 (after
// recording the error) when the token cannot be written.
__device__ __forceinline__ int token_block(int num_blocks, const int32_t* seq_ids, const int32_t* positions, int i,
                                           const int32_t* table, int num_seqs, int max_blocks, uint32_t* dev_err,
                                           int& seq, int& pos) {
  seq = seq_ids != nullptr ? seq_ids[i] : i;
  pos = positions[i];
  if (seq < 0 || seq >= num_seqs) {
    report(dev_err, QMLA_DEVERR_BAD_SEQ);
    return -1;
  }
  if (pos < 0 || pos >= max_blocks * kBlockTokens) {
    report(dev_err, QMLA_DEVERR_BAD_POSITION);
    return -1;
  }
  const int blk = table[static_cast<size_t>(seq) * max_blocks + pos / kBlockTokens];
  if (blk < 0 || blk >= num_blocks) {
    report(dev_err, QMLA_DEVERR_BAD_BLOCK);
    return -1;
  }
  return blk;
}

// Sink/recent BF16 protection rows (App. C.5, "BF16 protection and cache
// lifecycle"): position p of a request whose length after this write is L goes
// to row p when p < 4 and to row 4 + p mod 128 when p >= L - 128; each lane stores
// its own 16 bytes of the token's 1152.

constexpr int kAppendThreads = kGroups * 32;

// Quantises and packs n tokens. CB: content bits (4, 2) or kC4R4 for the paper's
// page (INT4 codes). NT: tokens per lane, 1 or 4 (a block writes 4 NT). VEC: latent
// and k_pe are 16-byte aligned (one 16-byte load per lane, else four 4-byte ones).
// prot / lens: the protection buffer [num_seqs][132][576] bf16 and the requests'
// lengths after this write, or null for an unprotected cache.
//
// What bounds it: for a prefill the issue slots, then the HBM traffic (1152 bytes
// read and 324 written per token, INT4); for a decode step's few tokens the latency
// of load -> extrema -> scale -> codes -> store. So one pass holds eight coordinates
// per lane, the extrema take three packed shuffles for minimum and maximum together,
// and the codes take two values per instruction (codes8). With four tokens per lane
// the eight lanes of a token share what is per token: lane i of four looks token i's
// destination up and works out its scale, and shuffles hand them round. Groups
// outside codes8's argument (quotients above 2^14, infinite values or scales) and
// the fp32 RoPE scale of the paper's page, whose codes are defined by the rounded
// fp32 quotient, divide value by value. 32,797 tokens of eight ragged prompts (INT4, calls
// on buffers larger together than L2) take 16.5 us, 2.9 TB/s of 6.8; a warp per (token,
// group) with two coordinates per lane and a division per code took 61.5.
template <int CB, int NT, bool VEC>
__global__ void __launch_bounds__(kAppendThreads) quant_append_kernel(
    uint8_t* __restrict__ pool, int num_blocks, const uint32_t* __restrict__ latent,
    const uint32_t* __restrict__ k_pe, const int32_t* __restrict__ seq_ids,
    const int32_t* __restrict__ positions, int n, const int32_t* __restrict__ table, int num_seqs,
    int max_blocks, uint32_t* dev_err, uint4* __restrict__ prot, const int32_t* __restrict__ lens) {
  static_assert(NT == 1 || NT == 4, "tokens per lane");
  using L = BlockLayout<CB>;
  // The decode's prep kernel may start meanwhile: it does not read the cache, and it
  // neither writes anything nor ends before this kernel has ended. (A decode step with
  // prep after the writer / beside it, us: 8 sequences x 128 heads, 300..2,500 tokens,
  // protected 36.9 / 35.2; 64 x 4,097 INT4 116.8 / 115.5; 128 x 16 heads 186.9 / 185.4.)
  griddep_launch_dependents();
  const int g = threadIdx.x >> 5;  // this warp's group
  const int lane = threadIdx.x & 31;
  const int piece = lane & 7;
  const int tok0 = blockIdx.x * (4 * NT) + (lane >> 3);  // token i of the lane: tok0 + 4 i
  const int bits = g < 8 ? (CB == kC4R4 ? 4 : CB) : kPeBits;
  const int m = (1 << bits) - 1;
  // The groups' loads do not wait for the seq_ids -> block-table lookups, which
  // only the stores need.
  uint4 raw[NT];
#pragma unroll
  for (int i = 0; i < NT; ++i) {
    const int tok = tok0 + 4 * i;
    raw[i] = make_uint4(0, 0, 0, 0);
    if (tok < n) {
      const uint32_t* src = g < 8 ? latent + static_cast<size_t>(tok) * (kDc / 2) + g * 32 + piece * 4
                                  : k_pe + static_cast<size_t>(tok) * (kDr / 2) + piece * 4;
      if constexpr (VEC) {
        raw[i] = *reinterpret_cast<const uint4*>(src);
      } else {
        raw[i] = make_uint4(src[0], src[1], src[2], src[3]);
      }
    }
  }
  // This lane's share: token `own` of the lane's NT. dst is the block's slot, the
  // block id times 64 plus the slot, or -1; rows the protection rows (sink, ring), or
  // -1. Errors are reported once per token, by its group-0 warp.
  const int own = piece & (NT - 1);
  int dst = -1, sink = -1, ring = -1;
  if (tok0 + 4 * own < n) {
    const int tok = tok0 + 4 * own;
    int seq = 0, pos = 0;
    const int blk = token_block(num_blocks, seq_ids, positions, tok, table, num_seqs, max_blocks,
                                piece == own && g == 0 ? dev_err : nullptr, seq, pos);
    if (blk >= 0) {
      dst = blk * kBlockTokens + pos % kBlockTokens;
      if (prot != nullptr) {
        if (pos < kSinkTokens) sink = seq * kProtRows + pos;
        if (pos >= lens[seq] - kRecentTokens) ring = seq * kProtRows + kSinkTokens + pos % kRecentTokens;
      }
    }
  }
  // Extrema of each token's 64 values: (min, -max) as a bf16 pair, so that one packed
  // minimum per shuffle serves both. bf16 minima are exact, and NaNs lose against
  // numbers as in fminf / fmaxf.
  uint32_t ext = 0;  // of token `own`
#pragma unroll
  for (int i = 0; i < NT; ++i) {
    const uint32_t w[4] = {raw[i].x, raw[i].y, raw[i].z, raw[i].w};
    __nv_bfloat162 lo = *reinterpret_cast<const __nv_bfloat162*>(&w[0]), hi = lo;
#pragma unroll
    for (int e = 1; e < 4; ++e) {
      const __nv_bfloat162 v = *reinterpret_cast<const __nv_bfloat162*>(&w[e]);
      lo = __hmin2(lo, v);
      hi = __hmax2(hi, v);
    }
    lo = __hmin2(lo, __lowhigh2highlow(lo));
    hi = __hmax2(hi, __lowhigh2highlow(hi));
    uint32_t pk =
        __byte_perm(*reinterpret_cast<uint32_t*>(&lo), *reinterpret_cast<uint32_t*>(&hi) ^ 0x80008000u, 0x7610);
#pragma unroll
    for (int off = 1; off < 8; off <<= 1) {
      const uint32_t o = __shfl_xor_sync(0xffffffffu, pk, off);
      const __nv_bfloat162 r = __hmin2(*reinterpret_cast<const __nv_bfloat162*>(&pk),
                                       *reinterpret_cast<const __nv_bfloat162*>(&o));
      pk = *reinterpret_cast<const uint32_t*>(&r);
    }
    if (i == own) ext = pk;
  }
  const float xmin = __uint_as_float(ext << 16), xmax = -__uint_as_float(ext & 0xFFFF0000u);
  float s_own, z_own;
  if constexpr (CB == kC4R4) {
    paper_scale(xmin, xmax, g < 8, s_own, z_own);
  } else {
    group_scale(xmin, xmax, m, s_own, z_own);
  }
  // 1 / s, or 0 for a group whose values divide one by one (an infinite or NaN
  // quotient among them; 1 / s is 0 when s is infinite)
  float y_own = __frcp_rn(s_own);
  if (!(fmaxf(fabsf(xmin), fabsf(xmax)) * y_own <= 16384.0f) || (CB == kC4R4 && g == 8)) y_own = 0.0f;
  if (piece == own && dst >= 0) {
    uint8_t* blk = pool + static_cast<size_t>(dst / kBlockTokens) * L::kBytes;
    const int slot = dst % kBlockTokens;
    if constexpr (CB == kC4R4) {
      if (g < 8) {
        *reinterpret_cast<__nv_bfloat16*>(blk + L::c_scale_off(g, slot)) = __float2bfloat16_rn(s_own);  // exact
      } else {
        *reinterpret_cast<float*>(blk + L::pe_scale_off(slot)) = s_own;
      }
      blk[L::zero_off(g, slot)] = static_cast<uint8_t>(z_own);
    } else {
      *reinterpret_cast<__half2*>(blk + L::sz_off(g, slot)) =
          __halves2half2(__float2half_rn(s_own), __float2half_rn(z_own));
    }
  }
#pragma unroll
  for (int i = 0; i < NT; ++i) {
    const uint32_t w[4] = {raw[i].x, raw[i].y, raw[i].z, raw[i].w};
    // (the token's values from its lane i)
    const int from = (lane & 24) | i;
    const float s = NT == 1 ? s_own : __shfl_sync(0xffffffffu, s_own, from);
    const float y = NT == 1 ? y_own : __shfl_sync(0xffffffffu, y_own, from);
    const float z = NT == 1 ? z_own : __shfl_sync(0xffffffffu, z_own, from);
    const int d = NT == 1 ? dst : __shfl_sync(0xffffffffu, dst, from);
    uint32_t c[4];  // codes 2 e and 2 e + 1 in the halves of c[e]
    if (y > 0.0f) {
      codes8(w, s, y, z, m, c);
    } else {
#pragma unroll
      for (int e = 0; e < 4; ++e)
        c[e] = quant_code(__uint_as_float(w[e] << 16), s, z, static_cast<float>(m)) |
               quant_code(__uint_as_float(w[e] & 0xFFFF0000u), s, z, static_cast<float>(m)) << 16;
    }
    // Packed low bits first: INT4 byte j = code 2 j | code 2 j + 1 << 4, INT2 byte j = codes 4 j .. 4 j + 3.
    uint32_t word;
    if (bits == 4) {
      const uint32_t a = c[0] | c[1] << 8, b = c[2] | c[3] << 8;
      word = __byte_perm(a | a >> 12, b | b >> 12, 0x5410);
    } else {
      const uint32_t a = c[0] | c[1] << 4 | c[2] << 8 | c[3] << 12;
      word = a | a >> 14;
    }
    if (prot != nullptr) {
      const int rows[2] = {NT == 1 ? sink : __shfl_sync(0xffffffffu, sink, from),
                           NT == 1 ? ring : __shfl_sync(0xffffffffu, ring, from)};
#pragma unroll
      for (int r = 0; r < 2; ++r)
        if (rows[r] >= 0) prot[static_cast<size_t>(rows[r]) * (kDqk * 2 / 16) + g * 8 + piece] = raw[i];
    }
    if (d < 0) continue;
    uint8_t* code = pool + static_cast<size_t>(d / kBlockTokens) * L::kBytes + L::code_off(g, d % kBlockTokens);
    if (bits == 4) {
      reinterpret_cast<uint32_t*>(code)[piece] = word;
    } else {
      reinterpret_cast<uint16_t*>(code)[piece] = static_cast<uint16_t>(word);
    }
  }
}

// Copies each token's 72 16-byte pieces (64 of the latent, 8 of the RoPE key)
// unchanged, one piece per thread. Bound by HBM for a prefill: whole 16-byte
// accesses on both sides, neighbouring threads on neighbouring pieces.
template <bool VEC>
__global__ void __launch_bounds__(256) bf16_append_kernel(
    uint8_t* __restrict__ pool, int num_blocks, const uint32_t* __restrict__ latent,
    const uint32_t* __restrict__ k_pe, const int32_t* __restrict__ seq_ids,
    const int32_t* __restrict__ positions, int n, const int32_t* __restrict__ table, int num_seqs,
    int max_blocks, uint32_t* dev_err) {
  constexpr int kPieces = kDqk * 2 / 16;
  griddep_launch_dependents();  // as in quant_append_kernel
  const long long idx = static_cast<long long>(blockIdx.x) * blockDim.x + threadIdx.x;
  const int tok = static_cast<int>(idx / kPieces);
  const int piece = static_cast<int>(idx - static_cast<long long>(tok) * kPieces);
  if (tok >= n) return;
  const uint32_t* src = piece < kDc / 8 ? latent + static_cast<size_t>(tok) * (kDc / 2) + piece * 4
                                        : k_pe + static_cast<size_t>(tok) * (kDr / 2) + (piece - kDc / 8) * 4;
  uint4 v;
  if constexpr (VEC) {
    v = *reinterpret_cast<const uint4*>(src);
  } else {
    v = make_uint4(src[0], src[1], src[2], src[3]);
  }
  int seq = 0, pos = 0;
  const int blk = token_block(num_blocks, seq_ids, positions, tok, table, num_seqs, max_blocks,
                              piece == 0 ? dev_err : nullptr, seq, pos);
  if (blk < 0) return;
  reinterpret_cast<uint4*>(pool + static_cast<size_t>(blk) * kBf16BlockBytes + pos % kBlockTokens * (kDqk * 2))[piece] =
      v;
}

bool aligned16(const void* a, const void* b) {
  return ((reinterpret_cast<uintptr_t>(a) | reinterpret_cast<uintptr_t>(b)) & 15) == 0;
}

template <int CB, int NT, bool VEC>
void launch_quant(void* pool, int num_blocks, const uint16_t* latent, const uint16_t* k_pe, const int32_t* seq_ids,
                  const int32_t* positions, int n, const int32_t* table, int num_seqs, int max_blocks,
                  uint32_t* dev_err, cudaStream_t stream, void* prot, const int32_t* lens) {
  const unsigned grid = static_cast<unsigned>((static_cast<long long>(n) + 4 * NT - 1) / (4 * NT));
  quant_append_kernel<CB, NT, VEC><<<grid, kAppendThreads, 0, stream>>>(
      static_cast<uint8_t*>(pool), num_blocks, reinterpret_cast<const uint32_t*>(latent),
      reinterpret_cast<const uint32_t*>(k_pe), seq_ids, positions, n, table, num_seqs, max_blocks, dev_err,
      static_cast<uint4*>(prot), lens);
}

// Tokens from which a lane takes four: below, one token per lane spreads the
// tokens over more SMs and ends sooner. One GB300, INT4 / the paper's page, eight
// prompts of equal length, buffers larger together than L2, four against one: 4,096
// tokens 4.1 against 3.9 / 5.4 against 4.5 us, 8,192 5.8 against 6.3 / 7.1 against 7.1,
// 32,768 15.1 against 19.5 / 19.8 against 20.7.
constexpr int kFourPerLane = 8192;

template <int CB>
void launch_quant(void* pool, int num_blocks, const uint16_t* latent, const uint16_t* k_pe, const int32_t* seq_ids,
                  const int32_t* positions, int n, const int32_t* table, int num_seqs, int max_blocks,
                  uint32_t* dev_err, cudaStream_t stream, void* prot, const int32_t* lens) {
  auto* f = !aligned16(latent, k_pe) ? launch_quant<CB, 1, false>
                                     : (n >= kFourPerLane ? launch_quant<CB, 4, true> : launch_quant<CB, 1, true>);
  f(pool, num_blocks, latent, k_pe, seq_ids, positions, n, table, num_seqs, max_blocks, dev_err, stream, prot, lens);
}

}  // namespace

cudaError_t launch_quant_append(void* pool, int c_bits, int num_blocks, const uint16_t* latent,
                                const uint16_t* k_pe, const int32_t* seq_ids,
                                const int32_t* positions, int n, const int32_t* table, int num_seqs,
                                int max_blocks, uint32_t* dev_err, cudaStream_t stream, void* prot,
                                const int32_t* lens) {
  if (n == 0) return cudaSuccess;
  auto* f = c_bits == kC4R4 ? launch_quant<kC4R4> : (c_bits == 4 ? launch_quant<4> : launch_quant<2>);
  f(pool, num_blocks, latent, k_pe, seq_ids, positions, n, table, num_seqs, max_blocks, dev_err, stream, prot, lens);
  return cudaGetLastError();
}

cudaError_t launch_bf16_append(void* pool, int num_blocks, const uint16_t* latent,
                               const uint16_t* k_pe, const int32_t* seq_ids,
                               const int32_t* positions, int n, const int32_t* table, int num_seqs,
                               int max_blocks, uint32_t* dev_err, cudaStream_t stream) {
  if (n == 0) return cudaSuccess;
  const unsigned grid = static_cast<unsigned>((static_cast<long long>(n) * (kDqk * 2 / 16) + 255) / 256);
  auto* f = aligned16(latent, k_pe) ? bf16_append_kernel<true> : bf16_append_kernel<false>;
  f<<<grid, 256, 0, stream>>>(static_cast<uint8_t*>(pool), num_blocks, reinterpret_cast<const uint32_t*>(latent),
                              reinterpret_cast<const uint32_t*>(k_pe), seq_ids, positions, n, table, num_seqs,
                              max_blocks, dev_err);
  return cudaGetLastError();
}

}  // namespace qmla
