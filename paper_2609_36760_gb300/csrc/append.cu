// Quantise-and-pack cache writer (App. C.4 quantiser; App. C.5 cache update:
// content- and RoPE-cache quantisation, integer packing and slot-mapped page
// insertion) for this library's block and for the paper's own page, and the
// plain BF16 writer for the comparison cache.
//
// A block of nine warps writes a few tokens: warp g quantises group g (64
// coordinates) of four tokens at a time, eight lanes per token with eight
// coordinates (16 bytes) each. A warp then reads four whole 128-byte lines and,
// where the tokens take consecutive slots (a prefill), writes their code rows
// and scales as contiguous runs; the bit width and the scale format are uniform
// in a warp. See quant_append_kernel for what bounds it.
#include <cuda_runtime.h>

#include "common.cuh"
#include "kernels.h"

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

// Two fp32 operations per instruction.
__device__ __forceinline__ uint64_t f32x2(float a, float b) {
  uint64_t r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(a), "f"(b));
  return r;
}
__device__ __forceinline__ uint64_t mul2(uint64_t a, uint64_t b) {
  uint64_t r;
  asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}
__device__ __forceinline__ uint64_t add2(uint64_t a, uint64_t b) {
  uint64_t r;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}
__device__ __forceinline__ uint64_t fma2(uint64_t a, uint64_t b, uint64_t c) {
  uint64_t r;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
  return r;
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

// Looks up and validates the destination of token i. Returns null (after
// recording the error) when the token cannot be written.
__device__ __forceinline__ uint8_t* token_block(uint8_t* pool, size_t block_bytes, int num_blocks,
                                                const int32_t* seq_ids, const int32_t* positions,
                                                int i, const int32_t* table, int num_seqs,
                                                int max_blocks, uint32_t* dev_err, int& slot) {
  const int seq = seq_ids != nullptr ? seq_ids[i] : i;
  const int pos = positions[i];
  if (seq < 0 || seq >= num_seqs) {
    report(dev_err, QMLA_DEVERR_BAD_SEQ);
    return nullptr;
  }
  if (pos < 0 || pos >= max_blocks * kBlockTokens) {
    report(dev_err, QMLA_DEVERR_BAD_POSITION);
    return nullptr;
  }
  const int blk = table[static_cast<size_t>(seq) * max_blocks + pos / kBlockTokens];
  if (blk < 0 || blk >= num_blocks) {
    report(dev_err, QMLA_DEVERR_BAD_BLOCK);
    return nullptr;
  }
  slot = pos % kBlockTokens;
  return pool + static_cast<size_t>(blk) * block_bytes;
}

// Sink/recent BF16 protection rows (App. C.5, "BF16 protection and cache
// lifecycle"): position p of a request whose length after this write is L goes
// to row p when p < 4 and to row 4 + p mod 128 when p >= L - 128. Each lane
// stores its own 16 bytes, piece `piece` (0..71) of the token's 1152.
__device__ __forceinline__ void protect_piece(uint4* prot, const uint4& v, int piece, int seq, int pos, int L) {
  uint4* base = prot + static_cast<size_t>(seq) * kProtRows * (kDqk * 2 / 16) + piece;
  if (pos < kSinkTokens) base[pos * (kDqk * 2 / 16)] = v;
  if (pos >= L - kRecentTokens) base[(kSinkTokens + pos % kRecentTokens) * (kDqk * 2 / 16)] = v;
}

constexpr int kAppendThreads = kGroups * 32;

// Quantises and packs n tokens. CB: content bits (4, 2) or kC4R4 for the paper's
// page (INT4 codes). NT: tokens per lane (a block writes 4 NT). VEC: latent and
// k_pe are 16-byte aligned (one 16-byte load per lane, else four 4-byte ones).
// prot / lens: the protection buffer [num_seqs][132][576] bf16 and the requests'
// lengths after this write, or null for an unprotected cache.
//
// What bounds it: for a prefill the issue slots and the HBM traffic (1152 bytes
// read and 324 written per token, INT4) weigh about the same; for a decode
// step's few tokens the latency of load -> extrema -> scale -> codes -> store.
// So one pass holds eight coordinates per lane, the extrema take three packed
// shuffles for minimum and maximum together, and the codes take two values per
// instruction (codes8). Groups outside codes8's argument (quotients above 2^14,
// infinite values or scales) and the fp32 RoPE scale of the paper's page, whose
// codes are defined by the rounded fp32 quotient, divide value by value.
template <int CB, int NT, bool VEC>
__global__ void __launch_bounds__(kAppendThreads) quant_append_kernel(
    uint8_t* __restrict__ pool, int num_blocks, const uint32_t* __restrict__ latent,
    const uint32_t* __restrict__ k_pe, const int32_t* __restrict__ seq_ids,
    const int32_t* __restrict__ positions, int n, const int32_t* __restrict__ table, int num_seqs,
    int max_blocks, uint32_t* dev_err, uint4* __restrict__ prot, const int32_t* __restrict__ lens) {
  using L = BlockLayout<CB>;
  const int g = threadIdx.x >> 5;  // this warp's group
  const int lane = threadIdx.x & 31;
  const int piece = lane & 7;
  const int tok0 = blockIdx.x * (4 * NT) + (lane >> 3);
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
  uint8_t* blk[NT];
  int slot[NT];
#pragma unroll
  for (int i = 0; i < NT; ++i) {
    const int tok = tok0 + 4 * i;
    blk[i] = nullptr;
    slot[i] = 0;
    // errors are reported once per token, by its group-0 warp
    if (tok < n)
      blk[i] = token_block(pool, L::kBytes, num_blocks, seq_ids, positions, tok, table, num_seqs, max_blocks,
                           piece == 0 && g == 0 ? dev_err : nullptr, slot[i]);
  }
#pragma unroll
  for (int i = 0; i < NT; ++i) {
    const uint32_t w[4] = {raw[i].x, raw[i].y, raw[i].z, raw[i].w};
    // Extrema of the token's 64 values: (min, -max) as a bf16 pair, so that one
    // packed minimum per shuffle serves both. bf16 minima are exact, and NaNs
    // lose against numbers as in fminf / fmaxf.
    __nv_bfloat162 lo = *reinterpret_cast<const __nv_bfloat162*>(&w[0]), hi = lo;
#pragma unroll
    for (int e = 1; e < 4; ++e) {
      const __nv_bfloat162 v = *reinterpret_cast<const __nv_bfloat162*>(&w[e]);
      lo = __hmin2(lo, v);
      hi = __hmax2(hi, v);
    }
    lo = __hmin2(lo, __lowhigh2highlow(lo));
    hi = __hmax2(hi, __lowhigh2highlow(hi));
    uint32_t pk = __byte_perm(*reinterpret_cast<uint32_t*>(&lo), *reinterpret_cast<uint32_t*>(&hi) ^ 0x80008000u, 0x7610);
#pragma unroll
    for (int off = 1; off < 8; off <<= 1) {
      const uint32_t o = __shfl_xor_sync(0xffffffffu, pk, off);
      const __nv_bfloat162 r = __hmin2(*reinterpret_cast<const __nv_bfloat162*>(&pk),
                                       *reinterpret_cast<const __nv_bfloat162*>(&o));
      pk = *reinterpret_cast<const uint32_t*>(&r);
    }
    const float xmin = __uint_as_float(pk << 16), xmax = -__uint_as_float(pk & 0xFFFF0000u);
    float s, z;
    if constexpr (CB == kC4R4) {
      paper_scale(xmin, xmax, g < 8, s, z);
    } else {
      group_scale(xmin, xmax, m, s, z);
    }
    const float y = __frcp_rn(s);
    // (false for an infinite or NaN quotient; y = 0 when s is infinite)
    const bool fast = y > 0.0f && fmaxf(fabsf(xmin), fabsf(xmax)) * y <= 16384.0f && !(CB == kC4R4 && g == 8);
    uint32_t c[4];  // codes 2 e and 2 e + 1 in the halves of c[e]
    if (fast) {
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
    if (blk[i] == nullptr) continue;
    const int tok = tok0 + 4 * i;
    if (prot != nullptr) {
      const int seq = seq_ids != nullptr ? seq_ids[tok] : tok;
      protect_piece(prot, raw[i], g * 8 + piece, seq, positions[tok], lens[seq]);
    }
    uint8_t* dst = blk[i] + L::code_off(g, slot[i]);
    if (bits == 4) {
      reinterpret_cast<uint32_t*>(dst)[piece] = word;
    } else {
      reinterpret_cast<uint16_t*>(dst)[piece] = static_cast<uint16_t>(word);
    }
    if (piece == 0) {
      if constexpr (CB == kC4R4) {
        if (g < 8) {
          *reinterpret_cast<__nv_bfloat16*>(blk[i] + L::c_scale_off(g, slot[i])) = __float2bfloat16_rn(s);  // exact
        } else {
          *reinterpret_cast<float*>(blk[i] + L::pe_scale_off(slot[i])) = s;
        }
        blk[i][L::zero_off(g, slot[i])] = static_cast<uint8_t>(z);
      } else {
        *reinterpret_cast<__half2*>(blk[i] + L::sz_off(g, slot[i])) =
            __halves2half2(__float2half_rn(s), __float2half_rn(z));
      }
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
  int slot = 0;
  uint8_t* blk = token_block(pool, kBf16BlockBytes, num_blocks, seq_ids, positions, tok, table,
                             num_seqs, max_blocks, piece == 0 ? dev_err : nullptr, slot);
  if (blk == nullptr) return;
  reinterpret_cast<uint4*>(blk + slot * kDqk * 2)[piece] = v;
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

// Tokens from which a lane takes two: below, one token per lane spreads the
// step's tokens over more SMs and ends sooner.
constexpr int kTwoPerLane = 8192;

template <int CB>
void launch_quant(void* pool, int num_blocks, const uint16_t* latent, const uint16_t* k_pe, const int32_t* seq_ids,
                  const int32_t* positions, int n, const int32_t* table, int num_seqs, int max_blocks,
                  uint32_t* dev_err, cudaStream_t stream, void* prot, const int32_t* lens) {
  auto* f = !aligned16(latent, k_pe) ? launch_quant<CB, 1, false>
                                     : (n >= kTwoPerLane ? launch_quant<CB, 2, true> : launch_quant<CB, 1, true>);
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
