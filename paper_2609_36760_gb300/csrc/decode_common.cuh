// Device code shared by the decode kernels: parameters, cache-row fetch and
// dequantisation (this library's blocks, the paper's page, BF16 rows, protection
// rows) and bounded waits.
#pragma once
#include <cuda_runtime.h>

#include <cstddef>

#include "common.cuh"
#include "kernels.h"
#include "ptx.cuh"

namespace qmla {

struct Params {
  const uint8_t* pool;
  // sink4/local128 protection buffer [batch][132][576] bf16, or null (unprotected).
  const uint8_t* prot;
  int num_blocks;
  const __nv_bfloat16* q_lat;
  const __nv_bfloat16* q_pe;
  // heads = q_tokens * hpt "virtual heads" (query token t, head h) -> t * hpt + h;
  // one query token per sequence: q_tokens = 1, hpt = heads.
  int batch, heads, n_hg;
  int n_img;  // query images (64-, 32- or 16-head groups) per sequence
  int q_tokens, hpt;
  const int32_t* table;
  int max_blocks;
  const int32_t* seq_lens;
  float scale_log2;  // softmax_scale * log2(e)
  float* out;
  float* lse;
  const int32_t* prefix;
  int32_t* prefix_w;
  // [grid] per CTA, written by the prep kernel with the prefix: {unit of the first
  // tile, prefix[unit], prefix[unit + 1], total tiles} and, for the first tile,
  // {table entry of rows 0..63, of rows 64..127, sequence length, tile index}, or for
  // a CTA pair {reference tile of row group 0, of group 1, sequence length, -}.
  int4* cta_info;
  int4* cta_first;
  int32_t* cta_t0;  // [grid + 1]: first tile of each CTA's range (cta_t0[grid] = total tiles)
  float* part_o;   // [(grid + units)][HG][512]
  float* part_ml;  // [(grid + units)][HG][2]
  uint8_t* qimg;   // [batch * n_img][9][HG][128 B]: swizzled fp16 query tiles
  uint32_t* dev_err;
  int grid;  // ranges the tile list is cut into
  int sms;
  unsigned long long* trace;  // trace builds only: per-CTA event clocks, else null
};

// Main kernel of the CTA-pair decode (decode_pair.cu) for a plan over 128-head
// units; pdl: it may overlap its predecessor's end.
cudaError_t launch_decode_pair(const Params& prm, int cache_kind, bool pdl, cudaStream_t stream);

namespace {

constexpr int kTileTokens = 128;                 // tokens per tile of the split plan
constexpr int kNumChunks = 9;                    // 8 content chunks of 64 channels + RoPE-key chunk
constexpr uint64_t kWaitNs = 2000000000ull;      // bound of every on-chip wait (2 s)
constexpr float kRescaleLog2 = 8.0f;             // rescale O only above 2^8 growth
constexpr float kLn2 = 0.6931471805599453f;


// Optional per-CTA timeline (clock64 at pipeline events), compiled in only
// for trace builds (-DQMLA_TRACE_BUILD); see qmla_trace_set in api.cu.
#ifdef QMLA_TRACE_BUILD
constexpr int kTraceCtas = 8, kTraceEvents = 128, kTraceTiles = 32;
// The buffer pointer travels in the kernel parameters (constant bank), so an
// event costs one clock read and one global store, no load.
#define QMLA_TRACE(ev, tile)                                                                     \
  do {                                                                                           \
    if (p.trace != nullptr && blockIdx.x < kTraceCtas && (tile) < kTraceTiles)                   \
      p.trace[(static_cast<size_t>(blockIdx.x) * kTraceEvents + (ev)) * kTraceTiles + (tile)] = \
          clock64();                                                                             \
  } while (0)
// All CTAs: wall-clock start/end (%globaltimer), SM id and tile count after the event area.
#define QMLA_TRACE_CTA(slot, value)                                                                       \
  do {                                                                                                    \
    if (p.trace != nullptr)                                                                               \
      p.trace[static_cast<size_t>(kTraceCtas) * kTraceEvents * kTraceTiles + blockIdx.x * 4 + (slot)] = \
          (value);                                                                                        \
  } while (0)
#else
#define QMLA_TRACE(ev, tile) \
  do {                       \
  } while (0)
#define QMLA_TRACE_CTA(slot, value) \
  do {                              \
  } while (0)
#endif

// Channel order inside each 8-channel (16-byte) piece of a reconstructed row:
// the unpacking below yields nibble/crumb pairs in this order, and the query
// tile and the output mapping use the same permutation.
template <int CB>
struct Perm {
  // position p of a piece holds channel at(p): INT4 swaps bits 0 and 1 of p
  // ([0,2,1,3,4,6,5,7]); INT2 rotates them ([0,4,1,5,2,6,3,7]); BF16 keeps p.
  __host__ __device__ static constexpr int at(int p) {
    if constexpr (CB == 4 || CB == kC4R4) {
      return (p & 4) | ((p & 1) << 1) | ((p >> 1) & 1);
    } else if constexpr (CB == 2) {
      return ((p & 1) << 2) | (p >> 1);
    } else {
      return p;
    }
  }
};
static_assert(Perm<4>::at(1) == 2 && Perm<4>::at(2) == 1 && Perm<4>::at(5) == 6 && Perm<4>::at(7) == 7, "INT4 order");
static_assert(Perm<2>::at(1) == 4 && Perm<2>::at(2) == 1 && Perm<2>::at(6) == 3 && Perm<2>::at(7) == 7, "INT2 order");

// --------------------------------------------------------------- helpers
__device__ __forceinline__ uint4 ldg_nc_v4(const void* ptr) {
  uint4 r;
  asm volatile("ld.global.nc.L1::no_allocate.v4.u32 {%0,%1,%2,%3}, [%4];"
               : "=r"(r.x), "=r"(r.y), "=r"(r.z), "=r"(r.w)
               : "l"(ptr));
  return r;
}
// 32 bytes in one request (the address is 32-byte aligned).
__device__ __forceinline__ void ldg_nc_v8(const void* ptr, uint4& a, uint4& b) {
  asm volatile("ld.global.nc.L1::no_allocate.v8.u32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
               : "=r"(a.x), "=r"(a.y), "=r"(a.z), "=r"(a.w), "=r"(b.x), "=r"(b.y), "=r"(b.z), "=r"(b.w)
               : "l"(ptr));
}
__device__ __forceinline__ uint32_t ldg_nc_u32(const void* ptr) {
  uint32_t r;
  asm volatile("ld.global.nc.L1::no_allocate.u32 %0, [%1];" : "=r"(r) : "l"(ptr));
  return r;
}
__device__ __forceinline__ uint32_t ldg_nc_u16(const void* ptr) {
  uint16_t r;
  asm volatile("ld.global.nc.L1::no_allocate.u16 %0, [%1];" : "=h"(r) : "l"(ptr));
  return r;
}
__device__ __forceinline__ uint32_t ldg_nc_u8(const void* ptr) {
  uint32_t r;
  asm volatile("ld.global.nc.L1::no_allocate.u8 %0, [%1];" : "=r"(r) : "l"(ptr));
  return r;
}
__device__ __forceinline__ void sts_v4(uint32_t addr, uint32_t a, uint32_t b, uint32_t c, uint32_t d) {
  asm volatile("st.shared.v4.b32 [%0], {%1,%2,%3,%4};" ::"r"(addr), "r"(a), "r"(b), "r"(c), "r"(d)
               : "memory");
}
// RN_f16((x - zz) * s) per half: the subtraction of two integers below 2048 is
// exact, so this is a single rounding of s (q - z).
__device__ __forceinline__ uint32_t dq2(uint32_t x, uint32_t zz, uint32_t ss) {
  uint32_t t, r;
  asm("sub.rn.f16x2 %0, %1, %2;" : "=r"(t) : "r"(x), "r"(zz));
  asm("mul.rn.f16x2 %0, %1, %2;" : "=r"(r) : "r"(t), "r"(ss));
  return r;
}
__device__ __forceinline__ uint32_t pack_h2(float lo, float hi) {
  const __half2 h = __floats2half2_rn(lo, hi);
  return *reinterpret_cast<const uint32_t*>(&h);
}
__device__ __forceinline__ float bf16_lo(uint32_t w) { return __uint_as_float(w << 16); }
__device__ __forceinline__ float bf16_hi(uint32_t w) { return __uint_as_float(w & 0xFFFF0000u); }
__device__ __forceinline__ float warp_max_f32(float v) {
  float r;
  asm volatile("redux.sync.max.f32 %0, %1, 0xffffffff;" : "=f"(r) : "f"(v));
  return r;
}

// Wait sites, reported in bits 8.. of the error word when a wait runs out.
enum WaitSite : uint32_t {
  kSiteDqSlot = 0, kSiteMmaQFull, kSiteMmaChunk, kSiteMmaPFull, kSiteMmaOFree,
  kSiteSmSFull, kSiteGrp, kSitePvEpi, kSiteMmaFin
};

// Marks the CTA aborted; a wait that ran out (rather than saw the abort)
// also records its site.
template <class C>
__device__ __forceinline__ void set_abort(C& c, uint32_t* dev_err) {
  *reinterpret_cast<volatile uint32_t*>(&c.abort) = 1u;
  report(dev_err, QMLA_DEVERR_TIMEOUT);
}
template <class C>
__device__ __forceinline__ bool wait_ok(int r, uint32_t site, C& c, uint32_t* dev_err) {
  if (r == 0) {
    report(dev_err, QMLA_DEVERR_TIMEOUT | (0x100u << site));
    *reinterpret_cast<volatile uint32_t*>(&c.abort) = 1u;
  }
  return r == 1;
}
// Warp-uniform bounded wait: every lane waits on the barrier itself. Letting
// one lane poll while the others sit at a warp-synchronising instruction was
// measured to be much slower on sm_103a: the parked warp delayed the draining
// of other warps' shared-memory stores by thousands of cycles, and its own
// wake-up after the phase completed took ~2k cycles.
template <class C>
__device__ __forceinline__ bool wwait(uint64_t* bar, uint32_t parity, C& c, uint32_t site,
                                      uint32_t* dev_err, uint64_t limit_ns = kWaitNs) {
  const int r = mbar_wait(bar, parity, limit_ns, &c.abort);
  const bool all_ok = __all_sync(0xffffffffu, r == 1);
  if (r == 0) wait_ok(r, site, c, dev_err);
  return all_ok;
}
// Barrier among the worker warps (one arrive per warp), bounded. Every worker
// passes the same sequence of these, so one mbarrier serves them all: a warp
// cannot arrive for phase n + 2 before every warp has arrived for n + 1.
template <class C>
__device__ __forceinline__ bool group_sync(C& c, uint32_t& phase, uint32_t* dev_err) {
  __syncwarp();
  mbar_arrive_if((threadIdx.x & 31) == 0 ? 1u : 0u, &c.grp);
  const bool ok = wwait(&c.grp, phase & 1u, c, kSiteGrp, dev_err);
  ++phase;
  return ok;
}

// -------------------------------------------------------- dequant warps
// Packed data of one token row for one chunk, fetched ahead of use.
struct Fetch {
  uint4 a, b;
  uint32_t sz;  // fp16 (s, z) pair; for the paper's page the scale as fp32 bits
  uint32_t z;   // the paper's page: the uint8 zero point
  bool ok;
};

// Block-table entry and sequence length of one token row of a tile, loaded a
// tile before they are needed (nothing branches on them until resolve_row).
// The table column is clamped so that rows past the sequence end never read
// beyond the sequence's table row.
struct RowRef {
  int entry, len, j, b;
  bool has;
};
template <int CB>
__device__ __forceinline__ const uint8_t* resolve_row(const Params& p, const RowRef& r, int row, bool& valid) {
  valid = false;
  if (!r.has || row >= min(kTileTokens, r.len - kTileTokens * r.j)) return nullptr;
  if (r.entry < 0 || r.entry >= p.num_blocks) {
    report(p.dev_err, QMLA_DEVERR_BAD_BLOCK);
    return nullptr;
  }
  valid = true;
  constexpr size_t kBlk = CB == 16 ? static_cast<size_t>(kBf16BlockBytes) : BlockLayout<CB == 16 ? 4 : CB>::kBytes;
  return p.pool + static_cast<size_t>(r.entry) * kBlk;
}

// The protection-buffer row a tile row attends with (App. C.5, "BF16
// protection and cache lifecycle": position p of a length-L request is
// protected iff p < min(4, L) or p >= L - 128), or null when the row is read
// from the packed cache. Sink positions read their sink row, which the writer
// always fills; recent ones the ring row 4 + p mod 128.
__device__ __forceinline__ const uint8_t* prot_row(const Params& p, const RowRef& r, int row) {
  if (p.prot == nullptr || !r.has) return nullptr;
  const int pos = kTileTokens * r.j + row;
  if (pos >= r.len) return nullptr;
  int pr;
  if (pos < kSinkTokens) {
    pr = pos;
  } else if (pos >= r.len - kRecentTokens) {
    pr = kSinkTokens + pos % kRecentTokens;
  } else {
    return nullptr;
  }
  return p.prot + (static_cast<size_t>(r.b) * kProtRows + pr) * (kDqk * 2);
}

template <int CB>
__device__ __forceinline__ Fetch fetch_chunk(const uint8_t* blk, bool valid, int k, int slot) {
  Fetch f;
  f.ok = valid;
  f.a = make_uint4(0, 0, 0, 0);
  f.b = f.a;
  f.sz = 0;
  f.z = 0;
  if (!valid) return f;
  using L = BlockLayout<CB>;
  const uint8_t* c = blk + L::code_off(k, slot);
  // a 32-byte code row in one request (half the requests of two 16-byte
  // loads, which made the next tile's fetch a quarter of the kernel's time)
  if (CB == 4 || CB == kC4R4 || k == 8) {
    ldg_nc_v8(c, f.a, f.b);
  } else {
    f.a = ldg_nc_v4(c);
  }
  if constexpr (CB == kC4R4) {
    // bf16 content scale -> fp32 bits by a 16-bit shift; the RoPE scale is fp32
    f.sz = k < 8 ? ldg_nc_u16(blk + L::c_scale_off(k, slot)) << 16 : ldg_nc_u32(blk + L::pe_scale_off(slot));
    f.z = ldg_nc_u8(blk + L::zero_off(k, slot));
  } else {
    f.sz = ldg_nc_u32(blk + L::sz_off(k, slot));
  }
  return f;
}

// Half h of a token row of the RoPE-key chunk (INT4 codes of channels 32 h ..
// 32 h + 31, bytes 16 h .. 16 h + 15): the two worker warps that share a row
// quarter split that chunk, so each dequantises 4.5 chunks per tile.
template <int CB>
__device__ __forceinline__ Fetch fetch_rope_half(const uint8_t* blk, bool valid, int slot, int h) {
  Fetch f;
  f.ok = valid;
  f.a = make_uint4(0, 0, 0, 0);
  f.b = f.a;
  f.sz = 0;
  f.z = 0;
  if (!valid) return f;
  using L = BlockLayout<CB>;
  f.a = ldg_nc_v4(blk + L::code_off(8, slot) + 16 * h);
  if constexpr (CB == kC4R4) {
    f.sz = ldg_nc_u32(blk + L::pe_scale_off(slot));  // the fp32 RoPE scale
    f.z = ldg_nc_u8(blk + L::zero_off(8, slot));
  } else {
    f.sz = ldg_nc_u32(blk + L::sz_off(8, slot));
  }
  return f;
}

// Unpacks one row (64 codes) of chunk k and stores RN_f16(s (q - z)) into the
// swizzled chunk tile. The code nibbles / crumbs are placed into the mantissa
// of 1024.0 (0x6400), giving 1024 + q exactly; subtracting 1024 + z is exact.
template <int CB>
__device__ __forceinline__ void store_row(uint32_t chunk_base, int row, const Fetch& f, bool int4) {
  if (!f.ok) {
#pragma unroll
    for (int i = 0; i < 8; ++i) sts_v4(chunk_base + swz_off(row, i, 128), 0, 0, 0, 0);
    return;
  }
  const __half2 sz = *reinterpret_cast<const __half2*>(&f.sz);
  const __half2 s2 = __half2half2(__low2half(sz));
  const __half2 zz2 = __half2half2(__hadd(__high2half(sz), __float2half_rn(1024.0f)));
  const uint32_t ss = *reinterpret_cast<const uint32_t*>(&s2);
  const uint32_t zz = *reinterpret_cast<const uint32_t*>(&zz2);
  constexpr uint32_t K = 0x64646464u;
  if (int4) {
    const uint32_t w[8] = {f.a.x, f.a.y, f.a.z, f.a.w, f.b.x, f.b.y, f.b.z, f.b.w};
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      const uint32_t lo = w[i] & 0x0F0F0F0Fu;          // e0 e2 e4 e6
      const uint32_t hi = (w[i] >> 4) & 0x0F0F0F0Fu;   // e1 e3 e5 e7
      sts_v4(chunk_base + swz_off(row, i, 128), dq2(__byte_perm(lo, K, 0x4140), zz, ss),
             dq2(__byte_perm(hi, K, 0x4140), zz, ss), dq2(__byte_perm(lo, K, 0x4342), zz, ss),
             dq2(__byte_perm(hi, K, 0x4342), zz, ss));
    }
  } else {
    const uint32_t w[4] = {f.a.x, f.a.y, f.a.z, f.a.w};
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const uint32_t c0 = w[i] & 0x03030303u;          // e0 e4 e8 e12
      const uint32_t c1 = (w[i] >> 2) & 0x03030303u;   // e1 e5 e9 e13
      const uint32_t c2 = (w[i] >> 4) & 0x03030303u;   // e2 e6 e10 e14
      const uint32_t c3 = (w[i] >> 6) & 0x03030303u;   // e3 e7 e11 e15
      sts_v4(chunk_base + swz_off(row, 2 * i, 128), dq2(__byte_perm(c0, K, 0x4140), zz, ss),
             dq2(__byte_perm(c1, K, 0x4140), zz, ss), dq2(__byte_perm(c2, K, 0x4140), zz, ss),
             dq2(__byte_perm(c3, K, 0x4140), zz, ss));
      sts_v4(chunk_base + swz_off(row, 2 * i + 1, 128), dq2(__byte_perm(c0, K, 0x4342), zz, ss),
             dq2(__byte_perm(c1, K, 0x4342), zz, ss), dq2(__byte_perm(c2, K, 0x4342), zz, ss),
             dq2(__byte_perm(c3, K, 0x4342), zz, ss));
    }
  }
}

// store_row split around the slot wait for the decode workers: dq_regs
// dequantises a packed row into registers before the wait, store_regs writes
// it into the swizzled chunk after it, so that only the stores remain between
// the slot's release and the chunk's arrival. Same arithmetic as store_row; a
// row that is not fetched (f.ok false) has zero codes, scale and zero point,
// so it dequantises to zeros without a branch.
__device__ __forceinline__ void dq_regs(uint32_t (&o)[32], const Fetch& f, bool int4) {
  const __half2 sz = *reinterpret_cast<const __half2*>(&f.sz);
  const __half2 s2 = __half2half2(__low2half(sz));
  const __half2 zz2 = __half2half2(__hadd(__high2half(sz), __float2half_rn(1024.0f)));
  const uint32_t ss = *reinterpret_cast<const uint32_t*>(&s2);
  const uint32_t zz = *reinterpret_cast<const uint32_t*>(&zz2);
  constexpr uint32_t K = 0x64646464u;
  const uint32_t w[8] = {f.a.x, f.a.y, f.a.z, f.a.w, f.b.x, f.b.y, f.b.z, f.b.w};
#pragma unroll
  for (int i = 0; i < 8; ++i) {
    if (int4) {
      const uint32_t lo = w[i] & 0x0F0F0F0Fu;
      const uint32_t hi = (w[i] >> 4) & 0x0F0F0F0Fu;
      o[4 * i + 0] = dq2(__byte_perm(lo, K, 0x4140), zz, ss);
      o[4 * i + 1] = dq2(__byte_perm(hi, K, 0x4140), zz, ss);
      o[4 * i + 2] = dq2(__byte_perm(lo, K, 0x4342), zz, ss);
      o[4 * i + 3] = dq2(__byte_perm(hi, K, 0x4342), zz, ss);
    } else {  // INT2: pieces 2m and 2m + 1 come from word m
      const uint32_t x = w[i >> 1];
      const uint32_t sel = (i & 1) ? 0x4342u : 0x4140u;
      o[4 * i + 0] = dq2(__byte_perm(x & 0x03030303u, K, sel), zz, ss);
      o[4 * i + 1] = dq2(__byte_perm((x >> 2) & 0x03030303u, K, sel), zz, ss);
      o[4 * i + 2] = dq2(__byte_perm((x >> 4) & 0x03030303u, K, sel), zz, ss);
      o[4 * i + 3] = dq2(__byte_perm((x >> 6) & 0x03030303u, K, sel), zz, ss);
    }
  }
}
__device__ __forceinline__ void store_regs(uint32_t chunk_base, int row, const uint32_t (&o)[32]) {
#pragma unroll
  for (int i = 0; i < 8; ++i)
    sts_v4(chunk_base + swz_off(row, i, 128), o[4 * i], o[4 * i + 1], o[4 * i + 2], o[4 * i + 3]);
}
// Half h of a RoPE-key row (fetch_rope_half): o[0..15] from the 32 INT4 codes
// of f.a, the same arithmetic as dq_regs; stored as pieces 4 h .. 4 h + 3.
__device__ __forceinline__ void dq_half(uint32_t (&o)[32], const Fetch& f) {
  const __half2 sz = *reinterpret_cast<const __half2*>(&f.sz);
  const __half2 s2 = __half2half2(__low2half(sz));
  const __half2 zz2 = __half2half2(__hadd(__high2half(sz), __float2half_rn(1024.0f)));
  const uint32_t ss = *reinterpret_cast<const uint32_t*>(&s2);
  const uint32_t zz = *reinterpret_cast<const uint32_t*>(&zz2);
  constexpr uint32_t K = 0x64646464u;
  const uint32_t w[4] = {f.a.x, f.a.y, f.a.z, f.a.w};
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const uint32_t lo = w[i] & 0x0F0F0F0Fu;
    const uint32_t hi = (w[i] >> 4) & 0x0F0F0F0Fu;
    o[4 * i + 0] = dq2(__byte_perm(lo, K, 0x4140), zz, ss);
    o[4 * i + 1] = dq2(__byte_perm(hi, K, 0x4140), zz, ss);
    o[4 * i + 2] = dq2(__byte_perm(lo, K, 0x4342), zz, ss);
    o[4 * i + 3] = dq2(__byte_perm(hi, K, 0x4342), zz, ss);
  }
}
__device__ __forceinline__ void store_half(uint32_t chunk_base, int row, const uint32_t (&o)[32], int h) {
#pragma unroll
  for (int i = 0; i < 4; ++i)
    sts_v4(chunk_base + swz_off(row, 4 * h + i, 128), o[4 * i], o[4 * i + 1], o[4 * i + 2], o[4 * i + 3]);
}

// Rows of the paper's page. store_row_c4r4 writes one row (64 INT4 codes) of
// chunk k as RN_f16(s (q - z)) with the stored bf16 (content) or fp32 (RoPE)
// scale. q - z is exact in fp16 (as in store_row); a bf16 scale in [2^-14,
// 65504] is an fp16 value, so the fp16 product is the single rounding of the
// exact product. Any other scale (the fp32 RoPE scale, a tiny or huge content
// scale) multiplies in fp32 and rounds to fp16 after (store_row_c4r4_f32): one
// rounding for content, whose fp32 product is exact, and
// RN_f16(RN_f32(s (q - z))) for the RoPE key.
__device__ __forceinline__ void store_row_c4r4_f32(uint32_t chunk_base, int row, const uint4& a, const uint4& b,
                                                   float s, uint32_t zz) {
  constexpr uint32_t K = 0x64646464u;
  const uint32_t w[8] = {a.x, a.y, a.z, a.w, b.x, b.y, b.z, b.w};
  auto dqf = [&](uint32_t x) {
    uint32_t t;
    asm("sub.rn.f16x2 %0, %1, %2;" : "=r"(t) : "r"(x), "r"(zz));
    const float2 d = __half22float2(*reinterpret_cast<const __half2*>(&t));
    return pack_h2(d.x * s, d.y * s);
  };
#pragma unroll
  for (int i = 0; i < 8; ++i) {
    const uint32_t lo = w[i] & 0x0F0F0F0Fu;
    const uint32_t hi = (w[i] >> 4) & 0x0F0F0F0Fu;
    sts_v4(chunk_base + swz_off(row, i, 128), dqf(__byte_perm(lo, K, 0x4140)), dqf(__byte_perm(hi, K, 0x4140)),
           dqf(__byte_perm(lo, K, 0x4342)), dqf(__byte_perm(hi, K, 0x4342)));
  }
}

template <bool kContent>
__device__ __forceinline__ void store_row_c4r4(uint32_t chunk_base, int row, const Fetch& f) {
  if (!f.ok) {
#pragma unroll
    for (int i = 0; i < 8; ++i) sts_v4(chunk_base + swz_off(row, i, 128), 0, 0, 0, 0);
    return;
  }
  const float s = __uint_as_float(f.sz);
  const __half2 zz2 = __half2half2(__float2half_rn(1024.0f + static_cast<float>(f.z)));
  const uint32_t zz = *reinterpret_cast<const uint32_t*>(&zz2);
  if constexpr (!kContent) {
    store_row_c4r4_f32(chunk_base, row, f.a, f.b, s, zz);
  } else {
    const __half sh = __float2half_rn(s);
    if (__half2float(sh) != s) {  // only a content scale outside fp16's normal range
      store_row_c4r4_f32(chunk_base, row, f.a, f.b, s, zz);
      return;
    }
    const __half2 s2 = __half2half2(sh);
    const uint32_t ss = *reinterpret_cast<const uint32_t*>(&s2);
    constexpr uint32_t K = 0x64646464u;
    const uint32_t w[8] = {f.a.x, f.a.y, f.a.z, f.a.w, f.b.x, f.b.y, f.b.z, f.b.w};
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      const uint32_t lo = w[i] & 0x0F0F0F0Fu;
      const uint32_t hi = (w[i] >> 4) & 0x0F0F0F0Fu;
      sts_v4(chunk_base + swz_off(row, i, 128), dq2(__byte_perm(lo, K, 0x4140), zz, ss),
             dq2(__byte_perm(hi, K, 0x4140), zz, ss), dq2(__byte_perm(lo, K, 0x4342), zz, ss),
             dq2(__byte_perm(hi, K, 0x4342), zz, ss));
    }
  }
}

// The paper's page into registers (the decode workers compute a chunk row
// before its stores, as dq_regs does for this library's block): NW code words
// of f (8 for a row, 4 for half a RoPE row) into o[0 .. 4 NW). Same arithmetic
// as store_row_c4r4: fp16 subtract-and-multiply for a content row whose bf16
// scale is an fp16 value, else (the RoPE key, or a content scale outside
// fp16's normal range) the fp32 product rounded once to fp16.
template <int NW>
__device__ __forceinline__ void dq_regs_c4r4(uint32_t (&o)[32], const Fetch& f, bool content) {
  const float s = __uint_as_float(f.sz);
  const __half2 zz2 = __half2half2(__float2half_rn(1024.0f + static_cast<float>(f.z)));
  const uint32_t zz = *reinterpret_cast<const uint32_t*>(&zz2);
  constexpr uint32_t K = 0x64646464u;
  const uint32_t w[8] = {f.a.x, f.a.y, f.a.z, f.a.w, f.b.x, f.b.y, f.b.z, f.b.w};
  const __half sh = __float2half_rn(s);
  if (content && __half2float(sh) == s) {
    const __half2 s2 = __half2half2(sh);
    const uint32_t ss = *reinterpret_cast<const uint32_t*>(&s2);
#pragma unroll
    for (int i = 0; i < NW; ++i) {
      const uint32_t lo = w[i] & 0x0F0F0F0Fu;
      const uint32_t hi = (w[i] >> 4) & 0x0F0F0F0Fu;
      o[4 * i + 0] = dq2(__byte_perm(lo, K, 0x4140), zz, ss);
      o[4 * i + 1] = dq2(__byte_perm(hi, K, 0x4140), zz, ss);
      o[4 * i + 2] = dq2(__byte_perm(lo, K, 0x4342), zz, ss);
      o[4 * i + 3] = dq2(__byte_perm(hi, K, 0x4342), zz, ss);
    }
  } else {
    auto dqf = [&](uint32_t x) {
      uint32_t t;
      asm("sub.rn.f16x2 %0, %1, %2;" : "=r"(t) : "r"(x), "r"(zz));
      const float2 d = __half22float2(*reinterpret_cast<const __half2*>(&t));
      return pack_h2(d.x * s, d.y * s);
    };
#pragma unroll
    for (int i = 0; i < NW; ++i) {
      const uint32_t lo = w[i] & 0x0F0F0F0Fu;
      const uint32_t hi = (w[i] >> 4) & 0x0F0F0F0Fu;
      o[4 * i + 0] = dqf(__byte_perm(lo, K, 0x4140));
      o[4 * i + 1] = dqf(__byte_perm(hi, K, 0x4140));
      o[4 * i + 2] = dqf(__byte_perm(lo, K, 0x4342));
      o[4 * i + 3] = dqf(__byte_perm(hi, K, 0x4342));
    }
  }
}

// A protected row's chunk k: 64 bf16 values (8 x 16 bytes) rounded to fp16 and
// placed in the same within-piece channel order as the packed rows
// (bf16 -> fp16 is exact for magnitudes in [2^-14, 65504]).
template <int CB>
__device__ __forceinline__ void store_row_prot(uint32_t chunk_base, int row, const uint4 (&v)[8], int k) {
#pragma unroll
  for (int i = 0; i < 8; ++i) {
    const uint32_t w[4] = {v[i].x, v[i].y, v[i].z, v[i].w};
    float f[8];
#pragma unroll
    for (int e = 0; e < 4; ++e) {
      f[2 * e] = bf16_lo(w[e]);
      f[2 * e + 1] = bf16_hi(w[e]);
    }
    uint32_t o[4];
    if (k < 8) {
#pragma unroll
      for (int e = 0; e < 4; ++e) o[e] = pack_h2(f[Perm<CB>::at(2 * e)], f[Perm<CB>::at(2 * e + 1)]);
    } else {
#pragma unroll
      for (int e = 0; e < 4; ++e) o[e] = pack_h2(f[Perm<4>::at(2 * e)], f[Perm<4>::at(2 * e + 1)]);
    }
    sts_v4(chunk_base + swz_off(row, i, 128), o[0], o[1], o[2], o[3]);
  }
}

// BF16 comparison cache: the row is copied and rounded to fp16.
__device__ __forceinline__ void store_row_bf16(uint32_t chunk_base, int row, const uint4 (&v)[8], bool ok) {
#pragma unroll
  for (int i = 0; i < 8; ++i) {
    uint32_t o[4] = {0, 0, 0, 0};
    if (ok) {
      const uint32_t w[4] = {v[i].x, v[i].y, v[i].z, v[i].w};
#pragma unroll
      for (int e = 0; e < 4; ++e) o[e] = pack_h2(bf16_lo(w[e]), bf16_hi(w[e]));
    }
    sts_v4(chunk_base + swz_off(row, i, 128), o[0], o[1], o[2], o[3]);
  }
}

// One row's chunk k of a packed cache (this library's block or the paper's
// page) as dq_row would store it (the eight 16-byte pieces in order),
// computed into registers: the protected bf16 row when ps is set, else the
// packed row f. The decode workers compute it ahead of its stores.
template <int CB, bool PROT>
__device__ __forceinline__ void row_regs(uint32_t (&o)[32], const Fetch& f, int k, const uint8_t* ps) {
  if (PROT && ps != nullptr) {
    uint4 pv[8];
#pragma unroll
    for (int i = 0; i < 8; ++i) pv[i] = __ldg(reinterpret_cast<const uint4*>(ps + k * 128) + i);
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      const uint32_t w[4] = {pv[i].x, pv[i].y, pv[i].z, pv[i].w};
      float v[8];
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        v[2 * e] = bf16_lo(w[e]);
        v[2 * e + 1] = bf16_hi(w[e]);
      }
      if (k < 8) {
#pragma unroll
        for (int e = 0; e < 4; ++e) o[4 * i + e] = pack_h2(v[Perm<CB>::at(2 * e)], v[Perm<CB>::at(2 * e + 1)]);
      } else {
#pragma unroll
        for (int e = 0; e < 4; ++e) o[4 * i + e] = pack_h2(v[Perm<4>::at(2 * e)], v[Perm<4>::at(2 * e + 1)]);
      }
    }
  } else if constexpr (CB == kC4R4) {
    dq_regs_c4r4<8>(o, f, k < 8);
  } else {
    dq_regs(o, f, CB == 4 || k == 8);
  }
  // Pin the results here: the (volatile) slot wait that follows must not be
  // hoisted above the arithmetic.
#pragma unroll
  for (int i = 0; i < 32; ++i) asm volatile("" : "+r"(o[i]));
}
// Half h of a RoPE-key row into o[0..15] (pieces 4 h .. 4 h + 3): the
// protection row's bf16 channels 32 h .. 32 h + 31 rounded to fp16 when the
// row is protected, else dq_half of the packed codes.
template <int CB, bool PROT>
__device__ __forceinline__ void row_regs_half(uint32_t (&o)[32], const Fetch& f, const uint8_t* ps, int h) {
  if (PROT && ps != nullptr) {
    uint4 pv[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) pv[i] = __ldg(reinterpret_cast<const uint4*>(ps + 8 * 128 + h * 64) + i);
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const uint32_t w[4] = {pv[i].x, pv[i].y, pv[i].z, pv[i].w};
      float v[8];
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        v[2 * e] = bf16_lo(w[e]);
        v[2 * e + 1] = bf16_hi(w[e]);
      }
#pragma unroll
      for (int e = 0; e < 4; ++e) o[4 * i + e] = pack_h2(v[Perm<4>::at(2 * e)], v[Perm<4>::at(2 * e + 1)]);
    }
  } else if constexpr (CB == kC4R4) {
    dq_regs_c4r4<4>(o, f, false);
  } else {
    dq_half(o, f);
  }
#pragma unroll
  for (int i = 0; i < 16; ++i) asm volatile("" : "+r"(o[i]));
}

// BF16 cache rows read coalesced: lane l of a warp handles piece l & 7 (16
// bytes) of rows r0 + 4 i + (l >> 3), i = 0..7, so every load instruction
// reads four whole 128-byte lines (32 rows x one chunk per warp). r0 is the
// warp's first row (its rows share a block, slots slot0 ..); vmask bit m is
// set when row r0 + m is to be read (else zeros).
__device__ __forceinline__ void bf16_load_t(uint4 (&v)[8], const uint8_t* blk, uint32_t vmask, int slot0, int k,
                                            int lane) {
#pragma unroll
  for (int i = 0; i < 8; ++i) {
    const int m = 4 * i + (lane >> 3);
    v[i] = (vmask >> m) & 1u ? ldg_nc_v4(blk + (slot0 + m) * (kDqk * 2) + k * 128 + (lane & 7) * 16)
                             : make_uint4(0, 0, 0, 0);
  }
}
// Writes those pieces rounded to fp16 into the swizzled chunk.
__device__ __forceinline__ void bf16_store_t(uint32_t chunk_base, int r0, const uint4 (&v)[8], int lane) {
#pragma unroll
  for (int i = 0; i < 8; ++i) {
    const int m = 4 * i + (lane >> 3);
    const uint32_t w[4] = {v[i].x, v[i].y, v[i].z, v[i].w};
    uint32_t o[4];
#pragma unroll
    for (int e = 0; e < 4; ++e) o[e] = pack_h2(bf16_lo(w[e]), bf16_hi(w[e]));
    sts_v4(chunk_base + swz_off(r0 + m, lane & 7, 128), o[0], o[1], o[2], o[3]);
  }
}

__device__ __forceinline__ float ex2_approx(float x) {
  float y;
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}

// The CTA whose range holds tile t (CTA c's range starts at c * T / grid).
__device__ __forceinline__ int cta_of(int t, int T, int grid) {
  return static_cast<int>((static_cast<long long>(t + 1) * grid - 1) / T);
}

// First tile of the reference range that tile j of 64-row group r lies in, in a unit of
// two such groups with tiles [pu0, pu1) of a list of T: ranges of the 64-row plan, 2 T /
// SMs tiles each, cut at unit ends (see decode_pair.cu).
__device__ __forceinline__ int ref_start(int r, int j, int pu0, int pu1, int T, int sms) {
  const int base = 2 * pu0 + r * (pu1 - pu0);
  const int c = cta_of(base + j, 2 * T, sms);
  return max(static_cast<int>(static_cast<long long>(c) * 2 * T / sms) - base, 0);
}

// Launches kern on stream; with pdl the launch may overlap the previous kernel
// in the stream (programmatic stream serialisation), which kern must wait for
// with griddep_wait before reading its results.
template <typename... Args>
cudaError_t launch_k(void (*kern)(Args...), dim3 grid, dim3 block, size_t smem, cudaStream_t stream, bool pdl,
                     Args... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = block;
  cfg.dynamicSmemBytes = smem;
  cfg.stream = stream;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = pdl ? 1 : 0;
  return cudaLaunchKernelEx(&cfg, kern, args...);
}

}  // namespace
}  // namespace qmla
