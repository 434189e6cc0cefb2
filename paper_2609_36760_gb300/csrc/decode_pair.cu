// Split-KV MLA decode for more than 64 query rows per sequence: a cluster of two
// CTAs handles a unit of 128 rows, 64 per CTA, with tcgen05 cta_group::2.
//
// Each tile is one 64-token cache block. As M = 128 MMAs over the pair,
//   S[h, t] = q[h, :] . C_hat[t, :]   A: each CTA's 64 rows of q, B: each CTA's 32
//                                     tokens (N = 64), K = 576,
//   O[h, c] += P[h, :] C_hat[:, c]    A: each CTA's 64 rows of P, B: each CTA's 256
//                                     channels (2 x N = 256), K = 64 tokens,
// so a CTA dequantises 32 tokens x 576 channels for the scores and, of the other
// CTA's 32 tokens, only its own 256 channels for the values: 832 instead of 1,152
// row-chunks of 64 channels per 64 tokens and 128 rows. Both operands of a tile
// and its scores are double-buffered, and separate warps dequantise, do the
// softmax and issue the MMAs, so that the tiles' phases overlap.
//
// Per 128 tokens and 64 rows decode_main's MMAs read 3,390 and its workers write 1,370
// wavefronts of 128 bytes of shared memory, one phase after the other; here the MMAs read
// 2,590 and the warps write 1,430, the reference tiles' among them, beside the softmax
// (ncu, the INT4 step below). Of 3.35k cycles per 64-token tile the tensor pipe then is
// active in 33% and the shared-memory port busy in 65%; the rest is the softmax warps'
// turn, mostly waits on shared memory and TMEM behind the other warps' bursts. One GB300, a
// decode step of 64 sequences x 128 heads x 4,097 tokens, decode_main / this: INT4 129.0 /
// 116.5 us, the paper's page with protection 174.2 / 136.8, BF16 237.4 / 165.1; INT2, 32 x
// 32,768 tokens: 395.5 / 363.
// (A second softmax group, one per alternate tile, was slower: 152 us on the INT4 step,
// its warps' extra waits and registers cost more than their overlap gave.)
//
// TMEM (per CTA, lanes 0..63 hold the first half of N for rows 0..63, lanes
// 64..127 the second): O 2 x 128 columns, S 4 buffers x 2 partials x 32 columns.
#include <cuda_runtime.h>

#include <cstddef>

#include "decode_common.cuh"

namespace qmla {
namespace {

constexpr int kPairTok = 64;       // tokens per tile: one cache block
constexpr int kSoftWarps = 4;      // warps 0..3, one per TMEM lane quarter
constexpr int kDqWarps = 13;       // warps 4..16, one 64-channel chunk of 32 tokens each
constexpr int kMmaWarp = kSoftWarps + kDqWarps;   // MMA issuer (leader), query loads (the other CTA)
constexpr int kPrefetchWarp = kMmaWarp + 1;       // L2 prefetch (the other CTA)
constexpr int kPairThreads = (kPrefetchWarp + 2) * 32;  // whole warpgroups (the last warp idles)
// Registers per thread after the launch's 96: the softmax warpgroup holds a row's
// scores and weights, the others give theirs up (4 x 8 = 32 per thread).
constexpr int kSoftRegs = 128, kOtherRegs = 88;
static_assert(kSoftRegs + 4 * kOtherRegs <= 5 * 96, "register split");
constexpr uint32_t kRows = 64;                           // query rows per CTA
constexpr uint32_t kQImg = kNumChunks * kRows * 128;     // query image
constexpr uint32_t kKChunk = 32 * 128, kKStage = kNumChunks * kKChunk;  // own tokens, K-major B of QK
constexpr uint32_t kVChunk = kPairTok * 128, kVStage = 4 * kVChunk;     // own channels, MN-major B of PV
constexpr uint32_t kPTile = kRows * 128;                 // P, K-major A of PV
constexpr uint32_t kKOff = kQImg, kVOff = kKOff + 2 * kKStage, kPOff = kVOff + 2 * kVStage;
constexpr uint32_t kCtrlOff = kPOff + 2 * kPTile;
constexpr uint32_t kColS = 256, kTmemPair = 512;
constexpr int kPrefetchTiles = 5;  // how far the L2 prefetch runs ahead

struct __align__(16) PairCtrl {
  // Waited on by the leader's issuers, arrived on by warps of both CTAs.
  uint64_t k_full[2], v_full[2];   // operand stage written (9 and 8 warps per CTA)
  uint64_t p_full[2], s_free[4];   // P written, S no longer needed (4 softmax warps per CTA)
  uint64_t p_fixed[2];             // CTA r rewrote P against a raised reference
  uint64_t o_free, q_peer;         // O read at a segment end; the other CTA's query is loaded
  // Arrived on by MMA commits, multicast to both CTAs.
  uint64_t s_full[4], k_free[2];   // scores complete; K stage free
  uint64_t pv_done[2];             // PV complete: V stage and P free
  uint64_t q_free;                 // every QK of a segment has completed
  uint64_t q_bar, fin;             // query copy (transaction count); end of the issuers
  uint64_t grp;                    // softmax warps among themselves
  uint32_t tmem_base, abort;
  uint32_t over[2];                // [v & 1] = v + 1 when real tile v has a weight above 2^8
  uint32_t raised[2][2];           // leader: the same for CTA [r]
  uint32_t progress;               // tile being dequantised, for the prefetch
  float xch[2][128];               // row values exchanged between the two halves of a row
};
constexpr int kPairSmem = 1024 + kCtrlOff + static_cast<int>(sizeof(PairCtrl));
static_assert(kPairSmem <= 232448, "shared memory per CTA");

// The tiles of one pair, in the order every role walks them: first the tiles
// that only give a softmax reference (see the softmax role), then the range, cut
// into segments at unit ends. Tile q is 64-token block q of a sequence.
struct PairSched {
  int q, qend;        // current tile, end of its run (segment or reference tile)
  int q0;             // first tile of the segment
  int unit, pu0, pu1; // unit and its 128-token tiles in the plan's list
  int b, g, len;
  int t0, t1;         // range in the plan's list
  int ref_next;       // second reference tile (128-token index), or -1
  bool ref, live;
  __device__ void enter_unit(const Params& p) {
    b = unit / p.n_hg;
    g = unit - b * p.n_hg;
    len = p.seq_lens[b];
  }
  __device__ int blocks() const { return (len + kPairTok - 1) / kPairTok; }
  __device__ void enter_segment(int j) {
    q = q0 = 2 * j;
    qend = min(2 * (min(t1, pu1) - pu0), blocks());
  }
  __device__ void init(const Params& p, int pair) {
    const int4 info = p.cta_info[pair], first = p.cta_first[pair];  // (see pair_start)
    t0 = p.cta_t0[pair];
    t1 = p.cta_t0[pair + 1];
    unit = info.x;
    pu0 = info.y;
    pu1 = info.z;
    b = unit / p.n_hg;
    g = unit - b * p.n_hg;
    len = first.z;
    ref_next = -1;
    ref = false;
    live = t0 < t1;
    q = qend = q0 = 0;
    if (!live) return;
    const int j0 = t0 - pu0, r0 = first.x, r1 = first.y;
    enter_segment(j0);
    if (r0 < j0 || r1 < j0) {
      ref = true;
      if (r0 < j0 && r1 < j0 && r0 != r1) ref_next = r1;
      q = 2 * (r0 < j0 ? r0 : r1);
      qend = min(q + 2, blocks());
    }
  }
  __device__ bool seg_first() const { return !ref && q == q0; }
  __device__ bool seg_last() const { return !ref && q + 1 == qend; }
  __device__ void next(const Params& p) {
    if (++q < qend) return;
    if (ref) {
      if (ref_next >= 0) {
        q = 2 * ref_next;
        qend = min(q + 2, blocks());
        ref_next = -1;
      } else {
        ref = false;
        enter_segment(t0 - pu0);
      }
      return;
    }
    const int t = min(t1, pu1);
    if (t >= t1) {
      live = false;
      return;
    }
    const int units = p.batch * p.n_hg;
    while (t >= pu1 && unit + 1 < units) {
      ++unit;
      pu0 = pu1;
      pu1 = p.prefix[unit + 1];
    }
    enter_unit(p);
    enter_segment(0);
  }
};

__device__ __forceinline__ int block_entry(const Params& p, const PairSched& sc) {
  return sc.live ? p.table[static_cast<size_t>(sc.b) * p.max_blocks + sc.q] : -1;
}

// A warp's arrival on a barrier of the leader (what the lanes did comes before a
// __syncwarp). Operands need no release to the other CTA: the tensor core of the SM that
// wrote them reads them, through the async proxy that fence_proxy_async_smem has ordered
// them for, and TMEM accesses are ordered by the tcgen05 fences. What the issuer itself
// reads (the mark of a raise), or what a rewrite depends on, is released to the cluster
// and acquired by the issuer's probe (arrive_leader_cluster, mbar_test_cluster). With
// that release in every arrival the INT4 step of 64 x 4,097 tokens takes 153 instead of
// 112 us.
__device__ __forceinline__ void arrive_leader(int lane, uint32_t bar_addr) { mbar_arrive_remote(bar_addr, lane == 0); }
__device__ __forceinline__ void arrive_leader_cluster(int lane, uint32_t bar_addr) {
  mbar_arrive_cluster(bar_addr, lane == 0);
}

// ------------------------------------------------------------ dequantisation
// Warp d: chunk d of the CTA's own 32 tokens (d < 9; the content chunks of the
// CTA's own channels go to the V stage too), or chunk 4 rank + d - 9 of the
// other CTA's 32 tokens for the V stage. One row per lane; the next tile's row
// is fetched as soon as this one's registers are free.
template <int CB, bool PROT>
__device__ void pair_dequant(const Params& p, PairSched sc, uint32_t smem, PairCtrl& ctl, int rank, int d, int lane) {
  const bool own = d < kNumChunks;
  const int k = own ? d : 4 * rank + d - kNumChunks;
  const int row = 32 * (own ? rank : 1 - rank) + lane;  // slot of the token in its block
  const bool to_v = !own || (k < 8 && (k >> 2) == rank);
  const uint32_t kdst = smem + kKOff + k * kKChunk;
  const uint32_t vdst = smem + kVOff + (k & 3) * kVChunk;
  const uint32_t kfull = cluster_map(smem_u32(&ctl.k_full[0]), 0), vfull = cluster_map(smem_u32(&ctl.v_full[0]), 0);
  uint32_t n = 0, v = 0;
  bool ok = true;
  // sc stands at the tile to be fetched next, whose block-table entry is loaded
  // an iteration ahead.
  bool live = sc.live, ref = sc.ref;
  int entry = block_entry(p, sc);
  Fetch f;
  uint4 raw[CB == 16 ? 8 : 1];
  const uint8_t* ps = nullptr;
  constexpr size_t kBlk = CB == 16 ? static_cast<size_t>(kBf16BlockBytes) : BlockLayout<CB == 16 ? 4 : CB>::kBytes;
  auto fetch = [&]() {
    // (a reference tile has no PV; a row past the sequence end is zero)
    bool valid = sc.live && (own || !sc.ref) && row < sc.len - kPairTok * sc.q;
    ps = nullptr;
    if constexpr (PROT) {
      RowRef r;
      r.has = valid;
      r.j = sc.q >> 1;
      r.len = sc.len;
      r.b = sc.b;
      ps = prot_row(p, r, (sc.q & 1) * kPairTok + row);
      if (ps != nullptr) valid = false;
    }
    if (valid && (entry < 0 || entry >= p.num_blocks)) {
      report(p.dev_err, QMLA_DEVERR_BAD_BLOCK);
      valid = false;
    }
    const uint8_t* blk = p.pool + static_cast<size_t>(entry) * kBlk;
    if constexpr (CB == 16) {
      bf16_load_t(raw, blk, __ballot_sync(0xffffffffu, valid), row & ~31, k, lane);
    } else {
      f = fetch_chunk<CB>(blk, valid, k, row);
    }
    if (sc.live) sc.next(p);
    entry = block_entry(p, sc);
  };
  fetch();
  while (ok && live) {
    const bool real = !ref;
    uint32_t o[32];
    const bool work = own || real;
    if (work) {
      if constexpr (CB == 16) {
#pragma unroll
        for (int i = 0; i < 8; ++i) {
          const uint32_t w[4] = {raw[i].x, raw[i].y, raw[i].z, raw[i].w};
#pragma unroll
          for (int e = 0; e < 4; ++e) o[4 * i + e] = pack_h2(bf16_lo(w[e]), bf16_hi(w[e]));
        }
      } else {
        row_regs<CB, PROT>(o, f, k, ps);
      }
    }
    if (d == 8 && lane == 0) *reinterpret_cast<volatile uint32_t*>(&ctl.progress) = n;
    live = sc.live;
    ref = sc.ref;
    fetch();
    auto store = [&](uint32_t base, int row0) {
#pragma unroll
      for (int i = 0; i < 8; ++i) {
        const uint32_t at = CB == 16 ? swz_off(row0 + 4 * i + (lane >> 3), lane & 7, 128)
                                     : swz_off(row0 + lane, i, 128);
        sts_v4(base + at, o[4 * i], o[4 * i + 1], o[4 * i + 2], o[4 * i + 3]);
      }
      fence_proxy_async_smem();
      __syncwarp();
    };
    if (own) {
      const uint32_t st = n & 1u;
      if (n >= 2 && !(ok = wwait(&ctl.k_free[st], ((n >> 1) - 1) & 1u, ctl, kSiteDqSlot, p.dev_err))) break;
      store(kdst + st * kKStage, 0);
      arrive_leader(lane, kfull + st * 8);
    }
    if (to_v && real) {
      const uint32_t st = v & 1u;
      if (v >= 2 && !(ok = wwait(&ctl.pv_done[st], ((v >> 1) - 1) & 1u, ctl, kSiteDqSlot, p.dev_err))) break;
      store(vdst + st * kVStage, row & 32);
      arrive_leader(lane, vfull + st * 8);
    }
    ++n;
    if (real) ++v;
  }
  if (!ok && lane == 0) set_abort(ctl, p.dev_err);
}

// ------------------------------------------------------------------- softmax
// lo += w.lo, hi += w.hi with w a pair of fp16 values.
__device__ __forceinline__ void add_h2(float& lo, float& hi, uint32_t w) {
  asm("{\n\t.reg .b16 l, h;\n\tmov.b32 {l, h}, %2;\n\tadd.rn.f32.f16 %0, l, %0;\n\tadd.rn.f32.f16 %1, h, %1;\n\t}"
      : "+f"(lo), "+f"(hi)
      : "r"(w));
}

// 32 columns of this thread's row of S (tokens 32 half .. 32 half + 31), in pairs:
// the sum of the two partials.
__device__ __forceinline__ void load_scores(uint32_t t_s, uint64_t (&x)[16]) {
  uint32_t a[32], b[32];
  tmem_ld32(t_s, a);
  tmem_ld32(t_s + 32, b);
  tmem_ld_wait();
#pragma unroll
  for (int i = 0; i < 16; ++i)
    x[i] = add2(f32x2(__uint_as_float(a[2 * i]), __uint_as_float(a[2 * i + 1])),
                f32x2(__uint_as_float(b[2 * i]), __uint_as_float(b[2 * i + 1])));
}
// Largest scaled score among the row's first `vis` of 32 columns (-inf if none).
__device__ __forceinline__ float scores_max(const uint64_t (&x)[16], float sl2, int vis) {
  float m = -INFINITY;
#pragma unroll
  for (int i = 0; i < 16; ++i) {
    m = fmaxf(m, 2 * i < vis ? __fmul_rn(lo2(x[i]), sl2) : -INFINITY);
    m = fmaxf(m, 2 * i + 1 < vis ? __fmul_rn(hi2(x[i]), sl2) : -INFINITY);
  }
  return m;
}

// The same straight from TMEM, a few columns at a time.
__device__ __forceinline__ float tmem_scores_max(uint32_t t_s, float sl2, int vis) {
  float m = -INFINITY;
#pragma unroll 1
  for (int c = 0; c < 32; c += 8) {
    uint32_t a[8], b[8];
    tmem_ld8(t_s + c, a);
    tmem_ld8(t_s + 32 + c, b);
    tmem_ld_wait();
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      const float x = __uint_as_float(a[i]) + __uint_as_float(b[i]);
      m = fmaxf(m, c + i < vis ? __fmul_rn(x, sl2) : -INFINITY);
    }
  }
  return m;
}

// Thread (row, half): query row `row` of the CTA and half the tokens of a tile;
// in O, half the channels. The weights are P = 2^(S scale log2e - m) with a
// reference m per row. The reference is renewed, as the maximum over a 128-token
// tile, at the first tile of every range of the 64-row plan (total / SMs tiles,
// cut at unit ends), wherever this pair's own range begins: the fp16 rounding
// of P depends on m, so the results then do not depend on which kernel or how
// many CTAs share a sequence. A pair whose range begins inside such a reference
// range first scores that range's first tile for its maximum (PairSched's
// reference tiles). A weight above 2^8 raises the reference in between.
template <int CB>
__device__ void pair_softmax(const Params& p, PairSched sc, uint32_t smem, PairCtrl& ctl, uint32_t tmem, int rank,
                             int warp, int lane, int pair) {
  const int half = warp >> 1, row = (warp & 1) * 32 + lane;
  const uint32_t lanes = static_cast<uint32_t>(warp * 32) << 16;
  const uint32_t t_o = tmem + lanes;
  const float sl2 = p.scale_log2;
  const uint32_t sfree = cluster_map(smem_u32(&ctl.s_free[0]), 0), pfull = cluster_map(smem_u32(&ctl.p_full[0]), 0);
  const uint32_t pfixed = cluster_map(smem_u32(&ctl.p_fixed[rank]), 0);
  const uint32_t ofree = cluster_map(smem_u32(&ctl.o_free), 0);
  uint32_t n = 0, v = 0, gph = 0, xbuf = 0, seg_v = 0;
  bool ok = true, whole = false;
  float m = -INFINITY, m_run = -INFINITY, l = 0.0f;
  int vis_end = 0;    // positions this row sees
  int next_ref = 0;   // tile j at which the next reference range begins
  int my_ref = -1;    // reference tile of this CTA's row group
  if (sc.live) {
    const int4 first = p.cta_first[pair];
    my_ref = rank == 0 ? first.x : first.y;
  }

  // The other half's value of a per-row quantity.
  auto exchange = [&](float mine, float& other) {
    ctl.xch[xbuf][half * 64 + row] = mine;
    ok = group_sync(ctl, gph, p.dev_err);
    other = ctl.xch[xbuf][(1 - half) * 64 + row];
    xbuf ^= 1u;
    return ok;
  };
  auto row_setup = [&]() {
    const int vh = (sc.g * 2 + rank) * static_cast<int>(kRows) + row;
    vis_end = min(sc.len, sc.len - p.q_tokens + vh / p.hpt + 1);
  };
  auto wait_s = [&](uint32_t i) {
    ok = wwait(&ctl.s_full[i & 3u], (i >> 2) & 1u, ctl, kSiteSmSFull, p.dev_err);
    tc_fence_after();
    return ok;
  };
  auto t_s = [&](uint32_t i) { return tmem + kColS + (i & 3u) * 64 + lanes; };
  auto release_s = [&](uint32_t i) {
    tc_fence_before();
    __syncwarp();
    arrive_leader(lane, sfree + (i & 3u) * 8);
  };
  // Moves the reference to mn before real tile i is accumulated: scales what O
  // and l hold by 2^(m - mn).
  auto move_ref = [&](float mn, uint32_t i) {
    const float a = m == mn || m == -INFINITY ? 1.0f : exp2f(m - mn);
    m = mn;
    m_run = fmaxf(m_run, mn);
    l *= a;
    if (i == seg_v) return true;  // O holds nothing yet
    if (!(ok = wwait(&ctl.pv_done[(i - 1) & 1u], ((i - 1) >> 1) & 1u, ctl, kSitePvEpi, p.dev_err))) return false;
    tc_fence_after();
    if (__any_sync(0xffffffffu, a != 1.0f)) {
#pragma unroll 1
      for (int c = 0; c < 256; c += 32) {
        uint32_t r[32];
        tmem_ld32(t_o + c, r);
        tmem_ld_wait();
#pragma unroll
        for (int e = 0; e < 32; ++e) r[e] = __float_as_uint(__uint_as_float(r[e]) * a);
        tmem_st32(t_o + c, r);
      }
      tmem_st_wait();
    }
    return true;
  };

  // The current real tile: scaled weights P = 2^(S scale log2e - m) in fp16 into pk.
  uint64_t x[16];
  uint32_t pk[16];
  int vis = 0;
  bool full = true;
  auto weights = [&]() {  // whether a weight is above 2^8 (as rounded)
    const uint64_t ss = f32x2(sl2, sl2);
    const uint64_t nm = f32x2(-m, -m);
    __half2 top = __float2half2_rn(0.0f);
#pragma unroll
    for (int i = 0; i < 16; ++i) {
      const uint64_t y = fma2(x[i], ss, nm);
      float y0 = lo2(y), y1 = hi2(y);
      if (!full) {
        y0 = 2 * i < vis ? y0 : -INFINITY;
        y1 = 2 * i + 1 < vis ? y1 : -INFINITY;
      }
      pk[i] = pack_h2(ex2_approx(y0), ex2_approx(y1));
      top = __hmax2(top, *reinterpret_cast<const __half2*>(&pk[i]));
    }
    return __hgt(__hmax(__low2half(top), __high2half(top)), __float2half_rn(256.0f));
  };
  auto store_p = [&](uint32_t st) {
    const uint32_t ptile = smem + kPOff + st * kPTile;
#pragma unroll
    for (int i = 0; i < 4; ++i)
      sts_v4(ptile + swz_off(row, half * 4 + i, 128), pk[4 * i], pk[4 * i + 1], pk[4 * i + 2], pk[4 * i + 3]);
    fence_proxy_async_smem();
    tc_fence_before();
    __syncwarp();
  };
  auto weight_sum = [&]() {
    float s[4] = {0.0f, 0.0f, 0.0f, 0.0f};
#pragma unroll
    for (int i = 0; i < 16; ++i) add_h2(s[2 * (i & 1)], s[2 * (i & 1) + 1], pk[i]);
    return (s[0] + s[1]) + (s[2] + s[3]);
  };
  // Settles the last tile (real tile v - 1, n - 1 among all) once every warp has given
  // its P: where one of them had a weight above 2^8, the reference is raised and P
  // rewritten (PV waits for p_fixed). Done at the next tile, so that nobody
  // waits for the other warps; until then its scores stay. The raised reference covers
  // the whole 128-token tile, as a renewed one does: an even block takes in the odd one
  // behind it (`next`: its scores are in the following buffer), an odd one the even one
  // before it, whose scores are therefore released with the odd one's.
  bool due = false;
  int vis_due = 0;
  float l_due = 0.0f;
  auto settle = [&](bool odd, bool next) {
    due = false;
    if (!(ok = wwait(&ctl.grp, gph & 1u, ctl, kSiteGrp, p.dev_err))) return false;
    ++gph;
    const uint32_t st = (v - 1) & 1u;
    if (*reinterpret_cast<volatile uint32_t*>(&ctl.over[st]) == v) {
      float mx = tmem_scores_max(t_s(n - 1), sl2, vis_due);
      if (odd || next)
        mx = fmaxf(mx, tmem_scores_max(t_s(odd ? n - 2 : n), sl2, odd ? vis_due + kPairTok : vis_due - kPairTok));
      float mo = 0.0f;
      if (!exchange(mx, mo)) return false;
      if (!move_ref(fmaxf(m, fmaxf(mx, mo)), v - 1)) return false;
      float l0 = 0.0f, l1 = 0.0f;
#pragma unroll 1
      for (int c = 0; c < 32; c += 8) {
        uint32_t a[8], b[8], w[4];
        tmem_ld8(t_s(n - 1) + c, a);
        tmem_ld8(t_s(n - 1) + 32 + c, b);
        tmem_ld_wait();
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          const float y0 = __fmaf_rn(__uint_as_float(a[2 * i]) + __uint_as_float(b[2 * i]), sl2, -m);
          const float y1 = __fmaf_rn(__uint_as_float(a[2 * i + 1]) + __uint_as_float(b[2 * i + 1]), sl2, -m);
          w[i] = pack_h2(c + 2 * i < vis_due ? ex2_approx(y0) : 0.0f, c + 2 * i + 1 < vis_due ? ex2_approx(y1) : 0.0f);
          add_h2(l0, l1, w[i]);
        }
        sts_v4(smem + kPOff + st * kPTile + swz_off(row, half * 4 + c / 8, 128), w[0], w[1], w[2], w[3]);
      }
      l_due = l0 + l1;
      fence_proxy_async_smem();
      tc_fence_before();
      __syncwarp();
      arrive_leader_cluster(lane, pfixed);
    }
    if (odd) release_s(n - 2);
    if (!next) release_s(n - 1);
    l += l_due;
    return true;
  };

  for (; ok && sc.live; sc.next(p)) {
    const int j = sc.q >> 1;
    const bool even = (sc.q & 1) == 0;
    if (n == 0) row_setup();
    if (sc.ref) {
      // Only the maximum of this tile is wanted, by the CTA whose range it starts.
      if (!wait_s(n)) break;
      if (j == my_ref) {
        const float mx = tmem_scores_max(t_s(n), sl2, vis_end - (kPairTok * sc.q + 32 * half));
        m = even ? mx : fmaxf(m, mx);
      }
      release_s(n);
      if (sc.q + 1 == sc.qend && j == my_ref) {
        float mo = 0.0f;
        if (!exchange(m, mo)) break;
        m = fmaxf(m, mo);
      }
      ++n;
      continue;
    }
    const bool first = sc.seg_first();
    bool renew = false;
    if (even) {
      if (first) {
        row_setup();
        l = 0.0f;
        seg_v = v;
        whole = sc.q == 0;
        next_ref = j > 0 ? my_ref : 0;  // (only the range's first segment starts inside a unit)
        if (next_ref < j) {
          // (m came from the reference tile)
          m_run = m;
        } else {
          m = m_run = -INFINITY;
        }
        renew = next_ref == j;
      } else {
        renew = j >= next_ref;
      }
      if (first || renew) {
        // start of the reference range after the one tile j lies in
        const int total = 2 * p.prefix[p.batch * p.n_hg];
        const int base = 2 * sc.pu0 + rank * (sc.pu1 - sc.pu0);
        const int c = cta_of(base + j, total, p.sms);
        next_ref = static_cast<int>(static_cast<long long>(c + 1) * total / p.sms) - base;
      }
    }
    if (!wait_s(n)) break;
    load_scores(t_s(n), x);
    if (due && !settle(even, !even)) break;
    vis = vis_end - (kPairTok * sc.q + 32 * half);
    if (renew) {
      float mx = scores_max(x, sl2, vis);
      if (sc.q + 1 < sc.qend) {  // the 128-token tile's second block, whose own turn comes next
        if (!wait_s(n + 1)) break;
        mx = fmaxf(mx, tmem_scores_max(t_s(n + 1), sl2, vis - kPairTok));
      }
      float mo = 0.0f;
      if (!exchange(mx, mo)) break;
      mx = fmaxf(mx, mo);
      // (kept when no key of the tile is seen, and never far below an earlier
      // reference, whose terms then carry the sum: 2^(m - mx) stays finite)
      if (!move_ref(mx == -INFINITY ? m : fmaxf(mx, m_run - 60.0f), v)) break;
    }
    full = __all_sync(0xffffffffu, vis >= 32);
    const bool over = __any_sync(0xffffffffu, weights());
    const uint32_t st = v & 1u;
    store_p(st);
    // A weight above 2^8 in any of the CTA's rows raises every row's reference (see
    // settle): the mark is written before the arrivals, so who has seen all of them
    // reads it.
    if (over) {
      if (lane == 0) {
        *reinterpret_cast<volatile uint32_t*>(&ctl.over[st]) = v + 1;
        st_cluster_u32(cluster_map(smem_u32(&ctl.raised[rank][st]), 0), v + 1);
      }
      arrive_leader_cluster(lane, pfull + st * 8);
    } else {
      arrive_leader(lane, pfull + st * 8);
    }
    mbar_arrive_if(lane == 0 ? 1u : 0u, &ctl.grp);
    l_due = weight_sum();
    due = true;
    vis_due = vis;
    ++n;
    ++v;
    if (!sc.seg_last()) continue;

    // ---- segment end: out = O / l, or the partial (m, l, o)
    if (due && !settle(!even, false)) break;
    whole = whole && sc.t1 >= sc.pu1;
    float lo = 0.0f;
    if (!exchange(l, lo)) break;
    const float lt = half == 0 ? l + lo : lo + l;
    const float inv = whole ? (lt > 0.0f ? 1.0f / lt : 0.0f) : 1.0f;
    if (!(ok = wwait(&ctl.pv_done[(v - 1) & 1u], ((v - 1) >> 1) & 1u, ctl, kSitePvEpi, p.dev_err))) break;
    tc_fence_after();
    // Through the P tiles (free until the next tile's weights), 32 columns at a time, so
    // that a warp stores whole 128-byte lines: a row per lane would touch 32 lines with
    // every store, 8k cycles a segment instead of about 2k.
    // (A warp's piece of them lies under other warps' weights. Those of the next segment
    // do not come before every warp is done: a segment that follows another starts its
    // unit, so its first tile renews the reference, with an exchange of all four warps.)
    const int h0 = (sc.g * 2 + rank) * static_cast<int>(kRows) + (warp & 1) * 32;  // the warp's first row
    const size_t orow0 = whole ? static_cast<size_t>(sc.b) * p.heads + h0
                               : (static_cast<size_t>(pair) + sc.unit) * 128 + rank * kRows + (warp & 1) * 32;
    float* const dst = (whole ? p.out : p.part_o) + orow0 * kDc + half * 256 + (lane & 7) * 4;
    const int rows = whole ? p.heads - h0 : 32;
    const uint32_t buf = smem + kPOff + warp * 4096;
#pragma unroll 1
    for (int c = 0; c < 256; c += 32) {
      uint32_t r[32];
      tmem_ld32(t_o + c, r);
      tmem_ld_wait();
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        uint32_t w[8];
#pragma unroll
        for (int e = 0; e < 8; ++e) w[Perm<CB>::at(e)] = __float_as_uint(__uint_as_float(r[8 * q + e]) * inv);
        sts_v4(buf + swz_off(lane, 2 * q, 128), w[0], w[1], w[2], w[3]);
        sts_v4(buf + swz_off(lane, 2 * q + 1, 128), w[4], w[5], w[6], w[7]);
      }
      __syncwarp();
#pragma unroll
      for (int i = 0; i < 8; ++i) {
        const int rr = 4 * i + (lane >> 3);
        const uint4 o = lds_v4(buf + swz_off(rr, lane & 7, 128));
        if (rr < rows) *reinterpret_cast<uint4*>(dst + static_cast<size_t>(rr) * kDc + c) = o;
      }
      __syncwarp();
    }
    if (half == 0 && lane < rows) {
      if (whole) {
        if (p.lse != nullptr) p.lse[orow0 + lane] = (m + log2f(lt)) * kLn2;
      } else {
        p.part_ml[(orow0 + lane) * 2] = m;
        p.part_ml[(orow0 + lane) * 2 + 1] = lt;
      }
    }
    tc_fence_before();
    __syncwarp();
    arrive_leader(lane, ofree);
  }
  if (!ok && lane == 0) set_abort(ctl, p.dev_err);
}

// ------------------------------------------------------------- single threads
__device__ __forceinline__ bool pwait(uint64_t* bar, uint32_t parity, PairCtrl& c, uint32_t site, uint32_t* dev_err) {
  return wait_ok(mbar_wait(bar, parity, kWaitNs, &c.abort), site, c, dev_err);
}

// The query image of the unit at sc, by bulk copies that complete on q_bar.
__device__ __forceinline__ void load_query(const Params& p, const PairSched& sc, uint8_t* sm, PairCtrl& ctl, int rank) {
  const uint8_t* src = p.qimg + (static_cast<size_t>(sc.b) * p.n_img + 2 * sc.g + rank) * kQImg;
  mbar_arrive_expect_tx(&ctl.q_bar, kQImg);
#pragma unroll 1
  for (int k = 0; k < kNumChunks; ++k)
    bulk_g2s(sm + k * kRows * 128, src + k * kRows * 128, kRows * 128, &ctl.q_bar);
}

// Leader: every MMA of the pair, from one thread (MMAs of two threads that
// interleave on the tensor core took 2,040 instead of 1,480 cycles per tile), PV of
// the older tile first, whichever has its operands.
__device__ void pair_mma(const Params& p, const PairSched& sc, uint8_t* sm, uint32_t smem, PairCtrl& ctl,
                         uint32_t tmem) {
  constexpr uint32_t kIdQK = idesc_f16_f32(128, kPairTok, false, false);
  constexpr uint32_t kIdPV = idesc_f16_f32(128, 256, false, true);
  const uint64_t qa = smem_desc(smem, 16, 1024, SWZ_128B), kb = smem_desc(smem + kKOff, 16, 1024, SWZ_128B);
  const uint64_t pa = smem_desc(smem + kPOff, 16, 1024, SWZ_128B);
  const uint64_t vb = smem_desc(smem + kVOff, kVChunk, 1024, SWZ_128B);
  PairSched sq = sc, sp = sc;
  uint32_t n = 0, v = 0, qseg = 0, pseg = 0, fixes[2] = {0u, 0u};
  int query = 0;  // of the segment at sq: 0 not asked for, 1 on its way, 2 there
  uint32_t refs = 0;  // reference tiles, which have no PV
  while (sp.live && sp.ref) {
    sp.next(p);
    ++refs;
  }
  uint64_t idle = 0;
  bool ok = true;
  while (ok && (sq.live || sp.live)) {
    bool did = false;
    if (sp.live) {
      const bool first = sp.seg_first();
      const uint32_t st = v & 1u, ph = (v >> 1) & 1u;
      bool ready = mbar_test_cluster(&ctl.p_full[st], ph) && mbar_test_cluster(&ctl.v_full[st], ph) &&
                   (!first || pseg == 0 || mbar_test_cluster(&ctl.o_free, (pseg - 1) & 1u));
      // A rewritten P is waited for by passing on to the QK below: the softmax settles a
      // tile when it has the next one's scores, which may not have been issued yet.
      bool fix[2] = {false, false};
      if (ready) {
#pragma unroll
        for (int r = 0; r < 2; ++r) {
          fix[r] = *reinterpret_cast<volatile uint32_t*>(&ctl.raised[r][st]) == v + 1;
          ready = ready && (!fix[r] || mbar_test_cluster(&ctl.p_fixed[r], fixes[r] & 1u));
        }
      }
      if (ready) {
        fixes[0] += fix[0] ? 1u : 0u;
        fixes[1] += fix[1] ? 1u : 0u;
        tc_fence_after();
        const uint64_t a1 = pa + ((st * kPTile) >> 4), b1 = vb + ((st * kVStage) >> 4);
        const uint32_t acc0 = first ? 0u : 1u;
#pragma unroll
        for (int blk = 0; blk < 2; ++blk) {
#pragma unroll
          for (int kk = 0; kk < 4; ++kk)
            umma2_f16_ss(tmem + blk * 128, a1 + ((kk * 32) >> 4), b1 + ((blk * 2 * kVChunk + kk * 2048) >> 4), kIdPV,
                         kk == 0 ? acc0 : 1u);
        }
        umma2_commit(&ctl.pv_done[st]);
        if (sp.seg_last()) ++pseg;
        ++v;
        sp.next(p);
        did = true;
      }
    }
    if (!did && sq.live) {
      if (query == 0 && (qseg == 0 || mbar_test(&ctl.q_free, (qseg - 1) & 1u))) {
        load_query(p, sq, sm, ctl, 0);
        query = 1;
      }
      if (query == 1 && mbar_test(&ctl.q_bar, qseg & 1u) && mbar_test_cluster(&ctl.q_peer, qseg & 1u)) query = 2;
      const uint32_t st = n & 1u;
      // (QK of real tile i goes after PV of tile i - 2: the softmax then knows that its P
      // tile is free once it has the scores)
      if (query == 2 && n < v + 2 + refs && mbar_test_cluster(&ctl.k_full[st], (n >> 1) & 1u) &&
          (n < 4 || mbar_test_cluster(&ctl.s_free[n & 3u], ((n >> 2) - 1) & 1u))) {
        tc_fence_after();
        const uint64_t b1 = kb + ((st * kKStage) >> 4);
        const uint32_t ts = tmem + kColS + (n & 3u) * 64;
        // (one partial after the other: switching the accumulator at every MMA costs 39
        // instead of 25.5 cycles each)
#pragma unroll
        for (int part = 0; part < 2; ++part) {
#pragma unroll
          for (int k = 0; k < kNumChunks; ++k) {
#pragma unroll
            for (int kk = part; kk < 4; kk += 2)
              umma2_f16_ss(ts + part * 32, qa + ((k * kRows * 128 + kk * 32) >> 4),
                           b1 + ((k * kKChunk + kk * 32) >> 4), kIdQK, k == 0 && kk < 2 ? 0u : 1u);
          }
        }
        umma2_commit(&ctl.s_full[n & 3u]);
        umma2_commit(&ctl.k_free[st]);
        if (sq.seg_last()) {
          umma2_commit(&ctl.q_free);
          query = 0;
          ++qseg;
        }
        ++n;
        sq.next(p);
        did = true;
      }
    }
    if (did) {
      idle = 0;
    } else {
      const uint64_t t = globaltimer_ns();
      if (idle == 0) idle = t;
      if (*reinterpret_cast<volatile uint32_t*>(&ctl.abort) != 0u) ok = false;
      if (t - idle > kWaitNs) ok = wait_ok(0, kSiteMmaChunk, ctl, p.dev_err);
    }
  }
  if (!ok) set_abort(ctl, p.dev_err);
}

// The other CTA: its query image of each segment, which replaces the previous
// segment's once all its QKs have completed (q_free).
__device__ void pair_query(const Params& p, PairSched sc, uint8_t* sm, PairCtrl& ctl, int rank) {
  uint32_t seg = 0;
  bool ok = true, loaded = false;
  for (; ok && sc.live; sc.next(p)) {
    if (!loaded) {
      if (seg > 0 && !(ok = pwait(&ctl.q_free, (seg - 1) & 1u, ctl, kSiteMmaQFull, p.dev_err))) break;
      load_query(p, sc, sm, ctl, rank);
      if (!(ok = pwait(&ctl.q_bar, seg & 1u, ctl, kSiteMmaQFull, p.dev_err))) break;
      arrive_leader_cluster(0, cluster_map(smem_u32(&ctl.q_peer), 0));
      loaded = true;
    }
    if (sc.seg_last()) {
      loaded = false;
      ++seg;
    }
  }
  // (the last commit's arrival here, so that it cannot reach a CTA that has left)
  if (ok && seg > 0) ok = pwait(&ctl.q_free, (seg - 1) & 1u, ctl, kSiteMmaFin, p.dev_err);
  if (!ok) set_abort(ctl, p.dev_err);
}

// The other CTA's idle issuer: brings the blocks of tiles ahead into L2 with one
// bulk request each, kPrefetchTiles ahead of the dequantisation.
template <int CB>
__device__ void pair_prefetch(const Params& p, PairSched sc, PairCtrl& ctl) {
  constexpr uint32_t kBytes = CB == 16 ? kBf16BlockBytes : BlockLayout<CB == 16 ? 4 : CB>::kBytes;
  uint32_t n = 0;
  const uint64_t begin = globaltimer_ns();
  for (; sc.live; sc.next(p), ++n) {
    while (n > *reinterpret_cast<volatile uint32_t*>(&ctl.progress) + kPrefetchTiles) {
      if (*reinterpret_cast<volatile uint32_t*>(&ctl.abort) != 0u || globaltimer_ns() - begin > 4 * kWaitNs) return;
      __nanosleep(400);
    }
    const int e = p.table[static_cast<size_t>(sc.b) * p.max_blocks + sc.q];
    if (n >= 2 && e >= 0 && e < p.num_blocks) bulk_prefetch_l2(p.pool + static_cast<size_t>(e) * kBytes, kBytes);
  }
}

template <int CB, bool PROT>
__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(kPairThreads, 1) decode_pair(const __grid_constant__ Params p) {
  extern __shared__ uint8_t smem_raw[];
  uint8_t* sm = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  const uint32_t smem = smem_u32(sm);
  PairCtrl& ctl = *reinterpret_cast<PairCtrl*>(sm + kCtrlOff);
  const int warp = __shfl_sync(0xffffffffu, static_cast<int>(threadIdx.x) >> 5, 0);
  const int lane = threadIdx.x & 31;
  const int rank = static_cast<int>(cluster_ctarank());
  const int pair = static_cast<int>(blockIdx.x >> 1);
  if (threadIdx.x == 0) {
    for (int i = 0; i < 2; ++i) {
      mbar_init(&ctl.k_full[i], 2 * kNumChunks);
      mbar_init(&ctl.v_full[i], 2 * 8);
      mbar_init(&ctl.p_full[i], 2 * kSoftWarps);
      mbar_init(&ctl.s_free[i], 2 * kSoftWarps);
      mbar_init(&ctl.s_free[i + 2], 2 * kSoftWarps);
      mbar_init(&ctl.s_full[i], 1);
      mbar_init(&ctl.s_full[i + 2], 1);
      mbar_init(&ctl.k_free[i], 1);
      mbar_init(&ctl.pv_done[i], 1);
    }
    mbar_init(&ctl.p_fixed[0], kSoftWarps);
    mbar_init(&ctl.p_fixed[1], kSoftWarps);
    mbar_init(&ctl.o_free, 2 * kSoftWarps);
    mbar_init(&ctl.q_peer, 1);
    mbar_init(&ctl.q_free, 1);
    mbar_init(&ctl.q_bar, 1);
    mbar_init(&ctl.fin, 1);
    mbar_init(&ctl.grp, kSoftWarps);
    ctl.abort = 0u;
    for (int i = 0; i < 2; ++i) ctl.over[i] = ctl.raised[0][i] = ctl.raised[1][i] = 0u;
    ctl.progress = 0u;
    fence_mbar_init();
  }
  if (warp == 0) {
    tmem_alloc2(&ctl.tmem_base, kTmemPair);
    tmem_relinquish2();
  }
  tc_fence_before();
  __syncthreads();
  cluster_sync_all();  // the other CTA's barriers are initialised
  tc_fence_after();
  const uint32_t tmem = __shfl_sync(0xffffffffu, ctl.tmem_base, 0);
  // The set-up above may overlap the prep kernel; everything below reads what
  // prep and the cache writer before it produced.
  griddep_wait();

  // (Each role makes its own schedule: one made before the branch, held across the
  // register split, spilled 244 bytes instead of 76 at most; 64 x 4,097 tokens, INT4: 120.8 us
  // instead of 115.1, BF16 168.5 instead of 163.3, INT2 32 x 32,768 386 instead of 368.)
  if (warp < kSoftWarps) {
    asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(kSoftRegs));
    PairSched sc;
    sc.init(p, pair);
    pair_softmax<CB>(p, sc, smem, ctl, tmem, rank, warp, lane, pair);
  } else {
    asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(kOtherRegs));
    if (warp < kMmaWarp) {
      PairSched sc;
      sc.init(p, pair);
      pair_dequant<CB, PROT>(p, sc, smem, ctl, rank, warp - kSoftWarps, lane);
    } else if (warp > kPrefetchWarp) {
      asm volatile("exit;");
    } else if (elect_one()) {  // the issuers are single threads
      PairSched sc;
      sc.init(p, pair);
      if (warp == kMmaWarp) {
        if (rank == 0) {
          pair_mma(p, sc, sm, smem, ctl, tmem);
        } else {
          pair_query(p, sc, sm, ctl, rank);
        }
      } else if (rank != 0) {
        pair_prefetch<CB>(p, sc, ctl);
      }
      if (warp == kMmaWarp && rank == 0) {
        // Every MMA must have landed before TMEM and shared memory are released;
        // this wait ignores the abort flag.
        umma2_commit_local(&ctl.fin);
        wait_ok(mbar_wait(&ctl.fin, 0, kWaitNs, nullptr), kSiteMmaFin, ctl, p.dev_err);
      }
    } else {
      // The other lanes leave: parked at a re-convergence point they delay the wake-up of
      // the elected one from its waits by more than a thousand cycles.
      asm volatile("exit;");
    }
  }
  griddep_launch_dependents();  // the merge may be scheduled as CTAs finish
  tc_fence_before();
  // Neither CTA leaves while the other may still arrive on its barriers or its
  // tensor core reads this CTA's operands (exited threads do not take part).
  cluster_arrive_wait();
  if (warp == 0) {
    tc_fence_after();
    tmem_dealloc2(tmem, kTmemPair);
  }
}

template <int CB, bool PROT>
cudaError_t launch_pair(const Params& prm, bool pdl, cudaStream_t stream) {
  static int configured_device = -1;
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  if (configured_device != dev) {
    e = cudaFuncSetAttribute(decode_pair<CB, PROT>, cudaFuncAttributeMaxDynamicSharedMemorySize, kPairSmem);
    if (e != cudaSuccess) return e;
    configured_device = dev;
  }
  return launch_k(decode_pair<CB, PROT>, dim3(2 * prm.grid), dim3(kPairThreads), kPairSmem, stream, pdl, prm);
}

}  // namespace

cudaError_t launch_decode_pair(const Params& prm, int cache_kind, bool pdl, cudaStream_t stream) {
  const bool prot = prm.prot != nullptr;
  if (cache_kind == kC4R4) return prot ? launch_pair<kC4R4, true>(prm, pdl, stream) : launch_pair<kC4R4, false>(prm, pdl, stream);
  if (cache_kind == 4) return prot ? launch_pair<4, true>(prm, pdl, stream) : launch_pair<4, false>(prm, pdl, stream);
  if (cache_kind == 2) return prot ? launch_pair<2, true>(prm, pdl, stream) : launch_pair<2, false>(prm, pdl, stream);
  return launch_pair<16, false>(prm, pdl, stream);
}

}  // namespace qmla
