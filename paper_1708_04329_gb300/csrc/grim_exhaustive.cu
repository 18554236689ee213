// All-bins filter over the token-major table (§GRIM-Filter steps 2-3;
// §Mapping GRIM-Filter: a row of p bins' existence bits per token is fetched
// and p counters are incremented, then p comparators give a pass bit per bin).
//
// GB300 mapping
// -------------
// * A persistent CTA (one per SM, 512 to 768 threads) takes work items (tile
//   of TW*32 bins, range of reads).  The tile -- 4^q rows x TW words of the
//   token-major table -- is staged in shared memory once per item and reused
//   by every read of the range.  TW = 32 (1024 bins, 128 KB at q = 5) up to q = 5 and
//   TW = 8 (256 bins, 128 KB) at q = 6.  Two extra rows follow the tile: all
//   zeros (for a q-gram holding a non-base: always a miss) and all ones
//   (padding after a read's last token: never a miss).
// * A warp holds 32/GL reads, one per group of GL = TW/4 lanes.  Lane i of a
//   group owns words 4i..4i+3 of the tile, i.e. 128 bins, and fetches them
//   for each token with one 16-byte shared load.  At TW = 32 a quarter warp
//   is one group reading one whole 128-byte row, so the four groups' loads of
//   four rows are four conflict-free wavefronts; at TW = 8 sixteen groups
//   load 32-byte rows whose bank group is row mod 4, and each group reads a
//   block-rotated copy of its read's class-cyclic token order (see
//   k_tokenise) so that every load covers the four bank groups evenly.
// * Each group copies the token row of the read it will take next into its
//   own shared-memory slot with cp.async while it works on the current one,
//   so the inner loop does not wait on global memory.  At TW = 8 a slot
//   holds a read's first blocks (up to four, as many as fit beside the tile
//   at the CTA size) and later blocks are loaded from L2.
// * Reads are swept in ranges whose token rows fit in L2, range by range,
//   so concurrent CTAs on different tiles share the same token rows.
// * Instead of p separate counters, each lane keeps bit-sliced vertical
//   counters: plane k of word w holds bit k of the counters of that word's 32
//   bins.  Counted are MISSES (tokens absent from the bin), started at
//   bias = 2^P - (D'+1) with D' = min(q*e, L-q+1), so the P-bit counter
//   overflows exactly when misses > D', i.e. when sum < T = (L-q+1) - q*e.
//   The overflow is kept in a sticky "dead" plane; a bin passes iff its dead
//   bit is clear at the end, and then its sum is (L-q+1) - (counter - bias).
//   P (5..8) is the smallest depth that holds the batch's largest D'.
// * Tokens are added 16 at a time with a carry-save (Harley-Seal) tree of
//   full adders (two 3-input LOP3s each), whose weight-16 carry ripples
//   through the P-4 upper planes: 2 logic ops per token per 32 bins at P = 5.
//   The logic ops run on the integer pipe, which bounds this kernel; the
//   token-to-address arithmetic is written as integer multiply-adds so that
//   it runs on the FMA pipe instead.
// * Early exit: a read leaves a tile once every one of its bins is dead --
//   exact, since a dead bin can never pass.
// * Two kernels differ in how a warp's groups, which run one instruction
//   stream, take their reads.  Taking one (new counters, the claim, the
//   prefetch of the read after it) costs the whole warp the same whether one
//   group or all do.  k_exhaustive (GRIM_SWITCH_GROUP) tests after each block
//   and switches every group whose read has ended.  k_lockstep
//   (GRIM_SWITCH_WARP, and every batch large enough to sort) takes reads with
//   as far to go together, tests nothing before the place where the tokeniser
//   expects a tile to be nearly done, and finishes what is live there apart.
//   Measured on GB300, k_exhaustive with a per-block test and a one-word tail
//   for uniform batches against k_lockstep (3.1 Gbp, ms): 250k reads of 100 bp,
//   coarse table 609 -> 589, 40k on the fine table 165 -> 156, 40k mixed
//   100-250 bp reads 102 -> 88, a plan of 4,096 of them 11.3 -> 9.6, 60k of 150
//   bp at q = 6 60.3 -> 56.8.  Both pipes are near their limit there (small
//   case: ALU 76%, shared-memory wavefronts 81%).
#include "grim_internal.cuh"

namespace grim {
namespace {

// CTA sizes built (the register cap follows from one CTA per SM): 512
// threads (128 registers), 640 (96) and 768 (80).  640 is the default: on
// GB300 it beat 768 threads (which spill a few words) by 4.7% at q = 5 and
// 2.4% at q = 6, and 512 by 2.6%; the autotuner can pick another.
constexpr uint32_t kDefaultThreads = 640;
constexpr uint32_t kNone = 0xFFFFFFFFu;
constexpr size_t kSmemLimit = kSmemMost - 128;  // dynamic shared memory per CTA (128 bytes are static)
// token rows of one read range: small enough to stay in L2 while every CTA
// sweeps its tiles against the range
constexpr uint64_t kDefaultRangeBytes = 48ull << 20;
constexpr uint32_t kSlotBlocksNarrow = 4;  // most slot blocks per read, 256-bin tiles
// per-warp scratch through which the lockstep kernel's live words change lanes:
// some planes of 32 words (what fits beside the slots) and 32 bytes that say
// where each came from
template <int TW>
constexpr int kScratchPlanes = TW == 8 ? 3 : 6;
template <int TW>
constexpr uint32_t kScratchBytes = kScratchPlanes<TW> * 128 + 32;

#define LOP3(d, a, b, c, lut) \
  asm("lop3.b32 %0, %1, %2, %3, " #lut ";" : "=r"(d) : "r"(a), "r"(b), "r"(c))

// full adder of three planes of the same weight: sum (a^b^c), carry maj(a,b,c)
__device__ __forceinline__ void fa(uint32_t a, uint32_t b, uint32_t c, uint32_t& s, uint32_t& k) {
  LOP3(s, a, b, c, 0x96);
  LOP3(k, a, b, c, 0xE8);
}
// full adder where b and c are existence words whose complements (misses) are
// added: sum a^~b^~c = a^b^c, carry maj(a,~b,~c)
__device__ __forceinline__ void fa_miss(uint32_t a, uint32_t b, uint32_t c, uint32_t& s,
                                        uint32_t& k) {
  LOP3(s, a, b, c, 0x96);
  LOP3(k, a, b, c, 0x71);
}

// integer multiply-adds (FMA pipe); the multipliers come from kernel
// arguments so they are not strength-reduced into shifts
__device__ __forceinline__ uint32_t imad(uint32_t a, uint32_t b, uint32_t c) {
  uint32_t d;
  asm("mad.lo.u32 %0, %1, %2, %3;" : "=r"(d) : "r"(a), "r"(b), "r"(c));
  return d;
}
// The full adder with its sum on the FMA pipe: as integers a + b + c is the sum
// word plus twice the carry word, so three multiply-adds stand in for one of
// the two logic ops.  Used for the adders of weight 4 and 8 of a block (12 of
// 60): 250k reads of 100 bp 593 -> 589.5 ms; with weight 2 as well 627.
__device__ __forceinline__ void fa_fma(uint32_t a, uint32_t b, uint32_t c, uint32_t& s, uint32_t& k,
                                       uint32_t one, uint32_t minus_two) {
  uint32_t m;
  LOP3(m, a, b, c, 0xE8);
  s = imad(m, minus_two, imad(c, one, imad(b, one, a)));
  k = m;
}
__device__ __forceinline__ uint32_t imul_hi(uint32_t a, uint32_t b) {
  uint32_t d;
  asm("mul.hi.u32 %0, %1, %2;" : "=r"(d) : "r"(a), "r"(b));
  return d;
}
__device__ __forceinline__ uint4 lds128(uint32_t addr) {
  uint4 v;
  asm volatile("ld.shared.v4.u32 {%0,%1,%2,%3}, [%4];"
               : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w)
               : "r"(addr));
  return v;
}

__device__ __forceinline__ uint32_t lds32(uint32_t addr) {
  uint32_t v;
  asm volatile("ld.shared.u32 %0, [%1];" : "=r"(v) : "r"(addr));
  return v;
}

template <int P, int NW = 4>
struct Counters {
  // per word: s1 s2 s4 s8 (weights 1..8), up[i] (weight 16 << i), dead
  uint32_t s1[NW], s2[NW], s4[NW], s8[NW], up[P - 4][NW], dead[NW];

  __device__ __forceinline__ void init(uint32_t bias) {
#pragma unroll
    for (int w = 0; w < NW; ++w) {
      s1[w] = 0u - (bias & 1u);
      s2[w] = 0u - ((bias >> 1) & 1u);
      s4[w] = 0u - ((bias >> 2) & 1u);
      s8[w] = 0u - ((bias >> 3) & 1u);
#pragma unroll
      for (int i = 0; i < P - 4; ++i) up[i][w] = 0u - ((bias >> (4 + i)) & 1u);
      dead[w] = 0u;
    }
  }

  // plane p of word w: the counter's planes by weight, then `dead`
  __device__ __forceinline__ uint32_t& plane(int p, int w) {
    return p == 0 ? s1[w] : p == 1 ? s2[w] : p == 2 ? s4[w] : p == 3 ? s8[w]
           : p < P ? up[p - 4][w] : dead[w];
  }

  // counter value of bin `bit` of word w
  __device__ __forceinline__ uint32_t value(int w, uint32_t bit) const {
    uint32_t v = ((s1[w] >> bit) & 1u) | (((s2[w] >> bit) & 1u) << 1) |
                 (((s4[w] >> bit) & 1u) << 2) | (((s8[w] >> bit) & 1u) << 3);
#pragma unroll
    for (int i = 0; i < P - 4; ++i) v |= ((up[i][w] >> bit) & 1u) << (4 + i);
    return v;
  }
};

struct ExhArgs {
  IndexView ix;
  ReadsView rv;
  RecordsView rec;
  uint32_t bin_bits;
  uint32_t n_tiles, sms;
  Live live;
  uint32_t row_stride;  // bytes of one token row in a group slot (multiple of 32)
  uint32_t slot_bytes;  // bytes of a group slot: two token rows
  uint32_t slot_blocks; // 16-token blocks a slot row holds; later blocks come from L2
  uint32_t c_row, c_hi, c_lo;  // TW*4, 65536, -65536: multipliers of the address math
  uint64_t range_bytes;        // token-row bytes of one read range (the read tile)
  uint32_t few_reads;          // batches of up to this many reads are k_exhaustive_few's
  const uint32_t* order;       // lockstep: the reads in the order they are taken (null: as given)
  uint32_t check_shift;        // lockstep: kMetaCheckCoarse or kMetaCheckFine
  uint32_t c_one, c_minus_two;  // multipliers of fa_fma
  uint32_t pad_pair;           // two never-miss tokens
  Ctl* ctl;
};

// the carries of a 16-token block between its quads
template <int NW>
struct CsaTemps {
  uint32_t t2a[NW], t2b[NW], t4a[NW], t4b[NW], t8a[NW], t8b[NW], t16[NW];
};

// Add the misses of four tokens, the quad-th of a 16-token block, whose
// existence words are a0..a3; the block's last quad carries into the upper
// planes.  FMA: fa_fma for the adders of weight 4 and 8.  k_exhaustive does
// without and is handed the row count in stage_tile, or it spills at P = 5: 4,000
// reads of 100 bp in one pass over 1.5M bins, GROUP, 2.32 -> 2.16 ms.
template <int P, int NW, bool FMA>
__device__ __forceinline__ void add_quad(Counters<P>& c, CsaTemps<NW>& t, int quad,
                                         const uint32_t (&a0)[NW], const uint32_t (&a1)[NW],
                                         const uint32_t (&a2)[NW], const uint32_t (&a3)[NW],
                                         uint32_t one, uint32_t m2) {
#pragma unroll
  for (int w = 0; w < NW; ++w) {
    uint32_t* t4 = (quad & 1) ? t.t4b : t.t4a;
    fa_miss(c.s1[w], a0[w], a1[w], c.s1[w], t.t2a[w]);
    fa_miss(c.s1[w], a2[w], a3[w], c.s1[w], t.t2b[w]);
    fa(c.s2[w], t.t2a[w], t.t2b[w], c.s2[w], t4[w]);
    auto fa_high = [&](uint32_t a, uint32_t b, uint32_t x, uint32_t& s, uint32_t& k) {
      if constexpr (FMA) fa_fma(a, b, x, s, k, one, m2);
      else fa(a, b, x, s, k);
    };
    if (quad == 1) fa_high(c.s4[w], t.t4a[w], t.t4b[w], c.s4[w], t.t8a[w]);
    if (quad == 3) {
      fa_high(c.s4[w], t.t4a[w], t.t4b[w], c.s4[w], t.t8b[w]);
      fa_high(c.s8[w], t.t8a[w], t.t8b[w], c.s8[w], t.t16[w]);
      // ripple the weight-16 carry through the upper planes; the carry out
      // of the top plane (counter >= 2^P: misses > D') sticks in `dead`
      uint32_t k = t.t16[w];
#pragma unroll
      for (int i = 0; i < P - 5; ++i) {
        const uint32_t nk = c.up[i][w] & k;
        c.up[i][w] ^= k;
        k = nk;
      }
      uint32_t d;
      LOP3(d, c.dead[w], c.up[P - 5][w], k, 0xF8);  // dead | (top & k)
      c.up[P - 5][w] ^= k;
      c.dead[w] = d;
    }
  }
}

// Add the misses of one 16-token block to the lane's four words.  tw holds 16
// table row indices as uint16 pairs; base is the shared address of this lane's
// words in row 0 (one 16-byte load per token).
template <int P, bool FMA>
__device__ __forceinline__ void add_block(Counters<P>& c, const uint32_t (&tw)[8], uint32_t base,
                                          const ExhArgs& a) {
  uint32_t addr[16];
#pragma unroll
  for (int j = 0; j < 8; ++j) {
    const uint32_t hi = imul_hi(tw[j], a.c_hi);     // token 2j+1
    const uint32_t lo = imad(hi, a.c_lo, tw[j]);    // token 2j
    addr[2 * j] = imad(lo, a.c_row, base);
    addr[2 * j + 1] = imad(hi, a.c_row, base);
  }
  CsaTemps<4> t;
#pragma unroll
  for (int quad = 0; quad < 4; ++quad) {
    const uint4 x0 = lds128(addr[4 * quad]), x1 = lds128(addr[4 * quad + 1]);
    const uint4 x2 = lds128(addr[4 * quad + 2]), x3 = lds128(addr[4 * quad + 3]);
    const uint32_t a0[4] = {x0.x, x0.y, x0.z, x0.w}, a1[4] = {x1.x, x1.y, x1.z, x1.w};
    const uint32_t a2[4] = {x2.x, x2.y, x2.z, x2.w}, a3[4] = {x3.x, x3.y, x3.z, x3.w};
    add_quad<P, 4, FMA>(c, t, quad, a0, a1, a2, a3, a.c_one, a.c_minus_two);
  }
}

// Add the misses of 8 tokens (half a block) to NW words: NW = 4 as add_block,
// NW = 1 the single word at `base`.
template <int P, int NW>
__device__ __forceinline__ void add_half(Counters<P, NW>& c, const uint4& tok, uint32_t base,
                                         const ExhArgs& a) {
  const uint32_t tw[4] = {tok.x, tok.y, tok.z, tok.w};
  uint32_t addr[8];
#pragma unroll
  for (int j = 0; j < 4; ++j) {
    const uint32_t hi = imul_hi(tw[j], a.c_hi);
    const uint32_t lo = imad(hi, a.c_lo, tw[j]);
    addr[2 * j] = imad(lo, a.c_row, base);
    addr[2 * j + 1] = imad(hi, a.c_row, base);
  }
  uint32_t x[8][NW];
#pragma unroll
  for (int j = 0; j < 8; ++j) {
    if constexpr (NW == 4) {
      const uint4 v = lds128(addr[j]);
      x[j][0] = v.x; x[j][1] = v.y; x[j][2] = v.z; x[j][3] = v.w;
    } else {
      x[j][0] = lds32(addr[j]);
    }
  }
#pragma unroll
  for (int w = 0; w < NW; ++w) {
    uint32_t t2a, t2b, t4a, t4b, k;
    fa_miss(c.s1[w], x[0][w], x[1][w], c.s1[w], t2a);
    fa_miss(c.s1[w], x[2][w], x[3][w], c.s1[w], t2b);
    fa(c.s2[w], t2a, t2b, c.s2[w], t4a);
    fa_miss(c.s1[w], x[4][w], x[5][w], c.s1[w], t2a);
    fa_miss(c.s1[w], x[6][w], x[7][w], c.s1[w], t2b);
    fa(c.s2[w], t2a, t2b, c.s2[w], t4b);
    fa(c.s4[w], t4a, t4b, c.s4[w], k);
    uint32_t nk = c.s8[w] & k;  // the weight-8 carry ripples on
    c.s8[w] ^= k;
    k = nk;
#pragma unroll
    for (int i = 0; i < P - 5; ++i) {
      nk = c.up[i][w] & k;
      c.up[i][w] ^= k;
      k = nk;
    }
    uint32_t d;
    LOP3(d, c.dead[w], c.up[P - 5][w], k, 0xF8);  // dead | (top & k)
    c.up[P - 5][w] ^= k;
    c.dead[w] = d;
  }
}

// Work items are (tile, range of reads): enough ranges (of at least 64 reads)
// to balance the persistent grid when tiles are few, and ranges whose token
// rows fit in L2 when there are many reads: items are then taken range by
// range, so the CTAs sweeping different tiles at the same time share one
// range's token rows in L2 instead of each streaming every read's tokens from
// DRAM.
struct Ranges {
  uint32_t n_ranges, per, n_items;
  bool range_major;
};
__device__ __forceinline__ Ranges read_ranges(const ExhArgs& a, uint32_t n_reads) {
  uint32_t n_ranges = (4u * a.sms + a.n_tiles - 1) / a.n_tiles;
  const uint64_t token_bytes = (uint64_t)n_reads * a.rv.ts * 2u * a.rv.copies;
  const uint32_t l2_ranges = (uint32_t)((token_bytes + a.range_bytes - 1) / a.range_bytes);
  n_ranges = max(n_ranges, l2_ranges);
  n_ranges = min(n_ranges, (n_reads + 63) / 64);
  n_ranges = max(n_ranges, 1u);
  const uint32_t per = (n_reads + n_ranges - 1) / n_ranges;
  n_ranges = (n_reads + per - 1) / per;
  return {n_ranges, per, a.n_tiles * n_ranges, a.n_tiles >= 4u * a.sms};
}

// the all-zeros and all-ones rows behind a tile, and 16 padding tokens
template <int TW>
__device__ __forceinline__ void fill_special_rows(uint32_t* tile, uint32_t r4, uint32_t pad_tokens,
                                                  uint32_t tid, uint32_t nthreads) {
  for (uint32_t i = tid; i < (uint32_t)TW; i += nthreads) {
    tile[rowInvalid(r4) * TW + i] = 0u;
    tile[rowPad(r4) * TW + i] = ~0u;
  }
  if (tid < 2) {  // 32 bytes
    const uint32_t pp = rowPad(r4) | (rowPad(r4) << 16);
    asm volatile("st.shared.v4.u32 [%0], {%1,%1,%1,%1};" ::"r"(pad_tokens + tid * 16u), "r"(pp));
  }
}

// start copying a tile: rows [0, r4), words [tile*TW, tile*TW+TW).  (r4 from a
// register in k_exhaustive, from the arguments in k_lockstep: the other way round
// the one spills, and the other's 4096-bin tiles lose 3%, 9.28 -> 9.55 ms for the
// existence counts at q = 4.)
template <int TW>
__device__ __forceinline__ void stage_tile(const ExhArgs& a, uint32_t r4, uint32_t tile,
                                           uint32_t sh_base, uint32_t tid, uint32_t nthreads) {
  constexpr uint32_t kChunks = TW / 4;  // 16-byte chunks per row
  const uint32_t* src = a.ix.tm + (uint64_t)tile * TW;
  for (uint32_t i = tid; i < r4 * kChunks; i += nthreads) {
    const uint32_t row = i / kChunks, chunk = i % kChunks;
    // (rows end on 1024 bins; the bins of a larger tile past them start out dead)
    if (TW > 32 && (uint64_t)tile * TW + chunk * 4u >= a.ix.wpad) continue;
    const uint32_t* g = src + (uint64_t)row * a.ix.wpad + chunk * 4u;
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(sh_base + row * TW * 4u +
                                                                  chunk * 16u),
                 "l"(g));
  }
  asm volatile("cp.async.commit_group;");
}

template <int P, int TW, int NT>
__global__ void __launch_bounds__(NT, 1) k_exhaustive(ExhArgs a) {
  constexpr uint32_t kRowBytes = TW * 4;     // one token's row of a tile
  constexpr uint32_t GL = TW / 4;            // lanes per group (one read)
  constexpr uint32_t kGroupMask = (1u << GL) - 1u;
  constexpr uint32_t kTileBinsT = TW * 32;
  // [tile: (r4 + 2) rows x TW words][group slots][16 padding tokens]
  extern __shared__ __align__(128) uint8_t smem[];
  __shared__ uint32_t s_item, s_next;
  const uint32_t tid = threadIdx.x, lane = tid & 31, grp = lane / GL, li = lane % GL;
  const uint32_t nthreads = blockDim.x;
  const uint32_t r4 = a.ix.r4;
  if (*(volatile uint32_t*)&a.ctl->status) return;  // set by the tokeniser before launch
  if (gated_off(a.ctl, a.live)) return;             // the batch takes the other path
  const uint32_t n_reads = live_reads(a.ctl, a.live, a.rv.n_reads);
  if (n_reads == 0) return;
  const Ranges rg = read_ranges(a, n_reads);

  uint32_t* s_tile = reinterpret_cast<uint32_t*>(smem);
  const uint32_t tile_bytes = (r4 + 2) * kRowBytes;
  const uint32_t sh_base = (uint32_t)__cvta_generic_to_shared(smem);
  const uint32_t slot = sh_base + tile_bytes + (tid / GL) * a.slot_bytes;
  const uint32_t pad_tokens = sh_base + tile_bytes + (nthreads / GL) * a.slot_bytes;
  fill_special_rows<TW>(s_tile, r4, pad_tokens, tid, nthreads);
  const uint32_t lane_base = sh_base + li * 16u;
  // the token copy this group reads (block-rotated copies spread the groups'
  // 32-byte rows over the bank groups at q = 6)
  const uint32_t copy = a.rv.copies > 1 ? grp % a.rv.copies : 0u;
  const uint32_t row_chunks = a.row_stride / 16u;  // 16-byte chunks of a slot row

  for (;;) {
    asm volatile("cp.async.wait_all;" ::: "memory");
    __syncthreads();  // previous item finished with the tile and the slots
    if (tid == 0) {
      s_item = atomicAdd(&a.ctl->item, 1u);
      s_next = 0;
    }
    __syncthreads();
    const uint32_t item = s_item;
    if (item >= rg.n_items) break;
    const uint32_t tile = rg.range_major ? item % a.n_tiles : item / rg.n_ranges;
    const uint32_t range = rg.range_major ? item / a.n_tiles : item % rg.n_ranges;
    const uint32_t r0 = range * rg.per;
    const uint32_t nr = min(rg.per, n_reads - r0);

    stage_tile<TW>(a, r4, tile, sh_base, tid, nthreads);

    // which bins of this lane's words exist (only the last tile is ragged)
    uint32_t vm[4];
#pragma unroll
    for (int w = 0; w < 4; ++w) {
      const uint64_t b0 = (uint64_t)tile * kTileBinsT + (li * 4u + w) * 32u;
      const uint64_t left = b0 < a.ix.num_bins ? a.ix.num_bins - b0 : 0;
      vm[w] = left >= 32 ? ~0u : ((1u << left) - 1u);
    }
    // per-group state (identical in the group's 8 lanes); the group's slot
    // holds two token rows: `buf` is the current read's, buf^1 the next's
    uint32_t cur = kNone, nxt = kNone, nxt_meta = 0, buf = 1;
    uint32_t nblk = 0, ntok = 0, bias = 0, executed = 0;
    bool fin = false;
    Counters<P> c;
    c.init(0);

    // take the first read and start copying its tokens
    {
      uint32_t k = 0;
      if (li == 0) k = atomicAdd(&s_next, 1u);
      k = __shfl_sync(0xFFFFFFFFu, k, grp * GL);
      if (k < nr) {
        nxt = r0 + k;
        nxt_meta = __ldg(a.rv.meta + nxt);
        const char* src = reinterpret_cast<const char*>(
            a.rv.tokens + ((uint64_t)nxt * a.rv.copies + copy) * a.rv.ts);
        for (uint32_t ch = li; ch < row_chunks; ch += GL)
          asm volatile("cp.async.ca.shared.global [%0], [%1], 16;" ::"r"(slot + ch * 16u),
                       "l"(src + ch * 16u));
      }
      asm volatile("cp.async.commit_group;");
    }
    asm volatile("cp.async.wait_all;" ::: "memory");
    __syncthreads();  // tile staged

    // (1) groups without a read switch to the one whose tokens were copied
    //     ahead, and start copying the read after it; `tp` is the shared
    //     address of a group's next 16-token block, `left` its blocks left
    //     (finished groups apply padding tokens, their results ignored)
    uint32_t tp = pad_tokens, step = 0, left = 0;
    auto switch_reads = [&](bool need) {
      asm volatile("cp.async.wait_all;" ::: "memory");
      __syncwarp();
      if (need) {
        if (nxt == kNone) {
          fin = true;
        } else {
          cur = nxt;
          buf ^= 1u;
          ntok = nxt_meta & 0xFFu;
          const uint32_t d = (nxt_meta >> 8) & 0xFFu;
          bias = (1u << P) - (d + 1u);
          nblk = (ntok + kBlockTokens - 1) / kBlockTokens;
          c.init(bias);
        }
        tp = fin ? pad_tokens : slot + buf * a.row_stride;
        step = fin ? 0u : 32u;
        left = fin ? ~0u : nblk;
      }
      const bool take = need && !fin;
      uint32_t k = 0;
      if (take && li == 0) k = atomicAdd(&s_next, 1u);
      k = __shfl_sync(0xFFFFFFFFu, k, grp * GL);
      if (take) {
        nxt = k < nr ? r0 + k : kNone;
        if (nxt != kNone) {
          nxt_meta = __ldg(a.rv.meta + nxt);
          const char* src = reinterpret_cast<const char*>(
              a.rv.tokens + ((uint64_t)nxt * a.rv.copies + copy) * a.rv.ts);
          const uint32_t dst = slot + (buf ^ 1u) * a.row_stride;
          for (uint32_t ch = li; ch < row_chunks; ch += GL)
            asm volatile("cp.async.ca.shared.global [%0], [%1], 16;" ::"r"(dst + ch * 16u),
                         "l"(src + ch * 16u));
        }
      }
      asm volatile("cp.async.commit_group;");
    };
    switch_reads(true);
    const uint32_t gmask = kGroupMask << (grp * GL);
    bool active = __any_sync(0xFFFFFFFFu, !fin);

    // the passing bins of the groups whose reads ended (emit), then new
    // reads for them (done); the warp runs this together
    auto emit_and_switch = [&](bool done, bool emit) {
      if (__any_sync(0xFFFFFFFFu, emit)) {
        uint32_t pm[4], cnt = 0;
#pragma unroll
        for (int w = 0; w < 4; ++w) {
          pm[w] = emit ? (~c.dead[w] & vm[w]) : 0u;
          cnt += __popc(pm[w]);
        }
        uint32_t incl = cnt;
#pragma unroll
        for (int d = 1; d < 32; d <<= 1) {
          const uint32_t t = __shfl_up_sync(0xFFFFFFFFu, incl, d);
          if (lane >= (uint32_t)d) incl += t;
        }
        const uint32_t tot = __shfl_sync(0xFFFFFFFFu, incl, 31);
        unsigned long long base = 0;
        if (lane == 0 && tot) base = atomicAdd(&a.ctl->n_rec, (unsigned long long)tot);
        base = __shfl_sync(0xFFFFFFFFu, base, 0);
        unsigned long long pos = base + incl - cnt;
        // past the capacity (count-only calls: always) records are only
        // counted, not walked bit by bit: 500 reads against 6.55M bins at
        // q = 4, six budgets, 9.5e9 passing pairs: 15.6 -> 10.4 ms
        if (base >= a.rec.cap) {
#pragma unroll
          for (int w = 0; w < 4; ++w) pm[w] = 0;
        }
#pragma unroll
        for (int w = 0; w < 4; ++w) {
          uint32_t m = pm[w];
          while (m) {
            const uint32_t bit = __ffs(m) - 1;
            m &= m - 1;
            const uint32_t misses = c.value(w, bit) - bias;
            const uint64_t bin = (uint64_t)tile * kTileBinsT + (li * 4u + w) * 32u + bit;
            if (pos < a.rec.cap) {
              a.rec.keys[pos] = ((unsigned long long)cur << a.bin_bits) | bin;
              a.rec.counts[pos] = (uint8_t)(ntok - misses);
            }
            ++pos;
          }
        }
      }
      if (done) cur = kNone;
      switch_reads(done);
      active = __any_sync(0xFFFFFFFFu, !fin);
    };

    while (active) {
      // (2) one 16-token block for all groups: from the slot, or for the blocks
      //     past the slot's rows (long reads at q = 6) from L2
      {
        uint4 t0, t1;
        const uint32_t bi = nblk - left;  // this read's block index
        // (1024-bin tiles: whole reads in slots)
        if (TW == 32 || fin || bi < a.slot_blocks) {
          t0 = lds128(tp);
          t1 = lds128(tp + 16u);
        } else {
          const uint4* g = reinterpret_cast<const uint4*>(
              a.rv.tokens + ((uint64_t)cur * a.rv.copies + copy) * a.rv.ts + bi * kBlockTokens);
          t0 = __ldg(g);
          t1 = __ldg(g + 1);
        }
        const uint32_t tw[8] = {t0.x, t0.y, t0.z, t0.w, t1.x, t1.y, t1.z, t1.w};
        add_block<P, false>(c, tw, lane_base, a);
      }
      tp += step;
      --left;

      // (3) a read ends when every bin of its tile is dead or its tokens are
      //     used up
      const uint32_t all_dead = c.dead[0] & c.dead[1] & c.dead[2] & c.dead[3];
      const uint32_t bal = __ballot_sync(0xFFFFFFFFu, all_dead == ~0u);
      const bool gdead = (bal & gmask) == gmask;
      const bool done = !fin && (gdead || left == 0);
      if (!__any_sync(0xFFFFFFFFu, done)) continue;
      if (done) executed += nblk - left;
      emit_and_switch(done, done && !gdead);
    }
    // one count per group (its lanes agree), one atomic per warp and item
    uint32_t ex = li == 0 ? executed : 0u;
    ex = __reduce_add_sync(0xFFFFFFFFu, ex);
    if (lane == 0 && ex) atomicAdd(&a.ctl->blocks, 2ull * ex);  // (counted in halves)
  }
}

// The lockstep kernel: the lane groups of a warp (4 on 1024-bin tiles, 16 on
// 256-bin tiles, 1 on the 4096-bin tiles of q <= 4) take reads of similar length to go (ExhArgs::order) together,
// run them for
// as many tokens as the tokeniser expects a tile to need, gather what is still
// live and finish that.
//
// * No end-of-read test until the check point (kMetaCheck*, the least of the
//   reads): whole 16-token blocks, and a half block where it is odd.
// * Then the warp counts the words (of its 128) that still hold a live bin.
//   As long as more than 32 do, it applies half blocks to all of them; 32 or
//   fewer are dealt out, one to a lane, through a scratch in shared memory
//   (planes, and where the word came from), and only those get the rest of
//   their reads' tokens: a quarter of the logic ops.  Exact: a word left
//   behind has no live bin, and a dead bin can never pass.
// * A read's last half blocks run into its row's padding (never a miss), so
//   shorter reads of a warp hold their counters.
// * Claims are a warp's: one shared atomic for its reads, two rounds ahead,
//   so the order's index and then the token row (cp.async) arrive in time.
template <int P, int TW, int NT>
__global__ void __launch_bounds__(NT, 1) k_lockstep(ExhArgs a) {
  constexpr uint32_t kRowBytes = TW * 4, kTileBinsT = TW * 32, GL = TW / 4, kGroups = 32 / GL;
  constexpr int kPlanes = kScratchPlanes<TW>;
  // [tile: (r4 + 2) rows x TW words][group slots][16 padding tokens][warp scratch]
  extern __shared__ __align__(128) uint8_t smem[];
  __shared__ uint32_t s_item, s_next;
  __shared__ unsigned long long s_counted;  // calls without room for records: passing bins
  const uint32_t tid = threadIdx.x, lane = tid & 31, grp = lane / GL, li = lane % GL;
  const uint32_t nthreads = blockDim.x;
  const uint32_t r4 = a.ix.r4;
  if (*(volatile uint32_t*)&a.ctl->status) return;
  if (gated_off(a.ctl, a.live)) return;
  const uint32_t n_reads = live_reads(a.ctl, a.live, a.rv.n_reads);
  if (n_reads == 0) return;
  const Ranges rg = read_ranges(a, n_reads);

  const uint32_t tile_bytes = (r4 + 2) * kRowBytes;
  const uint32_t sh_base = (uint32_t)__cvta_generic_to_shared(smem);
  const uint32_t slot = sh_base + tile_bytes + (tid / GL) * a.slot_bytes;
  const uint32_t pad_tokens = sh_base + tile_bytes + (nthreads / GL) * a.slot_bytes;
  const uint32_t scratch = pad_tokens + 32u + (tid >> 5) * kScratchBytes<TW>;
  if (tid == 0) s_counted = 0;
  fill_special_rows<TW>(reinterpret_cast<uint32_t*>(smem), r4, pad_tokens, tid, nthreads);
  const uint32_t lane_base = sh_base + li * 16u;
  const uint32_t row_chunks = a.row_stride / 16u;
  // 256-bin tiles: the token copy a group reads, and the halves its slot holds
  // (a read's later tokens come from L2)
  const uint32_t copies = TW == 8 ? a.rv.copies : 1u;
  const uint32_t slot_halves = TW == 8 ? 2u * a.slot_blocks : ~0u;
  auto token_row = [&](uint32_t r, uint32_t g) {
    return a.rv.tokens + ((uint64_t)r * copies + (TW == 8 ? g % copies : 0u)) * a.rv.ts;
  };

  for (;;) {
    asm volatile("cp.async.wait_all;" ::: "memory");
    __syncthreads();  // previous item finished with the tile and the slots
    if (tid == 0) {
      s_item = atomicAdd(&a.ctl->item, 1u);
      s_next = 0;
      if (a.rec.cap == 0) {
        if (s_counted) atomicAdd(&a.ctl->n_rec, s_counted);
        s_counted = 0;
      }
    }
    __syncthreads();
    const uint32_t item = s_item;
    if (item >= rg.n_items) break;
    const uint32_t tile = rg.range_major ? item % a.n_tiles : item / rg.n_ranges;
    const uint32_t range = rg.range_major ? item / a.n_tiles : item % rg.n_ranges;
    const uint32_t r0 = range * rg.per;
    const uint32_t nr = min(rg.per, n_reads - r0);
    stage_tile<TW>(a, a.ix.r4, tile, sh_base, tid, nthreads);
    // the last tile may be ragged: bins past the table's end start out dead
    const bool ragged = (uint64_t)(tile + 1) * kTileBinsT > a.ix.num_bins;

    auto claim = [&]() {
      uint32_t k = 0;
      if (lane == 0) k = atomicAdd(&s_next, kGroups);
      k = __shfl_sync(0xFFFFFFFFu, k, 0) + grp;
      return k >= nr ? kNone : a.order ? __ldg(a.order + r0 + k) : r0 + k;
    };
    auto fetch = [&](uint32_t r, uint32_t buf) {
      uint32_t m = 0;
      if (r != kNone) {
        m = __ldg(a.rv.meta + r);
        const char* src = reinterpret_cast<const char*>(token_row(r, grp));
        for (uint32_t ch = li; ch < row_chunks; ch += GL)
          asm volatile("cp.async.ca.shared.global [%0], [%1], 16;" ::"r"(
                           slot + buf * a.row_stride + ch * 16u),
                       "l"(src + ch * 16u));
      }
      asm volatile("cp.async.commit_group;");
      return m;
    };
    uint32_t nxt = claim(), buf = 0;
    uint32_t nxt_meta = fetch(nxt, 0);
    uint32_t nxt2 = claim();
    uint32_t ex = 0, tail_ex = 0, tail_words = 0;
    asm volatile("cp.async.wait_all;" ::: "memory");
    __syncthreads();  // tile staged

    for (;;) {
      const uint32_t cur = nxt, m = nxt_meta;
      const bool have = cur != kNone;
      if (!__any_sync(0xFFFFFFFFu, have)) break;
      asm volatile("cp.async.wait_all;" ::: "memory");
      __syncwarp();
      uint32_t tp = have ? slot + buf * a.row_stride : pad_tokens;
      const uint32_t step = have ? 16u : 0u;
      buf ^= 1u;
      nxt = nxt2;
      nxt_meta = fetch(nxt, buf);
      nxt2 = claim();

      // 0 without a read; rotated copies spread a block's tokens over both halves
      const uint32_t halves =
          TW == 8 ? ((m & 0xFFu) + 15u) >> 4 << 1 : ((m & 0xFFu) + 7u) >> 3;
      const uint32_t hmax = __reduce_max_sync(0xFFFFFFFFu, halves);
      uint32_t h = __reduce_min_sync(0xFFFFFFFFu, have ? (m >> a.check_shift) & 31u : 31u);
      // (256-bin tiles: whole blocks past the first half, whose 16 loads a half's 8
      // hardly undercut; 10k reads of 150 bp, one pass, e = 3 14.0 -> 11.9 ms)
      h = min(TW == 8 && h > 1u ? (h + 1u) & ~1u : h, hmax);
      const uint32_t bias = (1u << P) - (((m >> 8) & 0xFFu) + 1u);
      Counters<P> c;
      c.init(bias);
      if (!have || ragged) {
#pragma unroll
        for (int w = 0; w < 4; ++w) {
          const uint64_t b0 = (uint64_t)tile * kTileBinsT + (li * 4u + w) * 32u;
          const uint64_t left = b0 < a.ix.num_bins ? a.ix.num_bins - b0 : 0;
          c.dead[w] = !have ? ~0u : left >= 32 ? 0u : ~((1u << left) - 1u);
        }
      }
      // eight tokens of the group's read: half block `at`
      const uint4* far = reinterpret_cast<const uint4*>(token_row(have ? cur : 0u, grp));
      const uint4 pads = make_uint4(a.pad_pair, a.pad_pair, a.pad_pair, a.pad_pair);
      auto tokens_at = [&](uint32_t at, uint32_t near, const uint4* from, bool mine) {
        if (TW != 8 || at < slot_halves) return lds128(near);
        return mine ? __ldg(from + at) : pads;
      };
      for (uint32_t b = 0; b < h >> 1; ++b) {
        const uint4 t0 = tokens_at(2 * b, tp, far, have);
        const uint4 t1 = tokens_at(2 * b + 1, tp + 16u, far, have);
        const uint32_t tw[8] = {t0.x, t0.y, t0.z, t0.w, t1.x, t1.y, t1.z, t1.w};
        tp += 2u * step;
        add_block<P, true>(c, tw, lane_base, a);
      }
      if (h & 1u) {
        const uint4 t0 = tokens_at(h - 1u, tp, far, have);
        tp += step;
        add_half<P, 4>(c, t0, lane_base, a);
      }
      // live words, until few enough to gather, none, or the tokens are used up
      uint32_t live[4], n[4], total;
      for (;;) {
#pragma unroll
        for (int w = 0; w < 4; ++w) {
          live[w] = __ballot_sync(0xFFFFFFFFu, c.dead[w] != ~0u);
          n[w] = __popc(live[w]);
        }
        total = n[0] + n[1] + n[2] + n[3];
        if (total <= 32u || h >= hmax) break;
        const uint4 t0 = tokens_at(h, tp, far, have);
        tp += step;
        add_half<P, 4>(c, t0, lane_base, a);
        ++h;
      }
      ex += min(h, halves);
      if (total == 0) continue;

      // passing bins of NW words: their records, at consecutive places
      auto emit = [&](const uint32_t(&pm)[4], auto&& value, uint32_t read, uint32_t rm,
                      uint32_t bin0, uint32_t bin_step) {
        const uint32_t cnt = __popc(pm[0]) + __popc(pm[1]) + __popc(pm[2]) + __popc(pm[3]);
        if (a.rec.cap == 0) {
          // one global atomic per CTA and item instead of one per round, which
          // all warps would queue for when most bins pass
          const uint32_t all = __reduce_add_sync(0xFFFFFFFFu, cnt);
          if (lane == 0) atomicAdd(&s_counted, (unsigned long long)all);
          return;
        }
        uint32_t incl = cnt;
#pragma unroll
        for (int d = 1; d < 32; d <<= 1) {
          const uint32_t t = __shfl_up_sync(0xFFFFFFFFu, incl, d);
          if (lane >= (uint32_t)d) incl += t;
        }
        const uint32_t tot = __shfl_sync(0xFFFFFFFFu, incl, 31);
        unsigned long long base = 0;
        if (lane == 0 && tot) base = atomicAdd(&a.ctl->n_rec, (unsigned long long)tot);
        base = __shfl_sync(0xFFFFFFFFu, base, 0);
        if (base >= a.rec.cap) return;  // counted only
        unsigned long long pos = base + incl - cnt;
        const uint32_t ntok = rm & 0xFFu, bs = (1u << P) - (((rm >> 8) & 0xFFu) + 1u);
#pragma unroll
        for (int w = 0; w < 4; ++w) {
          uint32_t mask = pm[w];
          while (mask) {
            const uint32_t bit = __ffs(mask) - 1;
            mask &= mask - 1;
            if (pos < a.rec.cap) {
              a.rec.keys[pos] = ((unsigned long long)read << a.bin_bits) |
                                ((uint64_t)tile * kTileBinsT + bin0 + w * bin_step + bit);
              a.rec.counts[pos] = (uint8_t)(ntok - (value(w, bit) - bs));
            }
            ++pos;
          }
        }
      };
      if (h >= hmax) {
        const uint32_t pm[4] = {~c.dead[0], ~c.dead[1], ~c.dead[2], ~c.dead[3]};
        emit(pm, [&](int w, uint32_t bit) { return c.value(w, bit); }, cur, m, li * 128u, 32u);
        continue;
      }

      // gather: word w of this lane goes to lane at[w]
      const uint32_t below = (1u << lane) - 1u;
      uint32_t at[4], off = 0;
#pragma unroll
      for (int w = 0; w < 4; ++w) {
        at[w] = off + __popc(live[w] & below);
        off += n[w];
      }
      Counters<P, 1> g;
      uint32_t info = 0;
#pragma unroll
      for (int p0 = 0; p0 <= P; p0 += kPlanes) {
#pragma unroll
        for (int w = 0; w < 4; ++w) {
          if (c.dead[w] != ~0u) {
#pragma unroll
            for (int p = p0; p < p0 + kPlanes && p <= P; ++p)
              asm volatile("st.shared.u32 [%0], %1;" ::"r"(scratch + (p - p0) * 128u + at[w] * 4u),
                           "r"(c.plane(p, w)));
            if (p0 == 0)
              asm volatile("st.shared.u8 [%0], %1;" ::"r"(scratch + kPlanes * 128u + at[w]),
                           "r"(lane * 4u + w));
          }
        }
        __syncwarp();
#pragma unroll
        for (int p = p0; p < p0 + kPlanes && p <= P; ++p)
          g.plane(p, 0) = lds32(scratch + (p - p0) * 128u + lane * 4u);
        if (p0 == 0)
          asm volatile("ld.shared.u8 %0, [%1];" : "=r"(info) : "r"(scratch + kPlanes * 128u + lane));
        __syncwarp();
      }
      const bool on = lane < total;
      const uint32_t src = on ? info >> 2 : lane;  // the lane whose read and bins these are
      const uint32_t bin0 = (src % GL) * 128u + (info & 3u) * 32u;
      if (!on) g.dead[0] = ~0u;
      uint32_t gtp = __shfl_sync(0xFFFFFFFFu, tp, src);
      const uint32_t gstep = __shfl_sync(0xFFFFFFFFu, step, src);
      const uint32_t gbase = sh_base + (on ? bin0 >> 3 : 0u);
      {  // reads with a word left
        const uint32_t any = live[0] | live[1] | live[2] | live[3];
        if (TW == 128)
          off = 1;
        else if (TW == 32)
          off = ((any & 0xFFu) != 0) + ((any & 0xFF00u) != 0) + ((any & 0xFF0000u) != 0) +
                ((any & 0xFF000000u) != 0);
        else
          off = __popc((any | any >> 1) & 0x55555555u);
      }
      const uint4* gfar = far;
      if (TW == 8) {
        const uint32_t read = __shfl_sync(0xFFFFFFFFu, cur, src);
        gfar = reinterpret_cast<const uint4*>(token_row(on ? read : 0u, src / GL));
      }
      do {
        tail_words += g.dead[0] != ~0u;
        tail_ex += off;
        const uint4 t0 = tokens_at(h, gtp, gfar, on);
        gtp += gstep;
        add_half<P, 1>(g, t0, gbase, a);
        ++h;
      } while (h < hmax && __any_sync(0xFFFFFFFFu, g.dead[0] != ~0u));
      if (__any_sync(0xFFFFFFFFu, g.dead[0] != ~0u)) {
        const uint32_t pm[4] = {~g.dead[0], 0u, 0u, 0u};
        const uint32_t read = __shfl_sync(0xFFFFFFFFu, cur, src);
        const uint32_t rm = __shfl_sync(0xFFFFFFFFu, m, src);
        emit(pm, [&](int, uint32_t bit) { return g.value(0, bit); }, read, rm, bin0, 0u);
      }
    }
    // one count per group (its lanes agree), one atomic per warp and item
    // (4096-bin tiles count as four)
    constexpr uint32_t kUnits = TW == 128 ? 4 : 1;
    ex = __reduce_add_sync(0xFFFFFFFFu, li == 0 ? ex * kUnits : 0u);
    tail_words = __reduce_add_sync(0xFFFFFFFFu, tail_words);
    if (lane == 0) {
      atomicAdd(&a.ctl->blocks, (unsigned long long)ex);
      if (tail_ex) {
        atomicAdd(&a.ctl->tail_blocks, (unsigned long long)tail_ex * kUnits);
        atomicAdd(&a.ctl->tail_words, (unsigned long long)tail_words);
      }
    }
  }
}

// The same count for a handful of reads, straight from the token-major table.
// Staging every tile reads the whole table however few reads there are (4^q
// rows: 1 GB for the 3.1 Gbp coarse table at q = 5, 0.24 ms); here a warp holds
// one read and 4096 bins, loads only the rows that the read's tokens name,
// 512 contiguous bytes of each, and stops once all its bins are dead.  Warps
// on the same 4096 bins (all the reads) run side by side, so rows that reads
// share come from L2.  Bound by DRAM: 16 16-byte loads in flight a lane.
constexpr uint32_t kFewThreads = 256;
constexpr uint64_t kFewMinTable = 64ull << 20;  // bytes

template <int P>
__global__ void __launch_bounds__(kFewThreads, 2) k_exhaustive_few(ExhArgs a) {
  const uint32_t lane = threadIdx.x & 31;
  const uint32_t n_warps = gridDim.x * (kFewThreads / 32);
  const uint32_t r4 = a.ix.r4;
  if (*(volatile uint32_t*)&a.ctl->status) return;
  if (routed_off(a.ctl, a.live)) return;
  const uint32_t n_reads = live_reads(a.ctl, a.live, a.rv.n_reads);
  if (n_reads > a.few_reads) return;
  const uint64_t n_items = (a.ix.wpad + 127) / 128 * n_reads;
  for (uint64_t item = blockIdx.x * (kFewThreads / 32) + (threadIdx.x >> 5); item < n_items;
       item += n_warps) {
    const uint32_t r = (uint32_t)(item % n_reads);
    const uint64_t word0 = item / n_reads * 128 + lane * 4;  // this lane's words of a row
    const bool on = word0 < a.ix.wpad;                       // (rows are whole 1024-bin tiles)
    const uint32_t* col = a.ix.tm + (on ? word0 : 0);
    const uint32_t m = a.rv.meta[r];
    const uint32_t ntok = m & 0xFFu, d = (m >> 8) & 0xFFu;
    const uint32_t bias = (1u << P) - (d + 1u);
    const uint32_t nblk = (ntok + kBlockTokens - 1) / kBlockTokens;
    const uint4* tok =
        reinterpret_cast<const uint4*>(a.rv.tokens + (uint64_t)r * a.rv.copies * a.rv.ts);
    Counters<P> c;
    c.init(bias);
    uint32_t alive = 0;  // blocks after which this lane had a live bin
    bool ldead = !on;
    uint4 t0 = __ldg(tok), t1 = __ldg(tok + 1);
    for (uint32_t b = 0; b < nblk; ++b) {
      const uint32_t tw[8] = {t0.x, t0.y, t0.z, t0.w, t1.x, t1.y, t1.z, t1.w};
      if (b + 1 < nblk) {
        t0 = __ldg(tok + 2 * b + 2);
        t1 = __ldg(tok + 2 * b + 3);
      }
      // (the token is the same for the warp: no divergence)
      uint32_t x[16][4];
#pragma unroll
      for (int j = 0; j < 16; ++j) {
        const uint32_t row = (j & 1) ? tw[j >> 1] >> 16 : tw[j >> 1] & 0xFFFFu;
        const uint32_t fill = row == rowPad(r4) ? ~0u : 0u;
        uint4 v = make_uint4(fill, fill, fill, fill);
        if (row < r4) v = __ldg(reinterpret_cast<const uint4*>(col + (uint64_t)row * a.ix.wpad));
        x[j][0] = v.x; x[j][1] = v.y; x[j][2] = v.z; x[j][3] = v.w;
      }
      CsaTemps<4> t;
#pragma unroll
      for (int quad = 0; quad < 4; ++quad)
        add_quad<P, 4, true>(c, t, quad, x[4 * quad], x[4 * quad + 1], x[4 * quad + 2], x[4 * quad + 3],
                       a.c_one, a.c_minus_two);
      ldead = !on || (c.dead[0] & c.dead[1] & c.dead[2] & c.dead[3]) == ~0u;
      alive += ldead ? 0u : 1u;
      if (__all_sync(0xFFFFFFFFu, ldead)) break;
    }
    // blocks each tile (of 1024 bins, 256 at q = 6) needed, as the staged kernel
    // counts them
    const uint32_t tile_lanes = r4 <= 1024 ? 8u : 2u;
    uint32_t used = alive;
    used = max(used, __shfl_xor_sync(0xFFFFFFFFu, used, 1));
    if (tile_lanes == 8) {
      used = max(used, __shfl_xor_sync(0xFFFFFFFFu, used, 2));
      used = max(used, __shfl_xor_sync(0xFFFFFFFFu, used, 4));
    }
    used = lane % tile_lanes == 0 && on ? min(nblk, used + 1u) : 0u;
    used = __reduce_add_sync(0xFFFFFFFFu, used);
    if (lane == 0) atomicAdd(&a.ctl->blocks, 2ull * used);  // (counted in halves)
    if (__all_sync(0xFFFFFFFFu, ldead)) continue;
    uint32_t pm[4], cnt = 0;
#pragma unroll
    for (int w = 0; w < 4; ++w) {
      const uint64_t b0 = (word0 + w) * 32;
      const uint64_t left = on && b0 < a.ix.num_bins ? a.ix.num_bins - b0 : 0;
      pm[w] = ~c.dead[w] & (left >= 32 ? ~0u : (1u << left) - 1u);
      cnt += __popc(pm[w]);
    }
    uint32_t incl = cnt;
#pragma unroll
    for (int dd = 1; dd < 32; dd <<= 1) {
      const uint32_t t = __shfl_up_sync(0xFFFFFFFFu, incl, dd);
      if (lane >= (uint32_t)dd) incl += t;
    }
    const uint32_t tot = __shfl_sync(0xFFFFFFFFu, incl, 31);
    unsigned long long base = 0;
    if (lane == 0 && tot) base = atomicAdd(&a.ctl->n_rec, (unsigned long long)tot);
    base = __shfl_sync(0xFFFFFFFFu, base, 0);
    if (base >= a.rec.cap) continue;  // counted only
    unsigned long long pos = base + incl - cnt;
#pragma unroll
    for (int w = 0; w < 4; ++w) {
      uint32_t mask = pm[w];
      while (mask) {
        const uint32_t bit = __ffs(mask) - 1;
        mask &= mask - 1;
        if (pos < a.rec.cap) {
          a.rec.keys[pos] = ((unsigned long long)r << a.bin_bits) | ((word0 + w) * 32 + bit);
          a.rec.counts[pos] = (uint8_t)(ntok - (c.value(w, bit) - bias));
        }
        ++pos;
      }
    }
  }
}

template <typename Kernel>
void launch_k(Kernel kernel, const ExhArgs& a, size_t smem, uint32_t threads, uint32_t grid,
              cudaStream_t st, const char* name) {
  allow_smem(kernel, kSmemLimit);
  ProfScope ps(name, st);
  kernel<<<grid, threads, smem, st>>>(a);
}

// the counters need 2^P > D' (D' <= 255)
template <int TW, int NT>
void launch_nt(const ExhArgs& a, size_t smem, uint32_t threads, uint32_t grid, uint32_t max_d,
               bool lockstep, cudaStream_t st, const char* name) {
  auto run = [&](auto kernel) { launch_k(kernel, a, smem, threads, grid, st, name); };
  const int p = max_d < 32 ? 5 : max_d < 64 ? 6 : max_d < 128 ? 7 : 8;
  if (lockstep) {
    if (p == 5) run(k_lockstep<5, TW, NT>);
    else if (p == 6) run(k_lockstep<6, TW, NT>);
    else if (p == 7) run(k_lockstep<7, TW, NT>);
    else run(k_lockstep<8, TW, NT>);
    return;
  }
  if constexpr (TW != 128) {
    if (p == 5) run(k_exhaustive<5, TW, NT>);
    else if (p == 6) run(k_exhaustive<6, TW, NT>);
    else if (p == 7) run(k_exhaustive<7, TW, NT>);
    else run(k_exhaustive<8, TW, NT>);
  }
}

template <int TW>
void launch_tw(ExhArgs& a, const IndexView& ix, uint32_t max_d, uint32_t sms, uint32_t nt,
               bool warp_switch, cudaStream_t st, const char* name) {
  constexpr uint32_t kRowBytes = TW * 4, GL = TW / 4, kTileBinsT = TW * 32;
  a.n_tiles = (uint32_t)((ix.num_bins_pad + kTileBinsT - 1) / kTileBinsT);
  a.sms = sms;
  a.c_row = kRowBytes;
  // the largest CTA up to the built size whose tile and group slots fit in
  // shared memory
  const size_t tile_bytes = (size_t)(ix.r4 + 2) * kRowBytes;
  uint32_t threads = nt;
  const size_t scratch = warp_switch ? kScratchBytes<TW> : 0;  // per warp
  auto smem_of = [&](uint32_t t) {
    return tile_bytes + (size_t)(t / GL) * a.slot_bytes + 32 + t / 32 * scratch;
  };
  while (threads > 64 && smem_of(threads) > kSmemLimit) threads -= 32;
  const size_t smem = smem_of(threads);
  // small batches on few tiles need fewer CTAs (graph launches size for the
  // largest batch and let surplus CTAs find no work)
  uint32_t grid = sms;
  if (!a.live.on) {
    const uint32_t per_item = 64;
    const uint64_t items = (uint64_t)a.n_tiles * ((a.rv.n_reads + per_item - 1) / per_item);
    if (items < grid) grid = (uint32_t)(items ? items : 1);
  }
  if (nt == 512) launch_nt<TW, 512>(a, smem, threads, grid, max_d, warp_switch, st, name);
  else if (nt == 768) launch_nt<TW, 768>(a, smem, threads, grid, max_d, warp_switch, st, name);
  else launch_nt<TW, 640>(a, smem, threads, grid, max_d, warp_switch, st, name);
}

}  // namespace

uint32_t exhaustive_tile_bins(uint32_t r4) { return r4 <= 1024 ? 32u * 32u : 8u * 32u; }

bool exhaustive_shape_ok(const ExhShape& s) {
  const bool t_ok = s.threads == 0 || s.threads == 512 || s.threads == 640 || s.threads == 768;
  const bool r_ok = s.range_kb == 0 || (s.range_kb >= 1024 && s.range_kb <= (4u << 20));
  const bool w_ok = s.read_switch <= 2;
  return t_ok && r_ok && w_ok;
}

// A handful of reads go to k_exhaustive_few: it loads about n_reads * tokens
// rows, the staged kernel all 4^q, each once.  Measured on GB300 (few /
// staged, us): 3.1 Gbp coarse table at q = 5, mixed reads of an index for
// 250 bp, 1 read 14 / 230, 8 97 / 273, 16 153 / 279, 24 197 / 325, 32 372 /
// 341; 100 bp, 16 135 / 263, 48 290 / 321, 64 374 / 354; its fine table, 16
// 218 / 449, 64 607 / 603; q = 6, 64 165 / 361.  Tables that L2 holds stage
// as fast (50 Mbp: 18 / 15 at 16 reads).
uint32_t exhaustive_few_reads(const IndexView& ix, uint32_t ts) {
  return (uint64_t)ix.r4 * ix.wpad * 4u >= kFewMinTable ? 4u * ix.r4 / ts : 0u;
}

void launch_exhaustive(const IndexView& ix, const ReadsView& rv, RecordsView rec, uint32_t bin_bits,
                       uint32_t max_d, Ctl* ctl, cudaStream_t st, bool fine, const uint32_t* order,
                       Live live, ExhShape shape) {
  if (rv.n_reads == 0) return;
  const char* prof_name = fine ? "exhaustive" : "exhaustive_coarse";
  int dev = 0, sms = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  if (sms <= 0) sms = 1;
  ExhArgs a{};
  a.ix = ix;
  a.rv = rv;
  a.rec = rec;
  a.bin_bits = bin_bits;
  a.live = live;
  // a slot row holds a read's first blocks: all of them for the 1024-bin
  // tiles; for the 256-bin tiles of q = 6, whose 128 KB tile leaves little
  // room for the sixteen groups' slots of a warp, as many (up to
  // kSlotBlocksNarrow) as fit beside the tile at the CTA size -- the later
  // blocks come from L2 (warps matter more than slot blocks: at 768-thread
  // CTAs 1 block let 24 warps per SM fit, 7 blocks 11)
  const uint32_t nt = shape.threads ? shape.threads : kDefaultThreads;
  const uint32_t blocks = rv.ts / kBlockTokens;
  // slots of consecutive groups start 32 bytes apart modulo 128, so the
  // groups of a warp mostly read their tokens from different banks
  auto slot_bytes_of = [](uint32_t slot_blocks) {
    return (2u * slot_blocks * kBlockTokens * 2u + 127u) / 128u * 128u + 32u;
  };
  if (ix.r4 <= 1024) {
    a.slot_blocks = blocks;
  } else {
    const size_t tile_bytes = (size_t)(ix.r4 + 2) * 8u * 4u;
    const uint32_t groups = nt / 2u;  // 2-lane groups
    a.slot_blocks = 1;
    for (uint32_t sb = min(blocks, kSlotBlocksNarrow); sb > 1; --sb)
      if (tile_bytes + (size_t)groups * slot_bytes_of(sb) + 32 + nt / 32 * kScratchBytes<8> <=
          kSmemLimit) {
        a.slot_blocks = sb;
        break;
      }
  }
  a.row_stride = a.slot_blocks * kBlockTokens * 2u;
  a.slot_bytes = slot_bytes_of(a.slot_blocks);
  a.c_one = 1u;
  a.c_minus_two = 0u - 2u;
  a.c_hi = 65536u;
  a.c_lo = 0u - 65536u;
  a.range_bytes = shape.range_kb ? (uint64_t)shape.range_kb << 10 : kDefaultRangeBytes;
  a.ctl = ctl;
  // A graph launch decides by the batch's own count (k_plan_control leaves
  // ctl->path 0 for a few reads), so it enqueues both kernels.  (A count check
  // inside the staged kernel itself cost it 2.4% of its loop's schedule.)
  a.few_reads = exhaustive_few_reads(ix, rv.ts);
  if (a.few_reads && (live.on || rv.n_reads <= a.few_reads)) {
    const uint64_t n = min(rv.n_reads, a.few_reads);
    const uint64_t items = (ix.wpad + 127) / 128 * n;
    const uint64_t need = (items + kFewThreads / 32 - 1) / (kFewThreads / 32);
    const uint64_t most = (uint64_t)sms * 2;
    const unsigned grid = (unsigned)(need < most ? need : most);
    {
      ProfScope ps(prof_name, st);
      if (max_d < 32) k_exhaustive_few<5><<<grid, kFewThreads, 0, st>>>(a);
      else k_exhaustive_few<8><<<grid, kFewThreads, 0, st>>>(a);
    }
    if (!live.on || rv.n_reads <= a.few_reads) return;
  }
  a.order = order;
  a.pad_pair = rowPad(ix.r4) | (rowPad(ix.r4) << 16);
  a.check_shift = fine ? kMetaCheckFine : kMetaCheckCoarse;
  const bool ws = shape.read_switch == GRIM_SWITCH_WARP;
  // q <= 4: four times the bins fit a tile, a warp runs one read over all of
  // them, and a CTA has four times the rounds between two waits for a tile (500
  // reads at q = 4 are 6.25 rounds of its warps on 1024 bins, run as 7).  Where
  // there are tiles enough for every SM.  Existence counts of 500 reads against
  // 6.6M bins, six budgets: 9.3 -> 8.9 ms.
  if (ws && ix.r4 <= 256 && ix.num_bins_pad / 4096 >= (uint64_t)sms)
    launch_tw<128>(a, ix, max_d, (uint32_t)sms, nt, ws, st, prof_name);
  else if (ix.r4 <= 1024) launch_tw<32>(a, ix, max_d, (uint32_t)sms, nt, ws, st, prof_name);
  else launch_tw<8>(a, ix, max_d, (uint32_t)sms, nt, ws, st, prof_name);
}

}  // namespace grim
