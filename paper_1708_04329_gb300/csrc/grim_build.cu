// Index build (§GRIM-Filter: the reference is scanned once and every bin's
// bit vector is set from the tokens that occur in it; Fig. 2):
//   k_build_fused       q = 5, 6: ASCII straight to bin-major vectors and both
//                       token-major tables in one pass
//   k_pack_ref          ASCII -> 2-bit codes + not-a-base mask (the kernels below)
//   k_build_bin_major   one warp per bin, bit vector in shared memory
//   k_build_token_major one CTA per 1024-bin tile, the tile's [4^q rows x tile
//                       words] bitmap in shared memory (q <= 4)
//   k_tm_from_bm        q = 5, 6: token-major (and coarse token-major) tiles
//                       as bit transposes of the bin-major vectors, ORed over
//                       the members of each super-bin for the coarse table,
//                       where k_build_fused does not write them
#include "grim_internal.cuh"

namespace grim {
namespace {

// A/C/G/T (either case) -> 0/1/2/3; `ok` false for any other byte.
// Clearing bit 5 folds lowercase letters only ('a' 0x61 -> 'A' 0x41); the
// 2-bit code of the folded letter is ((u >> 1) ^ (u >> 2)) & 3 for exactly
// A (0x41), C (0x43), G (0x47) and T (0x54).
__device__ __forceinline__ uint32_t base_code(uint32_t c, bool& ok) {
  uint32_t u = c & 0xDFu;
  ok = (u == 0x41u) | (u == 0x43u) | (u == 0x47u) | (u == 0x54u);
  return ((u >> 1) ^ (u >> 2)) & 3u;
}

// Thread t packs bases [32t, 32t+32): two code words and one mask word.
__global__ void k_pack_ref(const char* __restrict__ ref, uint64_t n, uint32_t* __restrict__ codes,
                           uint32_t* __restrict__ invalid, uint64_t n32) {
  uint64_t t = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x;
  if (t >= n32) return;
  uint64_t base = t * 32;
  uint8_t b[32];
  if (base + 32 <= n && ((reinterpret_cast<uintptr_t>(ref) & 15u) == 0)) {
    const uint4* p = reinterpret_cast<const uint4*>(ref + base);
    uint4 v0 = __ldg(p), v1 = __ldg(p + 1);
    uint32_t w[8] = {v0.x, v0.y, v0.z, v0.w, v1.x, v1.y, v1.z, v1.w};
#pragma unroll
    for (int i = 0; i < 32; ++i) b[i] = (uint8_t)(w[i >> 2] >> (8 * (i & 3)));
  } else {
#pragma unroll
    for (int i = 0; i < 32; ++i) b[i] = (base + i < n) ? (uint8_t)ref[base + i] : (uint8_t)'N';
  }
  uint32_t c0 = 0, c1 = 0, inv = 0;
#pragma unroll
  for (int i = 0; i < 32; ++i) {
    bool ok;
    uint32_t c = base_code(b[i], ok);
    if (!ok) { inv |= 1u << i; c = 0; }
    if (i < 16) c0 |= c << (30 - 2 * i);
    else c1 |= c << (30 - 2 * (i - 16));
  }
  codes[2 * t] = c0;
  codes[2 * t + 1] = c1;
  invalid[t] = inv;
}

// Token starting at reference position p, or -1 if one of its q bases is not
// a base.  Needs p + q <= n (the packed arrays carry one spare word).
__device__ __forceinline__ int32_t token_at(const uint32_t* __restrict__ codes,
                                            const uint32_t* __restrict__ invalid, uint64_t p,
                                            uint32_t q) {
  uint64_t k = p >> 4;
  uint64_t w = ((uint64_t)__ldg(codes + k) << 32) | __ldg(codes + k + 1);
  uint32_t tok = (uint32_t)((w << (2 * (p & 15))) >> (64 - 2 * q));
  uint64_t m = p >> 5;
  uint64_t iw = (uint64_t)__ldg(invalid + m) | ((uint64_t)__ldg(invalid + m + 1) << 32);
  uint32_t bad = (uint32_t)(iw >> (p & 31)) & ((1u << q) - 1u);
  return bad ? -1 : (int32_t)tok;
}

// One warp per bin: set bit t of the bin's vector for every token wholly
// inside window [bB, min(bB+B+ext, n)).
__global__ void k_build_bin_major(const uint32_t* __restrict__ codes,
                                  const uint32_t* __restrict__ invalid, IndexView ix,
                                  uint32_t* __restrict__ bm) {
  extern __shared__ uint32_t s_vec[];  // [warps][wpb]
  const uint32_t warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const uint64_t b = blockIdx.x * (uint64_t)(blockDim.x >> 5) + warp;
  uint32_t* v = s_vec + warp * ix.wpb;
  for (uint32_t i = lane; i < ix.wpb; i += 32) v[i] = 0;
  __syncwarp();
  if (b < ix.num_bins) {
    uint64_t lo = b * ix.B;
    uint64_t hi = lo + ix.B + ix.ext;
    if (hi > ix.n) hi = ix.n;
    for (uint64_t p = lo + lane; p + ix.q <= hi; p += 32) {
      int32_t t = token_at(codes, invalid, p, ix.q);
      if (t >= 0) atomicOr(v + (t >> 5), 1u << (t & 31));
    }
  }
  __syncwarp();
  if (b < ix.num_bins)
    for (uint32_t i = lane; i < ix.wpb; i += 32) bm[b * ix.wpb + i] = v[i];
}

// One CTA per tile of tile_words*32 bins: every q-gram start p that lies in a
// window of the tile's bins sets its token's bit in each bin b whose window
// holds it, i.e. b*B <= p and p+q <= b*B+B+ext.
__global__ void __launch_bounds__(512) k_build_token_major(const uint32_t* __restrict__ codes,
                                                           const uint32_t* __restrict__ invalid,
                                                           IndexView ix, uint32_t tile_words,
                                                           uint32_t* __restrict__ tm) {
  extern __shared__ uint32_t s_tile[];  // [r4][tile_words]
  const uint32_t nwords = ix.r4 * tile_words;
  for (uint32_t i = threadIdx.x; i < nwords; i += blockDim.x) s_tile[i] = 0;
  __syncthreads();
  const uint64_t b0 = (uint64_t)blockIdx.x * tile_words * 32;
  uint64_t b1 = b0 + (uint64_t)tile_words * 32;
  if (b1 > ix.num_bins) b1 = ix.num_bins;
  if (b0 < b1) {
    const uint64_t p_lo = b0 * ix.B;
    // last start: p + q <= min(n, (b1-1)*B + B + ext)
    uint64_t end = b1 * ix.B + ix.ext;
    if (end > ix.n) end = ix.n;
    for (uint64_t p = p_lo + threadIdx.x; p + ix.q <= end; p += blockDim.x) {
      int32_t t = token_at(codes, invalid, p, ix.q);
      if (t < 0) continue;
      const uint64_t x = p + ix.q;
      uint64_t lo = x >= (uint64_t)ix.ext + 1 ? (x - ix.ext - 1) / ix.B : 0;
      uint64_t hi = p / ix.B;
      if (lo < b0) lo = b0;
      if (hi > b1 - 1) hi = b1 - 1;
      for (uint64_t b = lo; b <= hi; ++b) {
        uint32_t rel = (uint32_t)(b - b0);
        atomicOr(s_tile + (uint32_t)t * tile_words + (rel >> 5), 1u << (rel & 31));
      }
    }
  }
  __syncthreads();
  const uint64_t w0 = (uint64_t)blockIdx.x * tile_words;
  for (uint32_t i = threadIdx.x; i < nwords; i += blockDim.x) {
    uint32_t t = i / tile_words, w = i % tile_words;
    tm[(uint64_t)t * ix.wpad + w0 + w] = s_tile[i];
  }
}

template <int J>
__device__ __forceinline__ void transpose_round(uint32_t (&x)[32], uint32_t m) {
#pragma unroll
  for (int k = 0; k < 32; ++k) {
    if ((k & J) == 0) {
      const uint32_t t = ((x[k] >> J) ^ x[k + J]) & m;
      x[k + J] ^= t;
      x[k] ^= t << J;
    }
  }
}

// In-register transpose of a 32x32 bit matrix: on entry bit j of x[k] is
// element (k, j); on exit bit k of x[j] is.  Five rounds swap the
// off-diagonal halves of ever smaller diagonal blocks.
__device__ __forceinline__ void transpose32(uint32_t (&x)[32]) {
  transpose_round<16>(x, 0x0000FFFFu);
  transpose_round<8>(x, 0x00FF00FFu);
  transpose_round<4>(x, 0x0F0F0F0Fu);
  transpose_round<2>(x, 0x33333333u);
  transpose_round<1>(x, 0x55555555u);
}

// Token-major tile from the bin-major table (q >= 5, so a bin vector is a
// whole number of 32-word chunks).  One CTA of 32 warps per tile of TW*32
// (super-)bins; warp u takes bin group g = u % TW (32 bins) and token chunk
// c = u / TW (1024 tokens).  Lane l loads word 32c + l of each of the
// group's 32 vectors -- for a super-bin the OR of its f member bins, which
// is exactly the super-bin's vector (its window is the union of theirs) --
// transposes the 32x32 bits in registers, and leaves token rows in shared
// memory (row t at t*TW + (t >> 5): one padding word per 32 rows keeps the
// lanes' stores in distinct banks); the CTA then writes each token row's TW
// words to the token-major table.
template <int TW>
__global__ void __launch_bounds__(1024) k_tm_from_bm(const uint32_t* __restrict__ bm,
                                                     uint32_t wpb, uint32_t f, uint64_t units,
                                                     uint32_t r4, uint64_t wpad,
                                                     uint32_t* __restrict__ tm) {
  extern __shared__ uint32_t s_rows[];
  const uint32_t lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const uint32_t g = warp % TW, c = warp / TW;
  const uint64_t u0 = (uint64_t)blockIdx.x * TW * 32 + g * 32;  // first unit of the group
  uint32_t x[32];
#pragma unroll
  for (int k = 0; k < 32; ++k) {
    const uint64_t u = u0 + k;
    uint32_t w = 0;
    if (u < units)
      for (uint32_t m = 0; m < f; ++m) w |= __ldg(bm + (u * f + m) * wpb + c * 32 + lane);
    x[k] = w;
  }
  transpose32(x);  // x[j]: token 32*(32c + lane) + j, bit k = unit u0 + k
#pragma unroll
  for (int j = 0; j < 32; ++j) {
    const uint32_t t = 32u * (32u * c + lane) + j;
    s_rows[t * TW + g + (t >> 5)] = x[j];
  }
  __syncthreads();
  const uint64_t col0 = (uint64_t)blockIdx.x * TW;
  for (uint32_t i = threadIdx.x; i < r4 * TW; i += blockDim.x) {
    const uint32_t t = i / TW, col = i % TW;
    tm[(uint64_t)t * wpad + col0 + col] = s_rows[t * TW + col + (t >> 5)];
  }
}

// The number of set bits of each token row, i.e. how many (super-)bins hold
// the token: one CTA per row, 16 bytes a load (rows are whole 128-byte lines),
// four loads in flight a thread (0.17 ms for 1 GB; 0.45 with 4-byte loads).
__global__ void __launch_bounds__(512) k_row_popcount(const uint32_t* __restrict__ tm,
                                                      uint64_t words,
                                                      uint32_t* __restrict__ presence) {
  __shared__ unsigned long long part[32];
  const uint4* row = reinterpret_cast<const uint4*>(tm + (uint64_t)blockIdx.x * words);
  const uint64_t n = words / 4;
  unsigned long long c = 0;
#pragma unroll 4
  for (uint64_t i = threadIdx.x; i < n; i += blockDim.x) {
    const uint4 v = __ldg(row + i);
    c += __popc(v.x) + __popc(v.y) + __popc(v.z) + __popc(v.w);
  }
  for (int o = 16; o > 0; o >>= 1) c += __shfl_xor_sync(0xFFFFFFFFu, c, o);
  if ((threadIdx.x & 31) == 0) part[threadIdx.x >> 5] = c;
  __syncthreads();
  if (threadIdx.x < 32) {
    c = threadIdx.x < blockDim.x / 32 ? part[threadIdx.x] : 0ull;
    for (int o = 16; o > 0; o >>= 1) c += __shfl_xor_sync(0xFFFFFFFFu, c, o);
    if (threadIdx.x == 0) presence[blockIdx.x] = (uint32_t)(c > 0xFFFFFFFFull ? 0xFFFFFFFFull : c);
  }
}

// A token's rank among the tokens of its class (token % classes): how many of
// them fewer (super-)bins hold, ties by value; and the share of the `units`
// (super-)bins without it.  A warp per token, bound by the latency of its loads:
// with a thread per token the walk over the class took 37 us at q = 5, longer
// than the other kernels of a small build, this 12 (a launch that does nothing
// reads 5; 1 Mbp, B = 200, whole call 241 -> 211 us).
constexpr uint32_t kRanksWarps = 8;
__global__ void __launch_bounds__(kRanksWarps * 32) k_token_ranks(
    const uint32_t* __restrict__ presence, uint32_t rows, uint32_t classes, float units,
    uint16_t* __restrict__ rank, float* __restrict__ miss) {
  const uint32_t t = blockIdx.x * kRanksWarps + (threadIdx.x >> 5), lane = threadIdx.x & 31;
  if (t >= rows) return;
  const uint32_t mine = __ldg(presence + t);
  uint32_t r = 0;
#pragma unroll 16
  for (uint32_t i = t % classes + lane * classes; i < rows; i += 32 * classes) {
    const uint32_t p = __ldg(presence + i);
    r += p < mine || (p == mine && i < t);
  }
  r = __reduce_add_sync(0xFFFFFFFFu, r);
  if (lane == 0) {
    rank[t] = (uint16_t)r;
    miss[t] = fmaxf(0.f, 1.f - (float)mine / units);
  }
}

// 16 bases (bytes, first base lowest) to a code word (first base in the top
// bits) and a not-a-base mask.  A letter is a base iff folding its case and
// looking its 2-bit code up in "ACGT" gives it back.
__device__ __forceinline__ void pack16(const uint4& v, uint32_t& code, uint32_t& inv) {
  const uint32_t w[4] = {v.x, v.y, v.z, v.w};
  uint32_t x[4], m[4];
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const uint32_t u = w[i] & 0xDFDFDFDFu;
    const uint32_t c = ((u >> 1) ^ (u >> 2)) & 0x03030303u;
    uint32_t sel = (c | (c >> 4)) & 0x00FF00FFu;
    sel |= sel >> 8;  // the four codes as byte selectors (low 16 bits)
    x[i] = __byte_perm(0x54474341u, 0u, sel & 0xFFFFu) ^ u;
    m[i] = c * 0x40100401u;  // top byte: the four codes side by side, the first on top
  }
  code = __byte_perm(__byte_perm(m[3], m[2], 0x0073u), __byte_perm(m[1], m[0], 0x0073u), 0x5410u);
  inv = 0;
  if (x[0] | x[1] | x[2] | x[3]) {
#pragma unroll
    for (int k = 0; k < 16; ++k)
      if ((x[k >> 2] >> (8 * (k & 3))) & 0xFFu) inv |= 1u << k;
  }
}

// The whole build of a tile of kFusedBins bins by one CTA (q = 5, 6), from the
// reference's letters:
//   1. the tile's letters become 2-bit codes and a not-a-base mask in shared
//      memory (SWAR, 16 letters a thread and load);
//   2. each warp walks the cores (B positions) of its run of 32 bins and the
//      k + 1 cores after it, and sets the tokens starting in a core in a
//      vector of its own: P, those of the first `rem` positions, then A, all
//      of them.  A q-gram lies inside bin b's window iff it starts in
//      [bB, bB + B + ext - q], which with ext - q + 1 = k B + rem is
//      A(b) | ... | A(b + k) | P(b + k + 1): every token is set once, not once
//      for each of the bins whose windows overlap there;
//   3. (q = 5) the run's 32 vectors, one word a lane, are a 32 x 32 bit
//      transpose away from the token rows; both token-major tables leave
//      through shared memory in row pieces of 64 and 64 / f bytes.  At q = 6
//      the tile's 256 KB of vectors do not fit there: each thread reads the
//      words it has just written back from L2, 1024 tokens a pass.
// Bound by instruction issue (235 warp instructions a bin, 70% of the issue
// slots; the shared atomics take 29% of their pipe), not by its 8.1 GB of
// letters and tables at 3.1 Gbp, B = 200, q = 5: 4.1 ms there (4.3 with the
// runs' masks worked out for every core).  Packing the reference, setting each
// bin's bits from the codes and two transposes from DRAM took 16.0 ms.
// q = 6, 1.5 Gbp, B = 100: 6.2 ms for all tables (17.6 GB, 2.6 ms of copying;
// 295 instructions a bin, 58% of the slots, and the 64-byte row pieces), 13.5
// with the token rows and the super-bins' as transposes from DRAM, 2.6 for the
// vectors alone.
constexpr uint32_t kFusedBins = 512, kFusedWarps = kFusedBins / 32, kFusedMaxK = 3;
constexpr uint32_t kFusedGroups = kFusedBins / 32;  // tile words of a token row

struct FusedArgs {
  const char* ref;
  uint64_t n, num_bins, wpad, cwpad;
  uint32_t B, q, k, rem;
  uint32_t code_words;  // code words of the tile in shared memory (16 bases each)
  uint32_t region_words;  // shared memory before the warps' vectors
  uint32_t f;           // coarse factor (ctm set: 2, 4, 8 or 16; q = 6: 8 or 16)
  uint32_t* bm;
  uint32_t* tm;
  uint32_t* ctm;
};

// shared memory, in words.  q = 5: the tile's vectors, later row pieces; codes
// and mask, later the coarse row pieces; a vector per warp.  q = 6: codes and
// mask, later the row pieces of a token chunk and the super-bins' vectors; a
// vector per warp.
constexpr uint32_t kFusedRowWords = 1024u * kFusedGroups + 32u;
__host__ __device__ constexpr uint32_t fused_super_words(uint32_t f) {  // q = 6
  return f ? 4u * 32u * (kFusedBins / f) : 0u;
}

// WPL: words of a vector per lane, 1 (q = 5) or 4 (q = 6); K >= k; ROWS: the
// token rows too (at q = 6 a kernel of its own: their shared memory and code
// cost the vectors alone 7%)
template <uint32_t WPL, uint32_t K, bool ROWS>
__global__ void __launch_bounds__(kFusedWarps * 32, 2) k_build_fused(FusedArgs a) {
  extern __shared__ uint32_t s_fused[];
  uint32_t* s_rows = s_fused;
  uint32_t* s_code = s_fused + (WPL == 1 ? kFusedRowWords : 0u);
  uint16_t* inv16 = reinterpret_cast<uint16_t*>(s_code + a.code_words);  // 16 positions each
  uint32_t* s_vec = s_fused + a.region_words;
  const uint32_t tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const uint64_t bin0 = (uint64_t)blockIdx.x * kFusedBins;
  const uint64_t p0 = bin0 * a.B;  // a multiple of 512: 16-byte aligned in an aligned reference
  // 1. letters -> codes; positions past the reference are not bases
  bool any = false;
  const bool aligned = (reinterpret_cast<uintptr_t>(a.ref) & 15u) == 0;
  for (uint32_t i = tid; i < a.code_words; i += kFusedWarps * 32) {
    const uint64_t p = p0 + 16ull * i;
    uint32_t code = 0, inv = 0xFFFFu;
    if (aligned && p + 16 <= a.n) {
      pack16(__ldg(reinterpret_cast<const uint4*>(a.ref + p)), code, inv);
    } else if (p < a.n) {
      uint32_t w[4] = {0, 0, 0, 0};
      for (uint32_t j = 0; j < 16 && p + j < a.n; ++j)
        w[j >> 2] |= (uint32_t)(uint8_t)a.ref[p + j] << (8 * (j & 3));
      pack16(make_uint4(w[0], w[1], w[2], w[3]), code, inv);  // 0 is not a base
    }
    s_code[i] = code;
    inv16[i] = (uint16_t)inv;
    any |= inv != 0;
  }
  uint32_t* v = s_vec + warp * 32 * WPL;
#pragma unroll
  for (uint32_t w = 0; w < WPL; ++w) v[w * 32 + lane] = 0;
  any = __syncthreads_or(any);

  // 2. tokens starting at tile positions [lo, lo + len) into the warp's
  // vector: a lane takes `per` consecutive positions (a run), whose
  // per + q - 1 <= 16 bases it aligns into one register, so a token costs two
  // shifts for its bit, a shift and a mask for its word, and the atomic
  constexpr uint32_t kQ = WPL == 1 ? 5u : 6u, kMost = 17u - kQ;  // positions per lane
  constexpr uint32_t kBitShift = 32u - 2u * kQ, kWordMask = ((1u << (2u * kQ - 5u)) - 1u) << 2;
  const uint32_t v_base = (uint32_t)__cvta_generic_to_shared(v);
  auto set_run = [&](uint32_t p, uint32_t ok, uint32_t per) {
    const uint32_t* c = s_code + (p >> 4);
    const uint32_t x = __funnelshift_l(c[1], c[0], 2u * p);
    if (any) {
      const uint16_t* m16 = inv16 + (p >> 4);
      const uint32_t m = ((uint32_t)m16[0] | ((uint32_t)m16[1] << 16)) >> (p & 15u);
      uint32_t bad = m;
#pragma unroll
      for (uint32_t i = 1; i < kQ; ++i) bad |= m >> i;
      ok &= ~bad;
    }
    auto set = [&](uint32_t i) {
      asm volatile(
          "{\n.reg .pred p;\nsetp.ne.u32 p, %2, 0;\n@p red.shared.or.b32 [%0], %1;\n}" ::"r"(
              v_base + ((x >> (kBitShift + 3u - 2u * i)) & kWordMask)),
          "r"(1u << ((x >> (kBitShift - 2u * i)) & 31u)), "r"(ok & (1u << i))
          : "memory");
    };
#pragma unroll
    for (uint32_t i = 0; i < 3; ++i) set(i);
    if (per > 3) set(3);
    if (per > 4) {
#pragma unroll
      for (uint32_t i = 4; i < 8; ++i) set(i);
    }
    if (per > 8) {
#pragma unroll
      for (uint32_t i = 8; i < kMost; ++i) set(i);
    }
  };
  // a lane's first run in a core's first `rem` positions and in the rest: its
  // offset (0 for a lane without one) and which of its tokens exist
  const uint32_t rest = a.B - a.rem;
  const uint32_t per_p = max(1u, min(kMost, (a.rem + 31u) / 32u));
  const uint32_t per_r = min(kMost, (rest + 31u) / 32u);
  auto mask_of = [&](uint32_t at, uint32_t len, uint32_t per) {
    return at < len ? (1u << min(per, len - at)) - 1u : 0u;
  };
  const uint32_t ok_p = mask_of(lane * per_p, a.rem, per_p), at_p = ok_p ? lane * per_p : 0u;
  const uint32_t ok_r = mask_of(lane * per_r, rest, per_r), at_r = ok_r ? lane * per_r : 0u;
  auto set_tokens = [&](uint32_t lo, uint32_t len, uint32_t per, uint32_t at, uint32_t ok) {
    set_run(lo + at, ok, per);
    if (len > 32u * per)  // (more than 32 lanes' runs)
      for (at += 32u * per; at < len; at += 32u * per)
        set_run(lo + at, mask_of(at, len, per), per);
  };
  uint32_t pend[K + 1][WPL];  // bins c - k .. c so far (newest first)
#pragma unroll
  for (uint32_t i = 0; i <= K; ++i)
#pragma unroll
    for (uint32_t w = 0; w < WPL; ++w) pend[i][w] = 0;
  const uint32_t first = warp * 32;
  // this run's bins in the bin-major table
  const uint32_t rows = a.bm && bin0 + first < a.num_bins
                            ? (uint32_t)min((uint64_t)32u, a.num_bins - bin0 - first)
                            : 0u;
  uint32_t* out = a.bm + (bin0 + first) * (32 * WPL) + lane;
  uint32_t lo = first * a.B;
  for (uint32_t c = 0; c <= 32 + a.k; ++c, lo += a.B) {
    set_tokens(lo, a.rem, per_p, at_p, ok_p);
    __syncwarp();
    // core c's first positions complete bin c - k - 1
    if (c > a.k) {
      const uint32_t done = c - a.k - 1;
#pragma unroll
      for (uint32_t w = 0; w < WPL; ++w) {
        uint32_t x = v[w * 32 + lane];
#pragma unroll
        for (uint32_t i = 0; i <= K; ++i)
          if (i == a.k) x |= pend[i][w];
        if (done < rows) out[w * 32] = x;
        if (WPL == 1) s_rows[(first + done) * 32 + lane] = x;
      }
      out += 32 * WPL;
      if (done == 31) break;
      __syncwarp();  // the vector is read: the core's other tokens may be set
    }
    set_tokens(lo + a.rem, rest, per_r, at_r, ok_r);
    __syncwarp();
#pragma unroll
    for (uint32_t w = 0; w < WPL; ++w) {
      const uint32_t x = v[w * 32 + lane];
      v[w * 32 + lane] = 0;
#pragma unroll
      for (uint32_t i = K; i > 0; --i) pend[i][w] = pend[i - 1][w] | x;
      pend[0][w] = x;
    }
    __syncwarp();
  }
  if (!ROWS || (!a.tm && !a.ctm)) return;

  // 3. (q = 6) 1024 tokens at a time, a thread's words of its run's vectors
  // come back from L2, where it has just written them
  if constexpr (WPL == 4 && ROWS) {
    uint32_t* s_super = s_rows + kFusedRowWords;  // [chunk][super-bin of the tile][lane]
    const uint32_t supers = a.ctm ? kFusedBins / a.f : 0u;
    const uint32_t* in = a.bm + (bin0 + first) * 128 + lane;
    const uint64_t col0 = (uint64_t)blockIdx.x * kFusedGroups;
#pragma unroll 1
    for (uint32_t c = 0; c < 4; ++c) {
      uint32_t x[32];
#pragma unroll
      for (uint32_t k = 0; k < 32; ++k) x[k] = k < rows ? __ldcg(in + k * 128 + c * 32) : 0u;
      __syncthreads();  // codes, or the last chunk's rows, are no longer read
      if (supers) {
        uint32_t* to = s_super + (c * supers + first / a.f) * 32 + lane;
        uint32_t w = 0;
#pragma unroll
        for (uint32_t k = 0; k < 32; ++k) {
          w |= x[k];
          if (((k + 1) & (a.f - 1)) == 0) {
            *to = w;
            to += 32;
            w = 0;
          }
        }
      }
      if (col0 >= a.wpad) continue;
      transpose32(x);
#pragma unroll
      for (uint32_t j = 0; j < 32; ++j) s_rows[(32u * lane + j) * kFusedGroups + warp + lane] = x[j];
      __syncthreads();
      uint32_t* dst = a.tm + (1024u * c + tid / kFusedGroups) * a.wpad + col0 + tid % kFusedGroups;
#pragma unroll 8
      for (uint32_t j = 0; j < 32; ++j, dst += 32 * a.wpad)
        *dst = s_rows[tid + j * (32 * kFusedGroups + 1)];
    }
    __syncthreads();
    const uint32_t words = supers / 32;  // of a coarse row
    const uint64_t ccol0 = (uint64_t)blockIdx.x * words;
    if (ccol0 < a.cwpad) {
      for (uint32_t i = warp; i < 4 * words; i += kFusedWarps) {
        uint32_t x[32];
#pragma unroll
        for (uint32_t k = 0; k < 32; ++k)
          x[k] = s_super[(i / words * supers + i % words * 32 + k) * 32 + lane];
        transpose32(x);
        uint32_t* dst = a.ctm + (1024u * (i / words) + 32u * lane) * a.cwpad + ccol0 + i % words;
#pragma unroll
        for (uint32_t j = 0; j < 32; ++j, dst += a.cwpad) *dst = x[j];
      }
    }
    return;
  }

  // 3. token rows: the coarse table's from the ORs of f vectors, then the bins'
  __syncthreads();  // vectors complete, codes no longer read
  uint32_t* s_coarse = s_code;
  const uint32_t cgroups = a.ctm ? kFusedGroups / a.f : 0u;  // row words of the tile's super-bins
  uint32_t x[32];
  if (warp < cgroups) {
#pragma unroll
    for (uint32_t k = 0; k < 32; ++k) {
      uint32_t w = 0;
      for (uint32_t m = 0; m < a.f; ++m) w |= s_rows[((warp * 32 + k) * a.f + m) * 32 + lane];
      x[k] = w;
    }
    transpose32(x);
#pragma unroll
    for (uint32_t j = 0; j < 32; ++j) s_coarse[(32u * lane + j) * cgroups + warp + lane] = x[j];
  }
#pragma unroll
  for (uint32_t k = 0; k < 32; ++k) x[k] = s_rows[(first + k) * 32 + lane];
  transpose32(x);
  __syncthreads();  // every vector is in registers
  if (a.tm) {
#pragma unroll
    for (uint32_t j = 0; j < 32; ++j) s_rows[(32u * lane + j) * kFusedGroups + warp + lane] = x[j];
  }
  __syncthreads();
  // a thread keeps its column and steps down the rows
  static_assert(kFusedWarps * 32 == 32 * kFusedGroups, "one pass covers 32 token rows");
  const uint64_t col0 = (uint64_t)blockIdx.x * kFusedGroups;
  if (a.tm && col0 < a.wpad) {
    uint32_t* dst = a.tm + (uint64_t)(tid / kFusedGroups) * a.wpad + col0 + tid % kFusedGroups;
#pragma unroll 8
    for (uint32_t j = 0; j < 32; ++j, dst += 32 * a.wpad)
      *dst = s_rows[tid + j * (32 * kFusedGroups + 1)];
  }
  const uint64_t ccol0 = (uint64_t)blockIdx.x * cgroups;
  if (cgroups && ccol0 < a.cwpad) {
    const uint32_t per = kFusedWarps * 32 / cgroups;  // rows of a pass: 32 f
    uint32_t t = tid / cgroups;
    uint32_t* dst = a.ctm + (uint64_t)t * a.cwpad + ccol0 + tid % cgroups;
#pragma unroll 4
    for (uint32_t i = tid; i < 1024u * cgroups; i += kFusedWarps * 32, t += per, dst += per * a.cwpad)
      *dst = s_coarse[i + (t >> 5)];
  }
}

}  // namespace

void launch_tm_from_bm(const uint32_t* bm, const IndexView& unit_view, uint32_t wpb, uint32_t f,
                       uint32_t* tm, cudaStream_t st) {
  if (unit_view.num_bins == 0) return;
  const uint32_t r4 = unit_view.r4;
  const uint32_t tw = r4 <= 1024 ? 32u : 32768u / r4;  // tile words, as the filter's tiles
  const size_t smem = ((size_t)r4 * tw + r4 / 32) * sizeof(uint32_t);
  const uint64_t grid = unit_view.num_bins_pad / (tw * 32);
  ProfScope ps("transpose_token_major", st);
  if (tw == 32) {
    allow_smem(k_tm_from_bm<32>);
    k_tm_from_bm<32><<<(unsigned)grid, 1024, smem, st>>>(bm, wpb, f, unit_view.num_bins, r4,
                                                         unit_view.wpad, tm);
  } else {
    allow_smem(k_tm_from_bm<8>);
    k_tm_from_bm<8><<<(unsigned)grid, 1024, smem, st>>>(bm, wpb, f, unit_view.num_bins, r4,
                                                        unit_view.wpad, tm);
  }
}

void launch_presence(const uint32_t* tm, const IndexView& units, uint32_t* presence,
                     cudaStream_t st) {
  const uint32_t rows = units.r4;
  {
    ProfScope ps("row_popcount", st);
    k_row_popcount<<<rows, 512, 0, st>>>(tm, units.wpad, presence);
  }
  ProfScope ps("token_ranks", st);
  k_token_ranks<<<(rows + kRanksWarps - 1) / kRanksWarps, kRanksWarps * 32, 0, st>>>(
      presence, rows, rows > 1024 ? 4u : 1u, (float)units.num_bins, rank_table(presence, rows),
      miss_table(presence, rows));
}

namespace {
uint64_t fused_tile_words(const IndexView& v) {  // code words of a tile
  const uint32_t span = v.ext - v.q + 1;
  return ((uint64_t)(kFusedBins + span / v.B) * v.B + span % v.B + v.q + 15) / 16 + 1;
}
uint32_t fused_super_factor(uint32_t q, uint32_t f) {  // 0: not this kernel's
  // whole row words of super-bins in a tile; at q = 6 their vectors of all
  // 4096 tokens wait in shared memory (16 KB at f = 16, 128 KB at f = 2)
  return f > (q == 5 ? 1u : 7u) && kFusedGroups % f == 0 ? f : 0u;
}
uint32_t fused_region_words(const IndexView& v, uint32_t f, bool rows) {
  const uint32_t words = (uint32_t)fused_tile_words(v);
  const uint32_t codes = words + (words + 1) / 2 + 2;
  if (v.q == 5) return kFusedRowWords + std::max(codes, 1024u * (kFusedGroups / 2) + 32u);
  if (!rows) return codes;
  return std::max(codes, kFusedRowWords + fused_super_words(fused_super_factor(v.q, f)));
}
size_t fused_smem(const IndexView& v, uint32_t f, bool rows) {
  return sizeof(uint32_t) * (fused_region_words(v, f, rows) + kFusedWarps * v.wpb);
}
}  // namespace

uint32_t build_fused_layouts(const IndexView& v, uint32_t f) {
  if (v.q < 5 || (v.ext - v.q + 1) / v.B > kFusedMaxK || fused_tile_words(v) > 65536 ||
      fused_smem(v, f, true) > kSmemMost)
    return 0;
  return GRIM_LAYOUT_BIN_MAJOR | GRIM_LAYOUT_TOKEN_MAJOR |
         (fused_super_factor(v.q, f) ? GRIM_LAYOUT_COARSE : 0u);
}

void launch_build_fused(const char* ref, const IndexView& v, const IndexView& cv, uint32_t f,
                        uint32_t* bm, uint32_t* tm, uint32_t* ctm, cudaStream_t st) {
  const uint32_t span = v.ext - v.q + 1;
  FusedArgs a{};
  a.ref = ref;
  a.n = v.n;
  a.num_bins = v.num_bins;
  a.wpad = v.wpad;
  a.cwpad = cv.wpad;
  a.B = v.B;
  a.q = v.q;
  a.k = span / v.B;
  a.rem = span % v.B;
  a.code_words = (uint32_t)fused_tile_words(v);
  a.f = f;
  a.bm = bm;
  a.tm = tm;
  a.ctm = ctm;
  // tiles up to the padded ends of the rows (their vectors are zero there)
  uint64_t grid = (v.num_bins + kFusedBins - 1) / kFusedBins;
  if (tm) grid = v.num_bins_pad / kFusedBins;
  if (ctm && cv.num_bins_pad * f / kFusedBins > grid) grid = cv.num_bins_pad * f / kFusedBins;
  const bool rows = v.q == 5 || tm;
  a.region_words = fused_region_words(v, f, rows);
  const size_t smem = fused_smem(v, f, rows);
  ProfScope ps("build_fused", st);
  auto run = [&](auto kernel) {
    allow_smem(kernel);
    kernel<<<(unsigned)grid, kFusedWarps * 32, smem, st>>>(a);
  };
  const bool near = a.k <= 1;
  if (v.q == 5) run(near ? k_build_fused<1, 1, true> : k_build_fused<1, kFusedMaxK, true>);
  else if (rows) run(near ? k_build_fused<4, 1, true> : k_build_fused<4, kFusedMaxK, true>);
  else run(near ? k_build_fused<4, 1, false> : k_build_fused<4, kFusedMaxK, false>);
}

void launch_pack_ref(const char* ref, uint64_t n, uint32_t* codes, uint32_t* invalid,
                     cudaStream_t st) {
  uint64_t n32 = (n + 31) / 32;
  if (n32 == 0) return;
  ProfScope ps("pack_ref", st);
  k_pack_ref<<<(unsigned)((n32 + 255) / 256), 256, 0, st>>>(ref, n, codes, invalid, n32);
}

void launch_build_bin_major(const uint32_t* codes, const uint32_t* invalid, const IndexView& ix,
                            uint32_t* bm, cudaStream_t st) {
  if (ix.num_bins == 0) return;
  const uint32_t warps = 8;
  uint64_t grid = (ix.num_bins + warps - 1) / warps;
  ProfScope ps("build_bin_major", st);
  k_build_bin_major<<<(unsigned)grid, warps * 32, warps * ix.wpb * sizeof(uint32_t), st>>>(
      codes, invalid, ix, bm);
}

void launch_build_token_major(const uint32_t* codes, const uint32_t* invalid, const IndexView& ix,
                              uint32_t* tm, cudaStream_t st) {
  if (ix.num_bins == 0) return;
  // 128 KB of shared memory per tile: 32 words (1024 bins) up to q = 5,
  // 8 words (256 bins) at q = 6
  uint32_t tile_words = ix.r4 <= 1024 ? 32u : 32768u / ix.r4;
  size_t smem = (size_t)ix.r4 * tile_words * sizeof(uint32_t);
  allow_smem(k_build_token_major);
  uint64_t grid = (ix.num_bins_pad / 32) / tile_words;
  ProfScope ps("build_token_major", st);
  k_build_token_major<<<(unsigned)grid, 512, smem, st>>>(codes, invalid, ix, tile_words, tm);
}

}  // namespace grim
