// Candidate-list filter over the bin-major table (§GRIM-Filter: for each
// candidate location the mapper asks whether the bin holding it can possibly
// match; steps 2-3 and Fig. 5).
//
// GB300 mapping
// -------------
// * Warps claim chunks of 32-4096 consecutive candidates of the flattened lists
//   from a global counter (a chunk may hold many short lists; a long list is
//   spread over many warps, so no single 20,000-candidate list is left
//   running alone at the end).  For each read in its chunk the warp turns the
//   read's tokens into a multiplicity histogram (a byte per token value) and
//   then into bit planes P_k = {t : bit k of mult(t) is 1}, held in
//   registers, so that for any bin vector v the token sum is
//       sum = sum_k 2^k * popcount(v & P_k)
//   -- every position counts, repeats included, with a handful of AND +
//   POPC per 32 bits instead of one bit test per token.
// * Up to q = 5 a bin vector (4^q bits) is gathered by G lanes with 16-byte
//   loads (q = 5: 8 lanes x 16 B = 128 B, four candidates per warp step).  The
//   U vectors of a step are reduced over the lane group together (a butterfly
//   that halves the sums at each exchange), compared with
//   T = (L-q+1) - q*e, and one ballot places the passes.
// * At q = 6 (512-byte vectors) k_candidates_lookup looks up the read's tokens
//   instead, few lines of a vector at a time, and batches of reads with large
//   budgets go by whole vectors (lists_by_planes).
// * The path is random reads of 128-byte lines per (read, bin) pair: bound by
//   HBM, not by arithmetic.
#include "grim_internal.cuh"

namespace grim {
namespace {

template <int WPB>
struct Cfg {
  static constexpr int WL = WPB >= 4 ? 4 : WPB;  // words per lane
  static constexpr int G = WPB / WL;             // lanes per candidate
  static constexpr int CPW = 32 / G;             // candidates per warp step
};

template <int WL>
__device__ __forceinline__ void load_words(const uint32_t* p, uint32_t (&v)[WL]) {
  if constexpr (WL == 4) {
    // a vector is read once: it need not displace the ids and token rows in L1
    // (330M candidates: 8.66 -> 8.58 ms)
    asm("ld.global.nc.L1::no_allocate.v4.u32 {%0,%1,%2,%3}, [%4];"
        : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3])
        : "l"(p));
  } else if constexpr (WL == 2) {
    const uint2 x = __ldg(reinterpret_cast<const uint2*>(p));
    v[0] = x.x; v[1] = x.y;
  } else {
    v[0] = __ldg(p);
  }
}

struct CandArgs {
  IndexView ix;
  ReadsView rv;
  const int32_t* cand;
  const uint64_t* cand_off;
  RecordsView rec;
  Ctl* ctl;
  Live live;
};

constexpr int kWarps = 8;
// gathers in flight per lane group when the caller leaves it to the library
// (the autotuner's choice on GB300 for 128-byte vectors)
constexpr uint32_t kDefaultCandUnroll = 2;
// and candidates in flight per warp for the look-ups in 512-byte vectors
// (98.9M candidates through a plan, ms at 1 / 2 / 4 / 8: e = 7 4.4 / 5.4 / 4.4 /
// 4.35, e = 0 3.4 / 4.9 / 3.4 / 3.2)
constexpr uint32_t kDefaultLookupUnroll = 8;
constexpr int kRegPlanes = 2;  // bit planes held in registers: multiplicities up to 3

// Multiplicities of 4 and more (bits kRegPlanes.. of a token's count) are
// rare; they are kept as further bit planes in shared memory
// (xplanes[k - kRegPlanes][word]).
// per-warp shared memory: the multiplicity histogram, then the higher planes
__host__ __device__ constexpr uint32_t hist_words_of(uint32_t r4) { return r4 >= 4 ? r4 / 4 : 1; }
__host__ __device__ constexpr uint32_t warp_smem_words(uint32_t r4, uint32_t wpb) {
  return hist_words_of(r4) + (8 - kRegPlanes) * wpb;
}

// The read's multiplicity histogram (byte t = how many of its positions hold
// token t) and its bit planes P_k = {t : bit k of mult(t)} for this lane's WL
// words of a bin vector: planes below kRegPlanes in registers, the rest in
// shared memory.  Returns K, the number of planes in use, and the read's threshold in *thr.
// Warp-collective.
template <int WPB, int WL>
__device__ __forceinline__ uint32_t build_planes(const ReadsView& rv, uint32_t r, uint32_t r4,
                                                 uint32_t* hist, uint32_t* xplanes, uint32_t lane,
                                                 uint32_t sub, uint32_t (&P)[kRegPlanes][WL],
                                                 uint32_t* thr) {
  constexpr int kPlanesBuilt = 8;
  const uint32_t hist_words = hist_words_of(r4);
  // the warp has finished reading the previous read's histogram
  __syncwarp();
  for (uint32_t i = lane; i < hist_words; i += 32) hist[i] = 0;
  __syncwarp();
  const uint32_t m = rv.meta[r];
  const uint32_t ntok = m & 0xFFu, dmax = (m >> 8) & 0xFFu;
  const uint16_t* tk = rv.tokens + (uint64_t)r * rv.copies * rv.ts;
  for (uint32_t j = lane; j < ntok; j += 32) {
    const uint32_t t = tk[j];
    if (t < r4) atomicAdd(hist + (t >> 2), 1u << (8 * (t & 3u)));
  }
  __syncwarp();
  // the largest multiplicity decides how many bit planes the sums need
  // (almost always 1 or 2)
  uint32_t mx = 0;
  for (uint32_t i = lane; i < hist_words; i += 32) {
    const uint32_t h = hist[i];
    mx = max(mx, max(max(h & 0xFFu, (h >> 8) & 0xFFu), max((h >> 16) & 0xFFu, h >> 24)));
  }
  mx = __reduce_max_sync(0xFFFFFFFFu, mx);
  const uint32_t K = 32 - __clz(mx);  // planes in use
#pragma unroll
  for (int w = 0; w < WL; ++w) {
    const uint32_t wi = sub * WL + w;  // word index in the vector: tokens wi*32 .. wi*32+31
    uint32_t hw[8];
#pragma unroll
    for (int j = 0; j < 8; ++j) {
      const uint32_t h = wi * 8 + j;
      hw[j] = h < hist_words && (wi * 32 + 4 * j) < r4 ? hist[h] : 0u;
    }
#pragma unroll
    for (int k = 0; k < kPlanesBuilt; ++k) {
      if ((uint32_t)k < K) {
        uint32_t pk = 0;
#pragma unroll
        for (int j = 0; j < 8; ++j) {
          uint32_t x = (hw[j] >> k) & 0x01010101u;  // bit k of 4 byte counters
          x |= x >> 7;
          x |= x >> 14;
          pk |= (x & 0xFu) << (4 * j);
        }
        if (k < kRegPlanes) P[k < kRegPlanes ? k : 0][w] = pk;
        else xplanes[(k - kRegPlanes) * WPB + wi] = pk;
      } else if (k < kRegPlanes) {
        P[k < kRegPlanes ? k : 0][w] = 0;
      }
    }
  }
  *thr = ntok - dmax;  // pass iff sum >= (L-q+1) - min(q*e, L-q+1)
  return K;
}

// sum_k 2^k popc(v & P_k) over this lane's WL words
template <int WPB, int WL>
__device__ __forceinline__ uint32_t plane_sum(const uint32_t (&v)[WL],
                                              const uint32_t (&P)[kRegPlanes][WL], uint32_t K,
                                              const uint32_t* xplanes, uint32_t sub) {
  if constexpr (WL == 4 && kRegPlanes == 2) {
    if (K <= 2) {
      // the eight masked words (four of weight 1, four of weight 2) summed
      // bit-wise with a carry-save tree first: 4 POPC instead of 8
      const uint32_t a0 = v[0] & P[0][0], a1 = v[1] & P[0][1], a2 = v[2] & P[0][2],
                     a3 = v[3] & P[0][3];
      const uint32_t b0 = v[0] & P[1][0], b1 = v[1] & P[1][1], b2 = v[2] & P[1][2],
                     b3 = v[3] & P[1][3];
      const uint32_t s1 = a0 ^ a1 ^ a2, c1 = (a0 & a1) | (a2 & (a0 ^ a1));  // weights 1, 2
      const uint32_t s2 = s1 ^ a3, c2 = s1 & a3;                              // weights 1, 2
      const uint32_t s3 = c1 ^ c2 ^ b0, c3 = (c1 & c2) | (b0 & (c1 ^ c2));   // weights 2, 4
      const uint32_t s4 = b1 ^ b2 ^ b3, c4 = (b1 & b2) | (b3 & (b1 ^ b2));   // weights 2, 4
      const uint32_t s5 = s3 ^ s4, c5 = s3 & s4;                              // weights 2, 4
      const uint32_t s6 = c3 ^ c4 ^ c5, c6 = (c3 & c4) | (c5 & (c3 ^ c4));   // weights 4, 8
      return __popc(s2) + 2u * __popc(s5) + 4u * __popc(s6) + 8u * __popc(c6);
    }
  }
  uint32_t sum = 0;
#pragma unroll
  for (int p = 0; p < kRegPlanes; ++p) {
    if ((uint32_t)p < K) {
      uint32_t s = 0;
#pragma unroll
      for (int w = 0; w < WL; ++w) s += __popc(v[w] & P[p][w]);
      sum += s << p;
    }
  }
  for (uint32_t p = kRegPlanes; p < K; ++p) {
    uint32_t s = 0;
#pragma unroll
    for (int w = 0; w < WL; ++w) s += __popc(v[w] & xplanes[(p - kRegPlanes) * WPB + sub * WL + w]);
    sum += s << p;
  }
  return sum;
}

// Sums of U candidates over a lane group of G lanes (U <= G, powers of two):
// at each of the first log2(U) butterfly steps a lane keeps half of its
// sums and adds its partner's copy of them, sending the other half; the
// remaining steps reduce the one sum left.  Lane `sub` of the group returns
// the group total of candidate sub / (G / U).  log2(U) + log2(G/U) shuffles
// instead of U * log2(G).
template <int G, int U>
__device__ __forceinline__ uint32_t reduce_scatter(uint32_t (&s)[U], uint32_t sub) {
#pragma unroll
  for (int n = U, m = G / 2; n > 1; n >>= 1, m >>= 1) {
    const bool upper = (sub & (uint32_t)m) != 0;  // keep the upper half of the n sums
#pragma unroll
    for (int i = 0; i < n / 2; ++i) {
      const uint32_t lo = s[i], hi = s[i + n / 2];
      s[i] = (upper ? hi : lo) + __shfl_xor_sync(0xFFFFFFFFu, upper ? lo : hi, m);
    }
  }
#pragma unroll
  for (int m = G / (2 * U); m >= 1; m >>= 1) s[0] += __shfl_xor_sync(0xFFFFFFFFu, s[0], m);
  return s[0];
}

// ids of candidates seg[off + u*CPW + slot] (u < U) of a segment of n
// candidates, 0 past its end; 32-bit offsets within the segment
template <int U, int CPW>
__device__ __forceinline__ void load_ids(const int32_t* __restrict__ seg, uint32_t off, uint32_t n,
                                         uint32_t slot, uint32_t (&b)[U]) {
#pragma unroll
  for (int u = 0; u < U; ++u) {
    const uint32_t k = off + u * CPW + slot;
    b[u] = k < n ? (uint32_t)__ldg(seg + k) : 0u;
  }
}

// Candidates per work claim: large enough that the search for a chunk's
// first read and the planes of the reads split at chunk edges stay cheap,
// small enough that every warp gets about 16 chunks (an even finish).  Below
// that, calls too short to give every warp a chunk of 256 take smaller ones,
// down to a batch of 32: a chunk is one warp's serial work, and there are
// warps to spare (37 reads' lists, 10.8k candidates: 54 us at 256, 28 at 32).
constexpr uint64_t kChunkFew = 32, kChunkMin = 256, kChunkMax = 4096, kChunksPerWarp = 16;
__device__ __forceinline__ uint64_t chunk_size(uint64_t n_cand, uint64_t warps) {
  uint64_t c = kChunkMax;
  while (c > kChunkMin && c * kChunksPerWarp * warps > n_cand) c >>= 1;
  while (c > kChunkFew && c * warps > n_cand) c >>= 1;
  return c;
}

// The read holding candidate x: the largest r < n_reads with cand_off[r] <= x
// (empty lists in between are skipped), by a 32-way search.
__device__ __forceinline__ uint32_t read_of(const uint64_t* __restrict__ cand_off, uint32_t n_reads,
                                            uint64_t x, uint32_t lane) {
  uint32_t lo = 0, hi = n_reads;  // cand_off[lo] <= x < cand_off[hi]
  while (hi - lo > 1) {
    const uint32_t step = (hi - lo + 31) / 32;
    const uint32_t p = lo + lane * step;
    const bool le = p < hi && cand_off[p] <= x;
    const uint32_t bal = __ballot_sync(0xFFFFFFFFu, le);  // lane 0 always (cand_off[lo] <= x)
    const uint32_t last = 31 - __clz(bal);
    lo = lo + last * step;
    hi = min(hi, lo + step);
  }
  return lo;
}

// CTAs per SM: eight (64 warps, 32 registers a thread); the gathers are
// latency-bound, and the extra warps outweigh a few spilled words.
constexpr int kCandCtasPerSm = 8;

template <int WPB, int U>
__global__ void __launch_bounds__(kWarps * 32, kCandCtasPerSm) k_candidates(CandArgs a) {
  using C = Cfg<WPB>;
  constexpr int WL = C::WL, G = C::G, CPW = C::CPW;
  extern __shared__ uint32_t s_warp[];
  const uint32_t lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const uint32_t r4 = a.ix.r4;
  uint32_t* hist = s_warp + warp * warp_smem_words(r4, WPB);  // byte t = multiplicity of token t
  uint32_t* xplanes = hist + hist_words_of(r4);  // higher planes
  const uint32_t sub = lane % G;     // this lane's slice of a bin vector
  const uint32_t slot = lane / G;    // which of the warp's CPW candidates
  if (*(volatile uint32_t*)&a.ctl->status) return;
  const uint32_t n_reads = live_reads(a.ctl, a.live, a.rv.n_reads);
  if (n_reads == 0) return;
  // the batch's lists span candidates [c_begin, c_end); warps claim chunks
  // of `chunk` consecutive candidates, so a long list is shared by many warps
  const uint64_t c_begin = a.cand_off[0], c_end = a.cand_off[n_reads];
  const uint64_t chunk =
      c_end > c_begin ? chunk_size(c_end - c_begin, (uint64_t)gridDim.x * kWarps) : kChunkMin;
  const uint64_t n_chunks = c_end > c_begin ? (c_end - c_begin + chunk - 1) / chunk : 0;

  uint32_t cur = 0xFFFFFFFFu, K = 0, thr = 0;  // the read whose planes are built
  const uint32_t last_row = (uint32_t)(a.ix.bm_rows - 1);
  const uint32_t num_bins = (uint32_t)a.ix.num_bins;  // bins are uint32 (checked at build)
  bool bad = false;  // this lane saw a candidate id outside [0, num_bins)
  uint32_t P[kRegPlanes][WL];
  // the next chunk is claimed one chunk ahead, so the atomic's latency
  // overlaps the current chunk's work
  uint32_t cj_next = 0;
  if (lane == 0) cj_next = atomicAdd(&a.ctl->item, 1u);
  for (;;) {
    const uint32_t cj = __shfl_sync(0xFFFFFFFFu, cj_next, 0);
    if (cj >= n_chunks) break;
    if (lane == 0) cj_next = atomicAdd(&a.ctl->item, 1u);
    // positions inside the chunk are 32-bit, relative to its first candidate
    const uint64_t base = c_begin + (uint64_t)cj * chunk;
    const uint32_t clen = (uint32_t)min(chunk, c_end - base);
    uint32_t r = read_of(a.cand_off, n_reads, base, lane);
    // the end of read r's list, clipped to the chunk (> 0: r's list holds base)
    uint32_t c1 = (uint32_t)min(a.cand_off[r + 1] - base, (uint64_t)clen);
    uint32_t p = 0;
    while (p < clen) {
      // the segment [p, c1) of read r's list inside this chunk; the end of the
      // next read's list is fetched while this one is scored
      const uint32_t c1_next = r + 2 <= n_reads && c1 < clen
                                   ? (uint32_t)min(a.cand_off[r + 2] - base, (uint64_t)clen)
                                   : c1;
      if (c1 > p) {
        // the segment's candidates seg[0, n)
        const int32_t* seg = a.cand + base + p;
        const uint32_t n = c1 - p;
        // the first candidate ids are fetched while the planes are built
        uint32_t bc[U];
        load_ids<U, CPW>(seg, 0, n, slot, bc);
        if (r != cur) {
          cur = r;
          K = build_planes<WPB, WL>(a.rv, r, r4, hist, xplanes, lane, sub, P, &thr);
        }
        // U independent gathers in flight per lane group; the ids of the
        // next step are fetched before this step's vectors are used
        for (uint32_t off = 0; off < n; off += CPW * U) {
          uint32_t bn[U];
          load_ids<U, CPW>(seg, off + CPW * U, n, slot, bn);
          // the caller's ids are checked here, where they are read anyway: an
          // id outside [0, num_bins) fails the call, never passes, and its
          // gather is clamped inside the table
          uint32_t v[U][WL];
#pragma unroll
          for (int u = 0; u < U; ++u) {
            const bool in = off + u * CPW + slot < n;
            bad |= in && bc[u] >= num_bins;
            const uint32_t row = min(bc[u], last_row);
            if (in) load_words<WL>(a.ix.bm + (uint64_t)row * WPB + sub * WL, v[u]);
          }
          // passing candidates of the warp get consecutive record slots
          auto emit = [&](bool pass, uint32_t c, uint32_t sum) {
            const uint32_t bal = __ballot_sync(0xFFFFFFFFu, pass);
            if (bal) {
              unsigned long long first = 0;  // the warp's first record slot
              if (lane == 0) first = atomicAdd(&a.ctl->n_rec, (unsigned long long)__popc(bal));
              first = __shfl_sync(0xFFFFFFFFu, first, 0);
              if (pass) {
                const unsigned long long pos = first + __popc(bal & ((1u << lane) - 1u));
                if (pos < a.rec.cap) {
                  a.rec.keys[pos] = base + p + c;
                  a.rec.counts[pos] = (uint8_t)sum;
                }
              }
            }
          };
          uint32_t sums[U];
#pragma unroll
          for (int u = 0; u < U; ++u)
            sums[u] = off + u * CPW + slot < n ? plane_sum<WPB, WL>(v[u], P, K, xplanes, sub) : 0u;
          if constexpr (U > 1 && U <= G) {
            // the U sums reduced over the lane group at once: each lane ends
            // with the total of candidate uq, held by G/U lanes
            const uint32_t total = reduce_scatter<G, U>(sums, sub);
            const uint32_t uq = sub / (G / U);
            uint32_t id = bc[0];
#pragma unroll
            for (int u = 1; u < U; ++u) id = uq == (uint32_t)u ? bc[u] : id;
            const uint32_t c = off + uq * CPW + slot;
            emit(sub % (G / U) == 0 && c < n && id < num_bins && total >= thr, c, total);
          } else {
#pragma unroll
            for (int u = 0; u < U; ++u) {
              const uint32_t c = off + u * CPW + slot;
              uint32_t sum = sums[u];
#pragma unroll
              for (int o = G / 2; o >= 1; o >>= 1) sum += __shfl_xor_sync(0xFFFFFFFFu, sum, o);
              emit(c < n && bc[u] < num_bins && sub == 0 && sum >= thr, c, sum);
            }
          }
#pragma unroll
          for (int u = 0; u < U; ++u) bc[u] = bn[u];
        }
      }
      p = c1;
      ++r;
      c1 = c1_next;
    }
  }
  if (__any_sync(0xFFFFFFFFu, bad) && lane == 0) atomicOr(&a.ctl->status, kStatusBadCand);
}

// Whole vectors of 512 bytes (q = 6) against a read, for budgets so large that
// a bin is ruled out only by a hundred or more tokens that it lacks: a vector is
// ANDed with the set of the read's tokens and with the set of those it holds
// twice; the few it holds more often are looked up.  Bound by HBM's rate of random
// 512-byte rows: 20k reads of 250 bp, 6.6M candidates, 0.55 ms whatever the budget
// (12e9 rows/s of 13.7e9).  A binary plane for each bit of the multiplicity, from a
// histogram of the tokens, took 0.78; the look-ups 0.51 at e = 18, 0.88 at e = 20,
// 1.47 at e = 33.
constexpr uint32_t kPlaneWords = 128;
struct __align__(16) Planes {  // a warp's, in shared memory; a lane takes 4 words of each
  uint32_t once[kPlaneWords], twice[kPlaneWords];
  uint16_t more[256];  // a token for every further occurrence
};

// Sets the planes of a token row; the number of further occurrences.
// Warp-collective.
__device__ __forceinline__ uint32_t set_planes(Planes& p, const uint16_t* tok, uint32_t ntok,
                                               uint32_t r4, uint32_t lane) {
  constexpr int kRounds = 8;  // up to 255 tokens
  uint32_t t[kRounds];
#pragma unroll
  for (int i = 0; i < kRounds; ++i)
    t[i] = 32u * i + lane < ntok ? tok[32u * i + lane] : rowPad(r4);
  __syncwarp();  // the last read's planes are no longer read
  reinterpret_cast<uint4*>(p.once)[lane] = make_uint4(0u, 0u, 0u, 0u);
  reinterpret_cast<uint4*>(p.twice)[lane] = make_uint4(0u, 0u, 0u, 0u);
  __syncwarp();
  uint32_t n = 0;
#pragma unroll
  for (int i = 0; i < kRounds; ++i) {
    const uint32_t w = t[i] >> 5, bit = 1u << (t[i] & 31u);
    const bool further = t[i] < r4 && (atomicOr(p.once + w, bit) & bit) &&
                         (atomicOr(p.twice + w, bit) & bit);
    const uint32_t m = __ballot_sync(0xFFFFFFFFu, further);
    if (further) p.more[n + __popc(m & ((1u << lane) - 1u))] = (uint16_t)t[i];
    n += __popc(m);
  }
  __syncwarp();
  return n;
}

// popc(v & a) + popc(v & b) over the warp's 128 words, through a carry-save tree
// (4 POPC instead of 8)
__device__ __forceinline__ uint32_t planes_present(const uint4& v, const uint4& a, const uint4& b) {
  const uint32_t x0 = v.x & a.x, x1 = v.y & a.y, x2 = v.z & a.z, x3 = v.w & a.w;
  const uint32_t y0 = v.x & b.x, y1 = v.y & b.y, y2 = v.z & b.z, y3 = v.w & b.w;
  const uint32_t s0 = x0 ^ x1 ^ x2, c0 = (x0 & x1) | (x2 & (x0 ^ x1));
  const uint32_t s1 = x3 ^ y0 ^ y1, c1 = (x3 & y0) | (y1 & (x3 ^ y0));
  const uint32_t s2 = s0 ^ s1 ^ y2, c2 = (s0 & s1) | (y2 & (s0 ^ s1));
  const uint32_t s3 = s2 ^ y3, c3 = s2 & y3;                            // weight 1; carries of 2
  const uint32_t s4 = c0 ^ c1 ^ c2, c4 = (c0 & c1) | (c2 & (c0 ^ c1));  // weights 2, 4
  const uint32_t s5 = s4 ^ c3, c5 = s4 & c3;                            // weights 2, 4
  return __reduce_add_sync(0xFFFFFFFFu, __popc(s3) + 2u * __popc(s5) + 4u * __popc(c4 ^ c5) +
                                            8u * __popc(c4 & c5));
}

// Up to 32 bins (lane k < n: its bin's row) against the read: the lane's sum + 1
// where it is at least thr, else 0.  Warp-collective.
template <int U>
__device__ __forceinline__ uint32_t planes_check(const uint32_t* bm, const Planes& p,
                                                 uint32_t n_more, uint32_t thr, uint32_t row,
                                                 uint32_t n, uint32_t lane) {
  const uint4 p0 = reinterpret_cast<const uint4*>(p.once)[lane];
  const uint4 p1 = reinterpret_cast<const uint4*>(p.twice)[lane];
  const uint4* vecs = reinterpret_cast<const uint4*>(bm) + lane;
  uint32_t sum = 0;  // of the lane's bin
  for (uint32_t k = 0; k < n; k += U) {
    uint4 v[U];
#pragma unroll
    for (int u = 0; u < U; ++u)
      v[u] = __ldg(vecs + (uint64_t)__shfl_sync(0xFFFFFFFFu, row, k + u) * (kPlaneWords / 4));
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const uint32_t present = planes_present(v[u], p0, p1);
      sum = lane == k + u ? present : sum;
    }
  }
  // a lane's bin and one token at a time
  const uint32_t* mine = bm + (uint64_t)row * kPlaneWords;
  for (uint32_t i = 0; i < n_more; ++i) {
    const uint32_t t = p.more[i];
    sum += (__ldg(mine + (t >> 5)) >> (t & 31u)) & 1u;
  }
  return lane < n && sum >= thr ? sum + 1u : 0u;
}

// Survivors of reads with D' >= far at q = 6, one at a time: its f members' vectors
// are consecutive and share the read's planes.  3.4M survivors of 16 members, 250 bp,
// e = 20: 5.0 ms (28 GB of vectors, 0.81 of the copy rate), 12.2 with k_refine's
// look-ups; 5.1 + 1.1 for sorting and expanding them into lists.
__device__ __forceinline__ void refine_by_planes(const IndexView& ix, const ReadsView& rv,
                                                 const unsigned long long* __restrict__ keys,
                                                 uint64_t n_surv, uint32_t cbits, uint32_t f,
                                                 const RecordsView& rec, uint32_t bin_bits,
                                                 uint32_t far, Ctl* ctl, Planes& planes) {
  const uint32_t lane = threadIdx.x & 31;
  const uint64_t warp = (blockIdx.x * (uint64_t)blockDim.x + threadIdx.x) >> 5;
  const uint64_t n_warps = ((uint64_t)gridDim.x * blockDim.x) >> 5;
  uint32_t cur = 0xFFFFFFFFu, n_more = 0;  // the read whose planes are set
  uint32_t batch = 32;  // survivors
  while (batch > 1 && n_surv < n_warps * batch) batch >>= 1;
  for (uint64_t base = warp * batch; base < n_surv; base += n_warps * batch) {
    const bool in = lane < batch && base + lane < n_surv;
    const unsigned long long key = in ? keys[base + lane] : 0ull;
    const uint32_t mine = (uint32_t)(key >> cbits), m = in ? rv.meta[mine] : 0u;
    uint32_t todo = __ballot_sync(0xFFFFFFFFu, in && ((m >> 8) & 0xFFu) >= far);
    for (; todo; todo &= todo - 1u) {
      const int s = __ffs(todo) - 1;
      const uint32_t r = __shfl_sync(0xFFFFFFFFu, mine, s), mr = __shfl_sync(0xFFFFFFFFu, m, s);
      const uint32_t ntok = mr & 0xFFu, dmax = (mr >> 8) & 0xFFu;
      const uint32_t first = (uint32_t)(__shfl_sync(0xFFFFFFFFu, key, s) & ((1ull << cbits) - 1ull)) * f;
      const uint32_t end = (uint32_t)min((uint64_t)first + f, ix.num_bins);
      const uint16_t* tok = rv.tokens + (uint64_t)r * rv.copies * rv.ts;
      if (r != cur) {
        cur = r;
        n_more = set_planes(planes, tok, ntok, ix.r4, lane);
      }
      for (uint32_t b = first; b < end; b += 32) {
        const uint32_t n = min(end - b, 32u), row = b + min(lane, n - 1u);
        const uint32_t found = planes_check<4>(ix.bm, planes, n_more, ntok - dmax, row, n, lane);
        const uint32_t bal = __ballot_sync(0xFFFFFFFFu, found != 0);
        if (!bal) continue;
        unsigned long long at = 0;
        if (lane == 0) at = atomicAdd(&ctl->n_final, (unsigned long long)__popc(bal));
        at = __shfl_sync(0xFFFFFFFFu, at, 0) + __popc(bal & ((1u << lane) - 1u));
        if (found && at < rec.cap) {
          rec.keys[at] = ((unsigned long long)r << bin_bits) | (b + lane);
          rec.counts[at] = (uint8_t)(found - 1u);
        }
      }
    }
  }
}

// Exact check of the coarse pass's survivors, one (survivor, member bin) item
// at a time by a whole warp: lane j looks up the read's tokens j, j + 32, ...
// in the member's vector and a ballot counts the misses; the item ends once
// they exceed D'.  The tokens are in the all-bins order (rarest first), so
// most members end after one or two of these rounds.  Survivors come in the
// order the coarse pass found them: an item needs only its read's token row,
// so nothing is gained by sorting them by read first (the bit planes of
// k_candidates pay for themselves over a list, not over two members).
// Measured on GB300 against sorting the survivors, expanding them into lists
// and checking those with k_candidates: 6.4M survivors of 100 bp reads on the
// 3.1 Gbp tables 3.0 -> 1.8 ms; 2,383 survivors of a 1 Mbp genome 540 -> 25 us
// (19 chunks of short lists there, each one warp's serial work).  The chain of
// loads (token, then word of the vector) bounds it, so kRefineItems items run
// side by side in a warp.
// WIDE (q = 6): the survivors of reads with D' >= far are left to a second loop,
// refine_by_planes.  Look-ups cost with D', vectors do not (us, look-ups / vectors):
// 100 bp, D' = 36, 562k survivors of 16 1124 / 1034; 150 bp, D' = 48, 13k 244 / 234;
// D' = 60, 353k 1009 / 795, 2.0M of 8 2179 / 1218; with few members to share the
// planes, f = 2, 8k survivors at D' = 48 206 / 213.
constexpr int kRefineItems = 4;
constexpr uint32_t kRefineFar = 32, kRefineFarMembers = 8;

template <bool WIDE>
__global__ void __launch_bounds__(kWarps * 32, 4) k_refine(IndexView ix, ReadsView rv,
                                                           const unsigned long long* __restrict__ keys,
                                                           const unsigned long long* n_surv_at,
                                                           uint64_t room, uint32_t cbits, uint32_t f,
                                                           RecordsView rec, uint32_t bin_bits,
                                                           uint32_t far, Ctl* ctl, Live live) {
  constexpr int U = kRefineItems;
  if (*(volatile uint32_t*)&ctl->status) return;
  if (routed_off(ctl, live)) return;
  const uint64_t n_surv = *n_surv_at;
  if (n_surv > room) return;  // not all of them were kept: the call takes another way
  const uint32_t lane = threadIdx.x & 31;
  const uint64_t warp = (blockIdx.x * (uint64_t)blockDim.x + threadIdx.x) >> 5;
  const uint64_t n_warps = ((uint64_t)gridDim.x * blockDim.x) >> 5;
  const uint64_t n_items = n_surv * f;
  // items of a warp's batch: 32, or fewer when there are warps to spare (4,766
  // items: 25 us in batches of 32, 10 in batches of 4)
  uint32_t batch = 32;
  while (batch > (uint32_t)U && n_items < n_warps * batch) batch >>= 1;
  for (uint64_t base = warp * batch; base < n_items; base += n_warps * batch) {
    // lane i: the batch's item i
    const uint64_t i = base + lane;
    uint32_t r = 0, bin = 0, m = 0, found = 0;  // found: sum + 1 of a passing item
    bool in = i < n_items && lane < batch;
    if (in) {
      const uint64_t sv = i / f;
      const unsigned long long key = keys[sv];
      r = (uint32_t)(key >> cbits);
      const uint64_t b = (key & ((1ull << cbits) - 1ull)) * f + (i - sv * f);
      in = b < ix.num_bins;  // the last super-bin may have fewer members
      bin = (uint32_t)b;
      m = in ? rv.meta[r] : 0u;
      if (WIDE) in = in && ((m >> 8) & 0xFFu) < far;
    }
    const uint32_t todo = __ballot_sync(0xFFFFFFFFu, in);
    for (uint32_t k = 0; k < batch; k += U) {
      uint32_t live_items = (todo >> k) & ((1u << U) - 1u);
      if (!live_items) continue;
      const uint16_t* tok[U];
      const uint32_t* vec[U];
      uint32_t ntok[U], dmax[U], misses[U];
#pragma unroll
      for (int u = 0; u < U; ++u) {
        const uint32_t mu = __shfl_sync(0xFFFFFFFFu, m, k + u);
        tok[u] = rv.tokens + (uint64_t)__shfl_sync(0xFFFFFFFFu, r, k + u) * rv.copies * rv.ts + lane;
        vec[u] = ix.bm + (uint64_t)__shfl_sync(0xFFFFFFFFu, bin, k + u) * ix.wpb;
        ntok[u] = mu & 0xFFu;
        dmax[u] = (mu >> 8) & 0xFFu;
        misses[u] = 0;
      }
      for (uint32_t j = 0; live_items; j += 32) {
        uint32_t t[U], w[U];
#pragma unroll
        for (int u = 0; u < U; ++u)
          t[u] = (live_items >> u & 1u) && j + lane < ntok[u] ? tok[u][j] : rowPad(ix.r4);
#pragma unroll
        for (int u = 0; u < U; ++u) w[u] = t[u] < ix.r4 ? __ldg(vec[u] + (t[u] >> 5)) : 0u;
#pragma unroll
        for (int u = 0; u < U; ++u) {
          const bool miss = t[u] != rowPad(ix.r4) && !((w[u] >> (t[u] & 31u)) & 1u);
          misses[u] += __popc(__ballot_sync(0xFFFFFFFFu, miss));
          if (misses[u] > dmax[u]) {
            live_items &= ~(1u << u);
          } else if ((live_items >> u & 1u) && j + 32 >= ntok[u]) {  // every token looked up
            live_items &= ~(1u << u);
            if (lane == k + u) found = ntok[u] - misses[u] + 1u;
          }
        }
      }
    }
    const uint32_t bal = __ballot_sync(0xFFFFFFFFu, found != 0);
    if (bal) {
      unsigned long long first = 0;
      if (lane == 0) first = atomicAdd(&ctl->n_final, (unsigned long long)__popc(bal));
      first = __shfl_sync(0xFFFFFFFFu, first, 0);
      const unsigned long long pos = first + __popc(bal & ((1u << lane) - 1u));
      if (found && pos < rec.cap) {
        rec.keys[pos] = ((unsigned long long)r << bin_bits) | bin;
        rec.counts[pos] = (uint8_t)(found - 1u);
      }
    }
  }
  if constexpr (WIDE) {
    __shared__ Planes s_planes[kWarps];
    if (ctl->max_d >= far)
      refine_by_planes(ix, rv, keys, n_surv, cbits, f, rec, bin_bits, far, ctl,
                       s_planes[threadIdx.x >> 5]);
  }
}

// Candidate lists over large vectors (q = 6, 512 bytes), by token look-ups.
// A random 512-byte row costs DRAM its bytes (13.7e9 rows/s), and half of one
// half (27e9; a single 128-byte line 38e9), so the bin is ruled out from as
// few lines as possible: the tokeniser groups a read's tokens by line,
// fullest line first, and lane j looks up token 32*s + j of the first
// `stage` groups of 32 -- as many as leave more than D' misses expected -- in
// U candidates at once; one redux per candidate counts the tokens present.
// Only a bin that could still pass has the rest of its tokens looked up.
// Measured on GB300 (300k reads of 150 bp, e = 7, 98.9M candidates): 4.0 ms,
// 0.93 of the two-line rate; ANDing whole vectors with bit planes of the read
// took 9.48 ms at 91 warp instructions a candidate.  The same look-ups over
// 128-byte vectors (q = 5, mixed reads) lost to the planes, 9.8 against 8.6
// ms: one line is read either way, and a quarter warp per vector issues less.
// Batches of which a third of the reads or more have budgets too large to be
// settled by the first groups (Ctl::n_far) are checked with planes, whose time does
// not depend on the budget: 0.55 ms where the look-ups take 0.26 to 0.52 for the
// reads before that line and 0.82 to 1.47 for those past it.
constexpr uint32_t kFarShare = 3;

struct StageTokens {
  const char* at[kStageMax];  // the token's word in row 0, or a zero word
  uint32_t step[kStageMax];   // bytes from row to row (0 for the zero word)
  uint32_t bit[kStageMax];    // token & 31
};

// alive bits (candidate k of the batch) after the first S groups of tokens.
// At the most groups, reads with large budgets leave many bins alive, so lane
// k keeps candidate k's tokens present and the rest of the check goes on from
// there; with fewer groups almost every bin ends here and starts over if not.
template <int S, int U>
__device__ __forceinline__ uint32_t stage_scan(const StageTokens& st, uint32_t ids, uint32_t n,
                                               uint32_t need, uint32_t lane, uint32_t& present) {
  uint32_t alive = 0;
  for (uint32_t k = 0; k < n; k += U) {
    uint32_t w[U][S];
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const uint32_t row = __shfl_sync(0xFFFFFFFFu, ids, k + u);
#pragma unroll
      for (int s = 0; s < S; ++s)
        w[u][s] = __ldg(reinterpret_cast<const uint32_t*>(st.at[s] + (uint64_t)row * st.step[s]));
    }
    uint32_t a = 0;
#pragma unroll
    for (int u = 0; u < U; ++u) {
      uint32_t c = 0;
#pragma unroll
      for (int s = 0; s < S; ++s) c += (w[u][s] >> st.bit[s]) & 1u;
      c = __reduce_add_sync(0xFFFFFFFFu, c);
      if (c >= need) a |= 1u << u;
      if (S == kStageMax) present = lane == k + u ? c : present;
    }
    alive |= a << k;
  }
  return alive;
}

// The lists of a batch of reads with large budgets, in whole vectors.
__device__ __forceinline__ void lists_by_planes(const CandArgs& a, Planes& planes,
                                                uint32_t n_reads, uint32_t lane) {
  const uint64_t c_begin = a.cand_off[0], c_end = a.cand_off[n_reads];
  const uint64_t chunk = chunk_size(c_end - c_begin, (uint64_t)gridDim.x * kWarps);
  const uint64_t n_chunks = (c_end - c_begin + chunk - 1) / chunk;
  const uint32_t num_bins = (uint32_t)a.ix.num_bins, r4 = a.ix.r4;
  uint32_t cur = 0xFFFFFFFFu, thr = 0, n_more = 0;  // the read whose planes are set
  bool bad = false;
  for (;;) {
    uint32_t cj = 0;
    if (lane == 0) cj = atomicAdd(&a.ctl->item, 1u);
    cj = __shfl_sync(0xFFFFFFFFu, cj, 0);
    if (cj >= n_chunks) break;
    const uint64_t base = c_begin + (uint64_t)cj * chunk;
    const uint32_t clen = (uint32_t)min(chunk, c_end - base);
    uint32_t r = read_of(a.cand_off, n_reads, base, lane);
    for (uint32_t p = 0; p < clen; ++r) {
      const uint32_t c1 = (uint32_t)min(a.cand_off[r + 1] - base, (uint64_t)clen);
      if (c1 > p && r != cur) {
        cur = r;
        const uint32_t m = a.rv.meta[r], ntok = m & 0xFFu;
        thr = ntok - ((m >> 8) & 0xFFu);
        n_more = set_planes(planes, a.rv.tokens + (uint64_t)r * a.rv.copies * a.rv.ts, ntok, r4, lane);
      }
      for (; p < c1; p += 32) {
        const uint32_t n = min(c1 - p, 32u);
        const uint32_t id = lane < n ? (uint32_t)__ldg(a.cand + base + p + lane) : 0u;
        const bool ok = id < num_bins;
        bad |= !ok;
        uint32_t found = planes_check<4>(a.ix.bm, planes, n_more, thr, ok ? id : 0u, n, lane);
        if (!ok) found = 0;
        const uint32_t bal = __ballot_sync(0xFFFFFFFFu, found != 0);
        if (!bal) continue;
        unsigned long long at = 0;
        if (lane == 0) at = atomicAdd(&a.ctl->n_rec, (unsigned long long)__popc(bal));
        at = __shfl_sync(0xFFFFFFFFu, at, 0) + __popc(bal & ((1u << lane) - 1u));
        if (found && at < a.rec.cap) {
          a.rec.keys[at] = base + p + lane;
          a.rec.counts[at] = (uint8_t)(found - 1u);
        }
      }
      p = c1;
    }
  }
  if (__any_sync(0xFFFFFFFFu, bad) && lane == 0) atomicOr(&a.ctl->status, kStatusBadCand);
}

template <int U>
__global__ void __launch_bounds__(kWarps * 32, 6) k_candidates_lookup(CandArgs a, uint32_t miss256) {
  const uint32_t lane = threadIdx.x & 31;
  const uint32_t r4 = a.ix.r4, wpb = a.ix.wpb;
  if (*(volatile uint32_t*)&a.ctl->status) return;
  const uint32_t n_reads = live_reads(a.ctl, a.live, a.rv.n_reads);
  if (n_reads == 0) return;
  const uint64_t c_begin = a.cand_off[0], c_end = a.cand_off[n_reads];
  if (c_end <= c_begin) return;
  __shared__ Planes s_planes[kWarps];
  if ((uint64_t)a.ctl->n_far * kFarShare >= n_reads) {
    lists_by_planes(a, s_planes[threadIdx.x >> 5], n_reads, lane);
    return;
  }
  const uint64_t chunk = chunk_size(c_end - c_begin, (uint64_t)gridDim.x * kWarps);
  const uint64_t n_chunks = (c_end - c_begin + chunk - 1) / chunk;
  const uint32_t num_bins = (uint32_t)a.ix.num_bins;
  // a word of the control block that stays zero: what a q-gram with a
  // non-base, or a lane past the read's tokens, looks up
  const char* zero = reinterpret_cast<const char*>(a.ctl->pad);

  uint32_t cur = 0xFFFFFFFFu, ntok = 0, dmax = 0, stage = 0, need = 0;
  const uint16_t* tok = nullptr;
  StageTokens st;
  bool bad = false;
  uint32_t cj_next = 0;
  if (lane == 0) cj_next = atomicAdd(&a.ctl->item, 1u);
  for (;;) {
    const uint32_t cj = __shfl_sync(0xFFFFFFFFu, cj_next, 0);
    if (cj >= n_chunks) break;
    if (lane == 0) cj_next = atomicAdd(&a.ctl->item, 1u);
    const uint64_t base = c_begin + (uint64_t)cj * chunk;
    const uint32_t clen = (uint32_t)min(chunk, c_end - base);
    uint32_t r = read_of(a.cand_off, n_reads, base, lane);
    uint32_t c1 = (uint32_t)min(a.cand_off[r + 1] - base, (uint64_t)clen);
    uint32_t p = 0;
    while (p < clen) {
      const uint32_t c1_next = r + 2 <= n_reads && c1 < clen
                                   ? (uint32_t)min(a.cand_off[r + 2] - base, (uint64_t)clen)
                                   : c1;
      uint32_t id_next = p + lane < c1 ? (uint32_t)__ldg(a.cand + base + p + lane) : 0u;
      if (c1 > p && r != cur) {
        cur = r;
        const uint32_t m = a.rv.meta[r];
        ntok = m & 0xFFu;
        dmax = (m >> 8) & 0xFFu;
        tok = a.rv.tokens + (uint64_t)r * a.rv.copies * a.rv.ts;
        // groups of 32 tokens that leave D' + 6 misses expected
        stage = min(min(lookup_groups(dmax, miss256), (ntok + 31u) / 32u), (uint32_t)kStageMax);
#pragma unroll
        for (int s = 0; s < kStageMax; ++s) {
          const uint32_t t = s * 32u + lane < ntok ? tok[s * 32u + lane] : rowPad(r4);
          const bool on = t < r4 && (uint32_t)s < stage;
          st.at[s] = on ? reinterpret_cast<const char*>(a.ix.bm + (t >> 5)) : zero;
          st.step[s] = on ? wpb * 4u : 0u;
          st.bit[s] = t & 31u;
        }
        const uint32_t n1 = min(stage * 32u, ntok);
        need = n1 > dmax ? n1 - dmax : 0u;  // fewer of these present: more than D' misses
      }
      for (; p < c1; p += 32) {
        const uint32_t n = min(c1 - p, 32u);
        const uint32_t id = id_next;
        if (p + 32u + lane < c1) id_next = (uint32_t)__ldg(a.cand + base + p + 32u + lane);
        const bool ok = lane < n && id < num_bins;
        bad |= lane < n && !ok;
        const uint32_t row = ok ? id : 0u;
        uint32_t alive, present = 0;
        switch (stage) {
          case 1: alive = stage_scan<1, U>(st, row, n, need, lane, present); break;
          case 2: alive = stage_scan<2, U>(st, row, n, need, lane, present); break;
          case 3: alive = stage_scan<3, U>(st, row, n, need, lane, present); break;
          default: alive = stage_scan<kStageMax, U>(st, row, n, need, lane, present); break;
        }
        alive &= __ballot_sync(0xFFFFFFFFu, ok);
        // the few bins left: all their tokens, four bins side by side
        uint32_t found = 0;  // sum + 1 of this lane's candidate
        while (alive) {
          constexpr int V = 4;
          const uint32_t* vec[V];
          uint32_t k[V], misses[V], on = 0;
#pragma unroll
          for (int v = 0; v < V; ++v) {
            k[v] = alive ? (uint32_t)__ffs(alive) - 1u : 0u;
            if (alive) on |= 1u << v;
            alive &= alive - 1u;
            vec[v] = a.ix.bm + (uint64_t)__shfl_sync(0xFFFFFFFFu, row, k[v]) * wpb;
            misses[v] = 0;
            if (stage == (uint32_t)kStageMax)
              misses[v] = min(kStageMax * 32u, ntok) - __shfl_sync(0xFFFFFFFFu, present, k[v]);
          }
          for (uint32_t j = stage == (uint32_t)kStageMax ? kStageMax * 32u : 0u; on && j < ntok;
               j += 32) {
            const uint32_t t = j + lane < ntok ? tok[j + lane] : rowPad(r4);
            uint32_t w[V];
#pragma unroll
            for (int v = 0; v < V; ++v)
              w[v] = t < r4 && (on >> v & 1u) ? __ldg(vec[v] + (t >> 5)) : 0u;
#pragma unroll
            for (int v = 0; v < V; ++v) {
              const bool miss = t != rowPad(r4) && !((w[v] >> (t & 31u)) & 1u);
              misses[v] += __popc(__ballot_sync(0xFFFFFFFFu, miss));
              if (misses[v] > dmax) on &= ~(1u << v);
            }
          }
#pragma unroll
          for (int v = 0; v < V; ++v)
            if ((on >> v & 1u) && lane == k[v]) found = ntok - misses[v] + 1u;
        }
        const uint32_t bal = __ballot_sync(0xFFFFFFFFu, found != 0);
        if (bal) {
          unsigned long long first = 0;
          if (lane == 0) first = atomicAdd(&a.ctl->n_rec, (unsigned long long)__popc(bal));
          first = __shfl_sync(0xFFFFFFFFu, first, 0);
          const unsigned long long pos = first + __popc(bal & ((1u << lane) - 1u));
          if (found && pos < a.rec.cap) {
            a.rec.keys[pos] = base + p + lane;
            a.rec.counts[pos] = (uint8_t)(found - 1u);
          }
        }
      }
      p = c1;
      ++r;
      c1 = c1_next;
    }
  }
  if (__any_sync(0xFFFFFFFFu, bad) && lane == 0) atomicOr(&a.ctl->status, kStatusBadCand);
}

// CTAs of a list kernel: persistent, up to `most`, but no more warps than the
// smallest chunks that n_cand candidates make (every warp claims from one
// counter before it can know that none is left: 9,728 warps took 28 us over
// 338 chunks, 344 took 21)
uint64_t list_grid(uint64_t n_cand, uint64_t most) {
  const uint64_t need = n_cand / (kChunkFew * kWarps) + 1;
  return need < most ? need : most;
}

template <int U>
void launch_lookup(const CandArgs& a, uint64_t n_cand, cudaStream_t st) {
  int dev = 0, sms = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  const uint64_t grid = list_grid(n_cand, (uint64_t)(sms > 0 ? sms : 1) * 6u);
  ProfScope ps("candidates", st);
  k_candidates_lookup<U><<<(unsigned)grid, kWarps * 32, 0, st>>>(a, lookup_miss256(a.ix));
}

template <int WPB, int U>
void launch_u(const CandArgs& a, uint64_t n_cand, cudaStream_t st) {
  // at most 14 KB a CTA, so the launch bounds set how many an SM holds
  const size_t smem = (size_t)kWarps * warp_smem_words(a.ix.r4, WPB) * sizeof(uint32_t);
  static_assert(kWarps * warp_smem_words(1024, 32) * 4 * kCandCtasPerSm <= 227 * 1024,
                "eight CTAs of the largest vectors fit an SM");
  int dev = 0, sms = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  const uint64_t grid = list_grid(n_cand, (uint64_t)(sms > 0 ? sms : 1) * kCandCtasPerSm);
  ProfScope ps("candidates", st);
  k_candidates<WPB, U><<<(unsigned)grid, kWarps * 32, smem, st>>>(a);
}

template <int WPB>
void launch_t(const CandArgs& a, uint64_t n_cand, cudaStream_t st, uint32_t unroll) {
  if (unroll >= 8) launch_u<WPB, 8>(a, n_cand, st);
  else if (unroll >= 4) launch_u<WPB, 4>(a, n_cand, st);
  else if (unroll >= 2) launch_u<WPB, 2>(a, n_cand, st);
  else launch_u<WPB, 1>(a, n_cand, st);
}

}  // namespace

void launch_refine(const IndexView& ix, const ReadsView& rv, const unsigned long long* keys,
                   const unsigned long long* n_surv, uint64_t room, uint32_t cbits, uint32_t f,
                   RecordsView rec, uint32_t bin_bits, Ctl* ctl, cudaStream_t st, Live live) {
  if (room == 0) return;
  int dev = 0, sms = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  const uint64_t need = (room * f + 32 * kWarps - 1) / (32 * kWarps);
  const uint64_t most = (uint64_t)(sms > 0 ? sms : 1) * 4;
  const bool planes = ix.wpb == kPlaneWords && f >= kRefineFarMembers;
  auto kernel = planes ? k_refine<true> : k_refine<false>;
  ProfScope ps("candidates_refine", st);
  kernel<<<(unsigned)(need < most ? need : most), kWarps * 32, 0, st>>>(
      ix, rv, keys, n_surv, room, cbits, f, rec, bin_bits, kRefineFar, ctl, live);
}

void launch_candidates(const IndexView& ix, const ReadsView& rv, const int32_t* cand,
                       const uint64_t* cand_off, uint64_t n_cand, RecordsView rec, Ctl* ctl,
                       cudaStream_t st, Live live, uint32_t unroll) {
  if (unroll == 0) unroll = ix.wpb > 32 ? kDefaultLookupUnroll : kDefaultCandUnroll;
  if (rv.n_reads == 0) return;
  CandArgs a{ix, rv, cand, cand_off, rec, ctl, live};
  switch (ix.wpb) {
    case 1: launch_t<1>(a, n_cand, st, unroll); break;
    case 2: launch_t<2>(a, n_cand, st, unroll); break;
    case 8: launch_t<8>(a, n_cand, st, unroll); break;
    case 32: launch_t<32>(a, n_cand, st, unroll); break;
    case 128:
      if (unroll >= 8) launch_lookup<8>(a, n_cand, st);
      else if (unroll >= 4) launch_lookup<4>(a, n_cand, st);
      else if (unroll >= 2) launch_lookup<2>(a, n_cand, st);
      else launch_lookup<1>(a, n_cand, st);
      break;
    default: break;  // q outside 2..6 is rejected by grim_build
  }
}

}  // namespace grim
