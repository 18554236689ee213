// Read tokenising (§GRIM-Filter step 1: every token of the read is
// extracted) and the per-read threshold of Fig. 3, plus the validation of
// candidate-list offsets.
#include "grim_internal.cuh"

namespace grim {
namespace {

constexpr int kTokWarps = 8;
constexpr uint32_t kMaxStride = 256;  // token stride: <= 255 tokens rounded up to 16
constexpr int kTokRounds = 8;         // tokens per lane
constexpr int kTokCtasPerSm = 5;      // of the persistent grid
// A bin is out once it misses more than D' tokens.  After j tokens the misses
// of a random bin are about normal with mean S_j, the sum of the tokens' miss
// shares, and variance S_j (j - S_j) / j; the check comes at the first j whose
// mean is kCheckZ deviations past D'.
// (3 / 4 / 4.5 / 5 / 6 deviations: 250k reads of 100 bp, coarse table 602 / 599
// / 595 / 610 / 695 ms, 40k mixed reads 89.6 / 89.2 / 88.5 / 90.5 / 101.8, 60k of
// 150 bp at q = 6 57.6 / 56.8 / 56.9 / 57.3 / 63.9.)
constexpr float kCheckZ = 4.5f;
// The place is rounded to half blocks of 8 tokens: to the nearest, and of short
// ones most of them up, since a half block too many is cheaper there than looking
// again after each.  Uniform 100 bp reads, 600 Mbp, q = 5, sweeps in ms (rounded
// down / to the nearest / all up): one pass e = 0 2.85 / 2.82 / 2.85, e = 2 5.81 /
// 5.42 / 5.27, e = 5 9.20 / 9.05 / 8.93; coarse e = 0 1.80 / 1.78 / 1.68, e = 2 3.31 /
// 3.25 / 3.25, e = 5 5.99 / 6.01 / 6.06; 24 bp e = 0 3.73 / 3.68 / 3.42.
constexpr uint32_t kCheckShort = 48;
// Up to q = 4 most bins hold most tokens.  Where a token's share of misses is
// small their number is nearer a Poisson's than a normal's, and kCheckZ deviations
// put the check far too late: it comes there when the exponent of the tail
// (over ln(over / S) + (j - over) ln((j - over) / (j - S)), as much as kCheckZ
// deviations' kCheckZ^2 / 2) is large enough, cut down to halves.  Counts of 200
// reads of 150 bp against 15.1M bins, e = 0 743 -> 541 us, e = 2 1631 -> 1379; of 500
// reads of 80 bp against 19.7M, e = 0..5 17.8 -> 17.1 ms.  At q = 5 and 6 the two
// rules differ by less than 0.5%.
constexpr uint32_t kDenseRows = 256;

struct TokArgs {
  const char* reads;
  const uint64_t* offsets;
  const uint32_t* lens;
  const uint16_t* e;
  uint32_t n_reads, q, max_read_len, r4, ts, copies;
  const uint16_t* rank;  // IndexView::rank
  const float* miss;     // IndexView::miss
  float fine_power;      // fine_miss_power
  uint16_t* tokens;
  uint32_t* meta;
  Ctl* ctl;
  Live live;
  uint32_t max_e;
  uint64_t max_bases;
  const uint64_t* cand_off;  // list modes: the lists' CSR offsets
  uint64_t n_cand;
  uint32_t miss256;          // kLines: lookup_miss256
};

// One warp per read.  The read's tokens (row indices of the table: the token
// value for a clean q-gram, rowInvalid for one holding a non-base -- it still
// counts among the L-q+1 tokens and can never be found -- and rowPad after
// the last token) are written to tokens[(r*copies + k)*ts ...] in the order
// the filter kernel wants (a sum does not depend on it).  meta[r] =
// ntok | D' << 8 with D' = min(q*e, ntok): a bin passes iff at most D' of the
// read's tokens are missing from it, which is sum >= (L-q+1) - q*e.
//
// The bases become bit planes (one ballot for each of the code's bits and one
// for non-bases), so a lane cuts its q-grams out of registers with funnel
// shifts.
//
// kRarest (all bins, up to q = 5): q-grams with a non-base, which every bin
// misses, then the distinct tokens by ascending number of (super-)bins
// holding them, so that the all-bins kernels see misses as early as possible,
// then the repeats of a value already seen (a repeat misses exactly the bins
// its first occurrence misses; 1024-bin tiles: 1.7% fewer bit tests at q = 5).
// meta also gets the place in that order where a tile's bins are expected to
// be out but for a few (kCheckZ below): over 240 reads the number of tokens a
// tile really takes follows it with a correlation of 0.96 (reads of one length
// and budget) and 0.999 (mixed ones).
// The order is a counting sort without counters: every distinct token sets
// the bit of its rank in a bitmap of 4^q bits, and its place is the number of
// bits below.
//
// kCyclic (the 256-bin tiles of q = 6, copies = 4): a tile row is 32 bytes, so
// the row's bank group in shared memory is row & 3, and 16 reads of a warp
// loading random rows collide in bank groups.  The distinct tokens are dealt
// out round robin from the four row classes, each class rarest first (a
// bitmap for each), and copy k rotates every 16-token block by k positions.  A
// group g of the all-bins kernel reads copy g & 3, so at each load the warp's
// 16 groups cover the four bank groups four times each.  Every block holds the
// same tokens in every copy, so the per-block early exit and every sum are
// unchanged.
//
// kLines (candidate lists at q = 6): q-grams with a non-base first (misses
// that need no look-up), then the tokens grouped by the 128-byte line of a
// 512-byte bin vector that holds them (token >> 10), the line with the most
// tokens first, so that the list kernel's first look-ups touch as few lines
// of a vector as can rule the bin out.
//
// Bound by instruction issue.  Measured on GB300 against coding the bases
// through shared memory, q byte loads a token and a rank by comparing every
// pair of keys: 250k reads of 100 bp at q = 5 0.77 -> 0.29 ms, 60k of 150 bp at
// q = 6 0.91 -> 0.12 ms, 1M mixed reads in position order 0.85 -> 0.55 ms, a
// lone read of 250 bp 67 -> 16 us.
template <TokenOrder ORDER>
__global__ void __launch_bounds__(kTokWarps * 32, kTokCtasPerSm) k_tokenise(TokArgs a) {
  constexpr bool kRanked = ORDER == TokenOrder::kRarest || ORDER == TokenOrder::kCyclic;
  constexpr uint32_t kBitWords = ORDER == TokenOrder::kCyclic ? 128 : 32;
  __shared__ uint32_t s_bits[kRanked ? kTokWarps : 1][kBitWords];
  __shared__ __align__(16) uint16_t s_seq[kTokWarps][kMaxStride];
  const uint32_t lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const uint32_t below = (1u << lane) - 1u;
  const uint32_t n_warps = gridDim.x * kTokWarps;
  Ctl* ctl = a.ctl;
  const uint32_t q = a.q, r4 = a.r4;
  const uint32_t n_reads = live_reads(ctl, a.live, a.n_reads);
  // (an empty graph batch has lists to end somewhere too)
  if (n_reads == 0 && a.cand_off && blockIdx.x == 0 && threadIdx.x == 0 &&
      a.cand_off[0] != (a.live.on ? ctl->live_cand : a.n_cand))
    atomicOr(&ctl->status, kStatusBadCsr);
  // the extremes of this warp's reads (as in Ctl); raised once at the end: a
  // check of the shared words for every read is a load of one address for
  // every read, which takes longer than the tokens
  uint32_t max_d = 0, d_lo = 0, max_tight = 0, blk_max = 0, blk_lo = 0;
  uint32_t n_far = 0;  // kLines: reads past the look-ups
  for (uint64_t r = blockIdx.x * (uint64_t)kTokWarps + warp; r < n_reads; r += n_warps) {
    const uint32_t budget = a.e[r];
    if (budget > a.max_e && lane == 0) atomicOr(&ctl->status, kStatusArg);
    if (a.cand_off && lane == 0) {
      const uint64_t c0 = a.cand_off[r], c1 = a.cand_off[r + 1];
      if (c0 > c1 || (r + 1 == n_reads && c1 != (a.live.on ? ctl->live_cand : a.n_cand)))
        atomicOr(&ctl->status, kStatusBadCsr);
    }
    const uint32_t L = a.lens[r];
    const uint64_t off = a.offsets[r];
    bool bad = false;
    if (L < q) {
      if (lane == 0) atomicOr(&ctl->status, kStatusShort);
      bad = true;
    } else if (L > a.max_read_len || L - q + 1 > kMaxTokens) {
      if (lane == 0) atomicOr(&ctl->status, kStatusLong);
      bad = true;
    } else if (off > a.max_bases || L > a.max_bases - off) {  // past the end of the reads buffer
      if (lane == 0) atomicOr(&ctl->status, kStatusArg);
      bad = true;
    }
    const uint32_t ntok = bad ? 0 : L - q + 1;
    const uint32_t nb = bad ? 0 : L;

    // each base read once; every row starts as padding
    uint32_t ch[kTokRounds + 1];
#pragma unroll
    for (int i = 0; i <= kTokRounds; ++i)
      ch[i] = 32u * i + lane < nb ? (uint8_t)a.reads[off + 32u * i + lane] : 0u;
    const uint32_t pads = rowPad(r4) | (rowPad(r4) << 16);
    reinterpret_cast<uint4*>(s_seq[warp])[lane] = make_uint4(pads, pads, pads, pads);
    if constexpr (kRanked) {
#pragma unroll
      for (uint32_t w = 0; w < kBitWords; w += 32) s_bits[warp][w + lane] = 0;
    }
    __syncwarp();

    // bit planes of 32 bases: code bits and not-a-base (A0 C1 G2 T3, case folded)
    auto planes = [&](uint32_t c, uint32_t& lo, uint32_t& hi, uint32_t& inv) {
      const uint32_t u = c & 0xDFu;
      const uint32_t code = ((u >> 1) ^ (u >> 2)) & 3u;
      const bool ok = __byte_perm(0x54474341u, 0u, code | 0x4440u) == u;  // the code's letter
      lo = __ballot_sync(0xFFFFFFFFu, code & 1u);
      hi = __ballot_sync(0xFFFFFFFFu, code & 2u);
      inv = __ballot_sync(0xFFFFFFFFu, !ok);
    };
    const uint32_t qmask = (1u << q) - 1u;
    uint32_t row[kTokRounds], rk[kTokRounds], rep[kTokRounds];
    uint32_t lo0, hi0, inv0, n_inv = 0, n_rep = 0;
    uint32_t line_n[4] = {0, 0, 0, 0};  // kLines: tokens per line
    planes(ch[0], lo0, hi0, inv0);
#pragma unroll
    for (int i = 0; i < kTokRounds; ++i) {
      row[i] = rowPad(r4);
      rk[i] = rep[i] = 0;
      if (32u * i >= ntok) continue;  // the same for the warp
      uint32_t lo1, hi1, inv1;
      planes(ch[i + 1], lo1, hi1, inv1);
      const uint32_t lo = __funnelshift_r(lo0, lo1, lane) & qmask;
      const uint32_t hi = __funnelshift_r(hi0, hi1, lane) & qmask;
      const bool unclean = __funnelshift_r(inv0, inv1, lane) & qmask;
      lo0 = lo1;
      hi0 = hi1;
      inv0 = inv1;
      // interleave the two planes, first base most significant
      uint32_t z = __brev(lo | (hi << 16)) >> (16u - q);
      z = (z | (z << 4)) & 0x0F0F0F0Fu;
      z = (z | (z << 2)) & 0x33333333u;
      z = (z | (z << 1)) & 0x55555555u;
      const uint32_t t = ((z & 0xFFFFu) << 1) | (z >> 16);
      const bool in = 32u * i + lane < ntok;
      if (in) row[i] = unclean ? rowInvalid(r4) : t;
      if constexpr (ORDER == TokenOrder::kPosition) {
        if (in) s_seq[warp][32u * i + lane] = (uint16_t)row[i];
      } else {
        const uint32_t inv_mask = __ballot_sync(0xFFFFFFFFu, in && unclean);
        if (in && unclean)
          s_seq[warp][n_inv + __popc(inv_mask & below)] = (uint16_t)rowInvalid(r4);
        n_inv += __popc(inv_mask);
      }
      if constexpr (ORDER == TokenOrder::kLines) {
#pragma unroll
        for (uint32_t k = 0; k < 4; ++k)
          line_n[k] += __popc(__ballot_sync(0xFFFFFFFFu, row[i] < r4 && row[i] >> 10 == k));
      }
      if constexpr (kRanked) {
        const bool clean = row[i] < r4;
        bool seen = false;
        if (clean) {
          rk[i] = a.rank[row[i]];
          uint32_t w = rk[i] >> 5;
          if (ORDER == TokenOrder::kCyclic) w += 32u * (row[i] & 3u);
          seen = (atomicOr(&s_bits[warp][w], 1u << (rk[i] & 31u)) >> (rk[i] & 31u)) & 1u;
        }
        // of equal tokens in this round that are new to the read, exactly one
        // saw its bit clear, whichever came first; the lowest lane is taken as
        // the first occurrence so that the order is always the same
        uint32_t m = __ballot_sync(0xFFFFFFFFu, seen);
        for (uint32_t left = m; left;) {
          const uint32_t v = __shfl_sync(0xFFFFFFFFu, row[i], __ffs(left) - 1);
          const uint32_t same = __ballot_sync(0xFFFFFFFFu, row[i] == v);
          if (same & ~m) m = (m | same) & ~(same & (0u - same));
          left &= ~same;
        }
        rep[i] = m;
        n_rep += __popc(m);
      }
    }

    if constexpr (ORDER == TokenOrder::kLines) {
      uint32_t at[4];  // each line's first place
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        at[k] = n_inv;
#pragma unroll
        for (int i = 0; i < 4; ++i)
          if (line_n[i] > line_n[k] || (line_n[i] == line_n[k] && i < k)) at[k] += line_n[i];
      }
#pragma unroll
      for (int i = 0; i < kTokRounds; ++i) {
        if (32u * i >= ntok) continue;
#pragma unroll
        for (uint32_t k = 0; k < 4; ++k) {
          const bool mine = row[i] < r4 && row[i] >> 10 == k;
          const uint32_t m = __ballot_sync(0xFFFFFFFFu, mine);
          if (mine) s_seq[warp][at[k] + __popc(m & below)] = (uint16_t)row[i];
          at[k] += __popc(m);
        }
      }
    }
    if constexpr (kRanked) {
      __syncwarp();
      // bits below each word of the bitmap; kCyclic: of the four classes, a byte
      // each (at most 255 distinct tokens)
      uint32_t n = 0;
#pragma unroll
      for (uint32_t w = 0; w < kBitWords; w += 32) n |= __popc(s_bits[warp][w + lane]) << (w / 4);
      uint32_t incl = n;
#pragma unroll
      for (int d = 1; d < 32; d <<= 1) {
        const uint32_t t = __shfl_up_sync(0xFFFFFFFFu, incl, d);
        if (lane >= (uint32_t)d) incl += t;
      }
      const uint32_t pre = incl - n, tot = __shfl_sync(0xFFFFFFFFu, incl, 31);
      uint32_t rep_at = ntok - n_rep;
#pragma unroll
      for (int i = 0; i < kTokRounds; ++i) {
        if (32u * i >= ntok) continue;
        const uint32_t pw = __shfl_sync(0xFFFFFFFFu, pre, rk[i] >> 5);
        if (row[i] < r4) {
          uint32_t pos;
          if (rep[i] >> lane & 1u) {
            pos = rep_at + __popc(rep[i] & below);
          } else if constexpr (ORDER == TokenOrder::kCyclic) {
            const uint32_t c = row[i] & 3u;
            const uint32_t word = s_bits[warp][32u * c + (rk[i] >> 5)];
            const uint32_t x =
                ((pw >> (8 * c)) & 0xFFu) + __popc(word & ((1u << (rk[i] & 31u)) - 1u));
            // x rounds of the deal have passed, and the classes before c in this one
            pos = n_inv;
#pragma unroll
            for (uint32_t k = 0; k < 4; ++k) {
              const uint32_t tk = (tot >> (8 * k)) & 0xFFu;
              pos += min(tk, x + (k < c ? 1u : 0u));
            }
          } else {
            pos = n_inv + pw +
                  __popc(s_bits[warp][rk[i] >> 5] & ((1u << (rk[i] & 31u)) - 1u));
          }
          s_seq[warp][pos] = (uint16_t)row[i];
        }
        rep_at += __popc(rep[i]);
      }
    }
    __syncwarp();
    uint16_t* out = a.tokens + r * a.copies * a.ts;
    if constexpr (ORDER == TokenOrder::kCyclic) {
      // copy k: every 16-token block rotated by k positions
      for (uint32_t k = 0; k < a.copies; ++k) {
        uint32_t* o = reinterpret_cast<uint32_t*>(out + k * a.ts);
        for (uint32_t w = lane; w < a.ts / 2; w += 32) {
          const uint32_t p = 2u * w, blk = p & ~15u;
          o[w] = (uint32_t)s_seq[warp][blk | ((p + k) & 15u)] |
                 ((uint32_t)s_seq[warp][blk | ((p + 1u + k) & 15u)] << 16);
        }
      }
    } else {
      if (8u * lane < a.ts)
        reinterpret_cast<uint4*>(out)[lane] = reinterpret_cast<const uint4*>(s_seq[warp])[lane];
    }
    uint32_t d = q * budget;
    if (d > ntok) d = ntok;
    uint32_t meta = ntok | (d << 8);
    if constexpr (kRanked) {
      // (s_seq is complete: it was copied out above)
      const float over = (float)(d + 1u);
      float sum[2] = {0.f, 0.f};
      uint32_t at[2] = {0, 0};  // 1 + the check's place, coarse and fine
      const bool both = a.fine_power != 1.f;
      for (uint32_t j0 = 0; j0 < ntok && !(at[0] && at[1]); j0 += 32) {
        const uint32_t t = s_seq[warp][j0 + lane];
        const float miss = t < r4 ? a.miss[t] : t == rowInvalid(r4) ? 1.f : 0.f;
#pragma unroll
        for (int k = 0; k < 2; ++k) {
          if (k == 1 && !both) break;
          float incl = k == 0 ? miss : __powf(miss, a.fine_power);
#pragma unroll
          for (int dd = 1; dd < 32; dd <<= 1) {
            const float up = __shfl_up_sync(0xFFFFFFFFu, incl, dd);
            if (lane >= (uint32_t)dd) incl += up;
          }
          const float s = sum[k] + incl, n = (float)(j0 + lane + 1u), x = s - over;
          bool ok = j0 + lane < ntok && x > 0.f;
          if (r4 > kDenseRows)
            ok = ok && x * x * n >= kCheckZ * kCheckZ * s * (n - s);
          else  // (n - s is 0 for tokens that no bin holds)
            ok = ok && over * __logf(over / s) +
                               (n - over) * __logf((n - over) / fmaxf(n - s, 1e-6f)) >=
                           0.5f * kCheckZ * kCheckZ;
          const uint32_t hit = __ballot_sync(0xFFFFFFFFu, ok);
          if (hit && !at[k]) at[k] = j0 + __ffs(hit);
          sum[k] += __shfl_sync(0xFFFFFFFFu, incl, 31);
        }
        if (!both) at[1] = at[0];
      }
      // to halves: the nearest, or up where one makes a difference
      auto check = [&](uint32_t place) {
        const uint32_t p = place ? place : ntok;
        return min((p + (r4 <= kDenseRows ? 0u : p < kCheckShort ? 6u : 3u)) >> 3, 31u);
      };
      meta |= check(at[0]) << kMetaCheckCoarse;
      meta |= check(at[1]) << kMetaCheckFine;
      meta |= ((at[0] ? at[0] : ntok) >> 2) << kMetaOrder;
    }
    if (lane == 0) a.meta[r] = meta;
    const uint32_t nblk = (ntok + kBlockTokens - 1) / kBlockTokens;
    if constexpr (ORDER == TokenOrder::kLines) n_far += lookup_far(ntok, d, a.miss256);
    max_d = max(max_d, d);
    d_lo = max(d_lo, 255u - d);
    max_tight = max(max_tight, 255u - (ntok - d));
    blk_max = max(blk_max, nblk);
    blk_lo = max(blk_lo, 32u - nblk);
    __syncwarp();  // the row has been copied out
  }
  if (lane == 0) {
    // (skip the atomics once the extremes are reached)
    auto raise = [](uint32_t* p, uint32_t v) {
      if (v > *reinterpret_cast<volatile uint32_t*>(p)) atomicMax(p, v);
    };
    if (ORDER == TokenOrder::kLines && n_far) atomicAdd(&ctl->n_far, n_far);
    raise(&ctl->max_d, max_d);
    raise(&ctl->d_lo, d_lo);
    raise(&ctl->max_tight, max_tight);
    raise(&ctl->blk_max, blk_max);
    raise(&ctl->blk_lo, blk_lo);
  }
}

// Reads by descending order key, as given within a key (so that a batch is
// always grouped the same way): the keys of every block of reads are counted,
// then each block finds its places from the counts before it.
__global__ void __launch_bounds__(kOrderBlock) k_order_count(const uint32_t* __restrict__ meta,
                                                             uint32_t n_reads, uint32_t most,
                                                             uint32_t* __restrict__ order,
                                                             const Ctl* ctl, Live live) {
  __shared__ uint32_t s_n[kOrderKeys];
  if (ctl->status) return;
  n_reads = live_reads(ctl, live, n_reads);
  const uint32_t t = threadIdx.x, r = blockIdx.x * kOrderBlock + t;
  if (blockIdx.x * kOrderBlock >= n_reads) return;
  if (t < kOrderKeys) s_n[t] = 0;
  __syncthreads();
  if (r < n_reads) atomicAdd(&s_n[meta[r] >> kMetaOrder], 1u);
  __syncthreads();
  if (t < kOrderKeys) order[most + blockIdx.x * kOrderKeys + t] = s_n[t];
}

__global__ void __launch_bounds__(kOrderBlock) k_order_place(const uint32_t* __restrict__ meta,
                                                             uint32_t n_reads, uint32_t most,
                                                             uint32_t* __restrict__ order,
                                                             const Ctl* ctl, Live live) {
  constexpr uint32_t kWarps = kOrderBlock / 32;
  __shared__ uint32_t s_all[kOrderKeys], s_before[kOrderKeys];  // reads of a key; in earlier blocks
  __shared__ uint32_t s_warp[kWarps][kOrderKeys];
  if (ctl->status) return;
  n_reads = live_reads(ctl, live, n_reads);
  if (blockIdx.x * kOrderBlock >= n_reads) return;
  const uint32_t t = threadIdx.x, lane = t & 31, warp = t >> 5;
  const uint32_t r = blockIdx.x * kOrderBlock + t;
  const uint32_t blocks = (n_reads + kOrderBlock - 1) / kOrderBlock;
  if (t < kOrderKeys) s_all[t] = s_before[t] = 0;
  for (uint32_t i = t; i < kWarps * kOrderKeys; i += kOrderBlock) (&s_warp[0][0])[i] = 0;
  __syncthreads();
  {
    uint32_t all = 0, before = 0;
    for (uint32_t b = t / kOrderKeys; b < blocks; b += kOrderBlock / kOrderKeys) {
      const uint32_t n = order[most + b * kOrderKeys + t % kOrderKeys];
      all += n;
      if (b < blockIdx.x) before += n;
    }
    atomicAdd(&s_all[t % kOrderKeys], all);
    atomicAdd(&s_before[t % kOrderKeys], before);
  }
  const uint32_t key = r < n_reads ? meta[r] >> kMetaOrder : kOrderKeys;
  const uint32_t same = __match_any_sync(0xFFFFFFFFu, key);
  const uint32_t rank = __popc(same & ((1u << lane) - 1u));
  if (r < n_reads && rank == 0) s_warp[warp][key] = __popc(same);
  __syncthreads();
  if (r < n_reads) {
    uint32_t at = s_before[key] + rank;
    for (uint32_t k = key + 1; k < kOrderKeys; ++k) at += s_all[k];  // longer reads come first
    for (uint32_t w = 0; w < warp; ++w) at += s_warp[w][key];
    order[at] = r;
  }
}

// Reverse complement, one warp per read: out[off + L-1-j] = comp(reads[off + j])
// with A<->T and C<->G in either case (case kept); other bytes unchanged.
__global__ void k_reverse_complement(const char* __restrict__ reads,
                                     const uint64_t* __restrict__ offsets,
                                     const uint32_t* __restrict__ lens, uint32_t n_reads,
                                     char* __restrict__ out) {
  const uint64_t r = (blockIdx.x * (uint64_t)blockDim.x + threadIdx.x) >> 5;
  const uint32_t lane = threadIdx.x & 31;
  if (r >= n_reads) return;
  const uint64_t off = offsets[r];
  const uint32_t L = lens[r];
  for (uint32_t j = lane; j < L; j += 32) {
    const uint32_t c = (uint8_t)reads[off + j];
    const uint32_t u = c & 0xDFu, low = c & 0x20u;
    uint32_t d = c;
    if (u == 0x41u) d = 0x54u | low;       // A -> T
    else if (u == 0x54u) d = 0x41u | low;  // T -> A
    else if (u == 0x43u) d = 0x47u | low;  // C -> G
    else if (u == 0x47u) d = 0x43u | low;  // G -> C
    out[off + L - 1 - j] = (char)d;
  }
}

}  // namespace

void launch_reverse_complement(const char* reads, const uint64_t* offsets, const uint32_t* lens,
                               uint32_t n_reads, char* out, cudaStream_t st) {
  if (n_reads == 0) return;
  const uint32_t threads = 256;
  const uint64_t grid = ((uint64_t)n_reads * 32 + threads - 1) / threads;
  k_reverse_complement<<<(unsigned)grid, threads, 0, st>>>(reads, offsets, lens, n_reads, out);
}

void launch_tokenise(const char* reads, const uint64_t* offsets, const uint32_t* lens,
                     const uint16_t* e, const IndexView& ix, ReadsView rv, uint16_t* tokens,
                     uint32_t* meta, Ctl* ctl, cudaStream_t st, const uint64_t* cand_off,
                     uint64_t n_cand, float fine_power, Live live, uint32_t max_e,
                     uint64_t max_bases) {
  if (rv.n_reads == 0) return;
  const uint32_t threads = kTokWarps * 32;
  int dev = 0, sms = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  const uint64_t need = ((uint64_t)rv.n_reads + kTokWarps - 1) / kTokWarps;
  const uint64_t most = (uint64_t)(sms > 0 ? sms : 1) * kTokCtasPerSm;
  const uint64_t grid = need < most ? need : most;
  const TokArgs a{reads, offsets, lens,   e,    rv.n_reads, ix.q, ix.max_read_len, ix.r4,    rv.ts,
                  rv.copies, ix.rank, ix.miss, fine_power, tokens, meta, ctl, live, max_e, max_bases,
                  cand_off, n_cand, cand_off && ix.wpb > 32 ? lookup_miss256(ix) : 0u};
  // lists read whole token rows in any order up to 128-byte vectors; larger
  // ones (q = 6) are looked up line by line
  auto kernel = cand_off        ? (ix.wpb > 32 ? k_tokenise<TokenOrder::kLines>
                                               : k_tokenise<TokenOrder::kPosition>)
                : rv.copies > 1 ? k_tokenise<TokenOrder::kCyclic>
                                : k_tokenise<TokenOrder::kRarest>;
  ProfScope ps("tokenise", st);
  kernel<<<(unsigned)grid, threads, 0, st>>>(a);
}

void launch_order(const ReadsView& rv, uint32_t* order, const Ctl* ctl, cudaStream_t st,
                  Live live) {
  if (!order) return;
  const uint32_t grid = (rv.n_reads + kOrderBlock - 1) / kOrderBlock;
  ProfScope ps("order", st);
  k_order_count<<<grid, kOrderBlock, 0, st>>>(rv.meta, rv.n_reads, rv.n_reads, order, ctl, live);
  k_order_place<<<grid, kOrderBlock, 0, st>>>(rv.meta, rv.n_reads, rv.n_reads, order, ctl, live);
}

}  // namespace grim
