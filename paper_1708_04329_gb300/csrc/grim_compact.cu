// Stream compaction of the passing (read, bin, count) records
// (§Mapping GRIM-Filter: the filter's result per read is a vector over bins;
// here only the set entries are kept, read by read).
//
// The filter kernels append records in whatever order their warps finish, so
// the order is restored by a least-significant-digit radix sort on the record
// key -- (read << bin_bits | bin) in all-bins mode, the global candidate index
// in candidate mode; keys are unique, so the output order is unique too.
// Each 8-bit pass is a per-block digit histogram, a scan of each digit over
// the blocks, and a stable scatter (per-warp ranks from
// __match_any_sync, then warp order, then round order).  A last kernel splits
// the keys into the caller's read / bin / count arrays.  Short lists skip the
// radix sort: one kernel places each record by counting the smaller keys.
#include "grim_internal.cuh"

namespace grim {
namespace {

constexpr uint32_t kSortThreads = 256;
constexpr uint32_t kSortItems = 16;  // per thread per pass
constexpr uint32_t kSortTile = kSortThreads * kSortItems;

// Live record counts: *n_live (capped at n) when n_live is set, else n.
__device__ __forceinline__ uint64_t live_n(const unsigned long long* n_live, uint64_t n) {
  if (!n_live) return n;
  const uint64_t v = *n_live;
  return v < n ? v : n;
}

__global__ void __launch_bounds__(kSortThreads) k_rs_hist(const unsigned long long* __restrict__ keys,
                                                          uint64_t n, uint32_t shift,
                                                          uint32_t* __restrict__ hist, uint32_t nb,
                                                          const unsigned long long* n_live) {
  __shared__ uint32_t cnt[256];
  n = live_n(n_live, n);
  if ((uint64_t)blockIdx.x * kSortTile >= n) return;  // past the live records
  cnt[threadIdx.x] = 0;
  __syncthreads();
  const uint64_t base = (uint64_t)blockIdx.x * kSortTile;
  for (uint32_t i = 0; i < kSortItems; ++i) {
    const uint64_t idx = base + (uint64_t)i * kSortThreads + threadIdx.x;
    if (idx < n) atomicAdd(&cnt[(keys[idx] >> shift) & 0xFFu], 1u);
  }
  __syncthreads();
  hist[(uint64_t)threadIdx.x * nb + blockIdx.x] = cnt[threadIdx.x];
}

// Inclusive scan over the live blocks of each digit's row of the histogram
// (entry (d, blk) at h[d * nb + blk]), a CTA per digit; the scatter adds the
// smaller digits' totals, the rows' last entries.  One CTA scanning all 256
// rows took 35 us a pass at 1M records, this 6.
__device__ __forceinline__ uint32_t block_inclusive(uint32_t v, uint32_t* s_warp) {
  const uint32_t lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  uint32_t incl = v;
#pragma unroll
  for (int d = 1; d < 32; d <<= 1) {
    const uint32_t t = __shfl_up_sync(0xFFFFFFFFu, incl, d);
    if (lane >= (uint32_t)d) incl += t;
  }
  if (lane == 31) s_warp[warp] = incl;
  __syncthreads();
  for (uint32_t w = 0; w < warp; ++w) incl += s_warp[w];
  __syncthreads();
  return incl;
}

__global__ void __launch_bounds__(kSortThreads) k_rs_scan(uint32_t* __restrict__ h, uint64_t nb,
                                                          uint64_t n,
                                                          const unsigned long long* n_live) {
  __shared__ uint32_t s_warp[kSortThreads / 32], s_carry;
  n = live_n(n_live, n);
  const uint32_t nb_live = (uint32_t)((n + kSortTile - 1) / kSortTile);
  uint32_t* row = h + blockIdx.x * nb;
  uint32_t carry = 0;
  for (uint32_t c = 0; c < nb_live; c += kSortThreads) {
    const uint32_t i = c + threadIdx.x;
    const uint32_t incl = carry + block_inclusive(i < nb_live ? row[i] : 0u, s_warp);
    if (i < nb_live) row[i] = incl;
    if (threadIdx.x == kSortThreads - 1) s_carry = incl;
    __syncthreads();
    carry = s_carry;
  }
}

__global__ void __launch_bounds__(kSortThreads) k_rs_scatter(
    const unsigned long long* __restrict__ kin, const uint8_t* __restrict__ cin,
    unsigned long long* __restrict__ kout, uint8_t* __restrict__ cout, uint64_t n, uint32_t shift,
    const uint32_t* __restrict__ hist, uint32_t nb, const unsigned long long* n_live) {
  constexpr uint32_t kW = kSortThreads / 32;
  __shared__ uint32_t s_base[256];
  __shared__ uint32_t s_wcnt[kW][256];
  n = live_n(n_live, n);
  if ((uint64_t)blockIdx.x * kSortTile >= n) return;  // past the live records
  const uint32_t tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  {  // places of this block's first record of each digit
    static_assert(kSortThreads == 256, "a thread per digit");
    const uint32_t* row = hist + (uint64_t)tid * nb;
    const uint32_t all = row[(n + kSortTile - 1) / kSortTile - 1];
    const uint32_t before = block_inclusive(all, &s_wcnt[0][0]) - all;
    s_base[tid] = before + (blockIdx.x ? row[blockIdx.x - 1] : 0u);
  }
  const uint64_t base = (uint64_t)blockIdx.x * kSortTile;
  for (uint32_t round = 0; round < kSortItems; ++round) {
    for (uint32_t i = tid; i < kW * 256; i += kSortThreads) (&s_wcnt[0][0])[i] = 0;
    __syncthreads();
    const uint64_t idx = base + (uint64_t)round * kSortThreads + tid;
    const bool valid = idx < n;
    unsigned long long key = valid ? kin[idx] : 0ull;
    const uint8_t c = valid ? cin[idx] : (uint8_t)0;
    const uint32_t d = (uint32_t)(key >> shift) & 0xFFu;
    // invalid lanes get a value no valid digit has, so they never match
    const uint32_t peers = __match_any_sync(0xFFFFFFFFu, valid ? d : 256u + lane);
    const uint32_t rank = __popc(peers & ((1u << lane) - 1u));
    if (valid && rank == 0) s_wcnt[warp][d] = __popc(peers);
    __syncthreads();
    if (valid) {
      uint32_t off = s_base[d] + rank;
      for (uint32_t w = 0; w < warp; ++w) off += s_wcnt[w][d];
      kout[off] = key;
      cout[off] = c;
    }
    __syncthreads();
    uint32_t add = 0;
    for (uint32_t w = 0; w < kW; ++w) add += s_wcnt[w][tid];
    s_base[tid] += add;
    __syncthreads();  // s_wcnt is cleared again at the top of the next round
  }
}

// One record into the caller's arrays at position i.
struct EmitArgs {
  bool cand_mode;
  uint32_t bin_bits;
  const int32_t* cand;
  const uint64_t* cand_off;
  uint32_t n_reads;
  uint32_t* out_read;
  uint32_t* out_bin;
  uint8_t* out_count;
};
__device__ __forceinline__ void emit_record(const EmitArgs& e, uint64_t i, unsigned long long key,
                                            uint8_t count, uint32_t n_reads) {
  uint32_t r, b;
  if (e.cand_mode) {
    b = (uint32_t)e.cand[key];
    // largest r with cand_off[r] <= key
    uint32_t lo = 0, hi = n_reads - 1;
    while (lo < hi) {
      const uint32_t mid = lo + (hi - lo + 1) / 2;
      if (e.cand_off[mid] <= key) lo = mid;
      else hi = mid - 1;
    }
    r = lo;
  } else {
    r = (uint32_t)(key >> e.bin_bits);
    b = (uint32_t)(key & ((e.bin_bits >= 64) ? ~0ull : ((1ull << e.bin_bits) - 1ull)));
  }
  e.out_read[i] = r;
  e.out_bin[i] = b;
  e.out_count[i] = count;
}

__global__ void k_emit(const unsigned long long* __restrict__ keys,
                       const uint8_t* __restrict__ counts, uint64_t n, EmitArgs e,
                       const unsigned long long* n_live, const uint32_t* n_reads_live) {
  const uint64_t i = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x;
  if (i >= live_n(n_live, n)) return;
  emit_record(e, i, keys[i], counts[i], n_reads_live ? *n_reads_live : e.n_reads);
}

// Short pass lists: a record's place is the number of smaller keys, counted
// outright.  kRankSplit threads share a record and the block walks all keys
// through shared memory, so sorting and splitting n records is one launch of
// n^2 compares instead of the radix sort's three launches per key byte.
// Measured on GB300 (rank against radix with two-byte keys, events around each
// launch, us): 64 records 7 / 31, 2,048 9.5 / 61, 8,192 27 / 77, 16,384 75 /
// 78, 32,768 273 / 86: the line (kRankMax) is drawn where the compares still
// hide behind the launches they replace.  The number of records is read on the
// device, so the launch need not wait for the host to learn it.
constexpr uint32_t kRankThreads = 256;
constexpr uint32_t kRankSplit = 16;    // threads per record
constexpr uint32_t kRankChunk = 2048;  // keys in shared memory at a time
__global__ void __launch_bounds__(kRankThreads) k_rank_emit(
    const unsigned long long* __restrict__ keys, const uint8_t* __restrict__ counts,
    const unsigned long long* n_live, uint64_t limit, EmitArgs e, const Ctl* ctl) {
  __shared__ unsigned long long s_key[kRankChunk];
  if (ctl->status || *n_live > limit) return;
  const uint32_t n = (uint32_t)*n_live;
  if (blockIdx.x * (kRankThreads / kRankSplit) >= n) return;
  const uint32_t i = (blockIdx.x * kRankThreads + threadIdx.x) / kRankSplit;
  const uint32_t part = threadIdx.x % kRankSplit;
  const unsigned long long key = i < n ? keys[i] : 0ull;
  uint32_t rank = 0;
  for (uint32_t c0 = 0; c0 < n; c0 += kRankChunk) {
    const uint32_t m = min(kRankChunk, n - c0);
    __syncthreads();
    for (uint32_t j = threadIdx.x; j < m; j += kRankThreads) s_key[j] = keys[c0 + j];
    __syncthreads();
#pragma unroll 8
    for (uint32_t j = part; j < m; j += kRankSplit) rank += s_key[j] < key;
  }
#pragma unroll
  for (uint32_t d = 1; d < kRankSplit; d <<= 1) rank += __shfl_xor_sync(0xFFFFFFFFu, rank, d);
  if (i < n && part == 0) emit_record(e, rank, key, counts[i], e.n_reads);
}

}  // namespace

uint64_t sort_workspace_bytes(uint64_t cap) {
  const uint64_t nb = (cap + kSortTile - 1) / kSortTile;
  return 256ull * (nb ? nb : 1) * sizeof(uint32_t);
}

RecordsView sort_records(RecordsView a, RecordsView b, uint64_t n, uint32_t key_bits, void* hist,
                         cudaStream_t st, const unsigned long long* n_live) {
  if (n == 0) return a;
  const uint32_t nb = (uint32_t)((n + kSortTile - 1) / kSortTile);
  uint32_t* h = static_cast<uint32_t*>(hist);
  RecordsView src = a, dst = b;
  const uint32_t passes = (key_bits + 7) / 8;
  for (uint32_t p = 0; p < passes; ++p) {
    const uint32_t shift = 8 * p;
    {
      ProfScope ps("sort_hist", st);
      k_rs_hist<<<nb, kSortThreads, 0, st>>>(src.keys, n, shift, h, nb, n_live);
    }
    {
      ProfScope ps("sort_scan", st);
      k_rs_scan<<<256, kSortThreads, 0, st>>>(h, nb, n, n_live);
    }
    {
      ProfScope ps("sort_scatter", st);
      k_rs_scatter<<<nb, kSortThreads, 0, st>>>(src.keys, src.counts, dst.keys, dst.counts, n,
                                                shift, h, nb, n_live);
    }
    RecordsView t = src;
    src = dst;
    dst = t;
  }
  return src;
}

void rank_and_emit(const RecordsView& a, const unsigned long long* n_live, uint64_t limit,
                   bool candidate_mode, uint32_t bin_bits, const int32_t* cand,
                   const uint64_t* cand_off, uint32_t n_reads, uint32_t* out_read,
                   uint32_t* out_bin, uint8_t* out_count, const Ctl* ctl, cudaStream_t st) {
  if (limit > kRankMax) limit = kRankMax;
  if (limit == 0) return;
  const EmitArgs e{candidate_mode, bin_bits, cand, cand_off, n_reads, out_read, out_bin, out_count};
  ProfScope ps("rank_emit", st);
  k_rank_emit<<<(unsigned)((limit * kRankSplit + kRankThreads - 1) / kRankThreads), kRankThreads, 0,
                st>>>(a.keys, a.counts, n_live, limit, e, ctl);
}

void sort_and_emit(RecordsView a, RecordsView b, uint64_t n, uint32_t key_bits, void* hist,
                   bool candidate_mode, uint32_t bin_bits, const int32_t* cand,
                   const uint64_t* cand_off, uint32_t n_reads, uint32_t* out_read,
                   uint32_t* out_bin, uint8_t* out_count, cudaStream_t st,
                   const unsigned long long* n_live, const uint32_t* n_reads_live) {
  if (n == 0) return;
  const EmitArgs e{candidate_mode, bin_bits, cand, cand_off, n_reads, out_read, out_bin, out_count};
  const RecordsView src = sort_records(a, b, n, key_bits, hist, st, n_live);
  ProfScope ps("emit", st);
  k_emit<<<(unsigned)((n + 255) / 256), 256, 0, st>>>(src.keys, src.counts, n, e, n_live,
                                                      n_reads_live);
}

}  // namespace grim
