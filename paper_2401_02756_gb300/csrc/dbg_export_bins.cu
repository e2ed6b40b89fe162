// The sorted export by bins: the occupied slots' records are placed straight
// into the order of their keys' leading bits, and every stretch of a few
// thousand of them is then sorted in shared memory.
//
//   histogram -- the table read once: vertices per bin (the keys' top B bits),
//                and a bit for every slot that holds one;
//   plan      -- the bins' prefix sum; bins are joined into buckets of about
//                T records (bucket of a bin = its first position / T);
//   place     -- those slots read again: every record to the next free position
//                of its bin (one atomic a record on the bin's counter);
//   sort      -- a CTA per bucket: a counting sort by the bits that follow,
//                then every key's rank among the few that share its bin, and
//                keys and counter rows out in order, coalesced.
//
// So a record moves twice and no slot is read at random.  The radix sort of
// (32-bit prefix, slot index) pairs this replaces moved 16 bytes a record four
// times, gathered a random slot per vertex and put runs of equal prefixes in
// order in two more passes.  Export of 422.6 M vertices of a 20.8 GB table
// 35.4 -> 22.6 ms (histogram 4.1, place 12 to 12.9 from card to card, sort 5.9;
// 1.2 more with the counters at the slot's byte 8, two loads a row), of 57 M 5.1 ->
// 2.8 ms; k = 51, 75 M vertices (two 64-bit radix sorts before) 19.7 -> 4.2 ms.
//
// The place pass is at the rate of its stores.  A store to a sector that is
// not in the L2 costs one of about 4.1e10 misses a second however many of its
// line's other sectors were written just before (measured: 32-byte stores to
// 1,024 or to a million advancing tails alike, 128-byte ones four times the
// bytes), 10.3 ms for the 422.6 M; its reads and atomics hide behind that.
//
// The placed records go to 32-byte records of scratch when there is room for
// them -- a full sector per scattered store -- and otherwise straight to the
// outputs, which the sort then reorders in place (an 8- and a 16-byte store a
// record, 1.5 times the time, but no memory beyond the bins' is needed).
//
// Genomes of uneven base composition and repeats fill some bins far beyond the
// others.  A bucket with more records than its CTA's shared memory holds is
// skipped by the sort; the records of all such buckets are then sorted together
// by their whole keys, by a radix sort, and written back (56 bytes of scratch a
// record at most).  They are few: export of 432 M vertices (2^22 bins) at 50 / 40 /
// 35 / 30 % GC 22.9 / 22.9 / 23.8 / 28.7 ms, with none, none, 1 % and 11 % of the
// records in such buckets (a radix sort of all: 35.6 to 41.3).
// Graphs with a quarter of their records in such buckets are left to the radix
// sort as a whole.
#include <cub/device/device_radix_sort.cuh>

#include <algorithm>

#include "dbg_export.cuh"
#include "dbg_internal.cuh"

namespace dbg {
namespace {

constexpr int kSortBlock = 256;
constexpr int kLocalBits = 11;  // bins of the shared-memory counting sort
constexpr int kLocalBins = 1 << kLocalBits;
constexpr int kBinBits = 20, kBinLog2 = 7;  // bins: up to 2^20, or for 2^7 records each
constexpr int kPlanBins = 8192;  // up to this many: the plan is one CTA's work
constexpr int kPlanBlock = 1024;
constexpr int kChunkBlock = 256, kChunkPer = 16;  // more: a CTA for 4,096 bins
constexpr uint32_t kChunkBins = kChunkBlock * kChunkPer;
constexpr int kSlotsPerThread = 4;
constexpr int kCursorStride = 8;  // a bucket's cursor has a sector of its own
constexpr uint32_t kCursorBins = 1u << 17;  // in place: bucket cursors above so many bins
constexpr uint64_t kMaxPooledRecords = 4ull << 30;  // (what the pool keeps between calls)

constexpr uint32_t kBucketCap = 2048;  // records a bucket may hold
constexpr uint64_t kCrowdedShare = 4;  // at most one record in so many may lie in larger ones

struct ExportMeta {
  unsigned long long spilled;
  unsigned long long crowded;  // records in buckets of more than kBucketCap, at most
  uint32_t vertices, status;
};

// Everything the kernels share.
struct Plan {
  int key_bits;         // 2 (k - 1)
  int bin_bits;         // B
  int bucket_log2;      // T = 2^bucket_log2
  uint32_t buckets;     // last entry of the bucket arrays (a graph of more vertices is not placed)
  uint64_t max_rows;    // rows of the outputs
  uint64_t max_placed;  // records the scratch holds (place into 32-byte records)
  uint64_t max_crowded; // records that may lie in buckets above the cap
  uint2 *sums;          // [2^B / kChunkBins] records of a chunk of bins, of its last bin
  uint32_t *taken;      // a bit per slot: it holds a vertex (or null)
  uint32_t *bins;       // [2^B + 1] histogram, then exclusive prefix, then next free position
  uint32_t *start;      // [buckets + 2] first position of a bucket
  uint32_t *first_bin;  // [buckets + 2]
  uint32_t *cursor;     // [buckets + 2][kCursorStride] next free position, or null: the bins' own
  ExportMeta *meta;
  ExportMeta *report;   // the sort's copy of it in pinned host memory, or null
};

// Whether the placing and the sort may run: a complete graph, room for it,
// and few records in buckets above the cap.
__device__ __forceinline__ bool may_run(const Plan &p) {
  const ExportMeta m = *p.meta;
  return m.status == 0u && m.spilled == 0ull && m.vertices <= p.max_rows &&
         m.vertices <= p.max_placed && m.crowded <= p.max_crowded;
}

// Records a bin of n can put into a bucket above the cap: its own and those of
// the bins before it in its bucket (fewer than 2^bucket_log2).
__device__ __forceinline__ unsigned long long crowd(const Plan &p, uint32_t n) {
  const uint32_t T = 1u << p.bucket_log2;
  return n > kBucketCap - T ? (unsigned long long)n + T : 0ull;
}

// A key as one or two words.  aligned(): its leading 64 bits, from the top.
template <bool WIDE>
struct Key;
template <>
struct Key<false> {
  unsigned long long w;
  __device__ __forceinline__ uint64_t aligned(int bits) const { return w << (64 - bits); }
  __device__ __forceinline__ bool operator<(const Key &o) const { return w < o.w; }
  __device__ __forceinline__ bool empty() const { return w == kEmpty; }
};
template <>
struct Key<true> {
  unsigned long long hi, lo;
  __device__ __forceinline__ uint64_t aligned(int bits) const {
    const int h = bits - 64;  // bits of the high word, 0 .. 62
    return h == 0 ? lo : (hi << (64 - h)) | (lo >> h);
  }
  __device__ __forceinline__ bool operator<(const Key &o) const {
    return hi < o.hi || (hi == o.hi && lo < o.lo);
  }
  __device__ __forceinline__ bool empty() const { return hi == kEmpty; }
};

// The table goes past the L2 (evict_first), the bins' counters stay in it
// (evict_last): 2^22 bins of 432 M records 25.1 -> 23.9 ms an export, as 2^21 take
// (with four slots a thread in flight).
__device__ __forceinline__ uint32_t next_place(uint32_t *bin, uint64_t pol) {
  uint32_t at;
  asm volatile("atom.relaxed.gpu.global.add.L2::cache_hint.u32 %0, [%1], 1, %2;"
               : "=r"(at)
               : "l"(bin), "l"(pol)
               : "memory");
  return at;
}

// A 32-byte slot in one load, and a 32-byte record in one store.
struct Words {
  uint32_t w[8];
};
__device__ __forceinline__ Words ld_slot(const Slot *p) {
  Words v;
  asm volatile("ld.global.L1::no_allocate.L2::evict_first.v8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
               : "=r"(v.w[0]), "=r"(v.w[1]), "=r"(v.w[2]), "=r"(v.w[3]), "=r"(v.w[4]),
                 "=r"(v.w[5]), "=r"(v.w[6]), "=r"(v.w[7])
               : "l"(p));
  return v;
}
__device__ __forceinline__ void st_record(Slot *p, const Words &v) {
  st_sector(p, v.w[0], v.w[1], v.w[2], v.w[3], v.w[4], v.w[5], v.w[6], v.w[7]);
}

__device__ __forceinline__ unsigned long long word64(uint32_t lo, uint32_t hi) {
  return (unsigned long long)lo | ((unsigned long long)hi << 32);
}
template <bool WIDE>
__device__ __forceinline__ Key<WIDE> key_of(const Words &v) {
  if constexpr (WIDE)
    return Key<true>{word64(v.w[0], v.w[1]), word64(v.w[2], v.w[3])};
  else
    return Key<false>{word64(v.w[0], v.w[1])};
}
template <bool WIDE>
__device__ __forceinline__ uint4 row_of(const Words &v) {
  return WIDE ? make_uint4(v.w[4], v.w[5], v.w[6], v.w[7])
              : make_uint4(v.w[2], v.w[3], v.w[4], v.w[5]);
}
// A placed record: a one-word slot's counters come first, so that its row is
// one aligned 16-byte load in the sort (a two-word slot's row already is).
template <bool WIDE>
__device__ __forceinline__ Words record_of(const Words &v) {
  if constexpr (WIDE) return v;
  return Words{{v.w[2], v.w[3], v.w[4], v.w[5], v.w[0], v.w[1], 0u, 0u}};
}
template <bool WIDE>
__device__ __forceinline__ Key<WIDE> ld_record_key(const Slot *p) {
  if constexpr (WIDE) {
    const uint4 a = *reinterpret_cast<const uint4 *>(p);
    return Key<true>{word64(a.x, a.y), word64(a.z, a.w)};
  } else {
    return Key<false>{*(reinterpret_cast<const unsigned long long *>(p) + 2)};
  }
}
template <bool WIDE>
__device__ __forceinline__ Key<WIDE> ld_key(const Slot *p) {
  if constexpr (WIDE) {
    const uint4 a = __ldcs(reinterpret_cast<const uint4 *>(p));
    return Key<true>{word64(a.x, a.y), word64(a.z, a.w)};
  } else {
    return Key<false>{__ldcs(&p->key)};
  }
}

// Vertices per bin, and the slots that hold one.  Bound by one read of the table.
template <bool WIDE>
__global__ void __launch_bounds__(256) k_histogram(const Slot *t, uint64_t n, Plan p) {
  after_previous();
  const uint64_t stride = (uint64_t)gridDim.x * blockDim.x;
  const uint32_t lane = threadIdx.x & 31u;
  for (uint64_t i = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; i - lane < n;
       i += stride * kSlotsPerThread) {
    Key<WIDE> k[kSlotsPerThread];
#pragma unroll
    for (int u = 0; u < kSlotsPerThread; ++u) {
      const uint64_t j = i + u * stride;
      if (j < n)
        k[u] = ld_key<WIDE>(t + j);
      else
        memset(&k[u], 0xff, sizeof(k[u]));
    }
    if (p.taken) {
#pragma unroll
      for (int u = 0; u < kSlotsPerThread; ++u) {
        const uint32_t m = __ballot_sync(0xffffffffu, !k[u].empty());
        const uint64_t j = i + u * stride;
        if (lane == 0 && j < n) p.taken[j >> 5] = m;
      }
    }
#pragma unroll
    for (int u = 0; u < kSlotsPerThread; ++u)
      if (!k[u].empty())
        red_add_u32(&p.bins[k[u].aligned(p.key_bits) >> (64 - p.bin_bits)], 1u);
  }
}

// Bin i of the prefix (nbins: the end): opens every bucket from the one after
// the previous bin's to its own.
__device__ __forceinline__ void open_buckets(const Plan &p, uint32_t i, uint32_t nbins,
                                             uint32_t at, uint32_t before) {
  const uint32_t id = i < nbins ? at >> p.bucket_log2 : (at >> p.bucket_log2) + 1u;
  for (uint32_t b = i == 0 ? 0u : (before >> p.bucket_log2) + 1u; b <= min(id, p.buckets); ++b) {
    p.start[b] = at;
    if (p.cursor) p.cursor[b * kCursorStride] = at;
    p.first_bin[b] = i;
  }
}

__device__ __forceinline__ void fill_meta(const Plan &p, uint32_t vertices, const uint32_t *status,
                                          const unsigned long long *spilled) {
  p.meta->vertices = vertices;
  p.meta->status = ld_volatile_u32(status);
  p.meta->spilled = *(const volatile unsigned long long *)spilled;
}

// The plan of up to kPlanBins bins in one CTA: prefix, buckets, crowded bins.
__global__ void __launch_bounds__(kPlanBlock)
    k_plan(Plan p, const uint32_t *status, const unsigned long long *spilled) {
  after_previous();
  constexpr int kPer = kPlanBins / kPlanBlock;
  __shared__ uint32_t s_warp[32], s_last[kPlanBlock + 1];
  const uint32_t nbins = 1u << p.bin_bits;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const uint32_t i0 = threadIdx.x * kPer;
  uint32_t c[kPer], local = 0;
  unsigned long long crowded = 0;
#pragma unroll
  for (int q = 0; q < kPer; ++q) {
    c[q] = i0 + q < nbins ? p.bins[i0 + q] : 0u;
    local += c[q];
    crowded += crowd(p, c[q]);
  }
  uint32_t incl = local;
  for (int d = 1; d < 32; d <<= 1) {
    const uint32_t o = __shfl_up_sync(0xffffffffu, incl, d);
    if (lane >= d) incl += o;
  }
  if (lane == 31) s_warp[warp] = incl;
  __syncthreads();
  uint32_t w = s_warp[lane];
  for (int d = 1; d < 32; d <<= 1) {
    const uint32_t o = __shfl_up_sync(0xffffffffu, w, d);
    if (lane >= d) w += o;
  }
  const uint32_t total = __shfl_sync(0xffffffffu, w, 31);
  const uint32_t below = __shfl_sync(0xffffffffu, w, (warp + 31) & 31);
  uint32_t at = incl - local + (warp > 0 ? below : 0u);
  s_last[threadIdx.x + 1] = at + local - c[kPer - 1];  // the thread's last bin starts here
  __syncthreads();
  uint32_t before = threadIdx.x ? s_last[threadIdx.x] : 0u;
#pragma unroll
  for (int q = 0; q < kPer; ++q) {
    const uint32_t i = i0 + q;
    if (i > nbins) break;
    p.bins[i] = at;
    open_buckets(p, i, nbins, at, before);
    before = at;
    at += c[q];
  }
  if (threadIdx.x == kPlanBlock - 1 && nbins == kPlanBins) {  // the end comes after the last bin
    p.bins[nbins] = total;
    open_buckets(p, nbins, nbins, total, before);
  }
  if (crowded) atomicAdd(&p.meta->crowded, crowded);
  if (threadIdx.x == 0) fill_meta(p, total, status, spilled);
}

// kChunkPer bins of the calling thread in its CTA's chunk.
__device__ __forceinline__ void load_bins(const Plan &p, uint32_t (&c)[kChunkPer]) {
  const uint4 *in = reinterpret_cast<const uint4 *>(p.bins + (size_t)blockIdx.x * kChunkBins) +
                    threadIdx.x * (kChunkPer / 4);
#pragma unroll
  for (int q = 0; q < kChunkPer / 4; ++q) {
    const uint4 v = in[q];
    c[4 * q] = v.x;
    c[4 * q + 1] = v.y;
    c[4 * q + 2] = v.z;
    c[4 * q + 3] = v.w;
  }
}

// Sum over the CTA (kChunkBlock threads), for every thread.
__device__ __forceinline__ uint32_t chunk_sum(uint32_t v, uint32_t *s_warp) {
  v = __reduce_add_sync(0xffffffffu, v);
  if ((threadIdx.x & 31) == 0) s_warp[threadIdx.x >> 5] = v;
  __syncthreads();
  uint32_t sum = 0;
#pragma unroll
  for (int w = 0; w < kChunkBlock / 32; ++w) sum += s_warp[w];
  __syncthreads();
  return sum;
}

// More bins, first pass: the records of every chunk of bins (and of its last
// bin), and the crowded bins.
__global__ void __launch_bounds__(kChunkBlock) k_bin_sums(Plan p) {
  after_previous();
  __shared__ uint32_t s_warp[kChunkBlock / 32];
  uint32_t c[kChunkPer], local = 0;
  unsigned long long crowded = 0;
  load_bins(p, c);
#pragma unroll
  for (int q = 0; q < kChunkPer; ++q) {
    local += c[q];
    crowded += crowd(p, c[q]);
  }
  if (crowded) atomicAdd(&p.meta->crowded, crowded);
  const uint32_t sum = chunk_sum(local, s_warp);
  if (threadIdx.x == kChunkBlock - 1) p.sums[blockIdx.x] = make_uint2(sum, c[kChunkPer - 1]);
}

// Second pass: every chunk's prefix from the sums of those before it, and the
// buckets its bins open.
__global__ void __launch_bounds__(kChunkBlock)
    k_buckets(Plan p, const uint32_t *status, const unsigned long long *spilled) {
  after_previous();
  __shared__ uint32_t s_warp[kChunkBlock / 32], s_last[kChunkBlock + 1];
  const uint32_t nbins = 1u << p.bin_bits;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  uint32_t ahead = 0;
  for (uint32_t j = tid; j < blockIdx.x; j += kChunkBlock) ahead += p.sums[j].x;
  const uint32_t base = chunk_sum(ahead, s_warp);
  uint32_t c[kChunkPer], local = 0;
  load_bins(p, c);
#pragma unroll
  for (int q = 0; q < kChunkPer; ++q) local += c[q];
  uint32_t incl = local;
  for (int d = 1; d < 32; d <<= 1) {
    const uint32_t o = __shfl_up_sync(0xffffffffu, incl, d);
    if (lane >= d) incl += o;
  }
  if (lane == 31) s_warp[warp] = incl;
  __syncthreads();
  uint32_t at = base + incl - local;
  for (int w = 0; w < warp; ++w) at += s_warp[w];
  s_last[tid + 1] = at + local - c[kChunkPer - 1];  // the thread's last bin starts here
  if (tid == 0) s_last[0] = base - (blockIdx.x ? p.sums[blockIdx.x - 1].y : 0u);
  __syncthreads();
  uint32_t before = s_last[tid], prefix[kChunkPer];
  const uint32_t i0 = blockIdx.x * kChunkBins + tid * kChunkPer;
#pragma unroll
  for (int q = 0; q < kChunkPer; ++q) {
    prefix[q] = at;
    open_buckets(p, i0 + q, nbins, at, before);
    before = at;
    at += c[q];
  }
  uint4 *out = reinterpret_cast<uint4 *>(p.bins + i0);
#pragma unroll
  for (int q = 0; q < kChunkPer / 4; ++q)
    out[q] = make_uint4(prefix[4 * q], prefix[4 * q + 1], prefix[4 * q + 2], prefix[4 * q + 3]);
  if (i0 + kChunkPer == nbins) {  // the end comes after the last bin
    p.bins[nbins] = at;
    open_buckets(p, nbins, nbins, at, before);
    fill_meta(p, at, status, spilled);
  }
}

// Every record to its bin's next place: as a 32-byte record of `rec`, or (null)
// as a key and a counter row of the outputs.  Placed by bins, a bucket is in
// order but for the few records of a bin, which the sort's loads like (57 M
// records: sort 0.91 ms, 1.11 in any order).  A large graph's keys and rows go
// to the next place of their bucket instead: an 8- or 16-byte store that ends
// in a sector its neighbours also write is worth more there (24 graphs, 75 M
// records: place 3.26 -> 2.19 ms, sort 1.22 -> 1.30 ms).  A warp takes `run` words
// of 32 slots at a time and reads the slots whose bits are set (0.5 M
// vertices in 300 M slots: export 2.79 ms with every slot read again, 1.86 with a word
// a warp and load, 1.55 with 32; the table read once takes 1.34).  Eight slots a
// thread in flight for records, four in place (432 M records 23.9 -> 22.9 ms an
// export; 57 M in place 3.9 and 4.1).
template <bool WIDE, bool RECORDS>
__global__ void __launch_bounds__(256) k_place(const Slot *t, uint64_t n, uint32_t run, Plan p,
                                               Slot *rec, Key<WIDE> *keys, uint4 *counts) {
  after_previous();
  if (!may_run(p)) return;
  constexpr int kPer = RECORDS ? 8 : 4;
  const uint64_t pol = l2_policy_evict_last();
  const uint32_t lane = threadIdx.x & 31u;
  const uint64_t words = (n + 31) >> 5, warps = (uint64_t)gridDim.x * blockDim.x >> 5;
  for (uint64_t w0 = ((uint64_t)blockIdx.x * blockDim.x + threadIdx.x >> 5) * run; w0 < words;
       w0 += warps * run) {
    uint32_t taken = 0u;  // of the warp's word of this lane
    if (lane < run && w0 + lane < words)
      taken = p.taken ? p.taken[w0 + lane] : ~0u;
    uint32_t left = __ballot_sync(0xffffffffu, taken != 0u);
    while (left) {
      Words v[kPer];
      uint32_t at[kPer];
#pragma unroll
      for (int u = 0; u < kPer; ++u) {
        const uint32_t w = (uint32_t)__ffs((int)left) - 1u;  // (none: the slots of no word)
        const uint32_t m = __shfl_sync(0xffffffffu, taken, (int)(w & 31u));
        const uint64_t j = ((w0 + w) << 5) + lane;
        if (left && (m >> lane & 1u) && j < n)
          v[u] = ld_slot(t + j);
        else
          v[u].w[0] = v[u].w[1] = ~0u;
        left &= left - 1u;
      }
#pragma unroll
      for (int u = 0; u < kPer; ++u) {
        const Key<WIDE> k = key_of<WIDE>(v[u]);
        at[u] = ~0u;
        if (k.empty()) continue;
        uint32_t *bin = &p.bins[k.aligned(p.key_bits) >> (64 - p.bin_bits)];
        if (!RECORDS && p.cursor) bin = &p.cursor[(*bin >> p.bucket_log2) * kCursorStride];
        at[u] = next_place(bin, pol);
      }
#pragma unroll
      for (int u = 0; u < kPer; ++u) {
        if (at[u] == ~0u) continue;
        if constexpr (RECORDS) {
          st_record(rec + at[u], record_of<WIDE>(v[u]));
        } else {
          keys[at[u]] = key_of<WIDE>(v[u]);
          counts[at[u]] = row_of<WIDE>(v[u]);
        }
      }
    }
  }
}

template <bool WIDE, bool RECORDS>
constexpr size_t sort_smem() {
  return kBucketCap * (sizeof(Key<WIDE>) + (RECORDS ? sizeof(uint16_t) : sizeof(uint4))) +
         (kLocalBins + 1) * sizeof(uint32_t);
}

// A CTA per bucket, from `rec` or in place.  The bucket's keys lie in
// [first bin, next bucket's first bin): the bits below choose one of
// kLocalBins local bins; a key's place is its bin's start plus the number of
// smaller keys in the bin (vertices that differ in their last bases only
// share one: about eight at 50x and 1 % errors).
template <bool WIDE, bool RECORDS>
__global__ void __launch_bounds__(kSortBlock, RECORDS && !WIDE ? 6 : 4)
    k_bucket_sort(Plan p, const Slot *rec, Key<WIDE> *keys, uint4 *counts) {
  after_previous();
  constexpr int kPer = kBucketCap / kSortBlock;
  constexpr int kBinsPer = kLocalBins / kSortBlock;
  extern __shared__ __align__(16) unsigned char smem[];
  Key<WIDE> *s_key = reinterpret_cast<Key<WIDE> *>(smem);
  uint4 *s_row = reinterpret_cast<uint4 *>(s_key + kBucketCap);          // in place
  uint16_t *s_src = reinterpret_cast<uint16_t *>(s_key + kBucketCap);    // from records
  uint32_t *s_bin = reinterpret_cast<uint32_t *>(  // kLocalBins + 1
      RECORDS ? reinterpret_cast<unsigned char *>(s_src + kBucketCap)
              : reinterpret_cast<unsigned char *>(s_row + kBucketCap));
  __shared__ uint32_t s_warp[kSortBlock / 32];
  if (p.report && blockIdx.x == 0 && threadIdx.x == 0) *p.report = *p.meta;
  if (!may_run(p)) return;
  const uint32_t b = blockIdx.x;
  if (b > p.meta->vertices >> p.bucket_log2) return;
  const uint32_t s0 = p.start[b], n = p.start[b + 1] - s0;
  if (n == 0 || n > kBucketCap) return;  // (a larger one: k_crowd_gather's)
  const uint32_t bin0 = p.first_bin[b], span = p.first_bin[b + 1] - bin0;
  const uint64_t low = (uint64_t)bin0 << (64 - p.bin_bits);
  const int width = 64 - p.bin_bits + (span > 1 ? 32 - __clz((int)(span - 1)) : 0);
  const int shift = width > kLocalBits ? width - kLocalBits : 0;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  for (int j = tid; j < kLocalBins; j += kSortBlock) s_bin[j] = 0u;
  Key<WIDE> k[kPer];
  uint32_t where[kPer];  // local bin << 16 | place in it
#pragma unroll
  for (int q = 0; q < kPer; ++q) {
    const uint32_t i = q * kSortBlock + tid;
    if (i < n) {
      if constexpr (RECORDS)
        k[q] = ld_record_key<WIDE>(rec + s0 + i);
      else
        k[q] = keys[s0 + i];
    }
  }
  __syncthreads();
#pragma unroll
  for (int q = 0; q < kPer; ++q) {
    if (q * kSortBlock + tid < n) {
      const uint32_t l = (uint32_t)((k[q].aligned(p.key_bits) - low) >> shift);
      where[q] = (l << 16) | atomicAdd(&s_bin[l], 1u);
    }
  }
  __syncthreads();
  {
    uint32_t c[kBinsPer], local = 0;
#pragma unroll
    for (int q = 0; q < kBinsPer; ++q) {
      c[q] = s_bin[tid * kBinsPer + q];
      local += c[q];
    }
    uint32_t incl = local;
    for (int d = 1; d < 32; d <<= 1) {
      const uint32_t o = __shfl_up_sync(0xffffffffu, incl, d);
      if (lane >= d) incl += o;
    }
    if (lane == 31) s_warp[warp] = incl;
    __syncthreads();
    uint32_t w = lane < kSortBlock / 32 ? s_warp[lane] : 0u;
    for (int d = 1; d < kSortBlock / 32; d <<= 1) {
      const uint32_t o = __shfl_up_sync(0xffffffffu, w, d);
      if (lane >= d) w += o;
    }
    const uint32_t below = __shfl_sync(0xffffffffu, w, (warp + 31) & 31);
    uint32_t at = incl - local + (warp > 0 ? below : 0u);
#pragma unroll
    for (int q = 0; q < kBinsPer; ++q) {
      s_bin[tid * kBinsPer + q] = at;
      at += c[q];
    }
    if (tid == 0) s_bin[kLocalBins] = n;
  }
  __syncthreads();
#pragma unroll
  for (int q = 0; q < kPer; ++q)
    if (q * kSortBlock + tid < n) s_key[s_bin[where[q] >> 16] + (where[q] & 0xFFFFu)] = k[q];
  __syncthreads();
#pragma unroll
  for (int q = 0; q < kPer; ++q) {
    if (q * kSortBlock + tid < n) {
      const uint32_t a = s_bin[where[q] >> 16], e = s_bin[(where[q] >> 16) + 1];
      uint32_t f = a;
      if (e - a > 1)
        for (uint32_t j = a; j < e; ++j) f += s_key[j] < k[q] ? 1u : 0u;
      where[q] = f;
    }
  }
  __syncthreads();
#pragma unroll
  for (int q = 0; q < kPer; ++q) {
    const uint32_t i = q * kSortBlock + tid;
    if (i < n) {
      s_key[where[q]] = k[q];
      if constexpr (RECORDS)
        s_src[where[q]] = (uint16_t)i;
      else
        s_row[where[q]] = counts[s0 + i];
    }
  }
  __syncthreads();
  for (uint32_t i = tid; i < n; i += kSortBlock) {
    keys[s0 + i] = s_key[i];
    uint4 row;
    if constexpr (RECORDS) {  // (its sector was read with the key: an L2 hit)
      row = *(reinterpret_cast<const uint4 *>(rec + s0 + s_src[i]) + (WIDE ? 1 : 0));
    } else {
      row = s_row[i];
    }
    __stcs(counts + s0 + i, row);
  }
}

// The buckets above the cap.  Their records get consecutive numbers, in the
// buckets' order: off[b] is the first of bucket b.
constexpr int kOffBlock = 1024, kOffPer = 8;
__device__ __forceinline__ uint32_t crowded_in(const Plan &p, uint32_t b) {
  if (b > p.meta->vertices >> p.bucket_log2) return 0u;
  const uint32_t n = p.start[b + 1] - p.start[b];
  return n > kBucketCap ? n : 0u;
}
__global__ void __launch_bounds__(kOffBlock) k_crowd_offsets(Plan p, uint32_t *off) {
  after_previous();
  __shared__ uint32_t s_warp[32];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const uint32_t nb = (p.meta->vertices >> p.bucket_log2) + 1u;
  uint32_t run = 0;
  for (uint32_t b0 = 0; b0 < nb; b0 += kOffBlock * kOffPer) {
    const uint32_t b = b0 + threadIdx.x * kOffPer;
    uint32_t c[kOffPer], n = 0;
#pragma unroll
    for (int q = 0; q < kOffPer; ++q) n += c[q] = crowded_in(p, b + q);
    uint32_t incl = n;
    for (int d = 1; d < 32; d <<= 1) {
      const uint32_t o = __shfl_up_sync(0xffffffffu, incl, d);
      if (lane >= d) incl += o;
    }
    if (lane == 31) s_warp[warp] = incl;
    __syncthreads();
    uint32_t total = 0, below = 0;
    for (int w = 0; w < kOffBlock / 32; ++w) {
      if (w < warp) below += s_warp[w];
      total += s_warp[w];
    }
    uint32_t at = run + below + incl - n;
#pragma unroll
    for (int q = 0; q < kOffPer; ++q) {
      if (b + q < nb) off[b + q] = at;
      at += c[q];
    }
    run += total;
    __syncthreads();
  }
}

// What a record's number leads to: its key's words, its counter row, and for the
// sort the numbers themselves.
struct Crowd {
  uint32_t *off;
  uint64_t n;  // numbers there are (records, and a few that are none: they sort last)
  unsigned long long *lo[2], *hi[2];
  uint32_t *idx[2];
  uint4 *row;
};

__global__ void __launch_bounds__(256) k_crowd_none(Crowd c, int wide) {
  after_previous();
  const uint64_t stride = (uint64_t)gridDim.x * blockDim.x;
  for (uint64_t i = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; i < c.n; i += stride) {
    c.idx[0][i] = (uint32_t)i;
    c.lo[0][i] = ~0ull;
    if (wide) c.hi[0][i] = ~0ull;
  }
}

// A CTA takes kCrowdGroup buckets: f(position, number) for every
// record of those above the cap.
constexpr uint32_t kCrowdGroup = 16;
template <class F>
__device__ __forceinline__ void each_crowded(const Plan &p, const Crowd &c, F &&f) {
  __shared__ uint32_t s_n[kCrowdGroup];
  const uint32_t b0 = blockIdx.x * kCrowdGroup;
  if (threadIdx.x < kCrowdGroup) s_n[threadIdx.x] = crowded_in(p, b0 + threadIdx.x);
  __syncthreads();
  for (uint32_t q = 0; q < kCrowdGroup; ++q) {
    const uint32_t n = s_n[q];
    if (n == 0) continue;
    const uint32_t s0 = p.start[b0 + q], at = c.off[b0 + q];
    for (uint32_t i = threadIdx.x; i < n; i += blockDim.x) f(s0 + i, at + i);
  }
}

template <bool WIDE, bool RECORDS>
__global__ void __launch_bounds__(256)
    k_crowd_gather(Plan p, const Slot *rec, const Key<WIDE> *keys, const uint4 *counts, Crowd c) {
  after_previous();
  each_crowded(p, c, [&](uint32_t from, uint32_t at) {
    Key<WIDE> k;
    if constexpr (RECORDS) {
      k = ld_record_key<WIDE>(rec + from);
      c.row[at] = *(reinterpret_cast<const uint4 *>(rec + from) + (WIDE ? 1 : 0));
    } else {
      k = keys[from];
      c.row[at] = counts[from];
    }
    if constexpr (WIDE) {
      c.lo[0][at] = k.lo;
      c.hi[0][at] = k.hi;
    } else {
      c.lo[0][at] = k.w;
    }
  });
}

// hi[1] := hi[0] in the order of the first sort.
__global__ void __launch_bounds__(256) k_crowd_high(Crowd c) {
  after_previous();
  const uint64_t stride = (uint64_t)gridDim.x * blockDim.x;
  for (uint64_t i = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; i < c.n; i += stride)
    c.hi[1][i] = c.hi[0][c.idx[1][i]];
}

// The records of those buckets in order (idx: the sorted numbers).
template <bool WIDE>
__global__ void __launch_bounds__(256)
    k_crowd_write(Plan p, Crowd c, const uint32_t *idx, Key<WIDE> *keys, uint4 *counts) {
  after_previous();
  each_crowded(p, c, [&](uint32_t to, uint32_t at) {
    const uint32_t from = idx[at];
    Key<WIDE> k;
    if constexpr (WIDE) {
      k.lo = c.lo[0][from];
      k.hi = c.hi[0][from];
    } else {
      k.w = c.lo[0][from];
    }
    keys[to] = k;
    counts[to] = c.row[from];
  });
}

size_t al256(size_t x) { return (x + 255) & ~size_t(255); }

int ceil_log2(uint64_t x) {
  int r = 0;
  while ((1ull << r) < x) ++r;
  return r;
}

// Bins and buckets for at most `rows` vertices: buckets of T = 2^10 records
// or, in a small graph, few enough for about 512 CTAs; bins for 16 records, so
// that few atomics meet on one counter, up to 2^20 of them or one for 128 records
// (more of them cost uniform genomes time: 57 M vertices 2.92 ms, 3.02 with 2^22
// bins; fewer leave more to the crowded buckets' sort).  Outputs of a quarter of
// the table's slots or less may be too small for its vertices: the bins are then
// for that many, or the counting would meet on a few counters (57 M vertices
// counted for outputs of 1,000 rows: 16.8 ms, with the table's bins 0.6).
struct Shape {
  int bin_bits, bucket_log2;
  uint32_t nbins, buckets;
  size_t off_bins, off_start, off_first, off_cursor, off_sums, total;
  size_t taken;  // after them, if there is room: a bit per slot
};

void export_shape(int k, uint64_t rows, uint64_t n_slots, Shape &sh) {
  const int bits = ceil_log2(std::max<uint64_t>(rows, 2));
  sh.bucket_log2 = std::min(10, std::max(7, bits - 9));
  const int weight = ceil_log2(std::max<uint64_t>(std::max<uint64_t>(rows, 2), n_slots / 4));
  sh.bin_bits = std::min(std::min(std::max(kBinBits, weight - kBinLog2), 2 * (k - 1)),
                         std::max(1, weight - 4));
  sh.nbins = 1u << sh.bin_bits;
  sh.buckets = (uint32_t)(rows >> sh.bucket_log2) + 1u;
  sh.off_bins = 256;  // (the meta block first: cleared with the histogram)
  sh.off_start = sh.off_bins + al256(((size_t)sh.nbins + 1) * 4);
  sh.off_first = sh.off_start + al256(((size_t)sh.buckets + 2) * 4);
  sh.off_cursor = sh.off_first + al256(((size_t)sh.buckets + 2) * 4);
  sh.off_sums = sh.off_cursor +
                (sh.nbins > kCursorBins ? al256(((size_t)sh.buckets + 2) * 4 * kCursorStride) : 0);
  sh.total = sh.off_sums +
             (sh.nbins > (uint32_t)kPlanBins ? al256(sh.nbins / kChunkBins * sizeof(uint2)) : 0);
  sh.taken = al256((n_slots + 31) / 32 * 4);
}

// Scratch for the crowded buckets' records: the arrays of a Crowd of n and the
// radix sort's.
struct CrowdLayout {
  size_t off, lo[2], hi[2], idx[2], row, temp, temp_bytes, total;
};

int crowd_layout(int k, uint64_t n, uint32_t buckets, CrowdLayout &l) {
  l.temp_bytes = 0;
  DBG_CK(cub::DeviceRadixSort::SortPairs(nullptr, l.temp_bytes, (unsigned long long *)nullptr,
                                         (unsigned long long *)nullptr, (uint32_t *)nullptr,
                                         (uint32_t *)nullptr, (int64_t)n, 0, 64, (cudaStream_t)0));
  size_t at = 0;
  auto take = [&at](size_t bytes) {
    const size_t here = at;
    at += al256(bytes);
    return here;
  };
  l.off = take(((size_t)buckets + 2) * 4);
  for (int i = 0; i < 2; ++i) {
    l.lo[i] = take(n * 8);
    l.hi[i] = take(k > 32 ? n * 8 : 0);
    l.idx[i] = take(n * 4);
  }
  l.row = take(n * 16);
  l.temp = take(l.temp_bytes);
  l.total = at;
  return DBG_OK;
}

// Sort the buckets above the cap, `n` numbers for their records, after the others.
template <bool WIDE>
int sort_crowded(dbg_handle h, const Shape &sh, const Plan &p, uint64_t n, char *b,
                 const CrowdLayout &l, const Slot *rec, Key<WIDE> *keys, uint4 *counts,
                 cudaStream_t s) {
  Crowd c;
  c.off = reinterpret_cast<uint32_t *>(b + l.off);
  c.n = n;
  for (int i = 0; i < 2; ++i) {
    c.lo[i] = reinterpret_cast<unsigned long long *>(b + l.lo[i]);
    c.hi[i] = reinterpret_cast<unsigned long long *>(b + l.hi[i]);
    c.idx[i] = reinterpret_cast<uint32_t *>(b + l.idx[i]);
  }
  c.row = reinterpret_cast<uint4 *>(b + l.row);
  const int grid = (int)std::min<uint64_t>((n + 255) / 256, (uint64_t)std::max(1, h->sm_count) * 8);
  const int groups = (int)((sh.buckets + kCrowdGroup - 1) / kCrowdGroup);
  DBG_TRY(launch_after(k_crowd_offsets, 1, kOffBlock, 0, s, p, c.off));
  DBG_TRY(launch_after(k_crowd_none, grid, 256, 0, s, c, WIDE ? 1 : 0));
  if (rec)
    DBG_TRY(launch_after(k_crowd_gather<WIDE, true>, groups, 256, 0, s, p, rec, keys, counts, c));
  else
    DBG_TRY(launch_after(k_crowd_gather<WIDE, false>, groups, 256, 0, s, p, rec, keys, counts, c));
  size_t temp = l.temp_bytes;
  DBG_CK(cub::DeviceRadixSort::SortPairs(b + l.temp, temp, c.lo[0], c.lo[1], c.idx[0], c.idx[1],
                                         (int64_t)n, 0, std::min(64, p.key_bits), s));
  const uint32_t *idx = c.idx[1];
  if (WIDE && p.key_bits > 64) {  // the low words' order is kept among equal high words
    DBG_TRY(launch_after(k_crowd_high, grid, 256, 0, s, c));
    DBG_CK(cub::DeviceRadixSort::SortPairs(b + l.temp, temp, c.hi[1], c.lo[1], c.idx[1], c.idx[0],
                                           (int64_t)n, 0, p.key_bits - 64, s));
    idx = c.idx[0];
  }
  DBG_TRY(launch_after(k_crowd_write<WIDE>, groups, 256, 0, s, p, c, idx, keys, counts));
  DBG_CK(cudaGetLastError());
  DBG_CK(cudaStreamSynchronize(s));
  return DBG_OK;
}

// (buf_bytes: what there is of `buf`; the crowded buckets' scratch comes from its
// rest, or from the pool when buf is the pool's.  *too_dense: too many crowded
// records, or no scratch for them.)
template <bool WIDE>
int run(dbg_handle h, const Shape &sh, uint64_t max_rows, void *buf, uint64_t buf_bytes, bool pooled,
        Slot *rec, uint64_t rec_rows, uint64_t *keys_out, uint32_t *counts_out, ExportMeta &m,
        bool *too_dense, cudaStream_t s) {
  char *b = static_cast<char *>(buf);
  Plan p;
  p.key_bits = 2 * (h->k - 1);
  p.bin_bits = sh.bin_bits;
  p.bucket_log2 = sh.bucket_log2;
  p.buckets = sh.buckets;
  p.max_rows = max_rows;
  p.max_placed = rec ? rec_rows : ~0ull;
  p.max_crowded = std::max<uint64_t>(std::min(max_rows, h->n_slots) / kCrowdedShare, 1u << 16);
  p.sums = reinterpret_cast<uint2 *>(b + sh.off_sums);
  p.taken = buf_bytes >= sh.total + sh.taken ? reinterpret_cast<uint32_t *>(b + sh.total) : nullptr;
  p.meta = reinterpret_cast<ExportMeta *>(b);
  const ReportSlot slot;
  p.report = reinterpret_cast<ExportMeta *>(slot.p);
  p.bins = reinterpret_cast<uint32_t *>(b + sh.off_bins);
  p.start = reinterpret_cast<uint32_t *>(b + sh.off_start);
  p.first_bin = reinterpret_cast<uint32_t *>(b + sh.off_first);
  p.cursor = !rec && sh.nbins > kCursorBins ? reinterpret_cast<uint32_t *>(b + sh.off_cursor)
                                            : nullptr;
  Key<WIDE> *keys = reinterpret_cast<Key<WIDE> *>(keys_out);
  uint4 *counts = reinterpret_cast<uint4 *>(counts_out);
  const int sms = std::max(1, h->sm_count);
  const uint64_t n = h->n_slots;
  const int grid = (int)std::min<uint64_t>((n + 256 * kSlotsPerThread - 1) / (256 * kSlotsPerThread),
                                           (uint64_t)sms * 8);
  // (32 words a warp where every warp gets as many, else one load's)
  const uint32_t run = n >= (uint64_t)sms * 8 * 256 * 32 ? 32u : (uint32_t)kSlotsPerThread;
  DBG_CK(cudaMemsetAsync(b, 0, sh.off_start, s));  // meta and histogram
  DBG_TRY(launch_after(k_histogram<WIDE>, grid, 256, 0, s, h->table, n, p));
  DBG_CK(cudaGetLastError());
  if (sh.nbins <= (uint32_t)kPlanBins) {
    DBG_TRY(launch_after(k_plan, 1, kPlanBlock, 0, s, p, h->d_status, h->d_spill_count));
  } else {
    DBG_TRY(launch_after(k_bin_sums, sh.nbins / kChunkBins, kChunkBlock, 0, s, p));
    DBG_TRY(launch_after(k_buckets, sh.nbins / kChunkBins, kChunkBlock, 0, s, p, h->d_status,
                         h->d_spill_count));
  }
  DBG_CK(cudaGetLastError());
  if (rec) {
    constexpr size_t smem = sort_smem<WIDE, true>();
    DBG_TRY(launch_after(k_place<WIDE, true>, grid, 256, 0, s, h->table, n, run, p, rec, keys, counts));
    DBG_CK(cudaFuncSetAttribute(k_bucket_sort<WIDE, true>,
                                cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
    DBG_TRY(launch_after(k_bucket_sort<WIDE, true>, sh.buckets, kSortBlock, smem, s, p, rec, keys,
                         counts));
  } else {
    constexpr size_t smem = sort_smem<WIDE, false>();
    DBG_TRY(launch_after(k_place<WIDE, false>, grid, 256, 0, s, h->table, n, run, p, rec, keys, counts));
    DBG_CK(cudaFuncSetAttribute(k_bucket_sort<WIDE, false>,
                                cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
    DBG_TRY(launch_after(k_bucket_sort<WIDE, false>, sh.buckets, kSortBlock, smem, s, p, rec, keys,
                         counts));
  }
  DBG_CK(cudaGetLastError());
  if (!p.report) DBG_CK(cudaMemcpyAsync(&m, p.meta, sizeof(m), cudaMemcpyDeviceToHost, s));
  DBG_CK(cudaStreamSynchronize(s));
  if (p.report) m = *p.report;
  *too_dense = m.crowded > p.max_crowded;
  if (m.crowded == 0 || *too_dense || m.status != DBG_OK || m.spilled > 0 ||
      m.vertices > p.max_rows || m.vertices > p.max_placed)
    return DBG_OK;
  CrowdLayout l;
  const uint64_t nc = std::min<uint64_t>(m.crowded, m.vertices);
  DBG_TRY(crowd_layout(h->k, nc, sh.buckets, l));
  if (!pooled) {
    const uint64_t used = sh.total + (p.taken ? sh.taken : 0);
    *too_dense = buf_bytes - used < l.total;
    return *too_dense ? DBG_OK : sort_crowded<WIDE>(h, sh, p, nc, b + used, l, rec, keys, counts, s);
  }
  char *more = nullptr;
  if (scratch_alloc(reinterpret_cast<void **>(&more), l.total, s) != DBG_OK) {
    cudaGetLastError();
    *too_dense = true;
    return DBG_OK;
  }
  const int st = sort_crowded<WIDE>(h, sh, p, nc, more, l, rec, keys, counts, s);
  cudaFreeAsync(more, s);
  return st;
}

}  // namespace

int export_bins_scratch(int k, uint64_t rows, uint64_t n_slots, uint64_t &bytes) {
  Shape sh{};
  export_shape(k, rows, n_slots, sh);
  bytes = sh.total;
  return DBG_OK;
}

int export_bins(dbg_handle h, uint64_t *keys_out, uint32_t *counts_out, uint64_t max_rows,
                uint64_t *D, cudaStream_t s, void *scratch, uint64_t scratch_bytes,
                bool *too_dense, bool *no_records) {
  *too_dense = false;
  if (no_records) *no_records = false;
  const uint64_t rows = std::min(max_rows, h->n_slots);
  Shape sh{};
  export_shape(h->k, rows, h->n_slots, sh);
  char *buf = static_cast<char *>(scratch);
  uint64_t buf_bytes = scratch_bytes;
  if (!scratch) {
    buf_bytes = sh.total + sh.taken;
    if (scratch_alloc(reinterpret_cast<void **>(&buf), buf_bytes, s) != DBG_OK) {
      cudaGetLastError();  // (without the slots' bits, then)
      buf_bytes = sh.total;
      DBG_TRY(scratch_alloc(reinterpret_cast<void **>(&buf), buf_bytes, s));
    }
  }
  if (scratch && scratch_bytes < sh.total) return DBG_ERR_INVALID_ARG;
  // room for 32-byte records: the graph's own event buffer (idle between its
  // inserts; its event orders the two) when the graph has one that fits, or
  // the pool (k > 32, and outputs that only the sort may write)
  Slot *rec = nullptr;
  uint64_t rec_rows = 0;
  bool own = false;
  if (!scratch && h->bin.ev2) {
    rec = reinterpret_cast<Slot *>(h->bin.ev2);
    rec_rows = bin_ev2_bytes(h) / sizeof(Slot);
    own = rec_rows >= rows / 2;  // (a table is rarely more than two thirds full)
    if (!own) rec = nullptr;
  }
  const bool pooled = !rec && (h->k > 32 || no_records) && !scratch &&
                      rows * sizeof(Slot) <= kMaxPooledRecords;
  if (pooled) {
    rec_rows = rows;
    const int st = scratch_alloc(reinterpret_cast<void **>(&rec), rows * sizeof(Slot), s);
    if (st != DBG_OK) {  // (none to be had: into the outputs)
      cudaGetLastError();
      rec = nullptr;
    }
  }
  Slot *const from_pool = pooled ? rec : nullptr;
  int rc = DBG_OK;
  ExportMeta m{};
  for (;;) {
    if (no_records && !rec) {
      *no_records = true;
      break;
    }
    if (own) {
      const cudaError_t e = cudaStreamWaitEvent(s, h->bin.done, 0);
      if (e != cudaSuccess) { rc = cuda_fail(e, "cudaStreamWaitEvent"); break; }
    }
    rc = (h->k > 32 ? run<true> : run<false>)(h, sh, max_rows, buf, buf_bytes, !scratch, rec,
                                              rec_rows, keys_out, counts_out, m, too_dense, s);
    if (own && rc == DBG_OK) {
      const cudaError_t e = cudaEventRecord(h->bin.done, s);
      if (e != cudaSuccess) rc = cuda_fail(e, "cudaEventRecord");
    }
    if (rc != DBG_OK || !rec || m.vertices <= rec_rows || m.vertices > max_rows) break;
    rec = nullptr;  // more vertices than the event buffer holds: into the outputs
    own = false;
  }
  if (from_pool) cudaFreeAsync(from_pool, s);
  if (!scratch) {
    const cudaError_t e = cudaFreeAsync(buf, s);
    if (rc == DBG_OK && e != cudaSuccess) rc = cuda_fail(e, "cudaFreeAsync");
  }
  if (rc != DBG_OK || (no_records && *no_records)) return rc;
  if (m.status != DBG_OK) return (int)m.status;
  if (m.spilled > 0) return DBG_ERR_NEEDS_GROW;
  *D = m.vertices;
  return DBG_OK;
}

}  // namespace dbg
