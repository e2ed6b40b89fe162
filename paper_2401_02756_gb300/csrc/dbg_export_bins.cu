// The sorted export by bins: the occupied slots' records are placed straight
// into the order of their keys' leading bits, and every stretch of a few
// thousand of them is then sorted in shared memory.
//
//   histogram -- the table read once: vertices per bin (the keys' top B bits);
//   plan      -- the bins' prefix sum; bins are joined into buckets of about
//                T records (bucket of a bin = its first position / T);
//   place     -- the table read again: every record to the next free position
//                of its bin (one atomic a record on the bin's counter);
//   sort      -- a CTA per bucket: a counting sort by the bits that follow,
//                then every key's rank among the few that share its bin, and
//                keys and counter rows out in order, coalesced.
//
// So a record moves twice and no slot is read at random.  The radix sort of
// (32-bit prefix, slot index) pairs this replaces moved 16 bytes a record four
// times, gathered a random slot per vertex and put runs of equal prefixes in
// order in two more passes.  Export of 422.6 M vertices of a 20.8 GB table
// 35.4 -> 22 ms (histogram 4.0, place 10.8 to 12.3 from card to card, sort 6.5;
// 7.7 with the counters at the slot's byte 8, two loads a row), of 57 M 5.1 ->
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
// record, 1.5 times the time, but no memory beyond the bins' is needed).  A
// table whose keys crowd into one bin (more than a bucket's shared memory
// holds) is left to the radix sort.
#include <cub/device/device_scan.cuh>

#include <algorithm>

#include "dbg_export.cuh"
#include "dbg_internal.cuh"

namespace dbg {
namespace {

constexpr int kSortBlock = 256;
constexpr int kLocalBits = 11;  // bins of the shared-memory counting sort
constexpr int kLocalBins = 1 << kLocalBits;
constexpr int kMaxBinBits = 20;
constexpr int kPlanBins = 8192;  // up to this many: the plan is one CTA's work
constexpr int kPlanBlock = 1024;
constexpr int kSlotsPerThread = 4;
constexpr int kCursorStride = 8;  // a bucket's cursor has a sector of its own
constexpr uint32_t kCursorBins = 1u << 17;  // in place: bucket cursors above so many bins
constexpr uint64_t kMaxPooledRecords = 4ull << 30;  // (what the pool keeps between calls)

constexpr uint32_t kBucketCap = 2048;  // records a bucket may hold

struct ExportMeta {
  unsigned long long spilled;
  uint32_t vertices, max_bin, status;
};

// Everything the kernels share.
struct Plan {
  int key_bits;         // 2 (k - 1)
  int bin_bits;         // B
  int bucket_log2;      // T = 2^bucket_log2
  uint32_t buckets;     // last entry of the bucket arrays (a graph of more vertices is not placed)
  uint64_t max_rows;    // rows of the outputs
  uint64_t max_placed;  // records the scratch holds (place into 32-byte records)
  uint32_t *bins;       // [2^B + 1] histogram, then exclusive prefix, then next free position
  uint32_t *start;      // [buckets + 2] first position of a bucket
  uint32_t *first_bin;  // [buckets + 2]
  uint32_t *cursor;     // [buckets + 2][kCursorStride] next free position, or null: the bins' own
  ExportMeta *meta;
  ExportMeta *report;   // the sort's copy of it in pinned host memory, or null
};

// Whether the placing and the sort may run: a complete graph, room for it,
// and no bucket above the cap.
__device__ __forceinline__ bool may_run(const Plan &p) {
  const ExportMeta m = *p.meta;
  return m.status == 0u && m.spilled == 0ull && m.vertices <= p.max_rows &&
         m.vertices <= p.max_placed && (1u << p.bucket_log2) + m.max_bin <= kBucketCap;
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

// A 32-byte slot in one load, and a 32-byte record in one store.
struct Words {
  uint32_t w[8];
};
__device__ __forceinline__ Words ld_slot(const Slot *p) {
  Words v;
  asm volatile("ld.global.L1::no_allocate.v8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
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

// Vertices per bin.  Bound by one read of the table.
template <bool WIDE>
__global__ void __launch_bounds__(256) k_histogram(const Slot *t, uint64_t n, Plan p) {
  after_previous();
  const uint64_t stride = (uint64_t)gridDim.x * blockDim.x;
  for (uint64_t i = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n;
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

// The plan of up to kPlanBins bins in one CTA: prefix, buckets, largest bin.
__global__ void __launch_bounds__(kPlanBlock)
    k_plan(Plan p, const uint32_t *status, const unsigned long long *spilled) {
  after_previous();
  constexpr int kPer = kPlanBins / kPlanBlock;
  __shared__ uint32_t s_warp[32], s_last[kPlanBlock + 1];
  const uint32_t nbins = 1u << p.bin_bits;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const uint32_t i0 = threadIdx.x * kPer;
  uint32_t c[kPer], local = 0, most = 0;
#pragma unroll
  for (int q = 0; q < kPer; ++q) {
    c[q] = i0 + q < nbins ? p.bins[i0 + q] : 0u;
    local += c[q];
    most = max(most, c[q]);
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
  most = __reduce_max_sync(0xffffffffu, most);
  if (lane == 0 && most) atomicMax(&p.meta->max_bin, most);
  if (threadIdx.x == 0) fill_meta(p, total, status, spilled);
}

// The same from a finished prefix (more bins).  (The largest bin by one atomic a
// CTA, and only from a CTA that would raise it: one a warp on the one address
// took 24 us for 2^20 bins, now 8.)
__global__ void __launch_bounds__(256)
    k_buckets(Plan p, const uint32_t *status, const unsigned long long *spilled) {
  after_previous();
  __shared__ uint32_t s_most;
  if (threadIdx.x == 0) s_most = 0u;
  __syncthreads();
  const uint32_t nbins = 1u << p.bin_bits;
  const uint32_t i = blockIdx.x * blockDim.x + threadIdx.x;
  uint32_t n = 0;
  if (i <= nbins) {
    const uint32_t at = p.bins[i];
    open_buckets(p, i, nbins, at, i ? p.bins[i - 1] : 0u);
    if (i < nbins) n = p.bins[i + 1] - at;
    if (i == nbins) fill_meta(p, at, status, spilled);
  }
  n = __reduce_max_sync(0xffffffffu, n);
  if ((threadIdx.x & 31) == 0 && n) atomicMax(&s_most, n);
  __syncthreads();
  if (threadIdx.x == 0 && s_most > ld_volatile_u32(&p.meta->max_bin))
    atomicMax(&p.meta->max_bin, s_most);
}

// Every record to its bin's next place: as a 32-byte record of `rec`, or (null)
// as a key and a counter row of the outputs.  Placed by bins, a bucket is in
// order but for the few records of a bin, which the sort's loads like (57 M
// records: sort 0.91 ms, 1.11 in any order).  A large graph's keys and rows go
// to the next place of their bucket instead: an 8- or 16-byte store that ends
// in a sector its neighbours also write is worth more there (24 graphs, 75 M
// records: place 3.26 -> 2.19 ms, sort 1.22 -> 1.30 ms).
template <bool WIDE, bool RECORDS>
__global__ void __launch_bounds__(256) k_place(const Slot *t, uint64_t n, Plan p, Slot *rec,
                                               Key<WIDE> *keys, uint4 *counts) {
  after_previous();
  if (!may_run(p)) return;
  const uint64_t stride = (uint64_t)gridDim.x * blockDim.x;
  for (uint64_t i = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n;
       i += stride * kSlotsPerThread) {
    Words v[kSlotsPerThread];
    uint32_t at[kSlotsPerThread];
#pragma unroll
    for (int u = 0; u < kSlotsPerThread; ++u) {
      const uint64_t j = i + u * stride;
      if (j < n)
        v[u] = ld_slot(t + j);
      else
        v[u].w[0] = v[u].w[1] = ~0u;
    }
#pragma unroll
    for (int u = 0; u < kSlotsPerThread; ++u) {
      const Key<WIDE> k = key_of<WIDE>(v[u]);
      at[u] = ~0u;
      if (k.empty()) continue;
      uint32_t *bin = &p.bins[k.aligned(p.key_bits) >> (64 - p.bin_bits)];
      if (!RECORDS && p.cursor) bin = &p.cursor[(*bin >> p.bucket_log2) * kCursorStride];
      at[u] = atomicAdd(bin, 1u);
    }
#pragma unroll
    for (int u = 0; u < kSlotsPerThread; ++u) {
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
  if (n == 0) return;
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

size_t al256(size_t x) { return (x + 255) & ~size_t(255); }

int ceil_log2(uint64_t x) {
  int r = 0;
  while ((1ull << r) < x) ++r;
  return r;
}

// Bins and buckets for at most `rows` vertices: buckets of T = 2^10 records
// or, in a small graph, few enough for about 512 CTAs; bins for 16 records, so
// that few atomics meet on one counter, and at most 2^20 of them.  Outputs of a
// sixteenth of the table's slots or less may be too small for its vertices: the
// bins are then for that many, or the counting would meet on a few counters
// (57 M vertices counted for outputs of 1,000 rows: 16.8 ms, with the table's
// bins 0.5).
struct Shape {
  int bin_bits, bucket_log2;
  uint32_t nbins, buckets;
  size_t temp, off_bins, off_start, off_first, off_cursor, off_temp, total;
};

int export_shape(int k, uint64_t rows, uint64_t n_slots, Shape &sh) {
  const int bits = ceil_log2(std::max<uint64_t>(rows, 2));
  sh.bucket_log2 = std::min(10, std::max(7, bits - 9));
  sh.bin_bits = std::min(std::min(kMaxBinBits, 2 * (k - 1)),
                         std::max(1, ceil_log2(std::max<uint64_t>(rows, n_slots / 16)) - 4));
  sh.nbins = 1u << sh.bin_bits;
  sh.buckets = (uint32_t)(rows >> sh.bucket_log2) + 1u;
  sh.temp = 0;
  if (sh.nbins > (uint32_t)kPlanBins)
    DBG_CK(cub::DeviceScan::ExclusiveSum(nullptr, sh.temp, (uint32_t *)nullptr, (uint32_t *)nullptr,
                                         (int)sh.nbins + 1, (cudaStream_t)0));
  sh.off_bins = 256;  // (the meta block first: cleared with the histogram)
  sh.off_start = sh.off_bins + al256(((size_t)sh.nbins + 1) * 4);
  sh.off_first = sh.off_start + al256(((size_t)sh.buckets + 2) * 4);
  sh.off_cursor = sh.off_first + al256(((size_t)sh.buckets + 2) * 4);
  sh.off_temp = sh.off_cursor +
                (sh.nbins > kCursorBins ? al256(((size_t)sh.buckets + 2) * 4 * kCursorStride) : 0);
  sh.total = sh.off_temp + al256(sh.temp);
  return DBG_OK;
}

template <bool WIDE>
int run(dbg_handle h, const Shape &sh, uint64_t max_rows, void *buf, Slot *rec, uint64_t rec_rows,
        uint64_t *keys_out, uint32_t *counts_out, ExportMeta &m, cudaStream_t s) {
  char *b = static_cast<char *>(buf);
  Plan p;
  p.key_bits = 2 * (h->k - 1);
  p.bin_bits = sh.bin_bits;
  p.bucket_log2 = sh.bucket_log2;
  p.buckets = sh.buckets;
  p.max_rows = max_rows;
  p.max_placed = rec ? rec_rows : ~0ull;
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
  DBG_CK(cudaMemsetAsync(b, 0, sh.off_start, s));  // meta and histogram
  DBG_TRY(launch_after(k_histogram<WIDE>, grid, 256, 0, s, h->table, n, p));
  DBG_CK(cudaGetLastError());
  if (sh.nbins <= (uint32_t)kPlanBins) {
    DBG_TRY(launch_after(k_plan, 1, kPlanBlock, 0, s, p, h->d_status, h->d_spill_count));
  } else {
    size_t temp = sh.temp;
    DBG_CK(cub::DeviceScan::ExclusiveSum(b + sh.off_temp, temp, p.bins, p.bins,
                                         (int)sh.nbins + 1, s));
    DBG_TRY(launch_after(k_buckets, (sh.nbins + 256) / 256, 256, 0, s, p, h->d_status,
                         h->d_spill_count));
  }
  DBG_CK(cudaGetLastError());
  if (rec) {
    constexpr size_t smem = sort_smem<WIDE, true>();
    DBG_TRY(launch_after(k_place<WIDE, true>, grid, 256, 0, s, h->table, n, p, rec, keys, counts));
    DBG_CK(cudaFuncSetAttribute(k_bucket_sort<WIDE, true>,
                                cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
    DBG_TRY(launch_after(k_bucket_sort<WIDE, true>, sh.buckets, kSortBlock, smem, s, p, rec, keys,
                         counts));
  } else {
    constexpr size_t smem = sort_smem<WIDE, false>();
    DBG_TRY(launch_after(k_place<WIDE, false>, grid, 256, 0, s, h->table, n, p, rec, keys, counts));
    DBG_CK(cudaFuncSetAttribute(k_bucket_sort<WIDE, false>,
                                cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
    DBG_TRY(launch_after(k_bucket_sort<WIDE, false>, sh.buckets, kSortBlock, smem, s, p, rec, keys,
                         counts));
  }
  DBG_CK(cudaGetLastError());
  if (!p.report) DBG_CK(cudaMemcpyAsync(&m, p.meta, sizeof(m), cudaMemcpyDeviceToHost, s));
  DBG_CK(cudaStreamSynchronize(s));
  if (p.report) m = *p.report;
  return DBG_OK;
}

}  // namespace

int export_bins_scratch(int k, uint64_t rows, uint64_t n_slots, uint64_t &bytes) {
  Shape sh{};
  DBG_TRY(export_shape(k, rows, n_slots, sh));
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
  DBG_TRY(export_shape(h->k, rows, h->n_slots, sh));
  char *buf = static_cast<char *>(scratch);
  if (!scratch) DBG_TRY(scratch_alloc(reinterpret_cast<void **>(&buf), sh.total, s));
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
    rc = h->k > 32 ? run<true>(h, sh, max_rows, buf, rec, rec_rows, keys_out, counts_out, m, s)
                   : run<false>(h, sh, max_rows, buf, rec, rec_rows, keys_out, counts_out, m, s);
    if (own && rc == DBG_OK) {
      const cudaError_t e = cudaEventRecord(h->bin.done, s);
      if (e != cudaSuccess) rc = cuda_fail(e, "cudaEventRecord");
    }
    if (rc != DBG_OK || !rec || m.vertices <= rec_rows) break;
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
  *too_dense = m.vertices > 0 && (1u << sh.bucket_log2) + m.max_bin > kBucketCap;
  return DBG_OK;
}

}  // namespace dbg
