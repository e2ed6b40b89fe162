// Graphs with k from 33 to 64 (the paper's default is k = 51, Section "Code
// organization"): vertex keys of 32..63 bases need up to 126 bits.
//
// Slot (32 bytes, the same table as for k <= 32): word 0 = the key's high 64
// bits, word 1 = its low 64 bits, then the four 32-bit counters.  An empty
// slot has word 0 = all ones (never a key's high word: it holds at most 62
// bits) and word 1 = 0, which is what the table initialisation writes.
// Claims are one 128-bit atomicCAS (atom.cas.b128), probes one 128-bit atomic
// load, so a probe never sees half a key.
//
// The insert kernel takes tiles of reads: it stages the tiles' packed bytes
// in shared memory (coalesced, bounded by the stream's length), then gives
// each thread vertex positions of the tile; a key is cut from three 64-bit
// words of the staged stream and its 2-bit groups reversed so that the first
// base is most significant.
#include <cub/device/device_radix_sort.cuh>

#include <algorithm>

#include "dbg_wide.cuh"

namespace dbg {
namespace {

// Bound by the table's random sectors (a load that misses the L2, then the add
// that makes the sector dirty: 2.4e10 a second of a table far larger than the
// L2): 168 M positions into a 3.5 GB table 14.7 -> 12.5 ms (1.43 probes each,
// 241 M sector reads and as many sectors made dirty as positions), by one
// 128-bit load a probe, a warp-scanned prefix, 16-byte staging and tiles cut
// by the number of reads.  (CTAS: per SM.  A table that the L2 holds is bound by
// the probes' latency: 32 registers for 64 warps an SM, 4 M positions of 75-base
// reads into 80 MB 128 us at 40 registers -> 117, 4 M of 1 kb reads 158 -> 145; the
// 3.5 GB table is better off with 40, 12.5 ms against 12.9.)
template <int BLOCK, int CTAS>
__global__ void __launch_bounds__(BLOCK, CTAS)
    k_insert_wide(ItemDesc it, int tile_reads, const uint32_t *gate) {
  after_previous();
  if (gate != nullptr && ld_volatile_u32(gate) != 0u) return;
  if (blockIdx.x == 0 && threadIdx.x == 0) *small_counted(it.status) = 0u;  // (it grows, uncounted)
  __shared__ uint64_t s_off[kWideTile + 1];
  __shared__ uint64_t s_pre[kWideTile + 1];
  __shared__ __align__(16) uint64_t s_win[kWideWinBytes / 8 + 4];
  __shared__ uint64_t s_sum[kWideTile / 32];
  __shared__ uint32_t s_stop;
  static_assert(kWideTile <= BLOCK && kWideTile % 32 == 0, "a thread per read of a tile");
  const int k = it.k, m = k - 1;
  const uint64_t last = it.offsets[it.n_reads];
  const uint64_t nbytes = last >= it.origin ? (last - it.origin + 3) >> 2 : 0;
  WideSlot *table = reinterpret_cast<WideSlot *>(it.table);
  const uint64_t tiles = (it.n_reads + (uint64_t)tile_reads - 1) / (uint64_t)tile_reads;
  const int tid = threadIdx.x, lane = tid & 31;
  for (uint64_t t = blockIdx.x; t < tiles; t += gridDim.x) {
    const uint64_t r0 = t * (uint64_t)tile_reads;
    const int nr = (int)min((uint64_t)tile_reads, it.n_reads - r0);
    if (tid == 0) s_stop = ld_volatile_u32(it.status);
    for (int i = tid; i <= nr; i += BLOCK) s_off[i] = it.offsets[r0 + i];
    __syncthreads();
    if (s_stop) return;  // an earlier error stops the insert (the same value for every thread)
    // vertex positions per read, prefix; bad offsets stop the tile
    uint64_t nv = 0;
    bool wrong = false;
    if (tid < nr) {
      const uint64_t a = s_off[tid], b = s_off[tid + 1];
      wrong = b < a || a < it.origin;
      const uint64_t len = b >= a ? b - a : 0;
      nv = len >= (uint64_t)k ? len - k + 2 : 0;
    }
    uint64_t incl = nv;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
      const uint64_t o = __shfl_up_sync(0xffffffffu, incl, d);
      if (lane >= d) incl += o;
    }
    if (lane == 31 && tid < kWideTile) s_sum[tid >> 5] = incl;
    const bool bad = __syncthreads_or(wrong) != 0;
    if (tid < nr) {
      for (int w = 0; w < tid >> 5; ++w) incl += s_sum[w];
      s_pre[tid] = incl - nv;
      if (tid == nr - 1) s_pre[nr] = bad ? 0 : incl;
    }
    if (bad && tid == 0) set_sticky(it.status, DBG_ERR_BAD_OFFSETS);
    // the tile's bytes, staged if they fit the window: 16 bytes a load where
    // the stream allows, zeros past its end
    const uint64_t lo_b = s_off[0] >= it.origin ? ((s_off[0] - it.origin) >> 2) & ~15ull : 0;
    const uint64_t hi_b = s_off[nr] >= it.origin ? ((s_off[nr] - it.origin + 3) >> 2) : 0;
    const uint64_t b0 = lo_b;
    const uint64_t staged = (!bad && hi_b > lo_b && hi_b - lo_b + 24 <= (uint64_t)kWideWinBytes)
                                ? hi_b - lo_b + 24
                                : 0;
    if (staged) {
      const uint64_t end = min(hi_b, nbytes);  // (below lo_b when a later offset decreases)
      const uint64_t whole = it.vec_ok && end > lo_b ? (end - lo_b) >> 4 : 0;
      for (uint64_t i = tid; i < whole; i += BLOCK)
        reinterpret_cast<uint4 *>(s_win)[i] =
            __ldg(reinterpret_cast<const uint4 *>(it.packed + b0) + i);
      unsigned char *win = reinterpret_cast<unsigned char *>(s_win);
      for (uint64_t i = 16 * whole + tid; i < staged; i += BLOCK)
        win[i] = b0 + i < nbytes ? it.packed[b0 + i] : (unsigned char)0;
    }
    __syncthreads();
    const uint64_t total = s_pre[nr];
    for (uint64_t v = threadIdx.x; v < total; v += BLOCK) {
      int lo_r = 0, hi_r = nr - 1;  // the read holding vertex position v
      while (lo_r < hi_r) {
        const int mid = (lo_r + hi_r + 1) >> 1;
        if (s_pre[mid] <= v)
          lo_r = mid;
        else
          hi_r = mid - 1;
      }
      const uint64_t j = v - s_pre[lo_r];
      const uint64_t len = s_off[lo_r + 1] - s_off[lo_r];
      const uint64_t p = s_off[lo_r] - it.origin + j;  // first base of the vertex
      const bool edge = j + (uint64_t)k <= len;
      uint64_t w0, w1, w2, wl;
      uint32_t sh;
      if (staged) {
        const uint64_t bit = 2 * p - 8 * b0;
        const uint64_t wi = bit >> 6;
        sh = (uint32_t)(bit & 63);
        w0 = s_win[wi];
        w1 = s_win[wi + 1];
        w2 = s_win[wi + 2];
      } else {
        const uint64_t at = (p >> 2);
        sh = (uint32_t)(2 * (p & 3));
        w0 = word_at(it.packed, nbytes, at);
        w1 = word_at(it.packed, nbytes, at + 8);
        w2 = word_at(it.packed, nbytes, at + 16);
      }
      uint64_t hi, lo;
      wide_key(w0, w1, w2, sh, m, hi, lo);
      uint32_t label = 0;
      if (edge) {
        const uint64_t q = p + (uint64_t)m;  // the k-mer's last base
        if (staged) {
          const uint64_t bit = 2 * q - 8 * b0;
          wl = s_win[bit >> 6] >> (bit & 63);
        } else {
          wl = (uint64_t)__ldg(it.packed + (q >> 2)) >> (2 * (q & 3));
        }
        label = (uint32_t)(wl & 3u);
      }
      uint64_t s;
      if (wide_find_or_claim(table, it.n_slots, it.max_probes, hi, lo, s)) {
        if (edge) red_add_u32(&table[s].cnt[label], 1u);
      } else {
        set_sticky(it.status, DBG_ERR_CAPACITY);
      }
    }
    __syncthreads();
  }
}

// --- export -------------------------------------------------------------------

__global__ void k_wide_words(const WideSlot *t, const unsigned long long *idx, uint64_t n,
                             unsigned long long *out, int word) {
  const uint64_t stride = (uint64_t)gridDim.x * blockDim.x;
  for (uint64_t i = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += stride)
    out[i] = word ? t[idx[i]].w1 : t[idx[i]].w0;
}

__global__ void k_wide_gather(const WideSlot *t, const unsigned long long *idx, uint64_t n,
                              ulonglong2 *keys, uint4 *counts) {
  const uint64_t stride = (uint64_t)gridDim.x * blockDim.x;
  for (uint64_t i = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += stride) {
    const WideSlot &s = t[idx[i]];
    keys[i] = make_ulonglong2(s.w0, s.w1);
    counts[i] = make_uint4(s.cnt[0], s.cnt[1], s.cnt[2], s.cnt[3]);
  }
}

__global__ void k_wide_compact(const WideSlot *t, uint64_t n_slots, unsigned long long *idx,
                               unsigned long long *count, uint64_t cap) {
  const int lane = threadIdx.x & 31;
  const uint64_t warps = ((uint64_t)gridDim.x * blockDim.x) >> 5;
  const uint64_t w0 = (((uint64_t)blockIdx.x * blockDim.x) + threadIdx.x) >> 5;
  for (uint64_t base = w0 * 32; base < n_slots; base += warps * 32) {
    const uint64_t i = base + lane;
    const bool occ = i < n_slots && t[i].w0 != kEmpty;
    const unsigned mask = __ballot_sync(0xffffffffu, occ);
    unsigned long long pos = 0;
    if (lane == 0 && mask) pos = atomicAdd(count, (unsigned long long)__popc(mask));
    pos = __shfl_sync(0xffffffffu, pos, 0);
    const unsigned long long at = pos + __popc(mask & ((1u << lane) - 1u));
    if (occ && at < cap) idx[at] = i;
  }
}

size_t al256(size_t x) { return (x + 255) & ~size_t(255); }

}  // namespace

int launch_insert_wide(const ItemDesc &it, int sm_count, cudaStream_t s, const uint32_t *gate) {
  if (it.n_reads == 0) return DBG_OK;
  constexpr int B = 256;
  constexpr uint64_t kL2Bytes = 128ull << 20;
  const auto kern = it.n_slots * sizeof(WideSlot) <= kL2Bytes ? k_insert_wide<B, 8>
                                                              : k_insert_wide<B, 6>;
  int per_sm = 0;
  DBG_CK(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, B, 0));
  const uint64_t resident = (uint64_t)std::max(1, per_sm) * std::max(1, sm_count);
  const int tile_reads = std::min(kWideTile, auto_tile_reads(it.n_reads, resident));
  const uint64_t tiles = (it.n_reads + tile_reads - 1) / tile_reads;
  // (plainly behind a binned chain, see the one-word insert's launch)
  DBG_TRY(launch_next(gate == nullptr, kern, (int)std::min(tiles, resident), B, 0, s, it,
                      tile_reads, gate));
  DBG_CK(cudaGetLastError());
  return DBG_OK;
}

// Sorted export of a wide table: compaction, then two stable radix sorts
// (low words, then high words) carrying the slot indices, then a gather.
int export_sorted_wide(dbg_handle h, uint64_t D, uint64_t *keys_out, uint32_t *counts_out,
                       cudaStream_t s) {
  const int m = h->k - 1;
  const int hi_bits = 2 * m - 64;  // bits of the high word (0 .. 62)
  const WideSlot *t = reinterpret_cast<const WideSlot *>(h->table);
  size_t temp_bytes = 0;
  DBG_CK(cub::DeviceRadixSort::SortPairs(nullptr, temp_bytes, (unsigned long long *)nullptr,
                                         (unsigned long long *)nullptr,
                                         (unsigned long long *)nullptr,
                                         (unsigned long long *)nullptr, (int64_t)D, 0, 64, s));
  const size_t kb = al256(D * sizeof(unsigned long long));
  const size_t total = 4 * kb + al256(D * 16) + al256(D * 16) + 256 + al256(temp_bytes);
  char *buf = nullptr;
  DBG_TRY(scratch_alloc(reinterpret_cast<void **>(&buf), total, s));
  unsigned long long *w_a = reinterpret_cast<unsigned long long *>(buf);
  unsigned long long *w_b = reinterpret_cast<unsigned long long *>(buf + kb);
  unsigned long long *idx_a = reinterpret_cast<unsigned long long *>(buf + 2 * kb);
  unsigned long long *idx_b = reinterpret_cast<unsigned long long *>(buf + 3 * kb);
  ulonglong2 *keys = reinterpret_cast<ulonglong2 *>(buf + 4 * kb);
  uint4 *counts = reinterpret_cast<uint4 *>(buf + 4 * kb + al256(D * 16));
  unsigned long long *count =
      reinterpret_cast<unsigned long long *>(buf + 4 * kb + 2 * al256(D * 16));
  void *temp = buf + 4 * kb + 2 * al256(D * 16) + 256;
  const int grid = std::max(1, h->sm_count) * 8;
  int rc = DBG_OK;
  do {
    cudaError_t e = cudaMemsetAsync(count, 0, sizeof(unsigned long long), s);
    if (e != cudaSuccess) { rc = cuda_fail(e, "cudaMemsetAsync"); break; }
    k_wide_compact<<<grid, 256, 0, s>>>(t, h->n_slots, idx_a, count, D);
    k_wide_words<<<grid, 256, 0, s>>>(t, idx_a, D, w_a, 1);  // low words
    e = cub::DeviceRadixSort::SortPairs(temp, temp_bytes, w_a, w_b, idx_a, idx_b, (int64_t)D, 0,
                                        64, s);
    if (e != cudaSuccess) { rc = cuda_fail(e, "SortPairs(low words)"); break; }
    const unsigned long long *order = idx_b;
    if (hi_bits > 0) {  // stable: equal high words keep their low-word order
      k_wide_words<<<grid, 256, 0, s>>>(t, idx_b, D, w_a, 0);
      e = cub::DeviceRadixSort::SortPairs(temp, temp_bytes, w_a, w_b, idx_b, idx_a, (int64_t)D,
                                          0, hi_bits, s);
      if (e != cudaSuccess) { rc = cuda_fail(e, "SortPairs(high words)"); break; }
      order = idx_a;
    }
    k_wide_gather<<<grid, 256, 0, s>>>(t, order, D, keys, counts);
    e = cudaGetLastError();
    if (e != cudaSuccess) { rc = cuda_fail(e, "wide export kernels"); break; }
    if (keys_out) {
      e = cudaMemcpyAsync(keys_out, keys, D * 16, cudaMemcpyDefault, s);
      if (e != cudaSuccess) { rc = cuda_fail(e, "cudaMemcpyAsync(keys)"); break; }
    }
    if (counts_out) {
      e = cudaMemcpyAsync(counts_out, counts, D * sizeof(uint4), cudaMemcpyDefault, s);
      if (e != cudaSuccess) { rc = cuda_fail(e, "cudaMemcpyAsync(counts)"); break; }
    }
  } while (0);
  cudaError_t e = cudaFreeAsync(buf, s);
  if (rc == DBG_OK && e != cudaSuccess) rc = cuda_fail(e, "cudaFreeAsync");
  e = cudaStreamSynchronize(s);
  if (rc == DBG_OK && e != cudaSuccess) rc = cuda_fail(e, "cudaStreamSynchronize");
  return rc;
}

}  // namespace dbg
