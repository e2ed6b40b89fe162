// K1 (direct path): the fused read-tile insert kernel -- Alg. 2 "makeGraph"
// with Alg. 3 "addLeftVertex", Alg. 4 "findVertex" and the addRightVertex
// prose, done the GPU way.  The tile walk, shared-memory staging and key
// extraction are in dbg_tiles.cuh; this file is what happens to a vertex:
//
//   find or claim the key's slot: linear probing from the hash's home slot,
//   a relaxed load first and atomicCAS(EMPTY -> key) only on an empty slot,
//   so that a found vertex costs one L2 read and no atomic; then, if the
//   position starts a k-mer (j <= len - k), add 1 to the slot's counter for
//   the label s_{k-1} (a fire-and-forget atomicAdd at L2).
//
// Counters start at zero (table init), so a thread that loses the CAS race
// for a key can count at once: no allocate/retry/free loop (Alg. 3's
// do-while) is needed, and the result is independent of thread order.
//
// Warp aggregation (__match_any_sync; off in a new handle, whose tuning is all
// zeros; on where the tuning says 1 or leaves it to this file with -1): lanes of
// a warp holding the same key probe once (the lowest lane), and lanes adding to
// the same (slot, label) counter issue one atomicAdd of the group size.
//
// Probing is bounded by max_probes; a vertex that finds neither its key nor
// an empty slot sets the sticky DBG_ERR_CAPACITY and the CTA stops, and later
// tiles of the item are skipped, so an overfull table never spins.
#include <algorithm>

#include "dbg_tiles.cuh"

namespace dbg {
namespace {

template <bool AGG>
struct InsertVisitor {
  static constexpr bool kUniformRounds = false;
  volatile uint32_t *s_cap_hit;

  __device__ void tile_begin() {
    if (threadIdx.x == 0) *s_cap_hit = 0u;
  }
  __device__ bool stop(int) {
    if (AGG) return __any_sync(kFull, *s_cap_hit != 0u);
    return *s_cap_hit != 0u;
  }
  __device__ void round_end() {}

  __device__ void vertex(bool valid, uint64_t key, bool edge, uint32_t label, int lane, int,
                         const VertexCtx &c) {
    if (!AGG) {
      if (valid) {
        uint64_t slot;
        if (find_or_claim(c.table, c.n_slots, c.max_probes, key, slot)) {
          if (edge) red_add_u32(&c.table[slot].cnt[label], 1u);
        } else if (spill_or_fail(c.spill, c.spill_cap, c.spill_count, c.status, key, edge, label)) {
          *s_cap_hit = 1u;
        }
      }
    } else {
      const unsigned long long mk = valid ? key : kEmpty;
      const unsigned peers = __match_any_sync(kFull, mk);
      const int leader = __ffs(peers) - 1;
      uint64_t slot = 0;
      int ok = 0;
      if (valid && lane == leader) {
        ok = find_or_claim(c.table, c.n_slots, c.max_probes, key, slot) ? 1 : 0;
        if (!ok) {
          // every lane of the group spills its own position below
          ok = -1;
        }
      }
      slot = __shfl_sync(kFull, slot, leader);
      ok = __shfl_sync(kFull, ok, leader);
      if (valid && ok < 0) {
        if (spill_or_fail(c.spill, c.spill_cap, c.spill_count, c.status, key, edge, label))
          *s_cap_hit = 1u;
        ok = 0;
      }
      const bool add = valid && ok > 0 && edge;
      const unsigned long long ek = add ? ((slot << 2) | label) : kEmpty;
      const unsigned grp = __match_any_sync(kFull, ek);
      if (add && lane == __ffs(grp) - 1)
        atomicAdd(&c.table[slot].cnt[label], (uint32_t)__popc(grp));
    }
  }
};

// Reads per tile when the tuning leaves it open.  A tile is a CTA's unit of
// work, and a thread holds one position in flight, so a read set of few tiles
// leaves the chip idle: 1,000 reads in tiles of 256 ran on 4 CTAs (276 us;
// now 17).  The reads are cut into whole waves of the resident CTAs with at
// most kAutoTileReads reads a tile (20,000 reads on 1,216 CTAs: 94 us as one
// wave of 17, 109 as a wave of 16 and its rest), and at least kMinTileReads:
// a tile of one read would leave most of a CTA's threads idle.  That suits reads
// of 100 bases and more.  Tiles of 20 shorter ones hold too few positions for a
// CTA's threads and barriers, and only the device knows: a large read set's tiles
// take up to kShortTileReads of them, for kTilePositions positions (571,000 reads
// of 36 bases, k = 31: 174 us with tiles of 20, 110 with 109; 182,000 of 50: 110 ->
// 105).  Many read sets in one launch take up to kAutoTileReadsMany (128 sets of
// 36-base reads 0.67 ms with 20, 0.50 with 48 as with 256; of 150 bases 0.57, 0.56).
constexpr int kMinTileReads = 2, kAutoTileReads = 20, kAutoTileReadsMany = 48;
constexpr int kShortTileReads = 128;
constexpr uint64_t kTilePositions = 768;
constexpr uint64_t kAdaptReads = 12;  // reads per resident CTA from which the device is asked

__device__ __forceinline__ int short_tile_reads(const ItemDesc &it, int tile_reads) {
  const uint64_t bases = it.offsets[it.n_reads] - it.offsets[0];  // (decreasing: any size will do)
  const uint64_t length = bases / it.n_reads;
  const uint64_t positions = length + 2 > (uint64_t)it.k ? length + 2 - (uint64_t)it.k : 1ull;
  const uint64_t reads = kTilePositions / positions;
  return max(tile_reads, (int)min(reads, (uint64_t)kShortTileReads));
}

// Bound by the latency of dependent L2 round trips: a warp waits for its
// longest probe chain (about four loads and a CAS over its 32 positions), so
// the kernel is held to 32 registers for 64 warps an SM (a few words spill):
// 9.2 M positions into a 56 MB table 270 us at 48 registers -> 231 us.  A run
// of four positions per thread with their probes in flight together took
// 335 us: twice the instructions, at 13 active lanes instead of 19.
// (adapt, one read set: a tile may take up to kShortTileReads reads, when they are
// short -- see short_tile_reads)
template <int BLOCK, bool AGG, int N>
__global__ void __launch_bounds__(BLOCK, 2048 / BLOCK)
    k_insert(const __grid_constant__ ItemPack<N> pk, int tile_reads, bool adapt,
             const uint32_t *gate) {
  after_previous();
  if (gate != nullptr && ld_volatile_u32(gate) != 0u) return;
  if (blockIdx.x == 0)  // (the graphs grow, uncounted)
    for (int i = threadIdx.x; i < pk.n_items; i += BLOCK) *small_counted(pk.d[i].status) = 0u;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ volatile uint32_t s_cap_hit;
  InsertVisitor<AGG> vis{&s_cap_hit};
  uint64_t tiles = pk.total_tiles;
  if (N == 1 && adapt) {
    tile_reads = short_tile_reads(pk.d[0], tile_reads);
    tiles = (pk.d[0].n_reads + (uint64_t)tile_reads - 1) / (uint64_t)tile_reads;
  }
  for_each_vertex<BLOCK, N, 1>(pk, tile_reads, smem_raw, vis, blockIdx.x, tiles, gridDim.x);
}

// Number the items' tiles and launch.
template <int BLOCK, bool AGG, int N>
int launch_one(ItemPack<N> &pk, int tile_reads, int grid_ctas, int sm_count, cudaStream_t stream,
               const uint32_t *gate) {
  auto kern = k_insert<BLOCK, AGG, N>;
  int per_sm = 0;
  size_t smem = tile_smem_bytes(tile_reads > 0 ? tile_reads : kShortTileReads);
  if (smem > 48 * 1024)
    DBG_CK(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
  DBG_CK(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, BLOCK, smem));
  const int resident = std::max(1, per_sm) * std::max(1, sm_count);
  bool adapt = false;
  if (tile_reads <= 0) {
    uint64_t reads = 0;
    for (int i = 0; i < pk.n_items; ++i) reads += pk.d[i].n_reads;
    tile_reads = auto_tile_reads(reads, (uint64_t)resident,
                                 N == 1 ? kAutoTileReads : kAutoTileReadsMany);
    adapt = N == 1 && reads > kAdaptReads * (uint64_t)resident;
    if (!adapt) smem = tile_smem_bytes(tile_reads);
  }
  pk.total_tiles = 0;
  for (int i = 0; i < pk.n_items; ++i) {
    pk.d[i].tile_begin = pk.total_tiles;
    pk.total_tiles += (pk.d[i].n_reads + (uint64_t)tile_reads - 1) / (uint64_t)tile_reads;
  }
  if (pk.total_tiles == 0) return DBG_OK;
  int grid = grid_ctas > 0 ? grid_ctas : resident;
  if ((uint64_t)grid > pk.total_tiles) grid = (int)pk.total_tiles;
  // (a gated insert plainly: its CTAs stay on their SMs to the end, so they are not
  // to be placed while the binned chain's last kernel still runs.  323 M events of
  // 65,000 reads 5.7 ms, 5.7 to 6.5 launched over it; into a table that fills up on
  // the way 14.1 against 19.8)
  DBG_TRY(launch_next(gate == nullptr, kern, grid, BLOCK, smem, stream, pk, tile_reads, adapt,
                      gate));
  DBG_CK(cudaGetLastError());
  return DBG_OK;
}

template <int N>
int launch_pack(const ItemDesc *items, int n_items, int tile_reads, const dbg_tuning &t,
                int sm_count, cudaStream_t stream, const uint32_t *gate) {
  ItemPack<N> pk{};
  pk.n_items = n_items;
  for (int i = 0; i < n_items; ++i) pk.d[i] = items[i];
  const bool agg = t.warp_aggregate != 0;
#define DBG_LAUNCH(B)                                                                    \
  return agg ? launch_one<B, true, N>(pk, tile_reads, t.grid_ctas, sm_count, stream, gate) \
             : launch_one<B, false, N>(pk, tile_reads, t.grid_ctas, sm_count, stream, gate)
  switch (t.block_threads) {
    case 128: DBG_LAUNCH(128);
    case 256: DBG_LAUNCH(256);
    case 512: DBG_LAUNCH(512);
    default: return DBG_ERR_INVALID_ARG;
  }
#undef DBG_LAUNCH
}

}  // namespace

int auto_tile_reads(uint64_t reads, uint64_t resident, int most) {
  if (most <= 0) most = kAutoTileReads;
  const uint64_t waves = std::max<uint64_t>(1, (reads + resident * most - 1) / (resident * most));
  const uint64_t ctas = resident * waves;
  return (int)std::max<uint64_t>(kMinTileReads, (reads + ctas - 1) / ctas);
}

dbg_tuning resolve_tuning(const dbg_tuning &t) {
  dbg_tuning r = t;
  if (r.block_threads <= 0) r.block_threads = 256;
  if (r.tile_reads <= 0 || r.tile_reads > r.block_threads) r.tile_reads = r.block_threads;
  // warp aggregation left to us (-1): on, as it merges repeats (microsatellite
  // reads: 0.85 -> 0.18 ms) and costs nothing where the table's sectors are the
  // bound (100 Mbp direct insert: 155.9 ms either way)
  if (r.warp_aggregate < 0) r.warp_aggregate = 1;
  if (r.apply_unroll <= 0) r.apply_unroll = 4;
  if (r.apply_chunk <= 0) r.apply_chunk = 8;
  if (r.apply_counters <= 0) r.apply_counters = 16;
  return r;
}

int launch_insert(const ItemDesc *items, int n_items, const dbg_tuning &tuning, int sm_count,
                  cudaStream_t stream, const uint32_t *gate) {
  if (n_items <= 0) return DBG_OK;
  if (n_items > kBatchItems) return DBG_ERR_INVALID_ARG;
  const dbg_tuning t = resolve_tuning(tuning);
  // (0: chosen by the launch; resolve_tuning's default is the streaming walk's)
  const int tile_reads = tuning.tile_reads > 0 ? t.tile_reads : 0;
  return n_items == 1
             ? launch_pack<1>(items, n_items, tile_reads, t, sm_count, stream, gate)
             : launch_pack<kBatchItems>(items, n_items, tile_reads, t, sm_count, stream, gate);
}

}  // namespace dbg
