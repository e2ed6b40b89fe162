// K7: HyperLogLog sketch of a read set's vertex keys, the input of the
// capacity predictor (the table must be sized before the build; the number of
// distinct vertices is what sizes it).
//
// For every vertex position (the same positions the insert visits) the key is
// hashed with MurmurHash3's 64-bit finalizer after an XOR with a fixed salt
// (so the sketch hash is unrelated to the table's slot hash); the top 10 bits
// of the hash pick one of 1024 registers and the register keeps the maximum
// of rho = 1 + the number of leading zeros of the remaining 54 bits
// (Flajolet, Fusy, Gandouet, Meunier, "HyperLogLog", AofA 2007).  A maximum
// does not depend on order or repetition, so the registers are a function of
// the set of distinct keys only.
#include <math.h>

#include <algorithm>

#include "dbg_tiles.cuh"

namespace dbg {
namespace {

constexpr unsigned long long kSketchSalt = 0x9E3779B97F4A7C15ull;
constexpr int kSketchRegs = DBG_SKETCH_REGISTERS;
constexpr int kSketchRun = 16;  // positions of one read per thread and round
constexpr int kSketchCtas = 7;  // CTAs of 256 threads per SM (shared memory allows 7)
// read sets per launch: 256 descriptors (26.6 KB) still fit the kernel parameters
constexpr int kSketchItems = 2 * kBatchItems;

// Registers in shared memory (one read set per launch).  A register only
// grows, and after the first few thousand keys almost no key raises it: a key
// whose rho cannot exceed the smallest register (a lower bound the CTA
// refreshes at every tile start) is dropped after one compare, the others
// read their register first and take the atomic only to raise it.  At a tile
// start the CTA also exchanges registers with the item's global ones, which
// its other CTAs fill: the bound is then that of all keys seen so far, not of
// the CTA's share (64 samples on 1,052 CTAs: 1.61 -> 1.47 ms; with the
// CTA's own bound almost every step had a lane whose key passed it).  The
// registers are the same as without the bound.
struct SketchVisitor {
  static constexpr bool kUniformRounds = false;
  uint32_t *s_reg;
  uint32_t *g_reg;  // the item's registers in global memory
  volatile uint32_t *s_floor;  // every register is at least this (any value it held stays true)
  // The bits of the hash from 53 down to 32 are the leading bits of the 54 that
  // rho counts zeros in: a key for which they are above `lim` has rho <= floor
  // (a floor of 0 drops nothing; from 22 on, any set bit among them does).
  uint32_t lim = kLead;
  bool first = true;  // before the item's first tile
  static constexpr uint32_t kLead = (1u << 22) - 1u;
  __device__ void set_floor() {  // (the calling warp's; the minimum of all registers)
    uint32_t m = ~0u;
    for (int j = threadIdx.x & 31; j < kSketchRegs; j += 32)
      m = min(m, *reinterpret_cast<volatile uint32_t *>(&s_reg[j]));
    m = __reduce_min_sync(0xffffffffu, m);
    if ((threadIdx.x & 31) == 0) *s_floor = m;
  }
  // A read set's first tile: what its other CTAs know already.  (A CTA of the
  // first wave starts with the others: they know nothing yet, and asking would
  // be 2 us of a small read set's 34.)
  __device__ void item_begin(uint32_t *g, bool first_wave) {
    g_reg = g;
    first = true;
    for (int j = threadIdx.x; j < kSketchRegs; j += blockDim.x)
      s_reg[j] = first_wave ? 0u : ld_volatile_u32(g + j);
    if (threadIdx.x == 0) *s_floor = 0u;
    __syncthreads();
    if (first_wave) return;
    if (threadIdx.x < 32) set_floor();
    __syncthreads();
  }
  // Its last tile: what this CTA knows.  (ask: others have merged theirs by now,
  // and most registers need no atomic)
  __device__ void item_end(bool ask) {
    __syncthreads();
    for (int j = threadIdx.x; j < kSketchRegs; j += blockDim.x)
      if (s_reg[j] > (ask ? ld_volatile_u32(g_reg + j) : 0u)) atomicMax(&g_reg[j], s_reg[j]);
    __syncthreads();
  }
  __device__ void tile_begin() {
    const uint32_t f = *s_floor;
    lim = f < 22u ? kLead >> f : 0u;
    if (first) {  // (the registers are as item_begin left them)
      first = false;
      return;
    }
    for (int j = threadIdx.x; j < kSketchRegs; j += blockDim.x) {
      const uint32_t own = s_reg[j], all = ld_volatile_u32(g_reg + j);
      if (own > all)
        atomicMax(&g_reg[j], own);
      else
        s_reg[j] = all;  // (between tiles: no other thread touches it)
    }
    if (threadIdx.x < 32) set_floor();  // the next tile's (registers only grow: any moment's will do)
  }
  __device__ bool stop(int) { return false; }
  __device__ void round_end() {}
  __device__ void vertex(bool valid, uint64_t key, bool, uint32_t, int, int, const VertexCtx &) {
    if (!valid) return;
    // fmix64(key ^ salt) up to its last shift, which leaves the hash's high word
    // alone.  (The product's high word by itself first, the whole for the few keys
    // that pass, is more instructions: 64 samples 1.29 -> 1.25 ms, two tiles of
    // 10 kb reads, of which most keys pass, 1.36 -> 1.26.)
    uint64_t h = key ^ kSketchSalt;
    h = (h ^ (h >> 33)) * 0xff51afd7ed558ccdull;
    h = (h ^ (h >> 33)) * 0xc4ceb9fe1a85ec53ull;
    if (((uint32_t)(h >> 32) & kLead) > lim) return;  // 1 + clz(rest) <= floor: no register can rise
    h ^= h >> 33;
    const uint64_t rest = h << 10;
    const uint32_t idx = (uint32_t)(h >> 54);
    const uint32_t rho = rest ? (uint32_t)__clzll(rest) + 1u : 55u;
    if (rho > *reinterpret_cast<volatile uint32_t *>(&s_reg[idx])) atomicMax(&s_reg[idx], rho);
  }
};

template <int BLOCK>
__global__ void __launch_bounds__(BLOCK, kSketchCtas)
    k_sketch(const __grid_constant__ ItemPack<1> pk, int tile_reads, uint64_t chunk,
             uint32_t first_wave, uint32_t *regs) {
  after_previous();
  extern __shared__ __align__(16) unsigned char smem[];
  uint32_t *s_reg = reinterpret_cast<uint32_t *>(smem + tile_smem_bytes(tile_reads));
  __shared__ uint32_t s_floor;
  SketchVisitor vis{s_reg, nullptr, &s_floor};
  vis.item_begin(regs, blockIdx.x < first_wave);
  for_each_vertex<BLOCK, 1, kSketchRun>(pk, tile_reads, smem, vis, blockIdx.x * chunk,
                                        (blockIdx.x + 1) * chunk, 1);
  vis.item_end(gridDim.x > first_wave);
}

// Many read sets per launch.  Each CTA takes a contiguous range of tiles, so
// it meets few item boundaries; it keeps shared-memory registers for the
// item at hand and merges them into that item's global registers (carried in
// the descriptor's table pointer) when its tiles of the item end.
template <int BLOCK>
__global__ void __launch_bounds__(BLOCK, kSketchCtas)
    k_sketch_batch(const __grid_constant__ ItemPack<kSketchItems> pk, int tile_reads,
                   uint64_t chunk, uint32_t first_wave) {
  after_previous();
  extern __shared__ __align__(16) unsigned char smem[];
  uint32_t *s_reg = reinterpret_cast<uint32_t *>(smem + tile_smem_bytes(tile_reads));
  __shared__ uint32_t s_floor;
  SketchVisitor vis{s_reg, nullptr, &s_floor};
  const uint64_t t1 = min(pk.total_tiles, (blockIdx.x + 1) * chunk);
  for (uint64_t t = blockIdx.x * chunk; t < t1;) {
    const int it = find_item(pk, t);
    const uint64_t end = it + 1 < pk.n_items ? pk.d[it + 1].tile_begin : pk.total_tiles;
    const uint64_t tb = min(t1, end);
    vis.item_begin(reinterpret_cast<uint32_t *>(pk.d[it].table), blockIdx.x < first_wave);
    for_each_vertex<BLOCK, kSketchItems, kSketchRun>(pk, tile_reads, smem, vis, t, tb, 1);
    vis.item_end(gridDim.x > first_wave);
    t = tb;
  }
}

// Tiles per CTA: kSketchWaves CTAs for every one that is resident at a time, so
// that those which finish early leave their place to others (one CTA each left
// 30 % of the warps' time unused; 64 samples 1.47 ms at one, 1.40 at two, 1.41
// at four, 1.56 at eight).
constexpr uint64_t kSketchWaves = 2;
constexpr uint64_t kSketchMinReads = 8;  // reads a tile (dbg_sketch_reads)

uint64_t sketch_chunk(uint64_t tiles, uint64_t resident) {
  return std::max<uint64_t>(1, (tiles + kSketchWaves * resident - 1) / (kSketchWaves * resident));
}

// Every item's registers and status word := 0.
__global__ void k_zero_registers(const __grid_constant__ ItemPack<kSketchItems> pk) {
  after_previous();
  const int i = blockIdx.x;
  uint32_t *r = reinterpret_cast<uint32_t *>(pk.d[i].table);
  for (int j = threadIdx.x; j <= kSketchRegs; j += blockDim.x) r[j] = 0u;
}

}  // namespace
}  // namespace dbg

extern "C" int dbg_sketch_reads(int k, const uint8_t *packed, const uint64_t *offsets,
                                uint64_t n_reads, uint32_t *registers, void *stream) {
  using namespace dbg;
  if (k < 2 || k > 32 || !registers || (n_reads > 0 && (!packed || !offsets)))
    return DBG_ERR_INVALID_ARG;
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  DBG_CK(cudaMemsetAsync(registers, 0, (kSketchRegs + 1) * sizeof(uint32_t), s));
  if (n_reads == 0) return DBG_OK;
  constexpr int B = 256;
  int dev = 0, sms = 0, per_sm = 0;
  DBG_CK(cudaGetDevice(&dev));
  DBG_CK(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
  DBG_CK(cudaOccupancyMaxActiveBlocksPerMultiprocessor(
      &per_sm, k_sketch<B>, B, tile_smem_bytes(B) + kSketchRegs * sizeof(uint32_t)));
  const uint32_t resident = (uint32_t)(std::max(1, per_sm) * sms);
  // (a read set of few tiles is cut into one for every fourth resident CTA, as each
  // merges 1,024 registers: 500 reads of 10 kb ran on two CTAs, 1.33 -> 0.07 ms)
  const int tile_reads = (int)std::min<uint64_t>(
      B, std::max<uint64_t>(kSketchMinReads, (4 * n_reads + resident - 1) / resident));
  ItemPack<1> pk{};
  pk.n_items = 1;
  pk.total_tiles = (n_reads + tile_reads - 1) / tile_reads;
  ItemDesc &it = pk.d[0];
  it.packed = packed;
  it.offsets = offsets;
  it.n_reads = n_reads;
  it.origin = 0;
  it.table = nullptr;
  it.n_slots = 1;
  it.status = registers + kSketchRegs;  // bad offsets are reported here
  it.max_probes = 0;
  it.k = k;
  it.vec_ok = ((uintptr_t)packed & 15u) == 0 ? 1 : 0;
  const size_t smem = tile_smem_bytes(tile_reads) + kSketchRegs * sizeof(uint32_t);
  const uint64_t chunk = sketch_chunk(pk.total_tiles, resident);
  const int grid = (int)((pk.total_tiles + chunk - 1) / chunk);
  DBG_TRY(launch_after(k_sketch<B>, grid, B, smem, s, pk, tile_reads, chunk, resident, registers));
  DBG_CK(cudaGetLastError());
  return DBG_OK;
}

extern "C" int dbg_sketch_batch(const dbg_sketch_item *items, int n_items, void *stream) {
  using namespace dbg;
  if (n_items < 0 || (n_items > 0 && !items)) return DBG_ERR_INVALID_ARG;
  for (int i = 0; i < n_items; ++i)
    if (items[i].k < 2 || items[i].k > 32 || !items[i].registers ||
        (items[i].n_reads > 0 && (!items[i].packed || !items[i].offsets)))
      return DBG_ERR_INVALID_ARG;
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  constexpr int B = 256;
  const int tile_reads = B;
  const size_t smem = tile_smem_bytes(tile_reads) + kSketchRegs * sizeof(uint32_t);
  int dev = 0, sms = 0, per_sm = 0;
  DBG_CK(cudaGetDevice(&dev));
  DBG_CK(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
  if (smem > 48 * 1024)
    DBG_CK(cudaFuncSetAttribute(k_sketch_batch<B>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                (int)smem));
  DBG_CK(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_sketch_batch<B>, B, smem));
  for (int first = 0; first < n_items; first += kSketchItems) {
    const int cnt = std::min(kSketchItems, n_items - first);
    ItemPack<kSketchItems> pk{};
    pk.n_items = cnt;
    uint64_t tiles = 0;
    for (int i = 0; i < cnt; ++i) {
      const dbg_sketch_item &src = items[first + i];
      ItemDesc &it = pk.d[i];
      it.packed = src.packed;
      it.offsets = src.offsets;
      it.n_reads = src.n_reads;
      it.origin = 0;
      it.table = reinterpret_cast<Slot *>(src.registers);  // the item's registers
      it.n_slots = 1;
      it.status = src.registers + kSketchRegs;  // bad offsets are reported here
      it.max_probes = 0;
      it.k = src.k;
      it.tile_begin = tiles;
      it.vec_ok = ((uintptr_t)src.packed & 15u) == 0 ? 1 : 0;
      tiles += (src.n_reads + tile_reads - 1) / tile_reads;
    }
    pk.total_tiles = tiles;
    DBG_TRY(launch_after(k_zero_registers, cnt, 256, 0, s, pk));
    DBG_CK(cudaGetLastError());
    if (tiles == 0) continue;
    const uint32_t resident = (uint32_t)(std::max(1, per_sm) * sms);
    const uint64_t chunk = sketch_chunk(tiles, resident);
    const int grid = (int)((tiles + chunk - 1) / chunk);
    DBG_TRY(launch_after(k_sketch_batch<B>, grid, B, smem, s, pk, tile_reads, chunk, resident));
    DBG_CK(cudaGetLastError());
  }
  return DBG_OK;
}

extern "C" double dbg_sketch_estimate(const uint32_t *registers) {
  if (!registers) return -1.0;
  const double m = dbg::kSketchRegs;
  const double alpha = 0.7213 / (1.0 + 1.079 / m);
  double sum = 0.0;
  int zeros = 0;
  for (int j = 0; j < dbg::kSketchRegs; ++j) {
    sum += ldexp(1.0, -(int)registers[j]);
    zeros += registers[j] == 0u;
  }
  const double raw = alpha * m * m / sum;
  if (raw <= 2.5 * m && zeros > 0) return m * log(m / zeros);  // small-range correction
  return raw;
}
