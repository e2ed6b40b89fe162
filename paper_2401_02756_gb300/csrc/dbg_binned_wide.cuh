// The binned rebuild for k from 33 to 63 (included by dbg_binned.cu, whose
// region tables, buckets, units and scratch it shares): as the tiled path of
// one-word keys, with 16-byte events.
//
// An event is the key as two words of at most 61 and exactly 63 bits -- the
// key's bits from 63 up under the tag (edge << 2 | label) in the three top
// bits, and its 63 low bits -- so neither word of a key is ever all ones, and
// in shared memory each word can be claimed by a 64-bit CAS of its own: the
// first word of an empty slot, then the second.  Whoever claims the second
// word owns the slot; a thread that finds another key's second word under its
// own first word goes on to the next slot, as past any other key.
//
// Only rebuilds from empty (dbg_build_reads) come here: an insert into a held
// graph stays with the direct kernel.  Bound as the one-word path is, by issue
// and shared-memory latency, at twice the event bytes: 168 M positions into a
// table of 110 M slots 12.7 -> 5.1 ms (scatter 1.55, split 1.30, apply 2.16),
// where the direct insert is held by the table's random sectors.

namespace {

constexpr int kWideBlock = 512;
constexpr int kWideRun = 4;  // consecutive positions per thread and round
constexpr int kWideFlush = kWideBlock * kWideRun;
constexpr unsigned long long kLow63 = ~0ull >> 1;

struct __align__(16) WideEvent {
  unsigned long long a;  // tag << 61 | key bits 63 and up
  unsigned long long b;  // key bits 62 .. 0 (all ones: no event)
  __device__ __forceinline__ unsigned long long top() const { return a & (~0ull >> 3); }
  __device__ __forceinline__ uint32_t tag() const { return (uint32_t)(a >> 61); }
  __device__ __forceinline__ bool none() const { return b == ~0ull; }
};
__device__ __forceinline__ uint64_t wide_hi(unsigned long long a) { return a >> 1; }
__device__ __forceinline__ uint64_t wide_lo(unsigned long long a, unsigned long long b) {
  return (a << 63) | b;
}
__device__ __forceinline__ uint64_t event_hash(unsigned long long a, unsigned long long b) {
  return wide_hash(wide_hi(a), wide_lo(a, b));
}
__device__ __forceinline__ WideEvent ld_event(const WideEvent *p) {
  const ulonglong2 v = __ldcs(reinterpret_cast<const ulonglong2 *>(p));
  return WideEvent{v.x, v.y};
}

size_t wide_scatter_smem(int parts) {
  return (size_t)kWideFlush * (16 + 2) + (size_t)parts * (8 + 4 + 4) + 16;
}

// Tiles of kWideTile reads: every read is cut into runs of kWideRun positions,
// a thread takes a run a round (its first key cut from three words, the others
// rolled), and the round's events go to their regions' buckets in runs sorted
// in shared memory, one atomic a region and round.
__global__ void __launch_bounds__(kWideBlock, 2)
    k_wide_scatter(ItemDesc it, int shift, int parts, unsigned long long *cursor,
                   const unsigned long long *bucket_end, WideEvent *out, uint32_t *use_binned) {
  after_previous();
  if (ld_volatile_u32(use_binned) == 0u) return;
  extern __shared__ __align__(16) unsigned char smem[];
  WideEvent *sorted = reinterpret_cast<WideEvent *>(smem);
  unsigned long long *gbase = reinterpret_cast<unsigned long long *>(sorted + kWideFlush);
  uint32_t *hist = reinterpret_cast<uint32_t *>(gbase + parts);
  uint32_t *off = hist + parts;
  uint16_t *spid = reinterpret_cast<uint16_t *>(off + parts);
  __shared__ uint64_t s_off[kWideTile + 1];
  __shared__ uint32_t s_run[kWideTile + 1];  // first run of every read
  __shared__ __align__(16) uint64_t s_win[kWideWinBytes / 8 + 4];
  __shared__ uint32_t s_warp[kWideBlock / 32], s_stop;
  const int k = it.k, m = k - 1, tid = threadIdx.x;
  const uint64_t last = it.offsets[it.n_reads];
  const uint64_t nbytes = last >= it.origin ? (last - it.origin + 3) >> 2 : 0;
  if (last < it.origin && tid == 0) set_sticky(it.status, DBG_ERR_BAD_OFFSETS);
  const uint64_t tiles = (it.n_reads + kWideTile - 1) / kWideTile;
  const uint64_t mask_hi = (1ull << (2 * m - 64)) - 1ull;  // (2 m - 64 <= 60)
  for (int p = tid; p < parts; p += kWideBlock) hist[p] = 0u;
  for (uint64_t t = blockIdx.x; t < tiles; t += gridDim.x) {
    const uint64_t r0 = t * kWideTile;
    const int nr = (int)min((uint64_t)kWideTile, it.n_reads - r0);
    if (tid == 0) s_stop = ld_volatile_u32(it.status);
    for (int i = tid; i <= nr; i += kWideBlock) s_off[i] = it.offsets[r0 + i];
    __syncthreads();
    if (s_stop) return;  // an earlier error stops the insert (the same value for every thread)
    uint32_t runs = 0;
    bool wrong = false;
    if (tid < nr) {
      const uint64_t a = s_off[tid], b = s_off[tid + 1];
      wrong = b < a || a < it.origin;
      const uint64_t len = b >= a ? b - a : 0;
      if (len >= (uint64_t)k) runs = (uint32_t)((len - k + 2 + kWideRun - 1) / kWideRun);
    }
    uint32_t total_runs;
    const uint32_t first = cta_exclusive_prefix<kWideBlock>(runs, s_warp, total_runs);
    const bool bad = __syncthreads_or(wrong) != 0;
    if (tid <= nr) s_run[tid] = tid < nr ? first : total_runs;
    if (bad && tid == 0) set_sticky(it.status, DBG_ERR_BAD_OFFSETS);
    const uint64_t b0 = s_off[0] >= it.origin ? ((s_off[0] - it.origin) >> 2) & ~15ull : 0;
    const uint64_t hi_b = s_off[nr] >= it.origin ? ((s_off[nr] - it.origin + 3) >> 2) : 0;
    const uint64_t staged = (!bad && hi_b > b0 && hi_b - b0 + 24 <= (uint64_t)kWideWinBytes)
                                ? hi_b - b0 + 24
                                : 0;
    if (staged) {
      const uint64_t end = min(hi_b, nbytes);  // (below b0 when a later offset decreases)
      const uint64_t whole = it.vec_ok && end > b0 ? (end - b0) >> 4 : 0;
      for (uint64_t i = tid; i < whole; i += kWideBlock)
        reinterpret_cast<uint4 *>(s_win)[i] =
            __ldg(reinterpret_cast<const uint4 *>(it.packed + b0) + i);
      unsigned char *win = reinterpret_cast<unsigned char *>(s_win);
      for (uint64_t i = 16 * whole + tid; i < staged; i += kWideBlock)
        win[i] = b0 + i < nbytes ? it.packed[b0 + i] : (unsigned char)0;
    }
    __syncthreads();
    if (bad) return;
    for (uint32_t ub = 0; ub < total_runs; ub += kWideBlock) {
      const uint32_t u = ub + tid;
      WideEvent ev[kWideRun];
      uint32_t where[kWideRun];
      uint32_t cnt = 0, cnt_edge = 0, labels = 0;
      uint64_t hi = 0, lo = 0;
      if (u < total_runs) {
        int lr = 0, hr = nr - 1;  // the last read whose first run is at or before u
        while (lr < hr) {
          const int mid = (lr + hr + 1) >> 1;
          if (s_run[mid] <= u)
            lr = mid;
          else
            hr = mid - 1;
        }
        const uint64_t j0 = (uint64_t)(u - s_run[lr]) * kWideRun;
        const uint64_t nv = s_off[lr + 1] - s_off[lr] - (uint64_t)k + 2;  // > j0
        cnt = (uint32_t)min((uint64_t)kWideRun, nv - j0);
        cnt_edge = (uint32_t)min((uint64_t)kWideRun, nv - 1 - j0);
        const uint64_t p = s_off[lr] - it.origin + j0;  // first base of the run
        const uint64_t q = p + (uint64_t)m;              // base of its first label
        if (staged) {
          const uint32_t bit = (uint32_t)(2 * p - 8 * b0), wi = bit >> 6;
          wide_key(s_win[wi], s_win[wi + 1], s_win[wi + 2], bit & 63u, m, hi, lo);
          const uint32_t qb = (uint32_t)(2 * q - 8 * b0), sh = qb & 63u;
          const uint64_t w = s_win[qb >> 6], x = s_win[(qb >> 6) + 1];
          labels = (uint32_t)(sh ? (w >> sh) | (x << (64u - sh)) : w);
        } else {
          const uint64_t at = p >> 2;
          wide_key(word_at(it.packed, nbytes, at), word_at(it.packed, nbytes, at + 8),
                   word_at(it.packed, nbytes, at + 16), 2u * (uint32_t)(p & 3), m, hi, lo);
          labels = (uint32_t)(word_at(it.packed, nbytes, q >> 2) >> (2 * (q & 3)));
        }
      }
#pragma unroll
      for (int j = 0; j < kWideRun; ++j) {
        const uint32_t label = (labels >> (2 * j)) & 3u;
        where[j] = ~0u;
        if ((uint32_t)j < cnt) {
          const uint32_t tag = ((uint32_t)j < cnt_edge ? 4u : 0u) | label;
          ev[j].a = ((unsigned long long)tag << 61) | (hi << 1) | (lo >> 63);
          ev[j].b = lo & kLow63;
          const uint32_t p = (uint32_t)(wide_home(hi, lo, it.n_slots) >> shift);
          where[j] = (p << 16) | atomicAdd(&hist[p], 1u);
        }
        hi = ((hi << 2) | (lo >> 62)) & mask_hi;
        lo = (lo << 2) | label;
      }
      __syncthreads();
      // prefix over the regions; every region's run takes its place in its bucket
      const int per = (parts + kWideBlock - 1) / kWideBlock;
      const int p0 = min(parts, tid * per), p1 = min(parts, p0 + per);
      uint32_t local = 0;
      for (int p = p0; p < p1; ++p) local += hist[p];
      uint32_t total;
      uint32_t run = cta_exclusive_prefix<kWideBlock>(local, s_warp, total);
      for (int p = p0; p < p1; ++p) {
        const uint32_t h = hist[p];
        off[p] = run;
        if (h) {
          const unsigned long long at = atomicAdd(&cursor[p], (unsigned long long)h);
          if (at + h > bucket_end[p]) {  // the bucket is full: the direct insert takes over
            atomicExch(use_binned, 0u);
            gbase[p] = ~0ull;
          } else {
            gbase[p] = at - run;
          }
        }
        run += h;
        hist[p] = 0u;
      }
      __syncthreads();
#pragma unroll
      for (int j = 0; j < kWideRun; ++j) {
        if (where[j] != ~0u) {
          const uint32_t p = where[j] >> 16, at = off[p] + (where[j] & 0xFFFFu);
          sorted[at] = ev[j];
          spid[at] = (uint16_t)p;
        }
      }
      __syncthreads();
      for (uint32_t j = tid; j < total; j += kWideBlock) {
        const unsigned long long g = gbase[spid[j]];
        if (g != ~0ull) out[g + j] = sorted[j];  // (a bucket ends inside the buffer)
      }
    }
    __syncthreads();
  }
}

size_t wide_split_smem(int tpr) {
  return (size_t)kWideFlush * (16 + 4) + (size_t)tpr * 24;
}

// As k_tile_scatter: every event of a unit to its tile's bucket, each chunk of
// kWideFlush events sorted by tile in shared memory.
__global__ void __launch_bounds__(kWideBlock, 2)
    k_wide_split(const WideEvent *ev, WideEvent *ev2, uint64_t ev2_cap,
                 const unsigned long long *begin, const unsigned long long *counts, TileAux aux,
                 int parts, uint64_t unit, int tpr, uint32_t *use_binned) {
  after_previous();
  if (ld_volatile_u32(use_binned) == 0u) return;
  extern __shared__ __align__(16) unsigned char smem[];
  WideEvent *s_ev = reinterpret_cast<WideEvent *>(smem);                  // kWideFlush, in tile order
  uint32_t *s_tile = reinterpret_cast<uint32_t *>(s_ev + kWideFlush);     // kWideFlush
  uint32_t *s_hist = s_tile + kWideFlush;
  uint32_t *s_off = s_hist + tpr;
  uint32_t *s_fit = s_off + tpr;
  uint32_t *s_at = s_fit + tpr;
  uint32_t *s_ovf = s_at + tpr;
  uint32_t *s_dst = s_ovf + tpr;
  __shared__ uint32_t s_warp[kWideBlock / 32];
  const int tid = threadIdx.x;
  const int per = (tpr + kWideBlock - 1) / kWideBlock;
  const int j0 = min(tpr, tid * per), j1 = min(tpr, j0 + per);
  const uint64_t over_base = aux.region_base[parts];
  const uint64_t over_cap = ev2_cap > over_base ? (ev2_cap - over_base) / 2 : 0ull;
  WideEvent *over = ev2 + over_base;  // (event, region) pairs
  TileChunk c;
  bool have = tile_chunk_first(blockIdx.x, unit_region(aux.unit_base, parts, blockIdx.x), kWideFlush,
                               begin, counts, aux, parts, unit, c);
  while (have) {
    const uint32_t cap = aux.tile_cap[c.p];
    uint32_t *fill = aux.fill + aux.region_tile0[c.p];
    WideEvent *out = ev2 + aux.region_base[c.p];
    const uint64_t ns = aux.region_nslots[c.p];
    const uint64_t first_tile = aux.region_first[c.p] >> kTileLog2;
    WideEvent e[kWideRun];
#pragma unroll
    for (int r = 0; r < kWideRun; ++r) {
      const uint64_t i = c.x + (uint64_t)r * kWideBlock + tid;
      if (i < c.y)
        e[r] = ld_event(ev + i);
      else
        e[r].b = ~0ull;
    }
    for (int j = tid; j < tpr; j += kWideBlock) s_hist[j] = 0u;
    __syncthreads();
    uint32_t where[kWideRun];
#pragma unroll
    for (int r = 0; r < kWideRun; ++r) {
      if (!e[r].none()) {
        const uint64_t home = __umul64hi(event_hash(e[r].top(), e[r].b), ns);
        const uint32_t t = (uint32_t)((home >> kTileLog2) - first_tile);
        where[r] = (t << 16) | atomicAdd(&s_hist[t], 1u);
      }
    }
    __syncthreads();
    TileChunk nx = c;
    bool have_next;
    if (c.y < c.b) {
      nx.x = c.y;
      nx.y = min(nx.x + (uint64_t)kWideFlush, c.b);
      have_next = true;
    } else {
      have_next = tile_chunk_first(c.u + gridDim.x, c.p, kWideFlush, begin, counts, aux, parts, unit,
                                   nx);
    }
    uint32_t got[kMaxBinsPerThread];
#pragma unroll
    for (int q = 0; q < kMaxBinsPerThread; ++q) {
      const int j = j0 + q;
      const uint32_t h = j < j1 ? s_hist[j] : 0u;
      got[q] = h ? atomicAdd(&fill[j], h) : 0u;
    }
    uint32_t local = 0;
    for (int j = j0; j < j1; ++j) local += s_hist[j];
    uint32_t total;
    uint32_t run = cta_exclusive_prefix<kWideBlock>(local, s_warp, total);
#pragma unroll
    for (int q = 0; q < kMaxBinsPerThread; ++q) {
      const int j = j0 + q;
      if (j >= j1) break;
      const uint32_t h = s_hist[j];
      s_off[j] = run;
      if (h) {
        const uint32_t at = got[q];
        const uint32_t fit = at >= cap ? 0u : min(h, cap - at);
        s_fit[j] = fit;
        s_at[j] = (uint32_t)((uint64_t)j * cap + at);
        s_dst[j] = fit == h ? s_at[j] - run : ~0u;
        if (fit < h) {
          const unsigned long long o = atomicAdd(aux.overflow, (unsigned long long)(h - fit));
          if (o + (h - fit) > over_cap) {  // the area is full: the direct insert takes over
            atomicExch(use_binned, 0u);
            s_ovf[j] = ~0u;
          } else {
            s_ovf[j] = (uint32_t)o;
          }
        }
      }
      run += h;
    }
    __syncthreads();
#pragma unroll
    for (int r = 0; r < kWideRun; ++r) {
      if (!e[r].none()) {
        const uint32_t t = where[r] >> 16, i = s_off[t] + (where[r] & 0xFFFFu);
        s_ev[i] = e[r];
        s_tile[i] = t;
      }
    }
    __syncthreads();
    const uint32_t n = (uint32_t)(c.y - c.x);
    for (uint32_t i = tid; i < n; i += kWideBlock) {
      const uint32_t t = s_tile[i], dst = s_dst[t];
      if (dst != ~0u) {
        out[dst + i] = s_ev[i];
        continue;
      }
      const uint32_t r = i - s_off[t], fit = s_fit[t];
      if (r < fit) {
        out[(uint64_t)s_at[t] + r] = s_ev[i];
      } else if (s_ovf[t] != ~0u) {
        WideEvent *rec = over + 2 * ((uint64_t)s_ovf[t] + (r - fit));
        rec[0] = s_ev[i];
        rec[1] = WideEvent{(unsigned long long)c.p, 0ull};
      }
    }
    __syncthreads();
    c = nx;
    have = have_next;
  }
}

constexpr size_t kWideTileBytes = (size_t)kTileSlots * (8 + 8 + 16) + kFpBytes;

// As k_tile_apply for fresh tables: every tile of the table starts as EMPTY
// slots in shared memory, takes its events and is written once.
__global__ void __launch_bounds__(kWideBlock, 3)
    k_wide_apply(ItemDesc it, const WideEvent *ev2, WideEvent *ev,
                 const unsigned long long *begin, TileAux aux, int parts, int tpr_log2,
                 const uint32_t *use_binned) {
  after_previous();
  if (ld_volatile_u32(use_binned) == 0u) return;
  extern __shared__ __align__(16) unsigned char smem[];
  unsigned long long *ka = reinterpret_cast<unsigned long long *>(smem);
  unsigned long long *kb = ka + kTileSlots;
  uint32_t *cnt = reinterpret_cast<uint32_t *>(kb + kTileSlots);  // [4][kTileSlots]
  uint8_t *fp = reinterpret_cast<uint8_t *>(cnt + 4 * kTileSlots);
  uint32_t *fp32 = reinterpret_cast<uint32_t *>(fp);
  __shared__ uint32_t s_stop;
  const int tid = threadIdx.x;
  for (int i = tid; i < kTileSlots; i += kWideBlock) ka[i] = kb[i] = kEmpty;
  for (int i = tid; i < 4 * kTileSlots; i += kWideBlock) cnt[i] = 0u;
  for (int i = tid; i < kFpBytes / 4; i += kWideBlock) fp32[i] = 0u;
  __syncthreads();
  uint32_t claimed = 0;
  const uint64_t n_tiles = aux.region_tile0[parts], n_slots = it.n_slots;
  for (uint64_t t = blockIdx.x; t < n_tiles; t += gridDim.x) {
    const int p = (int)(t >> tpr_log2);
    const uint64_t j = t - aux.region_tile0[p];
    const uint32_t cap = aux.tile_cap[p];
    const uint64_t a = aux.region_base[p] + j * cap;
    const uint32_t n = min(aux.fill[t], cap);
    const uint64_t first = aux.region_first[p] + (j << kTileLog2);
    const int len = (int)min((uint64_t)kTileSlots, n_slots - first);
    if (n == 0) {
      for (int sl = tid; sl < len; sl += kWideBlock)
        st_sector(it.table + first + sl, ~0u, ~0u, 0u, 0u, 0u, 0u, 0u, 0u);
      continue;  // (shared memory untouched: still the EMPTY tile)
    }
    if (tid == 0) s_stop = ld_volatile_u32(it.status);
    __syncthreads();  // s_stop; the tile's EMPTY words (the previous copy-out re-made them)
    if (s_stop == 0u) {
      for (uint32_t base = 0; base < n; base += kWideBlock * kWideRun) {
        WideEvent e[kWideRun];
#pragma unroll
        for (int r = 0; r < kWideRun; ++r) {
          const uint32_t i = base + (uint32_t)(r * kWideBlock + tid);
          if (i < n)
            e[r] = ld_event(ev2 + a + i);
          else
            e[r].b = ~0ull;
        }
#pragma unroll
        for (int r = 0; r < kWideRun; ++r) {
          if (e[r].none()) continue;
          const unsigned long long ea = e[r].top(), eb = e[r].b;
          const uint64_t h = event_hash(ea, eb);
          const uint32_t f = slot_fp(h ^ (h >> 32)), f4 = f * 0x01010101u;
          int q = (int)(__umul64hi(h, n_slots) - first);
          const bool capped = it.max_probes <= (uint32_t)(len - q);
          const int limit = capped ? q + (int)it.max_probes : len;
          bool done = false;
          while (q < limit) {
            const uint32_t w = __funnelshift_r(fp32[q >> 2], fp32[(q >> 2) + 1], 8 * (q & 3));
            uint32_t cand = candidate_bytes(w, f4);
            if (limit - q < 4) cand &= (1u << (8 * (limit - q))) - 1u;
            if (cand == 0u) {
              q += 4;
              continue;
            }
            const int sl = q + (__ffs((int)cand) >> 3) - 1;
            unsigned long long prev = atomicCAS(&ka[sl], kEmpty, ea);
            if (prev == kEmpty || prev == ea) {
              prev = atomicCAS(&kb[sl], kEmpty, eb);
              if (prev == kEmpty) fp[sl] = (uint8_t)f;
              if (prev == kEmpty || prev == eb) {
                const uint32_t tag = e[r].tag();
                if (tag & 4u) atomicAdd(&cnt[(tag & 3u) * kTileSlots + sl], 1u);
                done = true;
                break;
              }
            }
            q = sl + 1;
          }
          if (done) continue;
          if (capped)  // max_probes slots inside the tile: as the direct insert
            set_sticky(it.status, DBG_ERR_CAPACITY);
          else
            ev[begin[p] + atomicAdd(&aux.deferred_n[p], 1ull)] = e[r];  // left the tile: later
        }
      }
    }
    __syncthreads();
    for (int sl = tid; sl < len; sl += kWideBlock) {
      const unsigned long long wa = ka[sl], wb = kb[sl];
      const unsigned long long hi = wa == kEmpty ? kEmpty : wide_hi(wa);
      const unsigned long long lo = wa == kEmpty ? 0ull : wide_lo(wa, wb);
      uint32_t *c = cnt + sl;
      st_sector(it.table + first + sl, (uint32_t)hi, (uint32_t)(hi >> 32), (uint32_t)lo,
                (uint32_t)(lo >> 32), c[0], c[kTileSlots], c[2 * kTileSlots], c[3 * kTileSlots]);
      ka[sl] = kb[sl] = kEmpty;
      c[0] = c[kTileSlots] = c[2 * kTileSlots] = c[3 * kTileSlots] = 0u;
    }
    for (int i = tid; i < kFpBytes / 4; i += kWideBlock) {
      const uint32_t w = fp32[i];  // four fingerprints: non-zero for a key
      claimed += (uint32_t)__popc((((w & 0x7F7F7F7Fu) + 0x7F7F7F7Fu) | w) & 0x80808080u);
      fp32[i] = 0u;
    }
    // (the next tile's barrier orders these writes before its events)
  }
  claimed = __reduce_add_sync(kFull, claimed);
  if ((tid & 31) == 0 && claimed)
    atomicAdd(small_built(it.status), (unsigned long long)claimed);
}

// As k_tile_deferred: the events that left their tile, then the overflow area,
// from their home slots.
__global__ void k_wide_deferred(const __grid_constant__ ItemPack<1> pk, const WideEvent *ev,
                                const WideEvent *ev2, const unsigned long long *begin,
                                TileAux aux, int parts, const uint32_t *use_binned) {
  after_previous();
  if (ld_volatile_u32(use_binned) == 0u) {
    hand_over(pk);
    return;
  }
  const ItemDesc &it = pk.d[0];
  WideSlot *table = reinterpret_cast<WideSlot *>(it.table);
  uint32_t claimed = 0;
  auto apply = [&](const WideEvent &e) {
    uint64_t s;
    bool fresh = false;
    const unsigned long long a = e.top();
    if (wide_find_or_claim(table, it.n_slots, it.max_probes, wide_hi(a), wide_lo(a, e.b), s, &fresh)) {
      if (e.tag() & 4u) red_add_u32(&table[s].cnt[e.tag() & 3u], 1u);
    } else {
      set_sticky(it.status, DBG_ERR_CAPACITY);
    }
    claimed += fresh ? 1u : 0u;
  };
  ListShare(parts).each_list([&](int p, uint64_t i, uint64_t step) {
    const uint64_t n = aux.deferred_n[p];
    if (n && i == 0) atomicAdd(aux.deferred, (unsigned long long)n);
    for (; i < n; i += step) apply(ev[begin[p] + i]);
  });
  const uint64_t no = *aux.overflow;  // (all of it written: the flag is still set)
  const WideEvent *over = ev2 + aux.region_base[parts];
  const uint64_t stride = (uint64_t)gridDim.x * blockDim.x;
  for (uint64_t i = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; i < no; i += stride)
    apply(over[2 * i]);
  claimed = __reduce_add_sync(kFull, claimed);
  if ((threadIdx.x & 31) == 0 && claimed)
    atomicAdd(small_built(it.status), (unsigned long long)claimed);
}

// What dbg_binned_counters tells, kept by the graph: the next graph's call
// overwrites the scratch's.
__global__ void k_wide_told(uint32_t *status, const uint32_t *use_binned, TileAux aux) {
  after_previous();
  if (threadIdx.x != 0) return;
  const bool binned = ld_volatile_u32(use_binned) != 0u;
  *small_word(status, kSmallOverflow) = binned ? *aux.overflow : 0ull;
  *small_word(status, kSmallDeferred) = binned ? *aux.deferred + 1ull : 0ull;
}

int wide_shift(dbg_handle h) {
  const int log2 = h->tuning.region_log2 > 0 ? h->tuning.region_log2
                                             : tiled_shift(h->n_slots, kTableRegions);
  return bin_geometry(h->n_slots, std::max(log2, kTileLog2)).shift;
}

// The units of 8 bytes that a graph's rebuild has room for: two an event.
uint64_t wide_units_wanted(dbg_handle h) {
  return 2 * (h->bin_want ? h->bin_want
                          : std::max(kBinMinEvents, kBinWideEventsPerSlot * h->n_slots));
}

// The scratch of the wide rebuilds, one a device, shared by its graphs: at about
// 100 bytes a slot by default it is three times the table, too much for every
// graph to keep.  The calls that use it follow one another on the GPU.  No
// captured call uses it (a replay would find it replaced or given back).
struct WideScratch {
  std::mutex mu;
  BinScratch sc;
};
WideScratch g_wide[kMaxDevices];
thread_local bool t_in_wide = false;  // (this thread holds a WideScratch's lock)

uint64_t scratch_bytes_of(const BinScratch &sc) {
  return sc.aux_bytes + (sc.meta ? kBinMetaBytes : 0) + (sc.ev ? sc.cap * sizeof(uint64_t) : 0) +
         (sc.ev2 ? ev2_capacity(sc.cap) * sizeof(uint64_t) : 0);
}

// Room for `want` 8-byte units, taken when there is not: no more than a quarter of the
// device's memory, and half of what is free beside the scratch's own.
bool ensure_wide(BinScratch &sc, uint64_t want, int parts, uint64_t tiles) {
  if (sc.cap < want) {
    size_t free_bytes = 0, all = 0;
    const uint64_t need = (want + ev2_capacity(want)) * sizeof(uint64_t) + kBinMetaBytes;
    if (cudaMemGetInfo(&free_bytes, &all) != cudaSuccess || need > all / 4 ||
        need > (free_bytes + scratch_bytes_of(sc)) / 2) {
      cudaGetLastError();
      return false;
    }
  }
  if ((sc.cap >= want || ensure_events(sc, want) == DBG_OK) &&
      ensure_tile_scratch(sc, parts, tiles, false))
    return true;
  cudaGetLastError();
  if (cudaDeviceSynchronize() == cudaSuccess) free_bin_scratch(sc);
  return false;
}

int wide_chain(dbg_handle h, const ItemDesc &it, BinScratch &sc, uint64_t want, int shift, int parts,
               uint64_t tiles, cudaStream_t s, int call) {
  const int tpr = 1 << (shift - kTileLog2), sms = std::max(1, h->sm_count);
  const bool overlap = tiles <= kOverlapTiles;
  const uint64_t cap = want / 2, cap2 = ev2_capacity(want) / 2;  // events
  const Marks mark{h, call};
  const MetaView mv = meta_view(sc);
  const TileAux aux = tile_aux(sc, parts, tiles);
  WideEvent *ev = reinterpret_cast<WideEvent *>(sc.ev);
  WideEvent *ev2 = reinterpret_cast<WideEvent *>(sc.ev2);
  ItemPack<1> pk{};
  pk.n_items = 1;
  pk.d[0] = it;
  pk.d[0].region0 = 0;
  DBG_CK(cudaMemsetAsync(mv.ctr, 0, kBinClearedBytes, s));
  mark(1, s);
  const int gx = (int)std::max<uint64_t>((uint64_t)sms * 4,
                                         std::min<uint64_t>(16384, (it.n_reads + 8191) / 8192));
  DBG_TRY(launch_next(overlap, k_bin_totals<1>, dim3(gx, 1), 256, 0, s, pk, mv.totals, mv.edges, 1,
                      aux.fill, tiles));
  DBG_TRY(launch_next(overlap, k_bin_buckets<1>, 1, 1024, 0, s, pk, mv.totals, mv.edges, 1, shift,
                      parts, mv.begin, mv.cursor, cap, mv.ctr, mv.flag, aux));
  DBG_CK(cudaGetLastError());
  mark(3, s);
  {
    const size_t smem = wide_scatter_smem(parts);
    DBG_CK(cudaFuncSetAttribute(k_wide_scatter, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
    int per_sm = 0;
    DBG_CK(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_wide_scatter, kWideBlock, smem));
    const uint64_t walk = (it.n_reads + kWideTile - 1) / kWideTile;
    DBG_TRY(launch_next(overlap, k_wide_scatter, (int)std::min<uint64_t>(walk, (uint64_t)std::max(1,
                        per_sm) * sms), kWideBlock, smem, s, pk.d[0], shift, parts, mv.cursor,
                        mv.begin + 1, ev, mv.flag));
    DBG_CK(cudaGetLastError());
  }
  mark(4, s);
  const uint64_t unit = tile_unit(tpr);
  DBG_TRY(launch_next(overlap, k_tile_units, 1, 1024, 0, s, mv.counts, mv.begin, mv.cursor, parts,
                      unit, cap2, aux, mv.flag));
  {
    const size_t smem = wide_split_smem(tpr);
    DBG_CK(cudaFuncSetAttribute(k_wide_split, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
    int per_sm = 0;
    DBG_CK(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_wide_split, kWideBlock, smem));
    DBG_TRY(launch_next(overlap, k_wide_split, std::max(1, per_sm) * sms, kWideBlock, smem, s, ev,
                        ev2, cap2, mv.begin, mv.counts, aux, parts, unit, tpr, mv.flag));
    DBG_CK(cudaGetLastError());
  }
  mark(5, s);
  {
    DBG_CK(cudaFuncSetAttribute(k_wide_apply, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                (int)kWideTileBytes));
    int per_sm = 0;
    DBG_CK(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_wide_apply, kWideBlock,
                                                         kWideTileBytes));
    DBG_TRY(launch_next(overlap, k_wide_apply, (int)std::min<uint64_t>(tiles, (uint64_t)std::max(1,
                        per_sm) * sms), kWideBlock, kWideTileBytes, s, pk.d[0], ev2, ev, mv.begin,
                        aux, parts, shift - kTileLog2, mv.flag));
    DBG_CK(cudaGetLastError());
  }
  mark(6, s);
  DBG_TRY(launch_next(overlap, k_wide_deferred, sms * 8, 256, 0, s, pk, ev, ev2, mv.begin, aux,
                      parts, mv.flag));
  DBG_CK(cudaGetLastError());
  // the direct insert runs only if the events did not fit (then nothing has
  // touched the table: the last kernel has emptied it)
  mark(7, s);
  DBG_TRY(launch_insert_wide(it, h->sm_count, s, mv.flag));
  mark(8, s);
  return launch_next(overlap, k_wide_told, 1, 32, 0, s, it.status, mv.flag, aux);
}

}  // namespace

int launch_binned_wide(dbg_handle h, const ItemDesc &it, cudaStream_t s, int call, bool *done) {
  *done = false;
  const int shift = wide_shift(h), parts = regions_of(h->n_slots, shift);
  const uint64_t want = wide_units_wanted(h), tiles = table_tiles(h->n_slots, shift);
  cudaStreamCaptureStatus capture = cudaStreamCaptureStatusNone;
  DBG_CK(cudaStreamIsCapturing(s, &capture));
  if (capture != cudaStreamCaptureStatusNone ||
      (1 << (shift - kTileLog2)) > kMaxBinsPerThread * kWideBlock ||
      want / 2 >= kMaxChainEvents ||  // (bucket positions are 32-bit)
      h->device >= kMaxDevices)
    return DBG_OK;
  WideScratch &w = g_wide[h->device];
  std::lock_guard<std::mutex> lock(w.mu);
  t_in_wide = true;
  int st = DBG_OK;
  if (ensure_wide(w.sc, want, parts, tiles)) {
    *done = true;
    cudaError_t e = cudaStreamWaitEvent(s, w.sc.done, 0);
    if (e == cudaSuccess) st = wide_chain(h, it, w.sc, want, shift, parts, tiles, s, call);
    if (e == cudaSuccess) e = cudaEventRecord(w.sc.done, s);  // (after an error, too)
    if (st == DBG_OK && e != cudaSuccess) st = cuda_fail(e, "wide scratch");
    h->built_counts = st == DBG_OK;  // (unless it fell back: see small_counted)
  }
  t_in_wide = false;
  return st;
}

uint64_t wide_scratch_bytes(int dev) {
  if (dev < 0 || dev >= kMaxDevices) return 0;
  std::lock_guard<std::mutex> lock(g_wide[dev].mu);
  return scratch_bytes_of(g_wide[dev].sc);
}

uint64_t release_wide_scratch(int dev) {
  if (dev < 0 || dev >= kMaxDevices || t_in_wide) return 0;
  std::lock_guard<std::mutex> lock(g_wide[dev].mu);
  BinScratch &sc = g_wide[dev].sc;
  const uint64_t held = scratch_bytes_of(sc);
  if (held == 0 || cudaDeviceSynchronize() != cudaSuccess) return 0;
  free_bin_scratch(sc);
  return held;
}
