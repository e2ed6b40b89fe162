// Downstream of the build: normalization (Section "Normalization of graph")
// and contigs (Section "Finding contigs", Alg. 5 findContigs with makePath),
// as passes over the resident table.
//
// Normalization replaces every counter c by floor(c / divisor + 0.5) in IEEE
// double (round to nearest, halves up), capped at 2^32 - 1: the counters stay
// integers, an error k-mer seen once falls to 0 and a genomic k-mer seen
// about `divisor` times stays 1.
//
// Contigs.  An outgoing edge of a vertex is a label with a nonzero counter.
// The first flag of the paper (no edge points to the vertex) is recomputed
// from the counters as they are.  A vertex starts contigs when its first flag
// is set or it has not exactly one outgoing edge, one contig per outgoing
// edge; a contig follows edges while the vertex it reaches has exactly one
// outgoing edge, and stops on reaching a vertex it has already visited
// (keeping the edge into it).  Contigs are listed by (start key, label): the
// start edges are emitted in any order and radix-sorted.
//
// One pass over the table finds every edge's target once: the target is
// marked in a bit per slot, and a vertex with one outgoing edge keeps its
// successor's slot in the slot's padding, so that a step of a walk is one
// 32-byte load.  A second pass over the bits emits the start edges.
//
// A walk is a chain of dependent loads (about half a microsecond each), so a
// long contig is cut at splitters: one in kSpacing of the single-exit vertices,
// chosen by the key's hash.  Every splitter walks to the next one, all in
// parallel, noting the labels; rounds of pointer doubling give jumps over up to
// 2^levels segments; a contig walks to its first splitter and jumps on from
// there, listing a unit of 2^levels segments per jump; and a lane per segment
// of a unit writes its bases.  A contig that meets a cycle (or a
// stretch of kMaxWalk steps without a splitter, which only a short cycle is)
// is walked by one thread instead: Brent's cycle detection (R. P. Brent, "An
// improved Monte Carlo factorization algorithm", BIT 20, 1980) finds the
// first repeated vertex with O(1) state.
//
// Measured against one thread per contig walking by table lookups, with a pass
// each to clear, mark, count and emit, twice over for the size query: a 50 kb
// error-free genome (one contig) 43 -> 0.25 ms, a 5 Mbp graph of 31,000
// contigs (2.75 GB table) 16.4 -> 1.6 ms, of which k_links takes 1.05 (the
// table read once: 0.41), segments 0.15 (5 M random slots: 0.12), units 0.09.
#include <cub/device/device_radix_sort.cuh>
#include <cub/device/device_scan.cuh>

#include <math.h>

#include <algorithm>
#include <vector>

#include "dbg_internal.cuh"

namespace dbg {
namespace {

constexpr uint64_t kNotFound = ~0ull;

struct View {
  Slot *t;
  uint64_t n;
  uint32_t max_probes;
  uint64_t mask;  // 2(k-1) low bits
  uint32_t *status;
};

// The slot of an existing key (the table is quiescent), or kNotFound.
__device__ __forceinline__ uint64_t find_key(const View &v, uint64_t key) {
  uint64_t s = home_slot(key, v.n);
  for (uint32_t p = 0; p < v.max_probes; ++p) {
    const unsigned long long cur = v.t[s].key;
    if (cur == key) return s;
    if (cur == kEmpty) return kNotFound;
    if (++s == v.n) s = 0;
  }
  return kNotFound;
}

// Every counter's quotient.  Bound by one read and one write of the table.
// The double-precision division is slow here (each slot's took 8.2 ms of a
// 2.6 GB table), so the CTA divides the counts below kQuot once, into a table
// in shared memory -- the same expression, so the same integers -- and only
// larger counts are divided one by one: 0.76 ms, the table read and its taken
// slots written at about 6 TB/s.  (wide: k > 32, the counters are the slot's
// second half)
constexpr uint32_t kQuot = 1024;

__device__ __forceinline__ uint32_t quotient(uint32_t c, double divisor) {
  const double q = floor((double)c / divisor + 0.5);
  return q >= 4294967295.0 ? 0xffffffffu : (uint32_t)q;
}

__global__ void __launch_bounds__(256) k_normalize(uint4 *t, uint64_t n, double divisor, int wide,
                                                 uint32_t *counted) {
  after_previous();
  if (blockIdx.x == 0 && threadIdx.x == 0) *counted = 0u;  // (the counters change)
  __shared__ uint32_t s_quot[kQuot];
  for (uint32_t c = threadIdx.x; c < kQuot; c += blockDim.x) s_quot[c] = quotient(c, divisor);
  __syncthreads();
  auto norm = [&](uint32_t c) { return c < kQuot ? s_quot[c] : quotient(c, divisor); };
  const uint64_t stride = (uint64_t)gridDim.x * blockDim.x;
  for (uint64_t i = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += stride) {
    uint4 lo = t[2 * i];
    uint4 hi = t[2 * i + 1];
    if ((lo.x & lo.y) == 0xffffffffu) continue;  // an empty slot
    if (wide) {
      hi = make_uint4(norm(hi.x), norm(hi.y), norm(hi.z), norm(hi.w));
    } else {
      lo.z = norm(lo.z);
      lo.w = norm(lo.w);
      hi.x = norm(hi.x);
      hi.y = norm(hi.y);
      t[2 * i] = lo;
    }
    t[2 * i + 1] = hi;
  }
}

constexpr uint32_t kSpacing = 4;       // one splitter in so many single-exit vertices (a power of two)
constexpr uint32_t kLabels = 32;
constexpr uint32_t kMaxWalk = 2048;    // steps without a splitter before a walk counts as a cycle's
constexpr uint32_t kEnd = ~0u;         // a segment's successor: the walk ends there
constexpr uint32_t kCyclic = ~0u - 1;  // it went kMaxWalk steps without meeting a splitter
constexpr unsigned long long kIsSplitter = 1ull << 63;  // in a slot's link: the rest is its number

// What the passes share.  A slot's link (its 8 bytes of padding), for a
// single-exit vertex: its successor's slot, or kIsSplitter | number.
struct Links {
  uint64_t w0, nw;                    // the words of 32 slots that the bits below are of
  uint32_t *marks;                    // a bit per slot: an edge points to its vertex
  uint2 *degree;                      // per 32 slots: bits of one exit, bits of several
  ulonglong2 *split;                  // a splitter's slot (label in the two top bits), successor's
  unsigned long long *labels;         // the first kLabels labels of its segment, two bits each
  uint32_t *next, *len;               // [levels + 1][kept]: the splitter 2^l segments on, the edges
  uint32_t cap;                       // splitters there is room for (the rest are ordinary vertices)
  uint32_t kept;                      // splitters there are
  unsigned long long *n_split;        // splitters found
  int levels;                         // jumps of up to 2^levels segments
};

__device__ __forceinline__ unsigned long long *link_of(Slot *t, uint64_t s) {
  return reinterpret_cast<unsigned long long *>(&t[s].pad[0]);
}

// A slot in two 16-byte loads: key, counters, link.
struct SlotWords {
  uint4 a, b;
  __device__ __forceinline__ SlotWords(const Slot *t, uint64_t s) {
    const uint4 *p = reinterpret_cast<const uint4 *>(t + s);
    a = p[0];
    b = p[1];
  }
  __device__ __forceinline__ unsigned long long key() const {
    return (unsigned long long)a.x | ((unsigned long long)a.y << 32);
  }
  __device__ __forceinline__ unsigned long long link() const {
    return (unsigned long long)b.z | ((unsigned long long)b.w << 32);
  }
  // Bits of the labels with a nonzero counter.
  __device__ __forceinline__ uint32_t exits() const {
    return (a.z ? 1u : 0u) | (a.w ? 2u : 0u) | (b.x ? 4u : 0u) | (b.y ? 8u : 0u);
  }
};

// Every edge marks its target; every single-exit vertex gets its link; the
// out-degrees as bits.  A warp takes kLinkWords times 32 consecutive slots (once in
// a table of few CTAs).  Bound by one read of the table, then by the random target
// lookups.  (Splitters are numbered by the CTA: an atomic per warp on the one
// counter, at one splitter in 4 vertices, took 2.6 ms of a 2.75 GB table where the
// rest takes 1.05.)
template <int kLinkWords>
__global__ void __launch_bounds__(256) k_links(View v, Links k) {
  after_previous();
  __shared__ uint32_t s_picks[2];
  __shared__ unsigned long long s_at;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, warps = blockDim.x >> 5;
  const uint64_t words = (v.n + 31) >> 5, step = (uint64_t)warps * kLinkWords;
  if (threadIdx.x < 2) s_picks[threadIdx.x] = 0u;
  __syncthreads();
  int turn = 0;
  for (uint64_t w0 = blockIdx.x * step; w0 < words; w0 += gridDim.x * step, turn ^= 1) {
    uint64_t target[kLinkWords];
    unsigned ones[kLinkWords], picks[kLinkWords];
    uint32_t at[kLinkWords], label[kLinkWords];
#pragma unroll
    for (int u = 0; u < kLinkWords; ++u) {
      const uint64_t w = w0 + (uint64_t)(u * warps + warp), i = (w << 5) + lane;
      unsigned long long key = kEmpty;
      uint32_t exits = 0;
      if (i < v.n) {
        const SlotWords sl(v.t, i);
        key = sl.key();
        if (key != kEmpty) exits = sl.exits();
      }
      target[u] = 0;
      for (uint32_t rest = exits; rest; rest &= rest - 1) {
        const uint32_t b = (uint32_t)__ffs((int)rest) - 1u;
        const uint64_t s = find_key(v, ((key << 2) | (uint64_t)b) & v.mask);
        if (s == kNotFound) {
          atomicCAS(v.status, 0u, (uint32_t)DBG_ERR_CAPACITY);  // a target is missing
          continue;
        }
        target[u] = s;
        if ((s >> 5) - k.w0 < k.nw) atomicOr(&k.marks[(s >> 5) - k.w0], 1u << (s & 31));
      }
      label[u] = (uint32_t)__ffs((int)exits) - 1u;  // (of a single-exit vertex)
      const bool one = exits != 0 && (exits & (exits - 1)) == 0;
      ones[u] = __ballot_sync(0xffffffffu, one);
      const unsigned several = __ballot_sync(0xffffffffu, exits != 0 && !one);
      if (lane == 0 && w - k.w0 < k.nw) k.degree[w - k.w0] = make_uint2(ones[u], several);
      picks[u] = __ballot_sync(0xffffffffu,
                               one && ((uint32_t)key_hash(key) & (kSpacing - 1u)) == 0u);
      at[u] = 0;
      if (lane == 0 && picks[u]) at[u] = atomicAdd(&s_picks[turn], (uint32_t)__popc(picks[u]));
    }
    __syncthreads();
    if (threadIdx.x == 0) {
      s_at = s_picks[turn] ? atomicAdd(k.n_split, (unsigned long long)s_picks[turn]) : 0ull;
      s_picks[turn ^ 1] = 0u;
    }
    __syncthreads();
#pragma unroll
    for (int u = 0; u < kLinkWords; ++u) {
      const uint64_t i = ((w0 + (uint64_t)(u * warps + warp)) << 5) + lane;
      const unsigned long long n = s_at + __shfl_sync(0xffffffffu, at[u], 0) +
                                   (unsigned)__popc(picks[u] & ((1u << lane) - 1u));
      if (!(ones[u] >> lane & 1u)) continue;
      const bool split = (picks[u] >> lane & 1u) && n < k.cap;
      if (split)
        k.split[n] = make_ulonglong2(i | ((unsigned long long)label[u] << 62), target[u]);
      *link_of(v.t, i) = split ? (kIsSplitter | n) : target[u];
    }
  }
}

// Start edges, (key << 2 | label), of every vertex that is first or has not
// exactly one outgoing edge: at most `cap` of them are written, *count
// receives their number.  A thread takes 32 slots' bits; a warp reserves its
// edges with one atomic.
__global__ void __launch_bounds__(256) k_start_edges(View v, Links k, unsigned long long *out,
                                                     unsigned long long *count, uint64_t cap) {
  after_previous();
  const int lane = threadIdx.x & 31;
  const uint64_t stride = (uint64_t)gridDim.x * blockDim.x;
  for (uint64_t base = (uint64_t)blockIdx.x * blockDim.x; base < k.nw; base += stride) {
    const uint64_t at_word = base + threadIdx.x, w = k.w0 + at_word;
    uint32_t starts = 0, ones = 0, edges = 0;
    if (at_word < k.nw) {
      const uint2 deg = k.degree[at_word];
      ones = deg.x & ~k.marks[at_word];
      starts = ones | deg.y;
      edges = (uint32_t)__popc(ones);
    }
    for (uint32_t rest = starts & ~ones; rest; rest &= rest - 1)
      edges += (uint32_t)__popc(SlotWords(v.t, (w << 5) + (uint32_t)__ffs((int)rest) - 1u).exits());
    uint32_t incl = edges;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const uint32_t y = __shfl_up_sync(0xffffffffu, incl, o);
      if (lane >= o) incl += y;
    }
    const uint32_t total = __shfl_sync(0xffffffffu, incl, 31);
    unsigned long long at = 0;
    if (lane == 31 && total) at = atomicAdd(count, (unsigned long long)total);
    at = __shfl_sync(0xffffffffu, at, 31) + (incl - edges);
    for (uint32_t rest = starts; rest; rest &= rest - 1) {
      const SlotWords sl(v.t, (w << 5) + (uint32_t)__ffs((int)rest) - 1u);
      for (uint32_t e = sl.exits(); e; e &= e - 1, ++at)
        if (at < cap) out[at] = (sl.key() << 2) | (unsigned long long)(__ffs((int)e) - 1);
    }
  }
}

// Every splitter walks to the next splitter or to the end of its chain and notes
// the labels on its way, so that writing the contigs need not walk again (a 5
// Mbp graph: units 0.30 -> 0.09 ms).
__global__ void __launch_bounds__(256) k_segments(View v, Links k) {
  after_previous();
  const uint64_t stride = (uint64_t)gridDim.x * blockDim.x;
  for (uint64_t i = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; i < k.kept; i += stride) {
    const ulonglong2 from = k.split[i];
    uint64_t s = from.y;
    unsigned long long labels = from.x >> 62;
    uint32_t edges = 1, next = kCyclic;
    for (; edges <= kMaxWalk; ++edges) {
      const SlotWords sl(v.t, s);
      const uint32_t e = sl.exits();
      if (e == 0 || (e & (e - 1))) {  // a dead end or a branch
        next = kEnd;
        break;
      }
      const unsigned long long link = sl.link();
      if (link & kIsSplitter) {
        next = (uint32_t)link;
        break;
      }
      if (edges < kLabels) labels |= (unsigned long long)(__ffs((int)e) - 1) << (2 * edges);
      s = link;
    }
    k.labels[i] = labels;
    k.next[i] = next;
    k.len[i] = edges;
  }
}

// Jumps of level l + 1 from those of level l.
__global__ void __launch_bounds__(256) k_double(Links k, int l) {
  after_previous();
  const uint32_t *next = k.next + (size_t)l * k.kept, *len = k.len + (size_t)l * k.kept;
  uint32_t *next2 = k.next + (size_t)(l + 1) * k.kept, *len2 = k.len + (size_t)(l + 1) * k.kept;
  const uint64_t stride = (uint64_t)gridDim.x * blockDim.x;
  for (uint64_t i = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; i < k.kept; i += stride) {
    const uint32_t a = next[i];
    const bool on = a < kCyclic;
    next2[i] = on ? next[a] : a;
    len2[i] = len[i] + (on ? len[a] : 0u);
  }
}

// One step of a walk by one thread: the successor of slot s, or kNotFound
// when its vertex does not have exactly one outgoing edge.  *base receives
// the label taken.
__device__ __forceinline__ uint64_t step(const View &v, const Links &k, uint64_t s, uint32_t *base) {
  const SlotWords sl(v.t, s);
  const uint32_t e = sl.exits();
  if (e == 0 || (e & (e - 1))) return kNotFound;
  *base = (uint32_t)__ffs((int)e) - 1u;
  const unsigned long long link = sl.link();
  return link & kIsSplitter ? k.split[(uint32_t)link].y : link;
}

// Number of edges of the contig whose first edge leads to slot x0, by one thread.
__device__ uint64_t contig_edges(const View &v, const Links &k, uint64_t x0, uint64_t guard) {
  uint32_t b;
  // Brent: the hare walks; the tortoise jumps to the hare at powers of two
  uint64_t tortoise = x0, hare = step(v, k, x0, &b);
  if (hare == kNotFound) return 1;  // x0 is a branch or a dead end
  uint64_t taken = 1, power = 1, lam = 1;
  while (tortoise != hare) {
    if (taken > guard) {  // cannot happen: a walk repeats within n steps
      atomicCAS(v.status, 0u, (uint32_t)DBG_ERR_CAPACITY);
      return 1;
    }
    if (power == lam) {
      tortoise = hare;
      power <<= 1;
      lam = 0;
    }
    const uint64_t nx = step(v, k, hare, &b);
    if (nx == kNotFound) return 1 + taken;  // ends at the hare, `taken` steps past x0
    hare = nx;
    ++taken;
    ++lam;
  }
  // a cycle of length lam; mu = index of its first vertex along x0, x1, ...
  // (every vertex up to x_{mu+lam} has one exit: the hare passed them all)
  uint64_t a = x0, c = x0;
  for (uint64_t i = 0; i < lam && c != kNotFound; ++i) c = step(v, k, c, &b);
  uint64_t mu = 0;
  while (a != c && a != kNotFound && c != kNotFound && mu <= guard) {
    a = step(v, k, a, &b);
    c = step(v, k, c, &b);
    ++mu;
  }
  if (a != c) {
    atomicCAS(v.status, 0u, (uint32_t)DBG_ERR_CAPACITY);
    return 1;
  }
  return 1 + mu + lam;  // the walk arrives at x_mu again after mu + lam steps
}

// A stretch of up to 2^levels segments of a contig, from splitter `split`,
// `rel` edges into the contig.
struct Unit {
  uint32_t contig, split;
  unsigned long long rel;
};
constexpr uint64_t kMaxUnitContigs = 0xFFFFFFFFull;
// A contig's own thread writes its first `own` edges (all of them when it
// does not go by splitters).
struct Contig {
  unsigned long long x0;   // slot of the first edge's target (kNotFound: missing)
  unsigned long long own;  // edges it writes itself
  uint32_t by_units;       // whether its units count
};

__global__ void __launch_bounds__(256)
    k_contig_lengths(View v, Links k, const unsigned long long *starts, uint64_t n_starts, int m,
                     uint64_t guard, Contig *contigs, unsigned long long *len, Unit *units,
                     unsigned long long *n_units, uint64_t units_cap) {
  after_previous();
  const uint32_t *jump = k.next + (size_t)k.levels * k.kept;
  const uint32_t *jlen = k.len + (size_t)k.levels * k.kept;
  const uint64_t stride = (uint64_t)gridDim.x * blockDim.x;
  for (uint64_t i = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n_starts; i += stride) {
    const uint64_t x0 = find_key(v, starts[i] & v.mask);
    Contig c{x0, 1ull, 0u};
    uint64_t edges = 1;
    if (x0 == kNotFound) {
      atomicCAS(v.status, 0u, (uint32_t)DBG_ERR_CAPACITY);  // a target is missing
    } else {
      uint64_t s = x0;
      uint32_t split = kCyclic;
      for (; edges <= kMaxWalk; ++edges) {
        const SlotWords sl(v.t, s);
        const uint32_t e = sl.exits();
        if (e == 0 || (e & (e - 1))) {
          split = kEnd;
          break;
        }
        const unsigned long long link = sl.link();
        if (link & kIsSplitter) {
          split = (uint32_t)link;
          break;
        }
        s = link;
      }
      c.own = edges;
      // on by jumps; the tortoise of Brent's method meets them again in a cycle
      uint32_t tortoise = split, power = 1, lam = 0;
      while (split < kCyclic) {
        c.by_units = 1;
        const unsigned long long at = atomicAdd(n_units, 1ull);
        if (at < units_cap) units[at] = Unit{(uint32_t)i, split, edges};
        edges += jlen[split];
        split = jump[split];
        if (split == tortoise) split = kCyclic;
        if (++lam == power) {
          tortoise = split;
          power <<= 1;
          lam = 0;
        }
      }
      if (split == kCyclic) {
        edges = contig_edges(v, k, x0, guard);
        c.own = edges;
        c.by_units = 0;
      }
    }
    contigs[i] = c;
    len[i] = (unsigned long long)m + edges;
  }
  if (blockIdx.x == 0 && threadIdx.x == 0) len[n_starts] = 0;
}

// Label 0..3 as its letter: A, C, G, T are the word's bytes from the lowest up.
__device__ __forceinline__ char letter(uint32_t label) { return (char)(0x54474341u >> (8 * label)); }

// Every contig's start vertex and the edges its own thread writes.
__global__ void __launch_bounds__(256)
    k_contig_heads(View v, Links k, const unsigned long long *starts, uint64_t n_starts, int m,
                   const Contig *contigs, const unsigned long long *off, char *out) {
  after_previous();
  const uint64_t stride = (uint64_t)gridDim.x * blockDim.x;
  for (uint64_t i = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n_starts; i += stride) {
    const unsigned long long e = starts[i];
    const unsigned long long key = e >> 2;
    const Contig c = contigs[i];
    char *o = out + off[i];
    for (int j = 0; j < m; ++j) o[j] = letter((uint32_t)(key >> (2 * (m - 1 - j))) & 3u);
    o[m] = letter((uint32_t)e & 3u);
    uint64_t s = c.x0;
    for (uint64_t j = 1; j < c.own && s != kNotFound; ++j) {
      uint32_t b = 0;
      s = step(v, k, s, &b);
      o[m + j] = letter(b);
    }
  }
}

// A lane per segment of a unit: the j-th is found by jumps of the bits of j, and
// its bases are written.
__global__ void __launch_bounds__(256)
    k_contig_units(View v, Links k, const Unit *units, uint64_t n_units, int m,
                   const Contig *contigs, const unsigned long long *off, char *out) {
  after_previous();
  const uint64_t stride = (uint64_t)gridDim.x * blockDim.x;
  for (uint64_t g = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; g >> k.levels < n_units;
       g += stride) {
    const uint32_t j0 = (uint32_t)g & ((1u << k.levels) - 1u);
    const Unit un = units[g >> k.levels];
    if (!contigs[un.contig].by_units) continue;  // a cycle: written by the contig's own thread
    uint32_t i = un.split;
    unsigned long long rel = un.rel;
    for (int l = k.levels - 1; l >= 0; --l) {  // (longest first: lanes past the end leave at once)
      if (((j0 >> l) & 1u) && i < kCyclic) {
        rel += k.len[(size_t)l * k.kept + i];
        i = k.next[(size_t)l * k.kept + i];
      }
    }
    if (i >= kCyclic) continue;
    char *o = out + off[un.contig] + m + rel;
    const uint32_t edges = k.len[i];
    if (edges <= kLabels) {
      unsigned long long labels = k.labels[i];
      for (uint32_t j = 0; j < edges; ++j, labels >>= 2) o[j] = letter((uint32_t)labels & 3u);
      continue;
    }
    uint64_t s = k.split[i].x & (~0ull >> 2);
    for (uint32_t j = 0; j < edges; ++j) {
      const SlotWords sl(v.t, s);
      o[j] = letter((uint32_t)__ffs((int)sl.exits()) - 1u);
      s = j == 0 ? k.split[i].y : sl.link();  // (no splitter inside a segment)
    }
  }
}

struct Guard {
  int prev = -1;
  bool changed = false;
  cudaError_t err = cudaSuccess;
  explicit Guard(int dev) {
    err = cudaGetDevice(&prev);
    if (err == cudaSuccess && prev != dev) {
      err = cudaSetDevice(dev);
      changed = err == cudaSuccess;
    }
  }
  ~Guard() {
    if (changed) cudaSetDevice(prev);
  }
};

// The passes that walk -- segments, lengths, heads, units -- take as long as
// their longest chain of half-microsecond steps: about kSpacing * ln(splitters)
// for a segment, and a jump per kSpacing * 2^levels edges of the longest contig.
// Splitters are dense, then, as far as there is room (a splitter takes 24 bytes
// and 8 a level): for every one of a table of up to 2^20 slots, for one in 32
// single-exit vertices of a full larger table, which a graph cleaned of its error
// k-mers seldom reaches.  One in 4 against one in 32: a 50 kb genome 500 -> 360 us
// with its build, the 31,000 contigs of a 5 Mbp one 2.1 -> 1.8 ms.
uint64_t room_splitters(uint64_t n_slots) {
  const uint64_t n = std::max(std::min<uint64_t>(n_slots / kSpacing, 1u << 18), n_slots / 32);
  return std::min<uint64_t>(n + n / 12 + 1024, 1ull << 30);
}
constexpr int kMaxLevels = 10;
int room_levels(uint64_t n_slots) { return n_slots <= 1ull << 23 ? kMaxLevels : 5; }
// Levels: jumps over 1024 edges at least, and over a contig's average number of
// segments, as far as `room` numbers are enough for the arrays.
int levels_of(uint64_t n_split, uint64_t contigs, uint64_t room) {
  int levels = 8;
  static_assert((kSpacing << 8) == 1024, "jumps over 1024 edges");
  while (levels < kMaxLevels && (n_split / contigs) >> levels) ++levels;
  return (int)std::min<uint64_t>(levels, room / n_split - 1);
}

size_t align256(size_t x) { return (x + 255) & ~size_t(255); }

// Temporary device memory of one call, given back to the pool in stream order
// when the call leaves.
struct Scratch {
  cudaStream_t s;
  std::vector<void *> held;
  int get(void **p, size_t bytes) {
    const int st = scratch_alloc(p, bytes, s);
    if (st == DBG_OK) held.push_back(*p);
    return st;
  }
  ~Scratch() {
    for (void *p : held) cudaFreeAsync(p, s);
  }
};

int read_status(dbg_handle h, cudaStream_t s) {
  const DeviceWord status{h->d_status, 4};
  uint64_t got = 0;
  DBG_TRY(read_words(&status, 1, &got, s));
  return (int)got;
}

}  // namespace
}  // namespace dbg

extern "C" int dbg_normalize(dbg_handle h, double divisor, void *stream) {
  using namespace dbg;
  if (!h || !(divisor > 0.0) || !isfinite(divisor)) return DBG_ERR_INVALID_ARG;
  h->built_counts = false;  // the counters change
  Guard g(h->device);
  if (g.err != cudaSuccess) return cuda_fail(g.err, "cudaSetDevice");
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  const int st = dbg_get_status(h, stream);  // complete graphs only
  if (st != DBG_OK) return st;
  const uint64_t want = (h->n_slots + 255) / 256;
  const int grid = (int)std::min<uint64_t>(want, (uint64_t)std::max(1, h->sm_count) * 8);
  DBG_TRY(launch_after(k_normalize, grid, 256, 0, s, reinterpret_cast<uint4 *>(h->table),
                       h->n_slots, divisor, h->k > 32 ? 1 : 0, small_counted(h->d_status)));
  DBG_CK(cudaGetLastError());
  return DBG_OK;
}

namespace dbg {
namespace {

// The contigs of a complete graph.  frugal: with memory for the contigs and a few
// bits a slot only -- no splitters (every contig is walked by its own thread), the
// start edges counted before they are listed, and, when a bit of each kind per
// slot is not to be had, bits for a part of the table and a pass for every part.
int find_contigs(dbg_handle h, char *bases_out, uint64_t max_bases, uint64_t *offsets_out,
                 uint64_t max_contigs, uint64_t *n_contigs, uint64_t *n_bases, cudaStream_t s,
                 bool frugal) {
  const int m = h->k - 1;
  const View v{h->table, h->n_slots, h->max_probes,
               m >= 32 ? ~0ull : ((1ull << (2 * m)) - 1ull), h->d_status};
  const int grid = std::max(1, h->sm_count) * 8;
  Scratch scr{s};
  // marks, degrees and splitters by the table's size
  const uint64_t words = (h->n_slots + 31) >> 5;
  const uint64_t cap = frugal ? 0 : room_splitters(h->n_slots);
  uint64_t nw = words;
  const uint64_t rounds = (uint64_t)room_levels(h->n_slots) + 1;
  auto bits_bytes = [](uint64_t w) { return 256 + align256(w * 4) + align256(w * 8); };
  auto split_bytes = [rounds](uint64_t c) {
    return align256(c * sizeof(ulonglong2)) + 2 * align256(c * 4 * rounds) + align256(c * 8);
  };
  char *buf = nullptr;
  for (;; nw = (nw + 1) / 2) {
    const int st = scr.get(reinterpret_cast<void **>(&buf), bits_bytes(nw) + split_bytes(cap));
    if (st == DBG_OK) break;
    if (st != DBG_ERR_OOM || !frugal || nw <= 1024) return st;
    cudaGetLastError();
  }
  unsigned long long *counts = reinterpret_cast<unsigned long long *>(buf);  // [3], see below
  const size_t mark_bytes = align256(nw * 4);
  Links k{};
  k.marks = reinterpret_cast<uint32_t *>(buf + 256);
  k.degree = reinterpret_cast<uint2 *>(buf + 256 + mark_bytes);
  k.split = reinterpret_cast<ulonglong2 *>(buf + bits_bytes(nw));
  k.next = reinterpret_cast<uint32_t *>(buf + bits_bytes(nw) + align256(cap * sizeof(ulonglong2)));
  k.len = reinterpret_cast<uint32_t *>(reinterpret_cast<char *>(k.next) +
                                       align256(cap * 4 * rounds));
  k.labels = reinterpret_cast<unsigned long long *>(
      reinterpret_cast<char *>(k.len) + align256(cap * 4 * rounds));
  k.cap = (uint32_t)cap;
  k.n_split = counts + 1;

  // the start edges into a buffer that holds as many as an ordinary graph has; a
  // second pass when there are more
  uint64_t starts_cap = frugal ? 0 : h->n_slots / 16 + 1024;
  unsigned long long *starts_a = nullptr;
  uint64_t got[4] = {0, 0, 0, 0};  // start edges, splitters, units, status
  for (bool linked = false;;) {
    if (starts_cap > 0)
      DBG_TRY(scr.get(reinterpret_cast<void **>(&starts_a), starts_cap * sizeof(unsigned long long)));
    // (the start edges of the parts add up; the splitters are numbered anew in each)
    const size_t kept = nw < words || linked ? sizeof(unsigned long long) : 0;
    if (kept) DBG_CK(cudaMemsetAsync(counts, 0, kept, s));
    for (k.w0 = 0; k.w0 < words; k.w0 += nw) {
      k.nw = std::min(nw, words - k.w0);
      if (!linked || nw < words) {
        DBG_CK(cudaMemsetAsync(buf + kept, 0, 256 - kept + mark_bytes, s));  // counts, marks
        if (h->n_slots <= 1u << 20)
          DBG_TRY(launch_after(k_links<1>, (int)std::min<uint64_t>((words + 7) / 8, (uint64_t)grid),
                               256, 0, s, v, k));
        else
          DBG_TRY(launch_after(k_links<2>, (int)std::min<uint64_t>((words + 15) / 16,
                               (uint64_t)grid), 256, 0, s, v, k));
      }
      DBG_TRY(launch_after(k_start_edges, (int)std::min<uint64_t>((k.nw + 255) / 256,
                           (uint64_t)grid), 256, 0, s, v, k, starts_a, counts, starts_cap));
    }
    DBG_CK(cudaGetLastError());
    const DeviceWord read[] = {{counts, 8}, {counts + 1, 8}, {counts + 2, 8}, {h->d_status, 4}};
    DBG_TRY(read_words(read, 4, got, s));
    if (got[3] != DBG_OK) return (int)got[3];
    if (got[0] <= starts_cap) break;
    starts_cap = got[0];
    linked = true;
  }
  const uint64_t S = got[0];
  const uint32_t n_split = (uint32_t)std::min<uint64_t>(got[1], cap);
  *n_contigs = S;
  *n_bases = 0;
  if (S == 0) {
    if (offsets_out)
      DBG_CK(cudaMemcpyAsync(offsets_out, n_bases, sizeof(uint64_t), cudaMemcpyDefault, s));
    DBG_CK(cudaStreamSynchronize(s));
    return DBG_OK;
  }
  // (contig numbers in a unit are 32-bit; the frugal form has no units)
  if (S > kMaxUnitContigs && !frugal) return DBG_ERR_OOM;

  k.kept = n_split;
  if (n_split > 0) {
    k.levels = levels_of(n_split, S, cap * rounds);
    const int sg = (int)std::min<uint64_t>(((uint64_t)n_split + 255) / 256, (uint64_t)grid);
    DBG_TRY(launch_after(k_segments, sg, 256, 0, s, v, k));
    for (int l = 0; l < k.levels; ++l)
      DBG_TRY(launch_after(k_double, sg, 256, 0, s, k, l));
    DBG_CK(cudaGetLastError());
  }
  size_t sort_bytes = 0, scan_bytes = 0;
  DBG_CK(cub::DeviceRadixSort::SortKeys(nullptr, sort_bytes, (unsigned long long *)nullptr,
                                        (unsigned long long *)nullptr, (int64_t)S, 0, 2 * m + 2,
                                        s));
  DBG_CK(cub::DeviceScan::ExclusiveSum(nullptr, scan_bytes, (unsigned long long *)nullptr,
                                       (unsigned long long *)nullptr, (int64_t)(S + 1), s));
  const size_t eb = align256((S + 1) * sizeof(unsigned long long));
  const size_t cb = align256(S * sizeof(Contig));
  char *buf2 = nullptr;
  DBG_TRY(scr.get(reinterpret_cast<void **>(&buf2),
                  3 * eb + cb + align256(std::max(sort_bytes, scan_bytes))));
  unsigned long long *starts_b = reinterpret_cast<unsigned long long *>(buf2);
  unsigned long long *len = reinterpret_cast<unsigned long long *>(buf2 + eb);
  unsigned long long *off = reinterpret_cast<unsigned long long *>(buf2 + 2 * eb);
  Contig *contigs = reinterpret_cast<Contig *>(buf2 + 3 * eb);
  void *temp = buf2 + 3 * eb + cb;
  DBG_CK(cub::DeviceRadixSort::SortKeys(temp, sort_bytes, starts_a, starts_b, (int64_t)S, 0,
                                        2 * m + 2, s));
  // a unit per jump: one or two a contig, and one in every 2^levels splitters
  // (again with as many as were counted when contigs share long tails)
  const uint64_t guard = 4 * h->n_slots + 64;
  const int cg = (int)std::min<uint64_t>((S + 255) / 256, (uint64_t)grid);
  uint64_t units_cap = n_split > 0 ? 2 * S + (n_split >> (k.levels - 1)) + 1024 : 0;
  Unit *units = nullptr;
  unsigned long long B = 0;
  for (;;) {
    if (units_cap > 0)
      DBG_TRY(scr.get(reinterpret_cast<void **>(&units), units_cap * sizeof(Unit)));
    DBG_TRY(launch_after(k_contig_lengths, cg, 256, 0, s, v, k, starts_b, S, m, guard, contigs, len,
                         units, counts + 2, units_cap));
    DBG_CK(cudaGetLastError());
    DBG_CK(cub::DeviceScan::ExclusiveSum(temp, scan_bytes, len, off, (int64_t)(S + 1), s));
    const DeviceWord words[] = {{counts + 2, 8}, {h->d_status, 4}, {off + S, 8}};
    uint64_t now[3];
    DBG_TRY(read_words(words, 3, now, s));
    got[2] = now[0];
    *n_bases = B = now[2];
    if (now[1] != DBG_OK) return (int)now[1];
    if (got[2] <= units_cap) break;
    units_cap = got[2];
    DBG_CK(cudaMemsetAsync(counts + 2, 0, sizeof(unsigned long long), s));
  }
  if (!bases_out || !offsets_out || S > max_contigs || B > max_bases) return DBG_ERR_BUFFER_TOO_SMALL;
  char *chars = nullptr;
  DBG_TRY(scr.get(reinterpret_cast<void **>(&chars), std::max<uint64_t>(B, 1)));
  DBG_TRY(launch_after(k_contig_heads, cg, 256, 0, s, v, k, starts_b, S, m, contigs, off, chars));
  DBG_CK(cudaGetLastError());
  if (got[2] > 0) {
    DBG_TRY(launch_after(k_contig_units, (int)std::min<uint64_t>(((got[2] << k.levels) + 255) / 256,
                         (uint64_t)grid), 256, 0, s, v, k, units, got[2], m, contigs, off, chars));
    DBG_CK(cudaGetLastError());
  }
  DBG_CK(cudaMemcpyAsync(offsets_out, off, (S + 1) * sizeof(uint64_t), cudaMemcpyDefault, s));
  DBG_CK(cudaMemcpyAsync(bases_out, chars, B, cudaMemcpyDefault, s));
  return read_status(h, s);
}

}  // namespace
}  // namespace dbg

extern "C" int dbg_find_contigs(dbg_handle h, char *bases_out, uint64_t max_bases,
                                uint64_t *offsets_out, uint64_t max_contigs, uint64_t *n_contigs,
                                uint64_t *n_bases, void *stream) {
  using namespace dbg;
  if (!h || !n_contigs || !n_bases || h->k > 32) return DBG_ERR_INVALID_ARG;
  Guard g(h->device);
  if (g.err != cudaSuccess) return cuda_fail(g.err, "cudaSetDevice");
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  DBG_TRY(dbg_get_status(h, stream));  // complete graphs only
  const int st = find_contigs(h, bases_out, max_bases, offsets_out, max_contigs, n_contigs, n_bases,
                              s, false);
  if (st != DBG_ERR_OOM) return st;
  cudaGetLastError();
  DBG_CK(cudaStreamSynchronize(s));  // (what the first attempt took is free again)
  trim_scratch_pool(h->device);
  return find_contigs(h, bases_out, max_bases, offsets_out, max_contigs, n_contigs, n_bases, s, true);
}
