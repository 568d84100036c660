// Device building blocks of one wavefront level, shared by the single-graph
// and the batched expansion kernels.
//
// Level i -> i+1 of Listing 1 (arXiv 1709.09990, Section 3.1): every set S of
// L_i is extended by every vertex v outside S with |Q(S, v)| <= k, and the
// extensions are deduplicated (Section 3.2) in an exact hash table.
#pragma once

#include <cstdint>

#include "tw_internal.h"
#include "tw_keys.cuh"

namespace tw {
namespace core {

constexpr unsigned kFull = 0xffffffffu;
// Resident warps per SM the register allocation must allow: 40 for the 32-bit
// kernel (on a geometric n=25 graph 1.67 ms of expand time against 1.77 with
// 32), 32 for the 64-bit one (with 40 it is 0.5% to 2% slower), 16 for the
// 128-bit one.
template <class K>
struct ResidentWarps {
  static constexpr int value = KeyTraits<K>::kBits <= 32 ? 40 : KeyTraits<K>::kBits <= 64 ? 32 : 16;
};

// Home slot of a hash: the high word of hash * slots (uniform over [0, slots)
// for any table size, so the table can be sized to the level).
__device__ __forceinline__ unsigned long long home_slot(unsigned long long h, unsigned long long slots) {
  return __umul64hi(h, slots);
}

// The component of G[S] that holds min(S) and its outer boundary N(comp) \ S
// (both empty for S = {}), by a bitset flood fill over the adjacency rows in
// shared memory.
template <class K>
__host__ __device__ __forceinline__ void min_component(const K S, const AdjRow<K>* __restrict__ sAdj, K& comp, K& bnd) {
  comp = kzero<K>();
  K q = kzero<K>();
  K front = klsb(S);
  while (!kempty(front)) {
    K ub = kzero<K>();
    const AdjRow<K> a = sAdj[pick(front, ub)];
    q |= a.row;
    comp |= bit_of(a, ub);
    front = (front | a.row) & S & ~comp;
  }
  bnd = q & ~S;
}

// The candidates v of state S (thread per state) that pass the cheap test: a
// lower bound of |Q(S, v)| from v's own row and, when v borders the component
// comp0 of min(S), that component's boundary b0, is at most k.
//
// With kCanonical only the canonical extensions are candidates: the v that lie
// in the component of G[S u {v}] holding the lowest vertex of S u {v}, i.e.
// v below min(S) or v in b0.  The level sets stay exactly those of Listing 1:
// Q(S, v) depends only on v's component of G[S u {v}] (a path from v whose
// interior lies in S never leaves it), so a set is feasible iff each of its
// components is, and a feasible set T is reached from T \ {u} with u the last
// vertex of a feasible ordering of T's lowest-vertex component.  Each new set
// is then produced by far fewer parents (on the geometric n=40 benchmark graph
// 3.3x fewer pairs).
//
// Candidates that border no other component of G[S] (two of three on the
// geometric n=40 graph) are settled by the test (done); the others still need
// the search (search).
template <class K>
struct Candidates {
  K done, search;
};
template <class K, bool kCanonical>
__host__ __device__ __forceinline__ Candidates<K> cheap_candidates(const K S, const K comp0, const K b0,
                                                          const AdjRow<K>* __restrict__ sAdj, const K valid, const K allowed,
                                                          const int k) {
  K cand = valid & allowed & ~S;
  if (kCanonical) cand &= kbelow_lowest(S) | b0;
  Candidates<K> c{kzero<K>(), kzero<K>()};
  while (!kempty(cand)) {
    K vb = kzero<K>();
    const AdjRow<K> a = sAdj[pick(cand, vb)];
    vb = bit_of(a, vb);
    const K nv = a.row;
    cand ^= vb;
    K t = nv, visit = nv & S;
    int most = k;
    if (kCanonical && !kempty(b0 & vb)) {
      t |= b0;
      visit &= ~comp0;
      most = k + 1;  // (b0 holds v itself)
    }
    if (kpopc(t & ~S) <= most) {
      if (kempty(visit))
        c.done |= vb;
      else
        c.search |= vb;
    }
  }
  return c;
}

// Is |Q(S, v)| <= k?  The search of Listing 1 as a bitset flood fill: it starts
// from N(v) and, when v borders the component of min(S) (v in b0), from that
// whole component at once (comp0, boundary b0), visits the vertices of S
// reachable from v and gathers their rows; it stops as soon as the vertices
// gathered outside S u {v} exceed k.
//
// vb is v's bit, nv its row.
template <class K>
__host__ __device__ __forceinline__ bool extension_feasible(const K S, const K comp0, const K b0, const K vb, const K nv,
                                                   const AdjRow<K>* __restrict__ sAdj, const int k) {
  const K out = ~(S | vb);
  K q = nv;
  K done = ~S;  // vertices that need no visit: those outside S and those visited
  if (!kempty(b0 & vb)) {
    done |= comp0;
    q |= b0;
  }
  K front = q & ~done;
  bool within;
  // (one way out of the loop, so that the warp's lanes meet again after it)
  while ((within = kpopc(q & out) <= k) && !kempty(front)) {
    K ub = kzero<K>();
    const AdjRow<K> a = sAdj[pick(front, ub)];
    q |= a.row;
    done |= bit_of(a, ub);
    front = (front | a.row) & ~done;
  }
  return within;
}

// Warp-wide minimum of (d, v), lowest v on ties; v < 0 means none.
__device__ __forceinline__ void warp_min_pair(int& d, int& v) {
#pragma unroll
  for (int off = 16; off > 0; off >>= 1) {
    const int od = __shfl_xor_sync(kFull, d, off);
    const int ov = __shfl_xor_sync(kFull, v, off);
    if (ov >= 0 && (v < 0 || od < d || (od == d && ov < v))) {
      d = od;
      v = ov;
    }
  }
}

// Does the minor-min-width bound of the graph H left after eliminating S
// exceed k (Section 3.3, with the second-smallest degree of each minor as the
// bound, which is also a treewidth lower bound)?  Warp-cooperative: every
// lane passes the same S; lane l owns the vertices l, l+32, ... and their rows
// of H (row of v = Q(S, v), found by a flood fill through S).  While H has
// more than k+1 vertices: take a minimum-degree vertex v (lowest index),
// record the second-smallest degree, delete v if isolated, else contract it
// into its minimum-degree neighbour (lowest index).  With at most k+1
// vertices left no degree can exceed k, so the answer is settled.
template <class K>
__device__ __forceinline__ bool mmw_exceeds(const K S, const AdjRow<K>* __restrict__ sAdj, const int n, const int k,
                                            const int lane) {
  constexpr int NV = KeyTraits<K>::kBits / 32;  // vertices per lane
  constexpr int kNone = 1 << 30;
  K alive = kfirst_n<K>(n) & ~S;
  K row[NV];
#pragma unroll
  for (int t = 0; t < NV; ++t) {
    const int v = lane + 32 * t;
    row[t] = kzero<K>();
    if (v < n && ktest(alive, v)) {
      const K nv = sAdj[v].row;
      K q = nv & ~S;
      K vis = nv & S;
      K front = vis;
      while (!kempty(front)) {
        K ub = kzero<K>();
        const AdjRow<K> a = sAdj[pick(front, ub)];
        front ^= bit_of(a, ub);
        const K r = a.row;
        q |= r & ~S;
        const K nw = r & S & ~vis;
        vis |= nw;
        front |= nw;
      }
      row[t] = q & ~kbit<K>(v);
    }
  }
  int count = kpopc(alive);
  int lb = 0;
  while (count > k + 1) {
    int deg[NV];
    int dmin = kNone, vmin = -1;
#pragma unroll
    for (int t = 0; t < NV; ++t) {
      const int v = lane + 32 * t;
      deg[t] = (v < n && ktest(alive, v)) ? kpopc(row[t] & alive) : kNone;
      if (deg[t] < dmin) {
        dmin = deg[t];
        vmin = v;
      }
    }
    warp_min_pair(dmin, vmin);
    int d2 = kNone, v2 = -1;
#pragma unroll
    for (int t = 0; t < NV; ++t) {
      const int v = lane + 32 * t;
      if (v != vmin && deg[t] < d2) {
        d2 = deg[t];
        v2 = v;
      }
    }
    warp_min_pair(d2, v2);
    lb = max(lb, d2);
    if (lb > k) return true;
    const K bv = kbit<K>(vmin);
    alive &= ~bv;
    --count;
    if (dmin == 0) continue;
    K mine = kzero<K>();
#pragma unroll
    for (int t = 0; t < NV; ++t)
      if (t == (vmin >> 5)) mine = row[t];
    const K rv = kshfl(mine, vmin & 31) & alive;
    int du = kNone, u = -1;
#pragma unroll
    for (int t = 0; t < NV; ++t) {
      const int v = lane + 32 * t;
      if (v < n && ktest(rv, v) && deg[t] < du) {
        du = deg[t];
        u = v;
      }
    }
    warp_min_pair(du, u);
#pragma unroll
    for (int t = 0; t < NV; ++t) {
      const int v = lane + 32 * t;
      if (v == u)
        row[t] |= rv & ~kbit<K>(u);
      else if (v < n && ktest(rv, v))
        row[t] |= kbit<K>(u);
    }
  }
  return false;
}

// Has this lane's state, if it is one of the extendable ones, a remaining graph
// with a minor-min-width bound above k?  (The warp examines its states one by
// one.)
template <class K>
__device__ __forceinline__ bool mmw_prunes(const K S, const bool extendable, const AdjRow<K>* __restrict__ sAdj, const int n,
                                           const int k, const int lane) {
  unsigned pending = __ballot_sync(kFull, extendable);
  bool mine = false;
  while (pending) {
    const int j = __ffs(pending) - 1;
    pending &= pending - 1;
    const bool prune = mmw_exceeds<K>(kshfl(S, j), sAdj, n, k, lane);
    if (prune && lane == j) mine = true;
  }
  return mine;
}

// One warp's scratch in shared memory: the 32 states of its chunk, the
// component of each state's lowest vertex with its boundary, the queue of
// (state, vertex) pairs (up to kTake of each state at a time), and the new sets
// that wait for a place in the output list.
constexpr int kTake = 16;
constexpr int kStage = 256;
template <class K>
struct WarpScratch {
  K state[32], comp[32], bnd[32];
  K stage_key[kStage];
  uint32_t stage_from[kStage];  // added vertex, or the parent's index (kParent)
  uint16_t queue[32 * kTake];
};

// Takes a vertex out of a non-empty set: by its row's bit for 64-bit sets (2%
// faster there), as the lowest one for the others.
template <class K>
__device__ __forceinline__ int take_vertex(K& set, const AdjRow<K>*) {
  const K b = klsb(set);
  set ^= b;
  return kindex(b);
}
template <>
__device__ __forceinline__ int take_vertex<unsigned long long>(unsigned long long& set,
                                                               const AdjRow<unsigned long long>* sAdj) {
  const int v = khighest(set);
  set ^= sAdj[v].bit;
  return v;
}

// Packs up to kTake (S, v) pairs of each of the warp's 32 states into the
// warp's queue (entry = lane << 8 | v) and takes them out of c; returns the
// number of pairs (warp uniform).  The pairs that need no search come first, so
// that the searches run in as few rounds of the warp as they fill (a round
// takes as long as its longest search).
template <class K>
__device__ __forceinline__ int build_queue(Candidates<K>& c, const int lane, const AdjRow<K>* __restrict__ sAdj,
                                           WarpScratch<K>& w) {
  const int n0 = min(kpopc(c.done), kTake);
  const int n1 = min(kpopc(c.search), kTake - n0);
  const int cnt = n0 | (n1 << 16);
  int incl = cnt;
#pragma unroll
  for (int d = 1; d < 32; d <<= 1) {
    const int t = __shfl_up_sync(kFull, incl, d);
    if (lane >= d) incl += t;
  }
  const int total = __shfl_sync(kFull, incl, 31);
  const int excl = incl - cnt;
  int pos = excl & 0xffff;
  for (int end = pos + n0; pos < end; ++pos) {
    const int v = take_vertex(c.done, sAdj);
    w.queue[pos] = (uint16_t)((lane << 8) | v);
  }
  pos = (total & 0xffff) + (excl >> 16);
  for (int end = pos + n1; pos < end; ++pos) {
    const int v = take_vertex(c.search, sAdj);
    w.queue[pos] = (uint16_t)((lane << 8) | v);
  }
  __syncwarp();
  return (total & 0xffff) + (total >> 16);
}
template <class K>
__device__ __forceinline__ bool any_left(const Candidates<K>& c) {
  return !kempty(c.done | c.search);
}

// The search's first half for one chunk: the component of min(S) and the cheap
// test; returns the surviving candidates of this lane's state.  Inactive lanes
// pass active = false.
template <class K, bool kCanonical, bool kMMW = false>
__device__ __forceinline__ Candidates<K> start_chunk(const K S, const bool active, const AdjRow<K>* __restrict__ sAdj,
                                                     const K valid, const K allowed, const int n, const int k,
                                                     const int lane, WarpScratch<K>& w) {
  K comp0 = kzero<K>(), b0 = kzero<K>();
  Candidates<K> c{kzero<K>(), kzero<K>()};
  if (active) {
    if (kCanonical) min_component<K>(S, sAdj, comp0, b0);
    c = cheap_candidates<K, kCanonical>(S, comp0, b0, sAdj, valid, allowed, k);
  }
  if (kMMW && mmw_prunes<K>(S, any_left(c), sAdj, n, k, lane)) c = Candidates<K>{kzero<K>(), kzero<K>()};
  w.state[lane] = S;
  w.comp[lane] = comp0;
  w.bnd[lane] = b0;
  return c;
}

// Tests the queued pairs (pair per lane) and packs the feasible ones to the
// front of the queue; returns their number (warp uniform).
template <class K>
__device__ __forceinline__ int keep_feasible(WarpScratch<K>& w, const int total, const int lane,
                                             const AdjRow<K>* __restrict__ sAdj, const int k) {
  int kept = 0;
  for (int base = 0; base < total; base += 32) {
    const int j = base + lane;
    uint16_t e = 0;
    bool ok = false;
    if (j < total) {
      e = w.queue[j];
      const AdjRow<K> av = sAdj[e & 0xff];
      ok = extension_feasible<K>(w.state[e >> 8], w.comp[e >> 8], w.bnd[e >> 8], own_bit(av, e & 0xff), av.row, sAdj,
                                 k);
    }
    const unsigned m = __ballot_sync(kFull, ok);  // (every lane has read its entry)
    if (ok) w.queue[kept + __popc(m & ((1u << lane) - 1u))] = e;
    kept += __popc(m);
    __syncwarp();
  }
  return kept;
}

// Where the winners of the inserts go.  With kParent the output records the
// index (parent_base + lane) of the parent state in its level; otherwise the
// added vertex.
// KO is the type of the list's keys (wider than the search's in the batched
// kernel, whose lists hold 64-bit keys).
template <class K, bool kParent, class KO = K>
struct LevelOut {
  KO* keys;
  uint8_t* pred;       // used when !kParent
  uint32_t* parent;    // used when kParent
  uint32_t parent_base;
  unsigned long long cap;
  unsigned long long* count;
  unsigned int* overflow;  // bit 0: output full, bit 1: probe limit
};

// Writes the warp's staged new sets to the output list from position b on.  With
// kRanged no predecessor is stored and output positions from split on go to
// tail[position - split] when tail is given (a list continued in a second
// buffer).
template <class K, bool kParent, bool kRanged, class KO = K>
__device__ __forceinline__ void store_stage(const WarpScratch<K>& w, const int staged, const unsigned long long b,
                                            const int lane, const LevelOut<K, kParent, KO>& out, K* tail,
                                            const unsigned long long split) {
  for (int j = lane; j < staged; j += 32) {
    const unsigned long long o = b + (unsigned long long)j;
    if (o < out.cap) {
      if (kRanged && tail != nullptr && o >= split)
        kstore_cs(&tail[o - split], w.stage_key[j]);
      else
        kstore_cs(&out.keys[o], (KO)w.stage_key[j]);
      if (kParent)
        __stcs(&out.parent[o], w.stage_from[j]);
      else if (!kRanged)
        __stcs(reinterpret_cast<signed char*>(&out.pred[o]), (signed char)w.stage_from[j]);
    } else {
      atomicOr(out.overflow, 1u);
    }
  }
}

// Moves the warp's staged new sets to the output list: one atomic add for all of
// them.  (Every add of a level goes to the same counter, which takes about one
// in 2.6 ns; with one add per 64 pairs that was the whole time of a level, with
// one per 200 new sets it no longer shows.)
template <class K, bool kParent, bool kRanged, class KO = K>
__device__ __forceinline__ void flush_stage(WarpScratch<K>& w, int& staged, const int lane,
                                            const LevelOut<K, kParent, KO>& out, K* tail, const unsigned long long split) {
  if (staged == 0) return;
  __syncwarp();
  unsigned long long b = 0;
  if (lane == 0) b = atomicAdd(out.count, (unsigned long long)staged);
  b = __shfl_sync(kFull, b, 0);
  store_stage<K, kParent, kRanged, KO>(w, staged, b, lane, out, tail, split);
  staged = 0;
  __syncwarp();
}

// Slot of the sector in which key may be put: the first of its slots from `from`
// on that may be empty, kSlotPresent when key comes before that, kSlotNone when
// every slot holds another key.
constexpr int kSlotPresent = -1, kSlotNone = -2;
template <class K>
__device__ __forceinline__ int find_slot(const Sector<K>& s, const K key, const int from) {
  int pos = kSlotNone;
#pragma unroll
  for (int i = Sector<K>::kSlots - 1; i >= 0; --i) {
    if (i < from) break;
    if (s.x[i] == key)
      pos = kSlotPresent;
    else if (kmaybe_empty(s.x[i]))
      pos = i;
  }
  return pos;
}

// Inserts key into the table from the first slot of sector b on; true when this
// thread put it in, false when it was there or the probe limit was reached
// (*overflow then gets bit 1).
//
// The table is probed in 32-byte sectors (4, 8 or 2 slots for 64-, 32- and
// 128-bit keys): a key's home is the first slot of a sector, and probing goes on
// slot by slot.  One load of the whole sector shows whether the key is there
// (two of three pairs on the geometric n=40 graph) or where the first empty slot
// is, so a pair costs one load and a new set one compare-and-swap more; only
// full sectors and lost races take further round trips.  (Probing slot by slot
// with compare-and-swaps took 16 of them per chunk of 32 states, most for a few
// lanes and one after the other.)  Keys fill a sector from its front: a thread
// tries a slot only after it saw the earlier ones hold other keys, so two
// threads with the same key meet at the same slot.
template <class K>
__device__ __forceinline__ bool insert_key(K* __restrict__ table, const unsigned int sectors, const int max_sectors,
                                           unsigned int b, const K key, unsigned int* overflow) {
  constexpr int B = Sector<K>::kSlots;
  const K empty = kones<K>();
  K* at = table + (size_t)b * B;
  Sector<K> s;
  kload_sector(at, s);
  int pos = find_slot<K>(s, key, 0);
  if (pos == kSlotPresent) return false;
  if (pos >= 0) {
    const K o = kcas(at + pos, empty, key);
    if (o == empty) return true;
    if (o == key) return false;
  }
  // a full sector or a lost race (apart from the first probe: one loop for both
  // made the kernel 6 to 23% slower)
  int from = pos >= 0 ? pos + 1 : B;
  for (int looked = 1;;) {
    if (from >= B) {
      if (++looked > max_sectors) {
        atomicOr(overflow, 2u);
        return false;
      }
      b = b + 1u == sectors ? 0u : b + 1u;
      at = table + (size_t)b * B;
      from = 0;
    }
    kload_sector(at, s);
    pos = find_slot<K>(s, key, from);
    if (pos == kSlotPresent) return false;
    if (pos == kSlotNone) {
      from = B;
      continue;
    }
    const K o = kcas(at + pos, empty, key);
    if (o == empty) return true;
    if (o == key) return false;
    from = pos + 1;
  }
}

// Tests the queued pairs (pair per lane) and inserts the feasible ones into the
// table; returns this lane's count of feasible pairs.
//
// One pair per lane at a time: with two in flight the kernel is 4% slower on the
// geometric n=40 graph (9.40 against 9.05 ms of expand time), with three 9%
// (more registers and code against latency that the other warps hide).
// Winners are staged in shared memory (staged of them wait) and flushed when
// the next round might not fit.
//
// With kRanged only the pairs whose new set hashes into range `range` of
// `ranges` equal ranges of the hash space are inserted (all feasible ones are
// pairs of one of the ranges); the table is the slice of that range (the home
// spreads the range's hashes over the slice: the high word of (hash * ranges
// mod 2^64) * sectors).
template <class K, bool kParent, bool kRanged = false, class KO = K>
__device__ __forceinline__ int search_insert(WarpScratch<K>& w, const int total, int& staged, const int lane,
                                             const AdjRow<K>* __restrict__ sAdj, const int k, K* __restrict__ table,
                                             const unsigned long long slots, const int max_probes,
                                             const LevelOut<K, kParent, KO>& out, const unsigned long long ranges = 1,
                                             const unsigned long long range = 0, K* tail = nullptr,
                                             const unsigned long long split = 0) {
  constexpr int B = Sector<K>::kSlots;
  // (the 2^32 - 1 sectors that an index holds are 128 GB)
  const unsigned int sectors = (unsigned int)min(slots / B, 0xffffffffull);
  const int max_sectors = (max_probes + B - 1) / B;
  int generated = 0;
  for (int base = 0; base < total; base += 32) {
    const bool have = base + lane < total;
    const int e = have ? w.queue[base + lane] : 0;
    const K S = w.state[e >> 8];
    const AdjRow<K> av = sAdj[e & 0xff];
    const K vb = own_bit(av, e & 0xff);
    const K key = S | vb;
    bool ok = have && extension_feasible<K>(S, w.comp[e >> 8], w.bnd[e >> 8], vb, av.row, sAdj, k);
    unsigned int home;
    if (kRanged) {
      const unsigned long long hash = khash(key);
      ok = ok && __umul64hi(hash, ranges) == range;
      home = (unsigned int)home_slot(hash * ranges, sectors);
    } else {
      home = __umulhi(khash32(key), sectors);
    }
    generated += ok ? 1 : 0;
    // the lanes whose searches took longer are waited for here, so that the warp
    // probes the table together
    __syncwarp();
    const bool won = ok && insert_key<K>(table, sectors, max_sectors, home, key, out.overflow);
    __syncwarp();
    if (staged > kStage - 32) flush_stage<K, kParent, kRanged, KO>(w, staged, lane, out, tail, split);
    const unsigned wm = __ballot_sync(kFull, won);
    if (won) {
      const int o = staged + __popc(wm & ((1u << lane) - 1u));
      w.stage_key[o] = key;
      w.stage_from[o] = kParent ? out.parent_base + (uint32_t)(e >> 8) : (uint32_t)(e & 0xff);
    }
    staged += __popc(wm);
  }
  return generated;
}

// A key from two 64-bit words (low word first).
template <class K> __host__ __device__ __forceinline__ K kfrom_words(unsigned long long lo, unsigned long long hi);
template <> __host__ __device__ __forceinline__ uint32_t kfrom_words<uint32_t>(unsigned long long lo,
                                                                                unsigned long long) {
  return (uint32_t)lo;
}
template <> __host__ __device__ __forceinline__ unsigned long long kfrom_words<unsigned long long>(
    unsigned long long lo, unsigned long long) {
  return lo;
}
template <> __host__ __device__ __forceinline__ K128 kfrom_words<K128>(unsigned long long lo, unsigned long long hi) {
  return K128{lo, hi};
}

// Parameters of one level expansion.
template <class K>
struct ExpandParams {
  const K* in_keys;
  unsigned long long n_in;
  const K* adj;
  int n;
  int k;
  K* table;
  unsigned long long table_slots;
  int max_probes;
  K* out_keys;
  uint8_t* out_pred;        // predecessor vertex of each new set, or (kParent)
  uint32_t* out_parent;     // the index of its parent in the input level
  unsigned long long out_cap;
  LevelCounters* ctr;
  K allowed;  // vertices that may be added (all by default)
  int mmw;    // 1: minor-min-width pruning of the states before they are extended
  unsigned long long ranges;  // ranged kernels: the hash space is split in this many ranges,
  unsigned long long range;   // and only pairs of this one are inserted (the table is its slice)
};

// C(n, r), or cap when it is at least cap.  The products run over
// min(r, n - r) steps, along which b = C(n - r + j, j) only grows and each
// division is exact, so with cap <= 2^40 nothing overflows.
__host__ __device__ __forceinline__ unsigned long long binom_capped(int n, int r, unsigned long long cap) {
  if (r < 0 || r > n) return 0ull;
  if (r > n - r) r = n - r;
  unsigned long long b = 1ull;
  for (int j = 1; j <= r; ++j) {
    b = b * (unsigned long long)(n - r + j) / (unsigned long long)j;
    if (b >= cap) return cap;
  }
  return b;
}

// The table of level i -> i+1 without FP64 (slow on this part; the result is
// the same in every thread): the expected size is cnt times the last growth
// ratio cnt / prev_cnt clamped to [1/4, n - i] (n at i = 0), plus 25% and
// 1024, at most the number of sets level i+1 can have; slots = that at
// load_pct percent, at least 64.  The ratio is exact integer arithmetic below
// 2^32 sets and single precision above.  sets_max = C(n, i+1), capped at
// kSetsCap (64-bit divisions take a thread 0.1 us each: the callers compute the
// binomials once per run or graph, not level by level, which took 1 to 3 us).
constexpr unsigned long long kSetsCap = 1ull << 40;
__device__ __forceinline__ void plan_level(unsigned long long cnt, unsigned long long prev_cnt, int n, int i,
                                           int load_pct, unsigned long long sets_max, unsigned long long* table_est,
                                           unsigned long long* slots) {
  const unsigned long long most = cnt * (unsigned long long)(n - i);
  const unsigned long long bound = min(most, sets_max) + 1ull;
  unsigned long long est = (unsigned long long)n;
  if (i > 0) {
    if (prev_cnt == 0)
      est = cnt;
    else if (cnt < (1ull << 16) && prev_cnt < (1ull << 32))
      est = ((unsigned)cnt * (unsigned)cnt) / (unsigned)prev_cnt;
    else if (cnt < (1ull << 32))
      est = cnt * cnt / prev_cnt;
    else
      est = (unsigned long long)fminf((float)cnt * ((float)cnt / (float)prev_cnt), (float)most);
    est = max(est, cnt / 4ull);
    est = min(est, most);
  }
  *table_est = min(est + est / 4ull + 1024ull, bound);
  *slots = max(64ull, load_pct == 50 ? 2ull * *table_est
                                     : (*table_est * 100ull + (unsigned long long)load_pct - 1ull) /
                                           (unsigned long long)load_pct);
}

// Adds the lanes' counts and, in lane 0, adds the sum to *total.
__device__ __forceinline__ void add_warp_count(unsigned long long count, const int lane, unsigned long long* total) {
#pragma unroll
  for (int d = 16; d > 0; d >>= 1) count += __shfl_xor_sync(kFull, count, d);
  if (lane == 0 && count) atomicAdd(total, count);
}

// One level i -> i+1 by the whole block: the adjacency rows go to shared
// memory, then each warp takes chunks of 32 consecutive states (coalesced key
// loads), queues their candidate pairs (thread per state), and tests and
// inserts the pairs (pair per lane).  scratch holds one entry per warp.
//
// With kBlockLocal the block expands the whole level alone (its warps take the
// chunks in turn): a persistent kernel whose blocks work on different graphs.
// With kKeysL2 the input keys are read through L2 only: persistent kernels,
// whose arena other SMs rewrite while stale lines may sit in this SM's L1.
// With kGroup the level is expanded by a group of the grid's blocks (block
// group_block of group_blocks) instead of the whole grid, and the caller has
// put the adjacency rows in sAdj.  Ranged kernels may
// continue the output list in out_tail from position out_split on.
//
// A level of fewer than 32 states per warp is dealt out in smaller chunks, to at
// most kSpreadWarps warps (each adds to the level's counter once): a chunk takes
// as long as its rounds of 32 pairs, one after the other.
constexpr unsigned kSpreadWarps = 1024;
template <class K, int kWarps, bool kMMW = false, bool kRanged = false, bool kBlockLocal = false,
          bool kKeysL2 = false, bool kGroup = false, bool kParent = false>
__device__ __forceinline__ void expand_level(const ExpandParams<K>& p, AdjRow<K>* sAdj, WarpScratch<K>* scratch,
                                             const unsigned group_block = 0, const unsigned group_blocks = 0,
                                             K* out_tail = nullptr, const unsigned long long out_split = 0) {
  if (!kGroup) {
    fill_rows<K>(sAdj, p.adj, p.n, threadIdx.x, blockDim.x);
    __syncthreads();
  }
  const int lane = threadIdx.x & 31;
  const int warp = threadIdx.x >> 5;
  WarpScratch<K>& w = scratch[warp];
  const K valid = kfirst_n<K>(p.n);
  unsigned long long generated = 0;
  int staged = 0;
  const unsigned long long blk = kGroup ? (unsigned long long)group_block : (unsigned long long)blockIdx.x;
  const unsigned long long nblk = kGroup ? (unsigned long long)group_blocks : (unsigned long long)gridDim.x;
  const unsigned long long first = kBlockLocal ? (unsigned long long)warp : blk * kWarps + warp;
  const unsigned long long stride = kBlockLocal ? (unsigned long long)kWarps : nblk * kWarps;
  const unsigned spread = (unsigned)min(stride, (unsigned long long)kSpreadWarps);
  const unsigned per = p.n_in < 32ull * spread ? max(1u, ((unsigned)p.n_in + spread - 1u) / spread) : 32u;
  const unsigned long long n_chunks = per == 32u ? (p.n_in + 31ull) / 32ull : ((unsigned)p.n_in + per - 1u) / per;
  LevelOut<K, kParent> out;
  out.keys = p.out_keys;
  out.pred = p.out_pred;
  out.parent = p.out_parent;
  out.parent_base = 0;
  out.cap = p.out_cap;
  out.count = &p.ctr->out_count;
  out.overflow = &p.ctr->overflow;
  for (unsigned long long chunk = first; chunk < n_chunks; chunk += stride) {
    const unsigned long long idx = chunk * per + lane;
    const bool active = (unsigned)lane < per && idx < p.n_in;
    if (kParent) out.parent_base = (uint32_t)(chunk * per);
    const K S = active ? (kKeysL2 ? kload_cg(&p.in_keys[idx]) : kload_cs(&p.in_keys[idx])) : valid;
    // (minor-min-width pruning drops some parents, so it extends by every
    // feasible vertex)
    Candidates<K> c = start_chunk<K, !kMMW, kMMW>(S, active, sAdj, valid, p.allowed, p.n, p.k, lane, w);
    do {
      const int total = build_queue<K>(c, lane, sAdj, w);
      generated += (unsigned long long)search_insert<K, kParent, kRanged>(w, total, staged, lane, sAdj, p.k, p.table,
                                                                           p.table_slots, p.max_probes, out, p.ranges,
                                                                           p.range, out_tail, out_split);
      __syncwarp();
    } while (__any_sync(kFull, any_left(c)));
  }
  if (kGroup) {
    // the block's last sets and its pair count with one atomic add each: at a
    // small level the adds to the two counters, 2.6 ns each, are on the way to
    // the group's barrier
    __shared__ int sStaged[kWarps];
    __shared__ unsigned int sPairs[kWarps];
    __shared__ unsigned long long sFirst;
    const unsigned int pairs = __reduce_add_sync(kFull, (unsigned)generated);  // (a lane's pairs of a level: 32 bits)
    if (lane == 0) {
      sStaged[warp] = staged;
      sPairs[warp] = pairs;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
      unsigned int sets = 0;
      unsigned long long all = 0;
      for (int x = 0; x < kWarps; ++x) {
        sets += (unsigned)sStaged[x];
        all += sPairs[x];
      }
      if (all) atomicAdd(&p.ctr->generated, all);
      sFirst = sets ? atomicAdd(out.count, (unsigned long long)sets) : 0ull;
    }
    __syncthreads();
    unsigned long long b = sFirst;
    for (int x = 0; x < warp; ++x) b += (unsigned long long)sStaged[x];
    store_stage<K, kParent, kRanged>(w, staged, b, lane, out, out_tail, out_split);
    return;
  }
  flush_stage<K, kParent, kRanged>(w, staged, lane, out, out_tail, out_split);
  add_warp_count(generated, lane, &p.ctr->generated);
}

// The backward walk by one block: from the first set of level `last`, find
// the current set in level j (keys [level_off[j], + level_cnt[j])), take its
// predecessor vertex as order[j-1] and drop it, down to level 1; then the
// vertices outside the final set in increasing order.  sWalk, sFound: shared.
template <class K>
__device__ __forceinline__ void walk_block(const K* __restrict__ keys, const uint8_t* __restrict__ pred,
                                          const unsigned long long* level_off, const unsigned long long* level_cnt,
                                          int last, int n, int32_t* order, K* sWalk, int* sFound) {
  if (threadIdx.x == 0) *sWalk = kload_cg(&keys[__ldcg(&level_off[last])]);
  __syncthreads();
  const K fin = *sWalk;
  for (int j = last; j >= 1; --j) {
    if (threadIdx.x == 0) *sFound = 0;
    __syncthreads();
    const K target = *sWalk;
    __syncthreads();  // every thread has the target before the finder replaces it
    const unsigned long long lo = __ldcg(&level_off[j]), cnt = __ldcg(&level_cnt[j]);
    // the scan issues kWalkU loads per thread before comparing (one L2
    // round trip per kWalkU keys, not per key) and stops at the batch that
    // found the set
    constexpr int kWalkU = 8;
    for (unsigned long long x0 = 0; x0 < cnt; x0 += (unsigned long long)blockDim.x * kWalkU) {
      K key[kWalkU];
#pragma unroll
      for (int u = 0; u < kWalkU; ++u) {
        const unsigned long long x = x0 + (unsigned long long)u * blockDim.x + threadIdx.x;
        key[u] = x < cnt ? kload_cg(&keys[lo + x]) : kzero<K>();
      }
      bool hit = false;
#pragma unroll
      for (int u = 0; u < kWalkU; ++u) {
        const unsigned long long x = x0 + (unsigned long long)u * blockDim.x + threadIdx.x;
        if (x < cnt && key[u] == target) {
          hit = true;
          if (atomicExch(sFound, 1) == 0) {
            const int v = __ldcg(&pred[lo + x]);
            order[j - 1] = v;
            *sWalk = target & ~kbit<K>(v);
          }
        }
      }
      if (__syncthreads_or(hit)) break;
    }
    __syncthreads();
  }
  if (threadIdx.x == 0) {
    int pos = last;
    for (int v = 0; v < n; ++v)
      if (!ktest(fin, v)) order[pos++] = v;
  }
  __syncthreads();
}

// The backward walk by one thread through parent indices: the added vertex is
// the bit in which a set and its parent differ.  Two dependent loads per level
// (scanning a level of 10^5 sets for the predecessor took a block 50 us).
template <class K>
__device__ __forceinline__ void walk_parents(const K* __restrict__ keys, const uint32_t* __restrict__ parent,
                                             const unsigned long long* level_off, int last, int n, int32_t* order) {
  unsigned long long idx = 0;
  K S = kload_cg(&keys[__ldcg(&level_off[last])]);
  const K fin = S;
  for (int j = last; j >= 1; --j) {
    idx = __ldcg(&parent[__ldcg(&level_off[j]) + idx]);
    const K prev = kload_cg(&keys[__ldcg(&level_off[j - 1]) + idx]);
    order[j - 1] = kindex(S ^ prev);
    S = prev;
  }
  int pos = last;
  for (int v = 0; v < n; ++v)
    if (!ktest(fin, v)) order[pos++] = v;
}

// Tree decomposition from an ordering, by one block (thread per vertex):
// bag(v) = {v} u Q(prefix(v), v) and parent(v) = the vertex of Q(prefix(v), v)
// eliminated first after v (the last vertex of the order when Q is empty; the
// last vertex is the root, -1).  adj64 / bags: n rows x words64 uint64;
// sAdj, sPos: shared arrays of 128 entries.
__device__ __forceinline__ void td_block(const unsigned long long* __restrict__ adj64, int n, int words64,
                                         const int32_t* __restrict__ order, int32_t* parent,
                                         unsigned long long* bags, K128* sAdj, int* sPos) {
  for (int i = threadIdx.x; i < n; i += blockDim.x) {
    sAdj[i] = K128{adj64[(size_t)i * words64], words64 > 1 ? adj64[(size_t)i * words64 + 1] : 0ull};
    sPos[i] = n;
  }
  __syncthreads();
  for (int i = threadIdx.x; i < n; i += blockDim.x) {
    const int o = order[i];
    if (o >= 0 && o < n) sPos[o] = i;  // a malformed order never indexes out of range
  }
  __syncthreads();
  for (int v = threadIdx.x; v < n; v += blockDim.x) {
    const int pv = sPos[v];
    K128 prefix = kzero<K128>();
    for (int u = 0; u < n; ++u)
      if (sPos[u] < pv) prefix |= kbit<K128>(u);
    K128 q = sAdj[v] & ~prefix;
    K128 vis = sAdj[v] & prefix;
    K128 front = vis;
    while (!kempty(front)) {
      const int u = klowest(front);
      front = kdrop_lowest(front);
      const K128 r = sAdj[u];
      q |= r & ~prefix;
      const K128 nw = r & prefix & ~vis;
      vis |= nw;
      front |= nw;
    }
    q &= ~kbit<K128>(v);
    const K128 bag = q | kbit<K128>(v);
    bags[(size_t)v * words64] = bag.lo;
    if (words64 > 1) bags[(size_t)v * words64 + 1] = bag.hi;
    int best = -1;
    K128 t = q;
    while (!kempty(t)) {
      const int u = klowest(t);
      t = kdrop_lowest(t);
      if (best < 0 || sPos[u] < sPos[best]) best = u;
    }
    if (best < 0) best = (pv >= n - 1) ? -1 : order[n - 1];
    parent[v] = best;
  }
}

}  // namespace core
}  // namespace tw
