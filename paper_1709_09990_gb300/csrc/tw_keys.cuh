// Vertex-set bitsets used as wavefront states, for the three width classes of
// the expansion kernels: 32-bit (n <= 32), 64-bit (n <= 64) and 128-bit
// (n <= 128).  A state S is the set of eliminated vertices (arXiv 1709.09990,
// Section 3.1: the lists hold sets S of vertices with a feasible partial
// elimination ordering); bit v of the key is set iff v is in S.
#pragma once

#include <cstdint>

namespace tw {

struct K128 {
  unsigned long long lo, hi;
};

__host__ __device__ __forceinline__ K128 operator&(K128 a, K128 b) { return {a.lo & b.lo, a.hi & b.hi}; }
__host__ __device__ __forceinline__ K128 operator|(K128 a, K128 b) { return {a.lo | b.lo, a.hi | b.hi}; }
__host__ __device__ __forceinline__ K128 operator~(K128 a) { return {~a.lo, ~a.hi}; }
__host__ __device__ __forceinline__ bool operator==(K128 a, K128 b) { return a.lo == b.lo && a.hi == b.hi; }
__host__ __device__ __forceinline__ bool operator!=(K128 a, K128 b) { return !(a == b); }
__host__ __device__ __forceinline__ K128& operator|=(K128& a, K128 b) { a = a | b; return a; }
__host__ __device__ __forceinline__ K128& operator&=(K128& a, K128 b) { a = a & b; return a; }
__host__ __device__ __forceinline__ K128 operator^(K128 a, K128 b) { return {a.lo ^ b.lo, a.hi ^ b.hi}; }
__host__ __device__ __forceinline__ K128& operator^=(K128& a, K128 b) { a = a ^ b; return a; }

template <class K> struct KeyTraits;
template <> struct KeyTraits<uint32_t> { static constexpr int kBits = 32; static constexpr int kWords64 = 1; };
template <> struct KeyTraits<unsigned long long> { static constexpr int kBits = 64; static constexpr int kWords64 = 1; };
template <> struct KeyTraits<K128> { static constexpr int kBits = 128; static constexpr int kWords64 = 2; };

// ---- construction ---------------------------------------------------------
template <class K> __host__ __device__ __forceinline__ K kzero();
template <> __host__ __device__ __forceinline__ uint32_t kzero<uint32_t>() { return 0u; }
template <> __host__ __device__ __forceinline__ unsigned long long kzero<unsigned long long>() { return 0ull; }
template <> __host__ __device__ __forceinline__ K128 kzero<K128>() { return {0ull, 0ull}; }

template <class K> __host__ __device__ __forceinline__ K kones();
template <> __host__ __device__ __forceinline__ uint32_t kones<uint32_t>() { return ~0u; }
template <> __host__ __device__ __forceinline__ unsigned long long kones<unsigned long long>() { return ~0ull; }
template <> __host__ __device__ __forceinline__ K128 kones<K128>() { return {~0ull, ~0ull}; }

template <class K> __host__ __device__ __forceinline__ K kbit(int v);
template <> __host__ __device__ __forceinline__ uint32_t kbit<uint32_t>(int v) { return 1u << v; }
template <> __host__ __device__ __forceinline__ unsigned long long kbit<unsigned long long>(int v) { return 1ull << v; }
template <> __host__ __device__ __forceinline__ K128 kbit<K128>(int v) {
  return v < 64 ? K128{1ull << v, 0ull} : K128{0ull, 1ull << (v - 64)};
}

// The set {0, .., n-1}.
template <class K> __host__ __device__ __forceinline__ K kfirst_n(int n);
template <> __host__ __device__ __forceinline__ uint32_t kfirst_n<uint32_t>(int n) { return n >= 32 ? ~0u : ((1u << n) - 1u); }
template <> __host__ __device__ __forceinline__ unsigned long long kfirst_n<unsigned long long>(int n) {
  return n >= 64 ? ~0ull : ((1ull << n) - 1ull);
}
template <> __host__ __device__ __forceinline__ K128 kfirst_n<K128>(int n) {
  if (n >= 128) return {~0ull, ~0ull};
  if (n >= 64) return {~0ull, (n == 64) ? 0ull : ((1ull << (n - 64)) - 1ull)};
  return {(1ull << n) - 1ull, 0ull};
}

// ---- queries ----------------------------------------------------------------
// (What the search of a level uses also compiles for the host, where the tests
// run it.)
__host__ __device__ __forceinline__ int kpopc(uint32_t a) {
#ifdef __CUDA_ARCH__
  return __popc(a);
#else
  return __builtin_popcount(a);
#endif
}
__host__ __device__ __forceinline__ int kpopc(unsigned long long a) {
#ifdef __CUDA_ARCH__
  return __popcll(a);
#else
  return __builtin_popcountll(a);
#endif
}
__host__ __device__ __forceinline__ int kpopc(K128 a) { return kpopc(a.lo) + kpopc(a.hi); }

__host__ __device__ __forceinline__ bool kempty(uint32_t a) { return a == 0u; }
__host__ __device__ __forceinline__ bool kempty(unsigned long long a) { return a == 0ull; }
__host__ __device__ __forceinline__ bool kempty(K128 a) { return (a.lo | a.hi) == 0ull; }

// Index of the lowest set bit; the argument must be non-empty.
__device__ __forceinline__ int klowest(uint32_t a) { return __ffs(a) - 1; }
__device__ __forceinline__ int klowest(unsigned long long a) { return __ffsll(a) - 1; }
__device__ __forceinline__ int klowest(K128 a) { return a.lo ? __ffsll(a.lo) - 1 : 63 + __ffsll(a.hi); }

// a without its lowest set bit.
__device__ __forceinline__ uint32_t kdrop_lowest(uint32_t a) { return a & (a - 1u); }
__device__ __forceinline__ unsigned long long kdrop_lowest(unsigned long long a) { return a & (a - 1ull); }
__device__ __forceinline__ K128 kdrop_lowest(K128 a) {
  return a.lo ? K128{a.lo & (a.lo - 1ull), a.hi} : K128{0ull, a.hi & (a.hi - 1ull)};
}

// Lowest set bit of a as a one-bit set (a must be non-empty for an index).
__host__ __device__ __forceinline__ uint32_t klsb(uint32_t a) { return a & (0u - a); }
__host__ __device__ __forceinline__ unsigned long long klsb(unsigned long long a) { return a & (0ull - a); }
__host__ __device__ __forceinline__ K128 klsb(K128 a) {
  return a.lo ? K128{a.lo & (0ull - a.lo), 0ull} : K128{0ull, a.hi & (0ull - a.hi)};
}

// The vertices below the lowest element of a (every vertex when a is empty).
__host__ __device__ __forceinline__ uint32_t kbelow_lowest(uint32_t a) { return (a - 1u) & ~a; }
__host__ __device__ __forceinline__ unsigned long long kbelow_lowest(unsigned long long a) { return (a - 1ull) & ~a; }
__host__ __device__ __forceinline__ K128 kbelow_lowest(K128 a) {
  return a.lo ? K128{(a.lo - 1ull) & ~a.lo, 0ull} : K128{~0ull, (a.hi - 1ull) & ~a.hi};
}

// Index of the only set bit of a one-bit set.
__host__ __device__ __forceinline__ int kindex(uint32_t b) {
#ifdef __CUDA_ARCH__
  return 31 - __clz(b);
#else
  return 31 - __builtin_clz(b);
#endif
}
__host__ __device__ __forceinline__ int kindex(unsigned long long b) {
#ifdef __CUDA_ARCH__
  return 63 - __clzll(b);
#else
  return 63 - __builtin_clzll(b);
#endif
}
__host__ __device__ __forceinline__ int kindex(K128 b) { return b.lo ? kindex(b.lo) : 64 + kindex(b.hi); }

__device__ __forceinline__ bool ktest(uint32_t a, int v) { return (a >> v) & 1u; }
__device__ __forceinline__ bool ktest(unsigned long long a, int v) { return (a >> v) & 1ull; }
__device__ __forceinline__ bool ktest(K128 a, int v) { return v < 64 ? ((a.lo >> v) & 1ull) : ((a.hi >> (v - 64)) & 1ull); }

// Warp shuffle of a key from lane src.
__device__ __forceinline__ uint32_t kshfl(uint32_t a, int src) { return __shfl_sync(0xffffffffu, a, src); }
__device__ __forceinline__ unsigned long long kshfl(unsigned long long a, int src) {
  return __shfl_sync(0xffffffffu, a, src);
}
__device__ __forceinline__ K128 kshfl(K128 a, int src) {
  return K128{__shfl_sync(0xffffffffu, a.lo, src), __shfl_sync(0xffffffffu, a.hi, src)};
}

// ---- rows in shared memory -----------------------------------------------------
// Index of the highest set bit (a must be non-empty).
__host__ __device__ __forceinline__ int khighest(uint32_t a) {
#ifdef __CUDA_ARCH__
  int r;
  asm("bfind.u32 %0, %1;" : "=r"(r) : "r"(a));
  return r;
#else
  return 31 - __builtin_clz(a);
#endif
}
__host__ __device__ __forceinline__ int khighest(unsigned long long a) {
  const uint32_t hi = (uint32_t)(a >> 32);
  return khighest(hi ? hi : (uint32_t)a) + (hi ? 32 : 0);
}

// A vertex's adjacency row and its own bit side by side: one shared-memory load
// gives both, so that walking through the bits of a set needs no shifts and no
// isolated lowest bit (the ALU pipe is what bounds the expansion kernels: 7.65 ->
// 7.03 ms of expand time on the geometric n=40 graph).  For 128-bit sets, whose
// rows fill a load, the bit is made instead.
//
// pick() gives a vertex of a non-empty set; bit_of() its bit, from its row or
// from pick(); own_bit() the bit of vertex v, whose row is a.
template <class K> struct __align__(2 * sizeof(K)) AdjRow { K row, bit; };
template <> struct AdjRow<K128> { K128 row; };
template <class K> __host__ __device__ __forceinline__ int pick(const K set, K&) { return khighest(set); }
// (For 128-bit sets by selects, the lowest vertex of the word that has one: with
// a branch each for klsb and kindex a solve of G(70, 0.8) takes 1.00 ms instead
// of 0.91, one of G(128, 0.96) 0.59 instead of 0.53.)
template <> __host__ __device__ __forceinline__ int pick<K128>(const K128 set, K128& bit) {
  const bool low = set.lo != 0ull;
  const unsigned long long w = low ? set.lo : set.hi;
  const unsigned long long b = w & (0ull - w);
  bit = K128{low ? b : 0ull, low ? 0ull : b};
  return khighest(b) + (low ? 0 : 64);
}
template <class K> __host__ __device__ __forceinline__ K bit_of(const AdjRow<K>& a, const K) { return a.bit; }
template <> __host__ __device__ __forceinline__ K128 bit_of<K128>(const AdjRow<K128>&, const K128 bit) { return bit; }
template <class K> __host__ __device__ __forceinline__ K own_bit(const AdjRow<K>& a, const int) { return a.bit; }
template <> __host__ __device__ __forceinline__ K128 own_bit<K128>(const AdjRow<K128>&, const int v) { return kbit<K128>(v); }
__host__ __device__ __forceinline__ void set_row(AdjRow<uint32_t>& a, uint32_t row, int v) { a = {row, 1u << v}; }
__host__ __device__ __forceinline__ void set_row(AdjRow<unsigned long long>& a, unsigned long long row, int v) {
  a = {row, 1ull << v};
}
__host__ __device__ __forceinline__ void set_row(AdjRow<K128>& a, K128 row, int) { a.row = row; }

// Fills the rows of a search from the n rows at adj, this thread every step-th
// from first on.  Every row that a bit of a set can name is written, those of
// n and above as vertices without edges: the search loops take a visited vertex
// out of their set with the bit that stands beside its row, so a row that holds
// no bit would keep a set with a bit at or above n (tw_expand_level_static takes
// its sets unchecked) in the loop for ever.
template <class K>
__host__ __device__ __forceinline__ void fill_rows(AdjRow<K>* rows, const K* adj, int n, int first, int step) {
  for (int v = first; v < KeyTraits<K>::kBits; v += step) set_row(rows[v], v < n ? adj[v] : kzero<K>(), v);
}

// ---- hashing ----------------------------------------------------------------
// 64-bit finaliser of MurmurHash3 (Appleby); the paper also hashes states with
// Murmur3 (Section 3.2).
__host__ __device__ __forceinline__ unsigned long long fmix64(unsigned long long x) {
  x ^= x >> 33;
  x *= 0xff51afd7ed558ccdull;
  x ^= x >> 33;
  x *= 0xc4ceb9fe1a85ec53ull;
  x ^= x >> 33;
  return x;
}
__device__ __forceinline__ unsigned long long khash(uint32_t a) { return fmix64((unsigned long long)a); }
__device__ __forceinline__ unsigned long long khash(unsigned long long a) { return fmix64(a); }
__device__ __forceinline__ unsigned long long khash(K128 a) { return fmix64(a.lo ^ fmix64(a.hi ^ 0x9e3779b97f4a7c15ull)); }

// A 32-bit hash for the home of a key in the table of one level: the words of the
// key times odd constants, folded and mixed twice by multiply and xor-shift (a
// third of the instructions of khash; its value is no result, it only spreads
// the keys).
__device__ __forceinline__ unsigned int mix32(unsigned int x) {
  x ^= x >> 16;
  x *= 0x9e3779b1u;
  x ^= x >> 15;
  x *= 0xbb67ae85u;
  return x ^ (x >> 13);
}
__device__ __forceinline__ unsigned int khash32(uint32_t a) { return mix32(a * 0x3c6ef373u); }
__device__ __forceinline__ unsigned int khash32(unsigned long long a) {
  const unsigned long long m = (unsigned long long)(unsigned int)a * 0x6a09e667f3bcc909ull +
                               (unsigned long long)(unsigned int)(a >> 32) * 0xbb67ae8584caa73bull;
  return mix32((unsigned int)m ^ (unsigned int)(m >> 32));
}
__device__ __forceinline__ unsigned int khash32(K128 a) {
  return mix32(khash32(a.lo) + 0x510e527fu * khash32(a.hi ^ 0x3c6ef372fe94f82bull));
}

// Level fingerprint fp(S) = mix(w0 ^ mix(w1)) with mix the splitmix64 output
// function (Steele, Lea & Flood 2014).  Order independent once summed.
__device__ __forceinline__ unsigned long long splitmix_out(unsigned long long z) {
  z = (z ^ (z >> 30)) * 0xbf58476d1ce4e5b9ull;
  z = (z ^ (z >> 27)) * 0x94d049bb133111ebull;
  return z ^ (z >> 31);
}
__device__ __forceinline__ unsigned long long kfingerprint(uint32_t a) { return splitmix_out((unsigned long long)a ^ splitmix_out(0ull)); }
__device__ __forceinline__ unsigned long long kfingerprint(unsigned long long a) { return splitmix_out(a ^ splitmix_out(0ull)); }
__device__ __forceinline__ unsigned long long kfingerprint(K128 a) { return splitmix_out(a.lo ^ splitmix_out(a.hi)); }

// ---- atomics ----------------------------------------------------------------
__device__ __forceinline__ uint32_t kcas(uint32_t* p, uint32_t cmp, uint32_t val) {
  return atomicCAS(reinterpret_cast<unsigned int*>(p), cmp, val);
}
__device__ __forceinline__ unsigned long long kcas(unsigned long long* p, unsigned long long cmp,
                                                   unsigned long long val) {
  return atomicCAS(p, cmp, val);
}
// 16-byte compare-and-swap (PTX atom.cas.b128, sm_90 and later); p must be
// 16-byte aligned.
__device__ __forceinline__ K128 kcas(K128* p, K128 cmp, K128 val) {
  K128 old;
  asm volatile(
      "{\n\t.reg .b128 c, v, o;\n\t"
      "mov.b128 c, {%2, %3};\n\t"
      "mov.b128 v, {%4, %5};\n\t"
      "atom.global.cas.b128 o, [%6], c, v;\n\t"
      "mov.b128 {%0, %1}, o;\n\t}"
      : "=l"(old.lo), "=l"(old.hi)
      : "l"(cmp.lo), "l"(cmp.hi), "l"(val.lo), "l"(val.hi), "l"(p)
      : "memory");
  return old;
}

// One 32-byte sector of a hash table (32-byte aligned), read with one access that
// goes to the L2 (other SMs write the table during a level).  Words are read whole;
// the two halves of a 128-bit key may be of different times.  Such a torn key, one
// half of the set being written and one half still all ones, never equals a set
// that is looked for, because all sets of one table have the same number of
// vertices: equal to it, a set would have 64 of them in the half that reads as all
// ones, and as many as the set being written only if that one has all 64 there too
// and is the same set.  A table that held sets of several levels could not be probed
// this way.
template <class K> struct Sector { static constexpr int kSlots = 32 / (int)sizeof(K); K x[kSlots]; };
__device__ __forceinline__ void kload_sector(const uint32_t* p, Sector<uint32_t>& s) {
  asm volatile("ld.relaxed.gpu.global.v8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
               : "=r"(s.x[0]), "=r"(s.x[1]), "=r"(s.x[2]), "=r"(s.x[3]), "=r"(s.x[4]), "=r"(s.x[5]), "=r"(s.x[6]),
                 "=r"(s.x[7])
               : "l"(p)
               : "memory");
}
__device__ __forceinline__ void kload_sector(const unsigned long long* p, Sector<unsigned long long>& s) {
  asm volatile("ld.relaxed.gpu.global.v4.b64 {%0, %1, %2, %3}, [%4];"
               : "=l"(s.x[0]), "=l"(s.x[1]), "=l"(s.x[2]), "=l"(s.x[3])
               : "l"(p)
               : "memory");
}
__device__ __forceinline__ void kload_sector(const K128* p, Sector<K128>& s) {
  unsigned long long a, b, c, d;
  asm volatile("ld.relaxed.gpu.global.v4.b64 {%0, %1, %2, %3}, [%4];"
               : "=l"(a), "=l"(b), "=l"(c), "=l"(d)
               : "l"(p)
               : "memory");
  s.x[0] = K128{a, b};
  s.x[1] = K128{c, d};
}

// May the slot that was read as x be empty?  (A 128-bit slot whose halves were
// read around a write counts as maybe empty: its compare-and-swap tells.)
__device__ __forceinline__ bool kmaybe_empty(uint32_t x) { return x == ~0u; }
__device__ __forceinline__ bool kmaybe_empty(unsigned long long x) { return x == ~0ull; }
__device__ __forceinline__ bool kmaybe_empty(K128 x) { return x.lo == ~0ull || x.hi == ~0ull; }

// Load that bypasses L1 (the table is written by other SMs during a level).
__device__ __forceinline__ uint32_t kload_cg(const uint32_t* p) { return __ldcg(p); }
__device__ __forceinline__ unsigned long long kload_cg(const unsigned long long* p) { return __ldcg(p); }
__device__ __forceinline__ K128 kload_cg(const K128* p) {
  ulonglong2 v = __ldcg(reinterpret_cast<const ulonglong2*>(p));
  return {v.x, v.y};
}

// Streaming (evict-first) load and store for the level lists, which are read
// or written once per level, so that the hash table keeps the L2.
__device__ __forceinline__ uint32_t kload_cs(const uint32_t* p) { return __ldcs(p); }
__device__ __forceinline__ unsigned long long kload_cs(const unsigned long long* p) { return __ldcs(p); }
__device__ __forceinline__ K128 kload_cs(const K128* p) {
  const ulonglong2 v = __ldcs(reinterpret_cast<const ulonglong2*>(p));
  return {v.x, v.y};
}
__device__ __forceinline__ void kstore_cs(uint32_t* p, uint32_t v) { __stcs(p, v); }
__device__ __forceinline__ void kstore_cs(unsigned long long* p, unsigned long long v) { __stcs(p, v); }
__device__ __forceinline__ void kstore_cs(K128* p, K128 v) {
  __stcs(reinterpret_cast<ulonglong2*>(p), make_ulonglong2(v.lo, v.hi));
}

}  // namespace tw
