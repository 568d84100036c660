// The search of one level (tw_expand_core.cuh) run on the host: for sets with
// and without bits at or above n, the component of the lowest vertex, its
// boundary, and |Q(S, v)| <= k are compared with plain closures over the rows.
// Prints "ok <number of sets>".
#include <cstdint>
#include <cstdio>
#include <vector>

#include "../../paper_1709_09990_gb300/csrc/tw_expand_core.cuh"

using namespace tw;

namespace {

uint64_t g_state = 88172645463325252ull;
uint64_t next_random() {
  g_state ^= g_state << 13;
  g_state ^= g_state >> 7;
  g_state ^= g_state << 17;
  return g_state;
}

template <class K> bool has(const K& s, int v) { return !kempty(s & kbit<K>(v)); }

// The vertices of `inside` reachable from start through inside (rows of n and
// above: no edges).
template <class K>
K closure(const K start, const K inside, const std::vector<K>& adj) {
  K seen = start;
  for (bool grown = true; grown;) {
    grown = false;
    for (int v = 0; v < (int)adj.size(); ++v)
      if (has(seen, v)) {
        const K more = adj[v] & inside & ~seen;
        if (!kempty(more)) {
          seen |= more;
          grown = true;
        }
      }
  }
  return seen;
}
template <class K>
K rows_of(const K set, const std::vector<K>& adj) {
  K q = kzero<K>();
  for (int v = 0; v < (int)adj.size(); ++v)
    if (has(set, v)) q |= adj[v];
  return q;
}

template <class K>
int check(int n, int sets) {
  constexpr int kBits = KeyTraits<K>::kBits;
  std::vector<K> adj(n, kzero<K>());
  for (int a = 0; a < n; ++a)
    for (int b = 0; b < a; ++b)
      if (next_random() % 6 == 0) {
        adj[a] |= kbit<K>(b);
        adj[b] |= kbit<K>(a);
      }
  AdjRow<K> rows[kBits];
  for (int t = 0; t < 3; ++t) fill_rows<K>(rows, adj.data(), n, t, 3);  // (as three threads)
  const K valid = kfirst_n<K>(n);
  for (int j = 0; j < sets; ++j) {
    K S = kzero<K>();
    const int upto = j % 2 ? kBits : n;  // every second set may hold bits at or above n
    for (int v = 0; v < upto; ++v)
      if (next_random() % 3 == 0) S |= kbit<K>(v);
    if (kempty(S)) S |= kbit<K>(upto - 1);
    K comp, bnd;
    core::min_component<K>(S, rows, comp, bnd);
    const K want = closure<K>(klsb(S), S, adj);
    if (!(comp == want) || !(bnd == (rows_of<K>(want, adj) & ~S))) return -1;
    for (int k = 0; k < n; k += 1 + n / 5) {
      const core::Candidates<K> c = core::cheap_candidates<K, true>(S, comp, bnd, rows, valid, kones<K>(), k);
      for (int v = 0; v < n; ++v) {
        if (has(S, v)) {
          if (has(c.done | c.search, v)) return -2;
          continue;
        }
        const K vb = kbit<K>(v);
        const K reached = closure<K>(adj[v] & S, S, adj);
        const int q = kpopc((adj[v] | rows_of<K>(reached, adj)) & ~(S | vb));
        const bool got = core::extension_feasible<K>(S, comp, bnd, own_bit(rows[v], v), rows[v].row, rows, k);
        if (got != (q <= k)) return -3;
        if (has(c.done, v) && q > k) return -4;
      }
    }
  }
  return sets;
}

}  // namespace

int main() {
  int total = 0;
  for (int n : {1, 2, 5, 20, 31, 32}) {
    const int r = check<uint32_t>(n, 200);
    if (r < 0) return std::printf("32-bit n=%d: %d\n", n, r), 1;
    total += r;
  }
  for (int n : {1, 20, 33, 63, 64}) {
    const int r = check<unsigned long long>(n, 200);
    if (r < 0) return std::printf("64-bit n=%d: %d\n", n, r), 1;
    total += r;
  }
  for (int n : {65, 70, 127, 128}) {
    const int r = check<K128>(n, 60);
    if (r < 0) return std::printf("128-bit n=%d: %d\n", n, r), 1;
    total += r;
  }
  std::printf("ok %d\n", total);
  return 0;
}
