// Host utilities of libtw: host/device pointers, growing device buffers within
// the context's memory cap, graph validation and upload.
#include <cuda_runtime.h>

#include <algorithm>
#include <cstring>
#include <vector>

#include "tw_host.h"

namespace tw {
namespace host {

bool is_device_ptr(const void* p) {
  if (p == nullptr) return false;
  cudaPointerAttributes a;
  if (cudaPointerGetAttributes(&a, p) != cudaSuccess) {
    cudaGetLastError();
    return false;
  }
  return a.type == cudaMemoryTypeDevice || a.type == cudaMemoryTypeManaged;
}

// Copies bytes from a host or device pointer into host memory.
int fetch(void* dst_host, const void* src, size_t bytes) {
  if (bytes == 0) return TW_OK;
  if (is_device_ptr(src)) {
    TW_CK(cudaMemcpy(dst_host, src, bytes, cudaMemcpyDeviceToHost));
  } else {
    std::memcpy(dst_host, src, bytes);
  }
  return TW_OK;
}

// Writes bytes from host memory to a host or device pointer.
int put(tw_ctx* c, void* dst, const void* src_host, size_t bytes) {
  if (bytes == 0 || dst == nullptr) return TW_OK;
  if (is_device_ptr(dst)) {
    TW_CK(cudaMemcpyAsync(dst, src_host, bytes, cudaMemcpyHostToDevice, c->stream));
    TW_CK(cudaStreamSynchronize(c->stream));
  } else {
    std::memcpy(dst, src_host, bytes);
  }
  return TW_OK;
}

// Copies bytes from device scratch to a host or device pointer.
int put_from_device(tw_ctx* c, void* dst, const void* src_dev, size_t bytes) {
  if (bytes == 0 || dst == nullptr) return TW_OK;
  TW_CK(cudaMemcpyAsync(dst, src_dev, bytes, cudaMemcpyDefault, c->stream));
  TW_CK(cudaStreamSynchronize(c->stream));
  return TW_OK;
}

int fetch_solution(tw_ctx* c) {
  SmallLayout L;
  // the region order .. bags in one copy
  constexpr size_t kRegion = SmallLayout().bounds - SmallLayout().order;
  if (!c->h_out) {
    if (cudaHostAlloc(reinterpret_cast<void**>(&c->h_out), kRegion, cudaHostAllocDefault) != cudaSuccess) {
      c->h_out = nullptr;
      cudaGetLastError();
      return TW_ERR_CUDA;
    }
  }
  TW_CK(cudaMemcpyAsync(c->h_out, small_at(c, L.order), kRegion, cudaMemcpyDeviceToHost, c->stream));
  return TW_OK;
}

int put_solution(tw_ctx* c, int n, int words, int32_t* order, int32_t* td_parent, uint64_t* td_bags) {
  SmallLayout L;
  struct Part {
    void* dst;
    size_t off, bytes;
  } parts[3] = {{order, L.order, (size_t)n * 4},
                {td_parent, L.parent, (size_t)n * 4},
                {td_bags, L.bags, (size_t)n * (size_t)words * 8}};
  bool any_host = false;
  for (const Part& p : parts) {
    if (!p.dst) continue;
    if (is_device_ptr(p.dst))
      TW_CK(cudaMemcpyAsync(p.dst, small_at(c, p.off), p.bytes, cudaMemcpyDeviceToDevice, c->stream));
    else
      any_host = true;
  }
  const bool fresh = any_host && c->h_out_fresh;  // (the fused solve has copied it already)
  if (any_host && !fresh) {
    const int rc = fetch_solution(c);
    if (rc) return rc;
  }
  c->h_out_fresh = false;
  TW_CK(cudaStreamSynchronize(c->stream));
  if (any_host)
    for (const Part& p : parts)
      if (p.dst && !is_device_ptr(p.dst)) std::memcpy(p.dst, c->h_out + (p.off - L.order), p.bytes);
  return TW_OK;
}

size_t total_bytes(const tw_ctx* c) {
  return c->keys.bytes + c->pred.bytes + c->table.bytes + c->cand_key.bytes + c->cand_v.bytes + c->ooc_keys.bytes +
         (c->count_fused ? c->fused.bytes : 0);
}

void release(tw_ctx* c, DevBuf* b) {
  if (!b->ptr) return;
  cudaStreamSynchronize(c->stream);
  cudaFree(b->ptr);
  b->ptr = nullptr;
  b->bytes = 0;
}

bool release_fused(tw_ctx* c) {
  if (!c->fused.ptr) return false;
  release(c, &c->fused);
  c->fused_clean = false;
  return true;
}

void release_scratch(tw_ctx* c) {
  release_fused(c);
  for (DevBuf* b : {&c->keys, &c->pred, &c->table, &c->cand_key, &c->cand_v, &c->ooc_keys}) release(c, b);
}

// Takes bytes (rounded up to 256) of pinned, device-mapped host memory from
// the context's chunks, allocating a chunk of at least kHostChunkBytes when
// the current ones are full; *out is the device-side address of the bytes.
// A failed allocation is TW_ERR_CAPACITY.
int host_take(tw_ctx* c, size_t bytes, char** out) {
  constexpr size_t kHostChunkBytes = 256ull << 20;
  bytes = (bytes + 255) & ~size_t(255);
  while (c->host_chunk < c->host_chunks.size()) {
    const tw_ctx::HostChunk& ch = c->host_chunks[c->host_chunk];
    if (c->host_used + bytes <= ch.bytes) {
      *out = ch.dptr + c->host_used;
      c->host_used += bytes;
      return TW_OK;
    }
    ++c->host_chunk;
    c->host_used = 0;
  }
  const size_t want = std::max(bytes, kHostChunkBytes);
  void* p = nullptr;
  if (cudaHostAlloc(&p, want, cudaHostAllocMapped | cudaHostAllocPortable) != cudaSuccess) {
    cudaGetLastError();
    return TW_ERR_CAPACITY;
  }
  void* d = nullptr;
  if (cudaHostGetDevicePointer(&d, p, 0) != cudaSuccess) {
    cudaGetLastError();
    cudaFreeHost(p);
    return TW_ERR_CUDA;
  }
  c->host_chunks.push_back({static_cast<char*>(p), static_cast<char*>(d), want});
  c->host_chunk = c->host_chunks.size() - 1;
  c->host_used = bytes;
  *out = static_cast<char*>(d);
  return TW_OK;
}

// Grows b to at least need bytes, keeping its first keep bytes.  Growth is
// geometric while the cap allows it.  The fused solve's buffer gives way to a
// level loop that needs its room (the run that used it has ended by then): under
// the cap where it counts, and where the device has no more memory.
int grow(tw_ctx* c, DevBuf* b, size_t need, size_t keep) {
  if (need <= b->bytes) return TW_OK;
  const bool may_release = b != &c->fused;
  auto held_without = [&]() { return total_bytes(c) - (b == &c->fused && !c->count_fused ? 0 : b->bytes); };
  if (c->count_fused && may_release && held_without() + need > c->mem_cap) release_fused(c);
  const size_t others = held_without();
  if (others + need > c->mem_cap) return TW_ERR_CAPACITY;
  size_t want = std::max(need, b->bytes * 2);
  if (others + want > c->mem_cap) want = need;
  want = (want + 255) & ~size_t(255);
  void* p = nullptr;
  if (cudaMalloc(&p, want) != cudaSuccess) {
    cudaGetLastError();
    if (may_release) release_fused(c);
    want = (need + 255) & ~size_t(255);
    if (cudaMalloc(&p, want) != cudaSuccess) {
      cudaGetLastError();
      return TW_ERR_CAPACITY;
    }
  }
  if (keep > 0 && b->ptr) {
    TW_CK(cudaMemcpyAsync(p, b->ptr, std::min(keep, b->bytes), cudaMemcpyDeviceToDevice, c->stream));
    TW_CK(cudaStreamSynchronize(c->stream));
  }
  if (b->ptr) {
    TW_CK(cudaStreamSynchronize(c->stream));
    cudaFree(b->ptr);
  }
  b->ptr = p;
  b->bytes = want;
  return TW_OK;
}

// Symmetric, no loops, no bit >= n: every edge rc with c > r must have its
// mirror, and there must be as many bits below the diagonal as above it.
int validate_rows(const uint64_t* rows, int n) {
  if (n < 1 || n > TW_MAX_N) return TW_ERR_INVALID;
  const int W = (n + 63) / 64;
  long above = 0, below = 0;
  for (int r = 0; r < n; ++r)
    for (int w = 0; w < W; ++w) {
      uint64_t x = rows[(size_t)r * W + w];
      const int used = std::min(64, n - 64 * w);
      if (used < 64 && (x >> used) != 0) return TW_ERR_INVALID;
      // the bits of this word below the diagonal, then the diagonal
      const int d = r - 64 * w;
      const uint64_t low = d < 0 ? 0ull : (d >= 64 ? ~0ull : (1ull << d) - 1ull);
      below += __builtin_popcountll(x & low);
      x &= ~low;
      if (d >= 0 && d < 64 && ((x >> d) & 1ull)) return TW_ERR_INVALID;
      above += __builtin_popcountll(x);
      for (; x; x &= x - 1) {
        const int c = 64 * w + __builtin_ctzll(x);
        if (!((rows[(size_t)c * W + (r >> 6)] >> (r & 63)) & 1ull)) return TW_ERR_INVALID;
      }
    }
  return above == below ? TW_OK : TW_ERR_INVALID;
}

int validate(const uint64_t* rows, int n, HostGraph* g) {
  const int rc = validate_rows(rows, n);
  if (rc) return rc;
  g->n = n;
  g->words = (n + 63) / 64;
  g->rows.assign(rows, rows + (size_t)n * g->words);
  return TW_OK;
}

int load_graph(const uint64_t* adj, int n, HostGraph* g) {
  if (adj == nullptr || n < 1 || n > TW_MAX_N) return TW_ERR_INVALID;
  const int W = (n + 63) / 64;
  std::vector<uint64_t> tmp((size_t)n * W);
  int rc = fetch(tmp.data(), adj, tmp.size() * sizeof(uint64_t));
  if (rc) return rc;
  return validate(tmp.data(), n, g);
}

char* small_at(tw_ctx* c, size_t off) { return static_cast<char*>(c->small.ptr) + off; }

// Uploads the adjacency in the key layout of class kc and in 64-bit rows: one
// copy of both from pinned memory.
int upload_graph(tw_ctx* c, const HostGraph& g, KeyClass kc) {
  SmallLayout L;
  c->count_fused = kc == kKey128;
  if (!c->h_up) {
    if (cudaHostAlloc(reinterpret_cast<void**>(&c->h_up), L.walk, cudaHostAllocDefault) != cudaSuccess) {
      c->h_up = nullptr;
      cudaGetLastError();
      return TW_ERR_CUDA;
    }
    TW_CK(cudaEventCreateWithFlags(&c->ev_up, cudaEventDisableTiming));
  } else {
    TW_CK(cudaEventSynchronize(c->ev_up));
  }
  const size_t w = key_bytes(kc);
  unsigned char* buf = c->h_up + L.adj;
  for (int r = 0; r < g.n; ++r) {
    const uint64_t lo = g.rows[(size_t)r * g.words];
    const uint64_t hi = g.words > 1 ? g.rows[(size_t)r * g.words + 1] : 0;
    if (kc == kKey32) {
      const uint32_t x = (uint32_t)lo;
      std::memcpy(&buf[r * w], &x, 4);
    } else if (kc == kKey64) {
      std::memcpy(&buf[r * w], &lo, 8);
    } else {
      std::memcpy(&buf[r * w], &lo, 8);
      std::memcpy(&buf[r * w + 8], &hi, 8);
    }
  }
  std::memcpy(c->h_up + L.adj64, g.rows.data(), g.rows.size() * 8);
  TW_CK(cudaMemcpyAsync(small_at(c, L.adj), c->h_up, L.adj64 + g.rows.size() * 8, cudaMemcpyHostToDevice, c->stream));
  TW_CK(cudaEventRecord(c->ev_up, c->stream));
  return TW_OK;
}

unsigned long long next_pow2(unsigned long long x) {
  unsigned long long p = 64;
  while (p < x) p <<= 1;
  return p;
}

double binom(int n, int r) {
  if (r < 0 || r > n) return 0.0;
  double b = 1.0;
  for (int i = 1; i <= r; ++i) b = b * (n - r + i) / i;
  return b;
}

}  // namespace host
}  // namespace tw
