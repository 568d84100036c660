// Persistent batched solve: one launch for a whole batch of graphs (n <= 64).
//
// Every block is a worker with its own workspace (a level arena and two
// tables in device memory).  A block takes the next graph from a queue (one
// atomic add), runs that graph's decide runs itself - Listing 1 level by level
// (Section 3.1), the block's warps taking the chunks of 32 states in turn, with
// only block barriers between levels - until the treewidth is certified (yes
// at tw, and no at tw-1 or tw equal to the lower bound), walks back through
// its levels for the ordering, and takes the next graph.  A block's levels are
// bound by latency (four warps, block barriers), and the launch lasts as long as
// its longest sweep: a graph of more than one_launch_n vertices is given up once
// a run holds `limit` sets (the host's choice, with both sides' times, is in
// run_batch_persistent).  The per-graph k
// sweep starts at the lower bound, or at a proposed bound (learned-k), and
// moves up on no and down on yes.  A graph whose levels outgrow the block's
// workspace is marked and left to the level-synchronous kernel (tw_batch.cu);
// nothing else leaves the device until the batch is done.
//
// In decide mode every graph runs one decide at its own k and reports its
// answer, level sizes and level fingerprints (tw_decide_batch).
#include <climits>

#include <cuda_runtime.h>

#include "tw_expand_core.cuh"
#include "tw_internal.h"
#include "tw_keys.cuh"

namespace tw {
namespace {

using core::ExpandParams;
using K = unsigned long long;
constexpr unsigned kFull = 0xffffffffu;


// What tw_stats reports of decide runs; thread 0 keeps them.  A run counts when it
// has ended: the next kernel makes a run that outgrew the workspace again from
// its empty set, and the yes runs of a graph that is left to it too, while the no
// runs are not made again.
struct RunCounts {
  unsigned long long states, candidates, generated, runs;
  __device__ void clear() { states = candidates = generated = runs = 0ull; }
  __device__ void add(const RunCounts& r) {
    states += r.states;
    candidates += r.candidates;
    generated += r.generated;
    runs += r.runs;
  }
};

// The block's view of its workspace.
struct Work {
  K* arena;
  uint8_t* pred;
  K* table[2];
  unsigned long long dirty[2];  // slots of each table to empty before use
  LevelCounters* ctr;
  unsigned long long* off;      // level offsets of the run in the arena
  unsigned long long* cnt;      // level sizes
};

// Sum and xor of the level fingerprints of keys[0, count) by the block.
__device__ void block_fingerprint(const K* keys, unsigned long long count, unsigned long long* sRed,
                                  unsigned long long* sum_out, unsigned long long* xor_out) {
  unsigned long long s = 0, x = 0;
  for (unsigned long long i = threadIdx.x; i < count; i += blockDim.x) {
    const unsigned long long f = kfingerprint(kload_cg(&keys[i]));
    s += f;
    x ^= f;
  }
#pragma unroll
  for (int d = 16; d > 0; d >>= 1) {
    s += __shfl_xor_sync(kFull, s, d);
    x ^= __shfl_xor_sync(kFull, x, d);
  }
  const int warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
  if ((threadIdx.x & 31) == 0) {
    sRed[2 * warp] = s;
    sRed[2 * warp + 1] = x;
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    unsigned long long ts = 0, tx = 0;
    for (int w = 0; w < nw; ++w) {
      ts += sRed[2 * w];
      tx ^= sRed[2 * w + 1];
    }
    *sum_out = ts;
    *xor_out = tx;
  }
  __syncthreads();
}

// decide(k) of one graph by one block into its workspace.  Returns false when
// the levels outgrow the workspace; else *yes and *last (the final level).
// With fp_sum / fp_xor (decide mode) the level fingerprints are written.  *run gets
// the run's counts.
template <int kWarps>
__device__ __noinline__ bool block_decide(const BatchSolveArgs& a, const K* adj, int n, int k, Work& w, AdjRow<K>* sAdj,
                             core::WarpScratch<K>* sScratch, const unsigned long long* sSets,
                             unsigned long long* sRed, bool* yes, int* last,
                             RunCounts* run, unsigned long long* fp_sum, unsigned long long* fp_xor) {
  if (threadIdx.x == 0) {
    run->clear();
    run->runs = 1ull;
  }
  for (int t = 0; t < 2; ++t) {
    for (unsigned long long j = threadIdx.x; j < w.dirty[t]; j += blockDim.x) w.table[t][j] = kones<K>();
    w.dirty[t] = 0;
  }
  if (threadIdx.x == 0) {
    w.arena[0] = kzero<K>();
    w.off[0] = 0ull;
    w.cnt[0] = 1ull;
  }
  if (fp_sum && threadIdx.x == 0) {
    fp_sum[0] = 0ull;  // fp of the empty set
    fp_xor[0] = 0ull;
  }
  __syncthreads();
  *last = 0;
  if (k >= n - 1) {
    *yes = true;
    return true;
  }
  const unsigned long long most = n <= a.one_launch_n ? a.A : a.limit;
  unsigned long long off = 0, cnt = 1, prev_cnt = 0;
  for (int i = 0; i <= n - k - 2; ++i) {
    // the plan of the level in integer arithmetic (FP64 is slow on this part)
    unsigned long long table_est = 0, slots = 0;
    core::plan_level(cnt, prev_cnt, n, i, a.load_pct, sSets[i + 1], &table_est, &slots);
    const unsigned long long out_off = off + cnt;
    if (out_off >= most || most - out_off < table_est) return false;
    if (slots > a.T) slots = a.T;
    const int t = i & 1;
    unsigned long long got = 0, gen = 0;
    for (;;) {
      // a table that fills is emptied and the level expanded again with a
      // larger one (up to the workspace's table size)
      if (threadIdx.x == 0) *w.ctr = LevelCounters{};
      __syncthreads();
      ExpandParams<K> p;
      p.in_keys = w.arena + off;
      p.n_in = cnt;
      p.adj = adj;
      p.n = n;
      p.k = k;
      p.table = w.table[t];
      p.table_slots = slots;
      p.max_probes = a.max_probes;
      p.out_keys = w.arena + out_off;
      p.out_pred = w.pred + out_off;
      p.out_parent = nullptr;
      p.out_cap = most - out_off;
      p.ctr = w.ctr;
      p.allowed = kones<K>();
      p.mmw = 0;
      p.ranges = 1;
      p.range = 0;
      core::expand_level<K, kWarps, false, false, true, true>(p, sAdj, sScratch);
      for (unsigned long long j = threadIdx.x; j < w.dirty[1 - t]; j += blockDim.x) w.table[1 - t][j] = kones<K>();
      w.dirty[1 - t] = 0;
      w.dirty[t] = max(w.dirty[t], slots);
      __syncthreads();
      got = __ldcg(&w.ctr->out_count);
      const unsigned int ovf = __ldcg(&w.ctr->overflow);
      gen = __ldcg(&w.ctr->generated);
      __syncthreads();
      if ((ovf & 1u) || got > p.out_cap) return false;  // the arena is full
      if (!(ovf & 2u) && got * 100ull <= slots * 90ull) break;
      if (slots >= a.T) return false;
      slots = min(a.T, max(2 * slots, (got * 100ull) / (unsigned long long)a.load_pct + 1024ull));
      for (unsigned long long j = threadIdx.x; j < w.dirty[t]; j += blockDim.x) w.table[t][j] = kones<K>();
      w.dirty[t] = 0;
      __syncthreads();
    }
    if (threadIdx.x == 0) {
      run->states += cnt;
      run->candidates += cnt * (unsigned long long)(n - i);
      run->generated += gen;
      w.off[i + 1] = out_off;
      w.cnt[i + 1] = got;
    }
    if (fp_sum) block_fingerprint(w.arena + out_off, got, sRed, &fp_sum[i + 1], &fp_xor[i + 1]);
    prev_cnt = cnt;
    off = out_off;
    cnt = got;
    *last = i + 1;
    if (got == 0ull) {
      *yes = false;
      __syncthreads();
      return true;
    }
  }
  *yes = true;
  __syncthreads();
  return true;
}

template <int kWarps>
__global__ void __launch_bounds__(kWarps * 32, 24 / kWarps) batch_solve_kernel(const BatchSolveArgs a) {
  __shared__ AdjRow<K> sAdj[64];
  __shared__ core::WarpScratch<K> sScratch[kWarps];
  __shared__ unsigned long long sRed[2 * kWarps];
  __shared__ unsigned long long sSets[65];  // C(n, j), capped
  __shared__ K sWalk;
  __shared__ int sFound;
  __shared__ int sGraph;
  const size_t slot = blockIdx.x;
  Work w;
  w.arena = a.arena + slot * a.A;
  w.pred = a.pred + slot * a.A;
  w.table[0] = a.tables + slot * 2 * a.T;
  w.table[1] = w.table[0] + a.T;
  w.dirty[0] = w.dirty[1] = a.T;  // the workspace starts with anything in it
  w.ctr = a.ctr + slot;
  w.off = a.level_off + slot * 130;
  w.cnt = a.level_cnt + slot * 130;
  __shared__ RunCounts sRun, sYes, sTotal;  // the run, the graph's yes runs, the block's counted runs
  if (threadIdx.x == 0) sTotal.clear();
  for (;;) {
    if (threadIdx.x == 0) sGraph = (int)atomicAdd(a.next_graph, 1u);
    __syncthreads();
    const int g = sGraph;
    __syncthreads();
    if (g >= a.num_graphs) break;
    const int n = a.n[g];
    const K* adj = a.adj + (size_t)g * 64;
    for (int j = threadIdx.x; j <= n; j += blockDim.x) sSets[j] = core::binom_capped(n, j, core::kSetsCap);
    bool yes = false;
    int last = 0;
    if (a.decide_mode) {
      unsigned long long* fs = a.fp_sum ? a.fp_sum + (size_t)g * 129 : nullptr;
      unsigned long long* fx = a.fp_xor ? a.fp_xor + (size_t)g * 129 : nullptr;
      const bool ok = block_decide<kWarps>(a, adj, n, a.k_start[g], w, sAdj, sScratch, sSets, sRed, &yes, &last,
                                           &sRun, fs, fx);
      if (threadIdx.x == 0) {
        if (ok) sTotal.add(sRun);
        a.status[g] = ok ? 0 : 2;
        a.yes[g] = yes ? 1 : 0;
        a.last[g] = last;
      }
      if (ok)
        for (int j = threadIdx.x; j <= last; j += blockDim.x) a.level_size[(size_t)g * 129 + j] = __ldcg(&w.cnt[j]);
      __syncthreads();
      continue;
    }
    // the k sweep with certification
    const int lb = a.lb[g];
    int k = a.k_start[g];
    int yes_min = INT_MAX, no_max = lb - 1, yes_in_arena = -1;
    bool ok = true;
    if (threadIdx.x == 0) sYes.clear();
    for (;;) {
      ok = block_decide<kWarps>(a, adj, n, k, w, sAdj, sScratch, sSets, sRed, &yes, &last, &sRun, nullptr, nullptr);
      if (!ok) break;
      if (threadIdx.x == 0) (yes ? sYes : sTotal).add(sRun);
      if (yes) {
        yes_min = min(yes_min, k);
        yes_in_arena = k;
      } else {
        no_max = max(no_max, k);
        yes_in_arena = -1;
      }
      if (yes_min == no_max + 1) break;
      k = yes_min == INT_MAX ? no_max + 1 : yes_min - 1;
    }
    if (ok && yes_in_arena != yes_min) {
      // the last run was a no: run the yes at tw again for its levels
      ok = block_decide<kWarps>(a, adj, n, yes_min, w, sAdj, sScratch, sSets, sRed, &yes, &last, &sRun, nullptr,
                                nullptr);
      if (threadIdx.x == 0) sYes.add(sRun);
    }
    if (!ok) {
      if (threadIdx.x == 0) {
        a.status[g] = 2;
        a.tw[g] = -1 - no_max;  // every k up to no_max answers no
      }
      __syncthreads();
      continue;
    }
    if (a.orders) core::walk_block<K>(w.arena, w.pred, w.off, w.cnt, last, n, a.orders + a.order_off[g], &sWalk, &sFound);
    if (threadIdx.x == 0) {
      sTotal.add(sYes);
      a.status[g] = 0;
      a.tw[g] = yes_min;
    }
    __syncthreads();
  }
  if (threadIdx.x == 0) {
    atomicAdd(&a.totals[0], sTotal.states);
    atomicAdd(&a.totals[1], sTotal.candidates);
    atomicAdd(&a.totals[2], sTotal.generated);
    atomicAdd(&a.totals[3], sTotal.runs);
  }
}

}  // namespace

int batch_solve_blocks(int warps) {
  int dev = 0, sms = 0, per_sm = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  if (warps == 8)
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, batch_solve_kernel<8>, 256, 0);
  else
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, batch_solve_kernel<4>, 128, 0);
  return sms * (per_sm > 0 ? per_sm : 1);
}

cudaError_t launch_batch_solve(const BatchSolveArgs& a, int blocks, int warps, cudaStream_t s) {
  if (a.num_graphs == 0) return cudaSuccess;
  if (warps == 8)
    batch_solve_kernel<8><<<blocks, 256, 0, s>>>(a);
  else
    batch_solve_kernel<4><<<blocks, 128, 0, s>>>(a);
  return cudaGetLastError();
}

}  // namespace tw
