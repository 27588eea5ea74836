// Offline preprocessing of the event stream: the source-based backward dependency scan
// (Algorithm 1) for every worker and synchronisation window at once, and the construction of one
// worker's mixed batches (Eq. 5) from the scan's result.
//
// The listing is a sequential backward walk whose frontier F grows as it goes.  Each (worker, window) pair is one thread
// block that walks the window in the same order, a chunk of one event per thread at a time:
//   position i   = index of an event in the walk (0 = last event of the window, counting backward);
//   entry[x]     = position from which node x is in F: the first position of batch s for the remote
//                  destinations of the batch's target events (they enter before the batch is walked),
//                  i + 1 for the remote endpoints of an auxiliary event at position i;
//   an event at position i whose source is remote is auxiliary iff min(entry[u], entry[v]) <= i.
// What an event decides depends only on entries set at smaller positions, so a chunk is settled once the chunks before it
// are and its own events, relaxed together (atomicMin on entry[]), have stopped changing anything: the number of rounds
// over a chunk is the length of the longest chain of its events pulling one another in, and no event is looked at again
// after its chunk.
#include <cstdarg>
#include <cstdio>

#include <cuda_runtime.h>
#include <stdint.h>

#include "../../include/tgnn.h"

namespace {

constexpr unsigned FULL = 0xffffffffu;
constexpr int kInf = 0x3fffffff;
constexpr int kOwned = 0x7fffffff;   // entry[] of a node the worker owns: never part of its frontier
constexpr int kMaxBlocks = TGNN_SCAN_MAX_BLOCKS;

int fail(char* err, int64_t size, int code, const char* fmt, ...) {
  if (err && size > 0) {
    va_list ap;
    va_start(ap, fmt);
    vsnprintf(err, (size_t)size, fmt, ap);
    va_end(ap);
  }
  return code;
}

// Bound by the rounds over each chunk (a block-wide vote each), so entry[] lies in shared memory when the node table fits
// (SMEM), events are fetched two chunks ahead, and a round is only followed by another when it lowered an entry.  Which
// nodes the worker owns is kept in entry[] too: looking owners up in global memory costs a warp up to 32 cache lines.
// 1.3 M events, 2 000 nodes, 8 workers, windows of 24 000 events: 80 us (1 105 us with sweeps over whole windows on tables
// in global memory).
template <bool SMEM>
__global__ void __launch_bounds__(1024) backward_scan_kernel(const int32_t* __restrict__ src, const int32_t* __restrict__ dst,
                                                             int64_t E, int batch, int K,
                                                             const int32_t* __restrict__ owner, int64_t N, int P, int Q,
                                                             uint8_t* __restrict__ role, int32_t* __restrict__ n_sync,
                                                             uint8_t* __restrict__ sync, int32_t* scratch,
                                                             int32_t* status) {
  extern __shared__ int32_t s_entry[];
  __shared__ int s_count;
  const int tid = threadIdx.x, T = blockDim.x;
  volatile int32_t* entry = SMEM ? s_entry : scratch + (int64_t)blockIdx.x * N;
  // hub nodes are lowered once and then found low enough by every later event: the atomic is the exception
  auto lower = [&](int x, int v) {
    if (entry[x] <= v) return false;
    atomicMin(const_cast<int32_t*>(entry) + x, v);
    return true;
  };
  for (int64_t pq = blockIdx.x; pq < (int64_t)P * Q; pq += gridDim.x) {
    const int p = (int)(pq / Q), q = (int)(pq % Q);
    const int64_t lo = (int64_t)q * K * batch;
    const int64_t hi = min(E, lo + (int64_t)K * batch);
    const int n = (int)(hi - lo);
    uint8_t* rl = role + (int64_t)p * E;
    for (int64_t x = tid; x < N; x += T) entry[x] = owner[x] == p ? kOwned : kInf;
    if (tid == 0) s_count = 0;
    __syncthreads();
    // remote destinations of the target events, at the first position of their batch
    // (the latest batch, whose position is the smallest, first; four events per thread in flight)
    for (int base = 0; base < n; base += 4 * T) {
      int u[4], v[4];
#pragma unroll
      for (int w = 0; w < 4; ++w) {
        const int i = base + w * T + tid;
        u[w] = i < n ? src[hi - 1 - i] : -1;
        v[w] = i < n ? dst[hi - 1 - i] : 0;
      }
#pragma unroll
      for (int w = 0; w < 4; ++w) {
        if (u[w] < 0 || entry[u[w]] != kOwned || entry[v[w]] == kOwned) continue;
        const int b = (n - 1 - (base + w * T + tid)) / batch;         // the event's batch within the window,
        lower(v[w], n - min(n, (b + 1) * batch));                     // whose last event is walked first
      }
    }
    __syncthreads();
    // the walk: endpoints are fetched two chunks ahead
    auto ends = [&](int i, int& fu, int& fv) {
      fu = i < n ? src[hi - 1 - i] : -1;
      fv = i < n ? dst[hi - 1 - i] : 0;
    };
    int u, v, u1, v1;
    ends(tid, u, v);
    ends(tid + T, u1, v1);
    bool settled = true;
    for (int base = 0; base < n; base += T) {
      const int i = base + tid;
      int u2, v2;
      ends(i + 2 * T, u2, v2);
      bool aux = false;
      const bool own = u >= 0 && entry[u] == kOwned, cand = u >= 0 && !own, remote = u >= 0 && entry[v] != kOwned;
      bool changed = true;
      for (int round = 0; changed && round <= T; ++round) {
        bool ch = false;
        if (cand && !aux && min(entry[u], entry[v]) <= i) {
          aux = true;   // (only a lowered entry can make a difference to another event of the chunk)
          ch = lower(u, i + 1);
          if (remote) ch = lower(v, i + 1) || ch;
        }
        changed = __syncthreads_or(ch) != 0;
      }
      settled = settled && !changed;
      if (i < n) rl[hi - 1 - i] = own ? 1 : (aux ? 2 : 0);
      u = u1; v = v1;
      u1 = u2; v1 = v2;
    }
    if (!settled && tid == 0) atomicExch(status, 1);
    // N_sync = the frontier after the walk
    int c = 0;
    for (int64_t x = tid; x < N; x += T) {
      const bool in = entry[x] < kInf;
      c += in;
      if (sync) sync[pq * N + x] = in ? 1 : 0;
    }
    for (int o = 16; o > 0; o >>= 1) c += __shfl_xor_sync(FULL, c, o);
    if ((tid & 31) == 0 && c) atomicAdd(&s_count, c);
    __syncthreads();
    if (tid == 0) n_sync[pq] = s_count;
    __syncthreads();
  }
}

// The same walk for four workers at once, while a table of 16 bytes per node fits shared memory: an event's endpoints are
// fetched and looked up once for all four (one 16-byte load per endpoint), and a chunk's rounds settle all four; the workers
// of a group differ only in which nodes they own.  A chunk is V events per thread: it is the chain of dependent lookups, additions
// and votes of a chunk that takes the time, not their number, and a longer chunk hardly needs more rounds (2.1 for 1 024 events,
// 2.3 for 2 048).  1.3 M events, 2 000 nodes, 8 workers, windows of 24 000 events: 48 us, 55 with one event per
// thread (82 with a block per worker and window; one byte per endpoint in front of the entries: 58).
constexpr int kGroup = 4, VG = 4;
template <int V>
__global__ void __launch_bounds__(1024) backward_scan_group_kernel(const int32_t* __restrict__ src, const int32_t* __restrict__ dst,
                                                                   int64_t E, int batch, int K, const int32_t* __restrict__ owner,
                                                                   int N, int P, int Q, uint8_t* __restrict__ role,
                                                                   int32_t* __restrict__ n_sync, uint8_t* __restrict__ sync,
                                                                   int32_t* status) {
  extern __shared__ __align__(16) int32_t s_tab[];   // [N][kGroup]
  __shared__ int s_count[kGroup];
  const int tid = threadIdx.x, T = blockDim.x;
  const auto look = [&](int x, int (&e)[kGroup]) {
    asm volatile("ld.shared.v4.b32 {%0, %1, %2, %3}, [%4];" : "=r"(e[0]), "=r"(e[1]), "=r"(e[2]), "=r"(e[3])
                 : "r"((uint32_t)__cvta_generic_to_shared(s_tab + kGroup * x)) : "memory");
  };
  const int groups = (P + kGroup - 1) / kGroup;
  for (int64_t pq = blockIdx.x; pq < (int64_t)groups * Q; pq += gridDim.x) {
    const int p0 = (int)(pq / Q) * kGroup, q = (int)(pq % Q), np = min(kGroup, P - p0);
    const int64_t lo = (int64_t)q * K * batch;
    const int64_t hi = min(E, lo + (int64_t)K * batch);
    const int n = (int)(hi - lo);
    for (int x = tid; x < N; x += T) {   // (a worker beyond the last owns nothing: its column is never written down)
      const int o = owner[x] - p0;
      *reinterpret_cast<int4*>(s_tab + kGroup * x) = make_int4(o == 0 ? kOwned : kInf, o == 1 ? kOwned : kInf, o == 2 ? kOwned : kInf, o == 3 ? kOwned : kInf);
    }
    if (tid < kGroup) s_count[tid] = 0;
    __syncthreads();
    // the next V events of a thread, endpoints of none: node 0 twice, and a position that nothing asks about
    const auto ends = [&](int base, int (&u)[V], int (&v)[V]) {
#pragma unroll
      for (int w = 0; w < V; ++w) {
        const int i = base + w * T + tid;
        u[w] = i < n ? src[hi - 1 - i] : -1;
        v[w] = i < n ? dst[hi - 1 - i] : 0;
      }
    };
    // remote destinations of the target events, at the first position of their batch (as above)
    int u[V], v[V], u1[V], v1[V];
    ends(0, u, v);
    for (int base = 0; base < n; base += V * T) {
      ends(base + V * T, u1, v1);
#pragma unroll
      for (int w = 0; w < V; ++w) {
        if (u[w] < 0) continue;
        int eu[kGroup], ev[kGroup];
        look(u[w], eu);
        look(v[w], ev);
        const int b = (n - 1 - (base + w * T + tid)) / batch, at = n - min(n, (b + 1) * batch);
#pragma unroll
        for (int g = 0; g < kGroup; ++g)
          if (eu[g] == kOwned && ev[g] != kOwned && ev[g] > at) atomicMin(s_tab + kGroup * v[w] + g, at);
      }
#pragma unroll
      for (int w = 0; w < V; ++w) { u[w] = u1[w]; v[w] = v1[w]; }
    }
    __syncthreads();
    ends(0, u, v);
    bool settled = true;
    for (int base = 0; base < n; base += V * T) {
      ends(base + V * T, u1, v1);
      unsigned own = 0u, aux = 0u, open = 0u;   // bit 4 w + g: event w is worker g's target, auxiliary to it, not decided yet
      bool changed = true;
      for (int round = 0; changed && round <= V * T; ++round) {
        bool ch = false;
#pragma unroll
        for (int w = 0; w < V; ++w) {
          const int i = base + w * T + tid;
          if (round == 0 ? u[w] < 0 : ((open >> (kGroup * w)) & ((1u << kGroup) - 1u)) == 0u) continue;
          int eu[kGroup], ev[kGroup];
          look(u[w], eu);
          look(v[w], ev);
#pragma unroll
          for (int g = 0; g < kGroup; ++g) {
            const unsigned bit = 1u << (kGroup * w + g);
            if (round == 0) {
              if (eu[g] == kOwned) { own |= bit; continue; }
              open |= bit;
            }
            if (!(open & bit) || min(eu[g], ev[g]) > i) continue;
            open &= ~bit;
            aux |= bit;
            // (only a lowered entry can make a difference to another event of the chunk)
            if (eu[g] > i + 1) { atomicMin(s_tab + kGroup * u[w] + g, i + 1); ch = true; }
            if (ev[g] != kOwned && ev[g] > i + 1) { atomicMin(s_tab + kGroup * v[w] + g, i + 1); ch = true; }
          }
        }
        changed = __syncthreads_or(ch) != 0;
      }
      settled = settled && !changed;
#pragma unroll
      for (int w = 0; w < V; ++w) {
        const int i = base + w * T + tid;
        if (i >= n) continue;
        uint8_t* r = role + (int64_t)p0 * E + (hi - 1 - i);
#pragma unroll
        for (int g = 0; g < kGroup; ++g, r += E)
          if (g < np) *r = (uint8_t)(((own >> (kGroup * w + g)) & 1u) | (((aux >> (kGroup * w + g)) & 1u) << 1));
      }
#pragma unroll
      for (int w = 0; w < V; ++w) { u[w] = u1[w]; v[w] = v1[w]; }
    }
    if (!settled && tid == 0) atomicExch(status, 1);
    // N_sync = the frontier after the walk
    int c[kGroup] = {};
    for (int x = tid; x < N; x += T) {
      int e[kGroup];
      look(x, e);
#pragma unroll
      for (int g = 0; g < kGroup; ++g) {
        const bool in = e[g] < kInf;
        c[g] += in;
        if (sync && g < np) sync[((int64_t)(p0 + g) * Q + q) * N + x] = in ? 1 : 0;
      }
    }
#pragma unroll
    for (int g = 0; g < kGroup; ++g) {
      const int t = __reduce_add_sync(FULL, c[g]);
      if ((tid & 31) == 0 && t) atomicAdd(&s_count[g], t);
    }
    __syncthreads();
    if (tid < np) n_sync[(int64_t)(p0 + tid) * Q + q] = s_count[tid];
    __syncthreads();
  }
}

// ---- mixed batches of one worker --------------------------------------------------------------
// off[s + 1] = events of batch s with role != 0, toff[s + 1] = with role == 1 (one block per batch)
__global__ void __launch_bounds__(256) mixed_count_kernel(const uint8_t* __restrict__ role, int64_t E, int batch,
                                                          int32_t* __restrict__ off, int32_t* __restrict__ toff) {
  __shared__ int s_a, s_t;
  const int s = blockIdx.x;
  if (threadIdx.x == 0) { s_a = 0; s_t = 0; }
  __syncthreads();
  const int64_t lo = (int64_t)s * batch, hi = min(E, lo + batch);
  int a = 0, t = 0;
  for (int64_t e = lo + threadIdx.x; e < hi; e += blockDim.x) {
    const uint8_t r = role[e];
    a += r != 0;
    t += r == 1;
  }
  for (int o = 16; o > 0; o >>= 1) {
    a += __shfl_xor_sync(FULL, a, o);
    t += __shfl_xor_sync(FULL, t, o);
  }
  if ((threadIdx.x & 31) == 0) { atomicAdd(&s_a, a); atomicAdd(&s_t, t); }
  __syncthreads();
  if (threadIdx.x == 0) { off[s + 1] = s_a; toff[s + 1] = s_t; }
}

// In-place inclusive prefix sums of off[1..nb] and toff[1..nb] (off[0] = toff[0] = 0): one block, chunks of 1024.
__global__ void __launch_bounds__(1024) mixed_offsets_kernel(int32_t* off, int32_t* toff, int nb) {
  __shared__ int s_warp[2][32];
  __shared__ int s_carry[2];
  const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
  if (tid == 0) { off[0] = 0; toff[0] = 0; s_carry[0] = 0; s_carry[1] = 0; }
  __syncthreads();
  for (int base = 0; base < nb; base += 1024) {
    const int j = base + tid;
    int a = j < nb ? off[j + 1] : 0, t = j < nb ? toff[j + 1] : 0;
    for (int o = 1; o < 32; o <<= 1) {
      const int a2 = __shfl_up_sync(FULL, a, o), t2 = __shfl_up_sync(FULL, t, o);
      if (lane >= o) { a += a2; t += t2; }
    }
    if (lane == 31) { s_warp[0][wid] = a; s_warp[1][wid] = t; }
    __syncthreads();
    if (wid == 0) {
      int wa = s_warp[0][lane], wt = s_warp[1][lane];
      for (int o = 1; o < 32; o <<= 1) {
        const int a2 = __shfl_up_sync(FULL, wa, o), t2 = __shfl_up_sync(FULL, wt, o);
        if (lane >= o) { wa += a2; wt += t2; }
      }
      s_warp[0][lane] = wa; s_warp[1][lane] = wt;
    }
    __syncthreads();
    const int pa = (wid ? s_warp[0][wid - 1] : 0) + s_carry[0], pt = (wid ? s_warp[1][wid - 1] : 0) + s_carry[1];
    if (j < nb) { off[j + 1] = a + pa; toff[j + 1] = t + pt; }
    __syncthreads();
    if (tid == 1023) { s_carry[0] = a + pa; s_carry[1] = t + pt; }
    __syncthreads();
  }
}

// Stable compaction of batch s: events with role != 0 in stream (= timestamp) order into the mixed-batch
// arrays at off[s], the targets among them into the target arrays at toff[s].
__global__ void __launch_bounds__(1024) mixed_fill_kernel(const int32_t* __restrict__ src, const int32_t* __restrict__ dst,
                                                         const double* __restrict__ t, const int32_t* __restrict__ neg,
                                                         const uint8_t* __restrict__ role, int64_t E, int batch,
                                                         const int32_t* __restrict__ off, const int32_t* __restrict__ toff,
                                                         int64_t cap_mixed, int64_t cap_tgt, int32_t* __restrict__ mb_src,
                                                         int32_t* __restrict__ mb_dst, double* __restrict__ mb_t,
                                                         int32_t* __restrict__ mb_eid, uint8_t* __restrict__ mb_aux,
                                                         int32_t* __restrict__ tg_src, int32_t* __restrict__ tg_dst,
                                                         double* __restrict__ tg_t, int32_t* __restrict__ tg_neg,
                                                         int32_t* __restrict__ tg_eid, int32_t* status) {
  // A warp takes a run of the batch: it counts its run, the block adds the runs up (the only barrier), and the warp goes through
  // its run again, whose events it can ask for without waiting for the others (325 batches of 4 000: 15.2 us; 17.1 with
  // a barrier and two round trips per 512 events).
  __shared__ int s_wa[32], s_wt[32];
  const int s = blockIdx.x, lane = threadIdx.x & 31, wid = threadIdx.x >> 5, nw = blockDim.x >> 5;
  const int64_t lo = (int64_t)s * batch, hi = min(E, lo + batch);
  const int run = (int)((hi - lo + 32 * nw - 1) / (32 * nw)) * 32;
  const int64_t w0 = lo + (int64_t)wid * run, w1 = min(hi, w0 + run);
  int na = 0, nt = 0;
#pragma unroll 4
  for (int64_t e = w0 + lane; e - lane < w1; e += 32) {
    const uint8_t r = e < w1 ? role[e] : 0;
    na += __popc(__ballot_sync(FULL, r != 0));
    nt += __popc(__ballot_sync(FULL, r == 1));
  }
  if (lane == 0) { s_wa[wid] = na; s_wt[wid] = nt; }
  __syncthreads();
  int pa = off[s], pt = toff[s];
  for (int w = 0; w < wid; ++w) { pa += s_wa[w]; pt += s_wt[w]; }
  const unsigned below = (1u << lane) - 1u;
#pragma unroll 2
  for (int64_t e = w0 + lane; e - lane < w1; e += 32) {
    const uint8_t r = e < w1 ? role[e] : 0;
    int es = 0, ed = 0, en = -1;
    double et = 0.0;
    if (e < w1) { es = src[e]; ed = dst[e]; et = t[e]; }   // (asked for before the role is known: most events are kept)
    if (r == 1 && neg && tg_neg) en = neg[e];
    const unsigned ba = __ballot_sync(FULL, r != 0), bt = __ballot_sync(FULL, r == 1);
    if (r != 0) {
      const int64_t o = pa + __popc(ba & below);
      if (o < cap_mixed) {
        mb_src[o] = es; mb_dst[o] = ed; mb_t[o] = et; mb_eid[o] = (int32_t)e; mb_aux[o] = r == 2;
      } else {
        atomicExch(status, 2);
      }
    }
    if (r == 1) {
      const int64_t o = pt + __popc(bt & below);
      if (o < cap_tgt) {
        tg_src[o] = es; tg_dst[o] = ed; tg_t[o] = et; tg_eid[o] = (int32_t)e;
        if (tg_neg) tg_neg[o] = en;
      } else {
        atomicExch(status, 2);
      }
    }
    pa += __popc(ba);
    pt += __popc(bt);
  }
}

}  // namespace

extern "C" {

int64_t tgnn_backward_scan_scratch(int64_t num_events, int batch, int K, int64_t num_nodes, int P) {
  if (num_events < 0 || batch < 1 || K < 1 || num_nodes < 1 || P < 1) return -1;
  const int64_t nb = (num_events + batch - 1) / batch;
  const int64_t Q = (nb + K - 1) / K;
  const int64_t blocks = P * Q < kMaxBlocks ? P * Q : kMaxBlocks;
  return (blocks > 0 ? blocks : 1) * num_nodes;
}

int tgnn_backward_scan(const int32_t* src, const int32_t* dst, int64_t num_events, int batch, int K,
                       const int32_t* owner, int64_t num_nodes, int P, uint8_t* role_out, int32_t* n_sync_out,
                       uint8_t* sync_out, int32_t* scratch, int32_t* status_out, void* stream, char* err_host,
                       int64_t err_size) {
  if (num_events < 0 || batch < 1 || K < 1 || num_nodes < 1 || P < 1)
    return fail(err_host, err_size, TGNN_EINVAL, "tgnn_backward_scan: size out of range");
  if ((int64_t)K * batch > 0x3ffffff0)
    return fail(err_host, err_size, TGNN_ECAPACITY, "tgnn_backward_scan: window of %lld events exceeds the position range",
                (long long)K * batch);
  if (num_events == 0) return TGNN_OK;
  if (!src || !dst || !owner || !role_out || !n_sync_out || !scratch || !status_out)
    return fail(err_host, err_size, TGNN_EINVAL, "tgnn_backward_scan: null pointer");
  const int64_t nb = (num_events + batch - 1) / batch;
  const int64_t Q = (nb + K - 1) / K;
  if (Q > 0x7fffffff / P) return fail(err_host, err_size, TGNN_ECAPACITY, "tgnn_backward_scan: too many windows");
  const int64_t pairs = (int64_t)P * Q;
  const int blocks = (int)(pairs < kMaxBlocks ? pairs : kMaxBlocks);
  cudaStream_t s = (cudaStream_t)stream;
  if (cudaMemsetAsync(status_out, 0, sizeof(int32_t), s) != cudaSuccess)
    return fail(err_host, err_size, TGNN_ECUDA, "tgnn_backward_scan: %s", cudaGetErrorString(cudaGetLastError()));
  // Chunk width: 512 (80 us on the stream above; 256: 97 us, 1024: 82 us), more while every pair has an SM to itself, less
  // for windows that small.  Node tables of up to 200 KB go to shared memory.
  const int64_t window = (int64_t)K * batch;
  const int threads = window < 512 ? 256 : (window < 1024 || pairs > 148 ? 512 : 1024);
  const size_t table = (size_t)num_nodes * sizeof(int32_t);
  // Workers in groups of four, where pairs would share SMs and a window is worth setting up a group's table for (whole passes of
  // scan and mixed batches, groups against pairs: 1 300 pairs of windows of 4 000 events 73 and 77 us, 2 600 pairs 102 and 118; but
  // 100 pairs of 8 000 events 44 and 40, two workers' 650 pairs 65 and 58, windows of 400 events on 12 000 nodes 43 and 38).
  if (P >= 3 && pairs > 148 && window >= 1024 && kGroup * table <= 200 * 1024) {
    const int64_t gpairs = (int64_t)((P + kGroup - 1) / kGroup) * Q;
    const auto kernel = window >= 4 * 1024 ? backward_scan_group_kernel<VG> : backward_scan_group_kernel<1>;
    if (kGroup * table > 48 * 1024 &&
        cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, 200 * 1024) != cudaSuccess)
      return fail(err_host, err_size, TGNN_ECUDA, "tgnn_backward_scan: %s", cudaGetErrorString(cudaGetLastError()));
    kernel<<<(int)(gpairs < 65536 ? gpairs : 65536), 1024, kGroup * table, s>>>(
        src, dst, num_events, batch, K, owner, (int)num_nodes, P, (int)Q, role_out, n_sync_out, sync_out, status_out);
  } else if (table <= 200 * 1024) {
    const cudaError_t ea = table > 48 * 1024
                               ? cudaFuncSetAttribute(backward_scan_kernel<true>, cudaFuncAttributeMaxDynamicSharedMemorySize, 200 * 1024)
                               : cudaSuccess;
    if (ea != cudaSuccess) return fail(err_host, err_size, TGNN_ECUDA, "tgnn_backward_scan: %s", cudaGetErrorString(ea));
    const int grid = (int)(pairs < 65536 ? pairs : 65536);
    backward_scan_kernel<true><<<grid, threads, table, s>>>(src, dst, num_events, batch, K, owner, num_nodes, P, (int)Q, role_out,
                                                            n_sync_out, sync_out, nullptr, status_out);
  } else {
    backward_scan_kernel<false><<<blocks, threads, 0, s>>>(src, dst, num_events, batch, K, owner, num_nodes, P, (int)Q, role_out,
                                                           n_sync_out, sync_out, scratch, status_out);
  }
  const cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return fail(err_host, err_size, TGNN_ECUDA, "tgnn_backward_scan: %s", cudaGetErrorString(e));
  return TGNN_OK;
}

int tgnn_build_mixed(const int32_t* src, const int32_t* dst, const double* t, const int32_t* neg, int64_t num_events,
                     int batch, const uint8_t* role, int32_t* mb_off_out, int32_t* tgt_off_out, int64_t cap_mixed,
                     int64_t cap_tgt, int32_t* mb_src, int32_t* mb_dst, double* mb_t, int32_t* mb_eid, uint8_t* mb_aux,
                     int32_t* tgt_src, int32_t* tgt_dst, double* tgt_t, int32_t* tgt_neg, int32_t* tgt_eid,
                     int32_t* status_out, void* stream, char* err_host, int64_t err_size) {
  if (num_events < 0 || batch < 1 || cap_mixed < 0 || cap_tgt < 0)
    return fail(err_host, err_size, TGNN_EINVAL, "tgnn_build_mixed: size out of range");
  if (num_events > 0x7fffffff) return fail(err_host, err_size, TGNN_ECAPACITY, "tgnn_build_mixed: event ids exceed int32");
  if (!mb_off_out || !tgt_off_out || !status_out) return fail(err_host, err_size, TGNN_EINVAL, "tgnn_build_mixed: null pointer");
  const int64_t nb = (num_events + batch - 1) / batch;
  if (nb > 0x7ffffff0) return fail(err_host, err_size, TGNN_ECAPACITY, "tgnn_build_mixed: too many batches");
  if (num_events > 0 && (!src || !dst || !t || !role || !mb_src || !mb_dst || !mb_t || !mb_eid || !mb_aux || !tgt_src ||
                         !tgt_dst || !tgt_t || !tgt_eid))
    return fail(err_host, err_size, TGNN_EINVAL, "tgnn_build_mixed: null pointer");
  cudaStream_t s = (cudaStream_t)stream;
  if (cudaMemsetAsync(status_out, 0, sizeof(int32_t), s) != cudaSuccess)
    return fail(err_host, err_size, TGNN_ECUDA, "tgnn_build_mixed: %s", cudaGetErrorString(cudaGetLastError()));
  if (nb > 0) mixed_count_kernel<<<(unsigned)nb, 256, 0, s>>>(role, num_events, batch, mb_off_out, tgt_off_out);
  mixed_offsets_kernel<<<1, 1024, 0, s>>>(mb_off_out, tgt_off_out, (int)nb);
  if (nb > 0)
    mixed_fill_kernel<<<(unsigned)nb, batch < 512 ? 256 : (nb > 148 ? 512 : 1024), 0, s>>>(src, dst, t, neg, role, num_events, batch, mb_off_out, tgt_off_out,
                                                   cap_mixed, cap_tgt, mb_src, mb_dst, mb_t, mb_eid, mb_aux, tgt_src,
                                                   tgt_dst, tgt_t, tgt_neg, tgt_eid, status_out);
  const cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return fail(err_host, err_size, TGNN_ECUDA, "tgnn_build_mixed: %s", cudaGetErrorString(e));
  return TGNN_OK;
}

}  // extern "C"
