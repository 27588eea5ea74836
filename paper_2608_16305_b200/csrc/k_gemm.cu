// Dense projections, fp32 FMA path: a strided tiled GEMM used for every
// projection and its two gradient products when math_mode is TGNN_MATH_FP32,
// and for products that do not fit the tensor-core kernels in the other modes.
#include <cstdio>

#include "tgnn_device.cuh"
#include "tgnn_internal.cuh"

namespace tgnn {
namespace {

// 64 x 64 tile, two teams of 128 threads, 8 x 4 outputs per thread: 32 multiply-adds per three 16-byte loads from shared
// memory.  Each team takes half of a step's contraction, and the teams' sums meet in shared memory at the end: the products of a
// batch are a few tiles per SM, whose warps do not hide each other's round trips.  (One team of four warps: the step of the
// smallest model 103.9 us, 93.6 with two; 1 800 x 744 x 100 with its launch 21.7 us, 20.9 with two.  64 threads with 8 x 8 outputs: a
// third slower.  Steps of 32: 23.7.  Multiply-adds of pairs: no change.)  Operand tiles are kept k-major ([k][m], [k][n]); the next
// step's tile is fetched into registers while the present one is used.
constexpr int BM = 64, BN = 64, BK = 16, TM = 8, TN = 4, TEAM = 128, NT = 2 * TEAM, PITCH = BM + 4;
constexpr int KQ = BK / 4;                    // runs of four along the contraction
constexpr int QUADS = BM * BK / 4 / NT;       // runs of four elements that a thread fetches per operand tile and step
static_assert(BM == BN, "both operand tiles use one loader");

// Four elements along the operand's contiguous index (es: its stride, 1 for every matrix of the step).  KC: that is the
// contraction index (element (r, k) at P[r * pitch + k * es], run q = 4 k's of row q / KQ), else the row index (element at
// P[k * pitch + r * es], run q = 4 rows of one k).
template <bool KC>
__device__ __forceinline__ float4 fetch_quad(const float* __restrict__ P, int64_t pitch, int64_t es, bool vec, int r0, int R, int k0,
                                             int k1, int q) {
  const int r = r0 + (KC ? q / KQ : 4 * (q & 15)), k = k0 + (KC ? 4 * (q % KQ) : q >> 4);
  float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
  if (r >= R || k >= k1) return v;
  const float* p = KC ? P + (int64_t)r * pitch + k * es : P + (int64_t)k * pitch + r * es;
  const int left = KC ? k1 - k : R - r;
  if (vec && left >= 4) return __ldg(reinterpret_cast<const float4*>(p));
  v.x = __ldg(p);
  if (left > 1) v.y = __ldg(p + es);
  if (left > 2) v.z = __ldg(p + 2 * es);
  if (left > 3) v.w = __ldg(p + 3 * es);
  return v;
}
template <bool KC>
__device__ __forceinline__ void store_quad(float (*S)[PITCH], const float4& v, int q) {
  if (KC) {
    const int r = q / KQ, k = 4 * (q % KQ);
    S[k][r] = v.x; S[k + 1][r] = v.y; S[k + 2][r] = v.z; S[k + 3][r] = v.w;
  } else {
    *reinterpret_cast<float4*>(&S[q >> 4][4 * (q & 15)]) = v;
  }
}

__device__ __forceinline__ void cluster_sync() {
  asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}

// (Not launched as a link of the chain itself: its blocks would take the places that the kernel before it leaves, three on some SMs
// and none on others, 21 -> 28 us for 1 800 x 100 x 845 behind the attention.)
// grid: (n tiles, m tiles, splits of the contraction).  Splits of a stored (not accumulated) product form a cluster: each
// leaves its partial tile in its own shared memory and sums a share of the rows over all of them.
template <bool AKC, bool BKC>
__global__ void __launch_bounds__(NT, 3) gemm_fp32_kernel(const GemmArgs g, int in_cluster) {
  __shared__ __align__(16) float tiles[2 * BM * PITCH];   // A and B tiles of two steps; at the end the teams' tiles
  __shared__ __align__(16) float s_bias[BN];
  static_assert(4 * BK <= 2 * BM, "the operand buffers fit the teams' tiles");
  float (*As)[BK][PITCH] = reinterpret_cast<float (*)[BK][PITCH]>(tiles), (*Bs)[BK][PITCH] = As + 2;
  const int M = g.dev_M ? min(*g.dev_M, g.M) : g.M;
  const int K = g.dev_K ? min(*g.dev_K, g.K) : g.K;
  const int m0 = blockIdx.y * BM, n0 = blockIdx.x * BN;
  if (m0 >= M || n0 >= g.N) return;   // (uniform over a cluster)
  // (asked for here and put into shared memory behind the products: loaded where it is added, it is waited for there)
  const float my_bias = threadIdx.x < BN && g.bias != nullptr && n0 + (int)threadIdx.x < g.N ? __ldg(g.bias + n0 + threadIdx.x) : 0.f;
  const int kchunk = ((K + g.split_k - 1) / g.split_k + BK - 1) / BK * BK;
  const int kbeg = blockIdx.z * kchunk, kend = min(K, kbeg + kchunk);
  if (kbeg >= kend && !in_cluster && !(blockIdx.z == 0 && g.bias)) return;

  const int tid = threadIdx.x, team = tid / TEAM, tx = tid & 15, ty = (tid >> 4) & 7;
  const int64_t ap = AKC ? g.a_rs : g.a_cs, bp = BKC ? g.b_cs : g.b_rs, ae = AKC ? g.a_cs : g.a_rs, be = BKC ? g.b_rs : g.b_cs;
  const bool avec = (((uintptr_t)g.A | (uintptr_t)g.a_tab) & 15) == 0 && ap % 4 == 0 && ae == 1 && (g.a_idx == nullptr || g.a_tab_cols % 4 == 0);
  const bool bvec = ((uintptr_t)g.B & 15) == 0 && bp % 4 == 0 && be == 1;
  // row-indirect A: the table row of each of this thread's runs
  int64_t arow[QUADS];
#pragma unroll
  for (int i = 0; i < QUADS; ++i) {
    const int r = m0 + (tid + i * NT) / KQ;
    int ti = -1;
    if (g.a_idx != nullptr && r < M) ti = g.a_idx[r];
    arow[i] = ti >= 0 && ti < g.a_tab_rows ? (int64_t)ti : -1;
  }
  auto fetch_a = [&](int k0, int i) {
    const int q = tid + i * NT;
    if (AKC && g.a_idx != nullptr && k0 + 4 * (q % KQ) < g.a_tab_cols) {
      if (arow[i] < 0) return make_float4(0.f, 0.f, 0.f, 0.f);
      return fetch_quad<true>(g.a_tab + arow[i] * g.a_tab_cols, 0, 1, avec, 0, BM, k0, min(kend, g.a_tab_cols), q);
    }
    return fetch_quad<AKC>(g.A, ap, ae, avec, m0, M, k0, kend, q);
  };

  float acc[TM][TN] = {};
  float rsum[TM] = {};
  const bool do_rowsum = g.rowsum_out != nullptr && blockIdx.x == 0 && tx == 0;
  float4 ra[QUADS], rb[QUADS];
  int buf = 0;
  if (kbeg < kend) {
#pragma unroll
    for (int i = 0; i < QUADS; ++i) {
      ra[i] = fetch_a(kbeg, i);
      rb[i] = fetch_quad<BKC>(g.B, bp, be, bvec, n0, g.N, kbeg, kend, tid + i * NT);
    }
#pragma unroll
    for (int i = 0; i < QUADS; ++i) {
      store_quad<AKC>(As[0], ra[i], tid + i * NT);
      store_quad<BKC>(Bs[0], rb[i], tid + i * NT);
    }
    __syncthreads();
  }
  for (int k0 = kbeg; k0 < kend; k0 += BK) {
    const bool more = k0 + BK < kend;
    if (more) {
#pragma unroll
      for (int i = 0; i < QUADS; ++i) {
        ra[i] = fetch_a(k0 + BK, i);
        rb[i] = fetch_quad<BKC>(g.B, bp, be, bvec, n0, g.N, k0 + BK, kend, tid + i * NT);
      }
    }
#pragma unroll
    for (int ks = 0; ks < BK / 2; ++ks) {
      const int kk = team * (BK / 2) + ks;
      const float4 a0 = *reinterpret_cast<const float4*>(&As[buf][kk][ty * TM]);
      const float4 a1 = *reinterpret_cast<const float4*>(&As[buf][kk][ty * TM + 4]);
      const float4 bv = *reinterpret_cast<const float4*>(&Bs[buf][kk][tx * TN]);
      const float a[TM] = {a0.x, a0.y, a0.z, a0.w, a1.x, a1.y, a1.z, a1.w}, b[TN] = {bv.x, bv.y, bv.z, bv.w};
      if (do_rowsum) {
#pragma unroll
        for (int i = 0; i < TM; ++i) rsum[i] += a[i];
      }
#pragma unroll
      for (int i = 0; i < TM; ++i)
#pragma unroll
        for (int j = 0; j < TN; ++j) acc[i][j] = fmaf(a[i], b[j], acc[i][j]);
    }
    if (more) {
#pragma unroll
      for (int i = 0; i < QUADS; ++i) {
        store_quad<AKC>(As[buf ^ 1], ra[i], tid + i * NT);
        store_quad<BKC>(Bs[buf ^ 1], rb[i], tid + i * NT);
      }
      __syncthreads();
      buf ^= 1;
    }
  }
  link_release();
  const bool cvec = ((uintptr_t)g.C & 15) == 0 && g.ldc % 4 == 0;
  auto put = [&](int gm, int gn, float4 v, bool bias) {   // row gm, columns gn .. gn + 3
    if (gm >= M || gn >= g.N) return;
    const int left = g.N - gn;
    if (bias) {
      const float4 b = *reinterpret_cast<const float4*>(s_bias + gn - n0);
      v.x += b.x; v.y += b.y; v.z += b.z; v.w += b.w;
    }
    float* c = g.C + (int64_t)gm * g.ldc + gn;
    if (g.accumulate) {
      if (cvec && left > 3) {
        atomicAdd(reinterpret_cast<float4*>(c), v);
      } else {
        atomicAdd(c, v.x);
        if (left > 1) atomicAdd(c + 1, v.y);
        if (left > 2) atomicAdd(c + 2, v.z);
        if (left > 3) atomicAdd(c + 3, v.w);
      }
      return;
    }
    if (g.relu) { v.x = fmaxf(v.x, 0.f); v.y = fmaxf(v.y, 0.f); v.z = fmaxf(v.z, 0.f); v.w = fmaxf(v.w, 0.f); }
    if (cvec && left > 3) {
      *reinterpret_cast<float4*>(c) = v;
    } else {
      c[0] = v.x;
      if (left > 1) c[1] = v.y;
      if (left > 2) c[2] = v.z;
      if (left > 3) c[3] = v.w;
    }
  };
  if (do_rowsum) {
#pragma unroll
    for (int i = 0; i < TM; ++i)
      if (m0 + ty * TM + i < M) atomicAdd(&g.rowsum_out[m0 + ty * TM + i], rsum[i]);
  }
  // the teams' tiles [64][64 + 4] over the operand buffers
  constexpr int TILE = BM * PITCH;
  float* part = tiles;
  if (tid < BN) s_bias[tid] = my_bias;
  __syncthreads();
#pragma unroll
  for (int i = 0; i < TM; ++i)
    *reinterpret_cast<float4*>(part + team * TILE + (ty * TM + i) * PITCH + tx * TN) = make_float4(acc[i][0], acc[i][1], acc[i][2], acc[i][3]);
  __syncthreads();
#pragma unroll 2
  for (int e = tid; e < BM * BN / 4; e += NT) {
    const int r = e / (BN / 4), c = 4 * (e % (BN / 4));
    float4 *own = reinterpret_cast<float4*>(part + r * PITCH + c), v = *own;
    const float4 w = *reinterpret_cast<const float4*>(part + TILE + r * PITCH + c);
    v.x += w.x; v.y += w.y; v.z += w.z; v.w += w.w;
    if (in_cluster) *own = v;
    else put(m0 + r, n0 + c, v, blockIdx.z == 0);
  }
  if (!in_cluster) return;
  cluster_sync();
  // This block's share of the tile summed over the cluster, into registers (two pieces of four columns per thread at most).  Only what will be stored
  // is asked for, and nothing is stored before the block has arrived at the last barrier: a block's shared memory may go when its peers have
  // arrived there, their loads of it have to be done by then, and a release with stores ahead of it would wait for those too. (0.3 us a
  // product more than an arrival that orders nothing: steps of the smallest model 83.0 -> 85.1 us.)
  const int S = gridDim.z;
  constexpr int PIECES = BM * BN / 4, MOST = PIECES / (2 * NT);
  static_assert(MOST * 2 * NT == PIECES, "a cluster is two blocks or more");
  float4 sum[MOST];
#pragma unroll
  for (int u = 0; u < MOST; ++u) {
    const int e = (u * S + blockIdx.z) * NT + tid, r = e / (BN / 4), c = 4 * (e % (BN / 4));
    float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
    if (e < PIECES && m0 + r < M && n0 + c < g.N) {
      const uint32_t own = (uint32_t)__cvta_generic_to_shared(part + r * PITCH + c);
      float4 x[8];   // (all of them on their way before the first is added)
#pragma unroll
      for (int z = 0; z < 8; ++z)
        if (z < S) {
          uint32_t peer;
          asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(peer) : "r"(own), "r"(z));
          asm volatile("ld.shared::cluster.v4.f32 {%0, %1, %2, %3}, [%4];"
                       : "=f"(x[z].x), "=f"(x[z].y), "=f"(x[z].z), "=f"(x[z].w) : "r"(peer) : "memory");
        }
#pragma unroll
      for (int z = 0; z < 8; ++z)
        if (z < S) { v.x += x[z].x; v.y += x[z].y; v.z += x[z].z; v.w += x[z].w; }
    }
    sum[u] = v;
  }
  __syncwarp();
  asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
#pragma unroll
  for (int u = 0; u < MOST; ++u) {
    const int e = (u * S + blockIdx.z) * NT + tid;
    if (e < PIECES) put(m0 + e / (BN / 4), n0 + 4 * (e % (BN / 4)), sum[u], true);
  }
  __syncwarp();
  asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
}

template <bool AKC, bool BKC>
cudaError_t launch_tiles(const GemmArgs& a, dim3 grid, bool in_cluster, cudaStream_t s) {
  if (!in_cluster) {
    gemm_fp32_kernel<AKC, BKC><<<grid, NT, 0, s>>>(a, 0);
    return cudaGetLastError();
  }
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid; cfg.blockDim = dim3(NT); cfg.stream = s;
  cudaLaunchAttribute at;
  at.id = cudaLaunchAttributeClusterDimension;
  at.val.clusterDim.x = 1; at.val.clusterDim.y = 1; at.val.clusterDim.z = grid.z;
  cfg.attrs = &at; cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, gemm_fp32_kernel<AKC, BKC>, a, 1);
}

}  // namespace

int launch_gemm(tgnn_ctx* ctx, const GemmArgs& g, const char* name, cudaStream_t s) {
  if (g.M <= 0 || g.N <= 0) return TGNN_OK;
  if (g.split_k > 1 && !g.accumulate) return set_error(ctx, TGNN_EINVAL, "gemm %s: split_k needs accumulate", name);
  if (ctx->cfg.math_mode != TGNN_MATH_FP32) {
    GemmArgs gp = g;
    if (ctx->cfg.math_mode != TGNN_MATH_TF32_FAST) gp.precise = 1;
    const int rc = launch_gemm_tf32(ctx, gp, name, s);
    if (rc != 1) return rc;  // 1: shape not handled by the tensor-core kernel, use the FMA tiles
    // not an error, but not silent either: the note stays in tgnn_last_error and the launches are counted
    ctx->fma_fallbacks++;
    snprintf(ctx->err, sizeof(ctx->err), "note: product %s (M=%d N=%d K=%d) does not fit the tensor-core kernel and ran on the "
             "fp32 FMA tiles (%lld such launches so far)", name, g.M, g.N, g.K, (long long)ctx->fma_fallbacks);
  }
  dim3 grid((g.N + BN - 1) / BN, (g.M + BM - 1) / BM, g.split_k < 1 ? 1 : g.split_k);
  GemmArgs a = g;
  if (a.split_k < 1) a.split_k = 1;
  // A stored product with few tiles and a long contraction: split over a cluster of up to eight blocks, as many as leave 48
  // contraction elements to each and all run at once (three per SM; with a device-side row count half the capacity is taken to
  // be in use).  Clusters of 5 to 7 do not pack: 1 800 x 100 x 845, launch included, by 4: 26.0 us, by 5: 28.0, by 7: 30.0.
  bool in_cluster = false;
  if (!a.accumulate && a.dev_K == nullptr) {
    const int64_t tiles = (int64_t)grid.x * (a.dev_M ? (grid.y + 1) / 2 : grid.y);
    int S = 1;
    for (const int c : {2, 3, 4, 8})
      if (tiles * c <= 3 * 148 && a.K >= 48 * c) S = c;
    if (S > 1) { in_cluster = true; a.split_k = S; grid.z = S; }
  }
  cudaError_t e;
  {
    KernelScope scope__(ctx, name, s);
    // which index of each operand is contiguous
    if (a.a_cs == 1 || a.a_rs != 1)
      e = a.b_rs == 1 || a.b_cs != 1 ? launch_tiles<true, true>(a, grid, in_cluster, s) : launch_tiles<true, false>(a, grid, in_cluster, s);
    else
      e = a.b_rs == 1 || a.b_cs != 1 ? launch_tiles<false, true>(a, grid, in_cluster, s) : launch_tiles<false, false>(a, grid, in_cluster, s);
  }
  if (e != cudaSuccess) return set_error(ctx, TGNN_ECUDA, "launch %s: %s", name, cudaGetErrorString(e));
  ctx->launches++;
  return TGNN_OK;
}

}  // namespace tgnn
