// Step (5) and its backward with the attention contracted on the query side.
//
// Per head h the textbook layer is  logit = q_h . (W_k,h z + b_k,h) / sqrt(dh),  a_h = sum_s p_s (W_v,h z_s + b_v,h),
// q_h = W_q,h [m_root || Phi(0)] + b_q,h,  out = ReLU(W_o [a || m_root] + b_o).  Nothing between a slot's input z and
// these sums is non-linear, so the weights can be applied to the root instead of to each of its k slots:
//   qp_h   = A_h m_root + c_h          A_h = W_k,h^T W_q,h,m / sqrt(dh),  c_h = W_k,h^T (W_q,h,phi Phi(0) + b_q,h) / sqrt(dh)
//   logit  = qp_h . z                  (b_k adds the same number to every slot of a root: the softmax does not see it)
//   zbar_h = sum_s p_s z_s
//   out    = ReLU(sum_h B_h zbar_h + [any slot] W_o,a b_v + W_o,m m_root + b_o)      B_h = W_o,a,h W_v,h
// The products over the n k slot rows (key/value projection, its input gradient, its weight gradient: 2 n k 2d d_kv
// flops each) become products over the n root rows, and a slot's input is only ever streamed: gathered, encoded, used
// for 2 H multiply-adds per column and forgotten, in the forward pass as in the backward pass.  No attention input,
// key, value or gradient row of a slot is written to memory.
//
// A row z lies as [memory (d) | time encoding (d) | features (d_e) | padding to 4] in everything of these files: ldz columns.
#include <cmath>

#include "k_attn.cuh"

namespace tgnn {
namespace {

constexpr unsigned FULL = 0xffffffffu;

// ---- the weights of the query side, and the way back from their gradients -----------------------------------------
// All of it is weight-sized (a few 10^7 multiply-adds): fp32 tiles of 32 x 32 outputs, one launch each way, with one
// block per tile of every head's products.
struct FoldArgs {
  int d, de, H, dh, dkv, ldz, ldc;
  float scale;
  const float *time_b, *wq, *bq, *wk, *wv, *bv, *wo;
  float *wA, *wAp, *cA, *cq, *wB;              // wA, wAp [H ldz, d]; cA [H ldz]; cq [d]; wB [d, ldc]
  const float *dOut, *T;                       // dOut [d, ldc]: gradient of wB;  T [d + 1, H ldz]: gradient of wA^T and cA
  float *g_wq, *g_bq, *g_wk, *g_wv, *g_bv, *g_wo;
  double* tg;
  const double* tg_part;                       // [parts][2 d]
  int parts;
  int seg[8];                                  // first block of each segment
};
// Column c of a head's row -> column of the weight matrices [memory | features | encoding]; -1 for padding.
__device__ __forceinline__ int z_col(const FoldArgs& f, int c) {
  if (c < f.d) return c;
  if (c < 2 * f.d) return c + f.de;
  return c - 2 * f.d < f.de ? c - f.d : -1;
}

// One tile of 32 x 32 outputs by 256 threads.  acc[i] += sum_k A(m0 + ty + 8 i, k) B(k, n0 + tx) over k in [k0, k1); tx = threadIdx % 32,
// ty = threadIdx / 32.  AM / BN: the operand is contiguous along m / along n (else along k): which index the loading threads run along.
// These tiles are a link of the step's chain with one or two blocks per SM, bound by round trips and by what a multiply-add
// costs around it: 64 k's are fetched at a time, the next 64 while these are used; a thread takes 4 x 4 outputs for a quarter of
// the k's (two 16-byte loads from shared memory per 16 multiply-adds, where a column of four outputs took five loads per four),
// and the quarters meet in shared memory.  Unfolding at d = 100, 172 features, launch included: 12.6 -> 10.6 us.
constexpr int FT = 32, FK = 64, FP = FT + 4;   // tile, k's per step, row pitch (16-byte rows)
template <bool AM, bool BN, typename FA, typename FB>
__device__ __forceinline__ void fold_tile(float* smem, float (&acc)[4], int m0, int M, int n0, int N, int k0, int k1, FA fa, FB fb) {
  // smem: A and B as [k][m | n], at the end the quarters' sums
  float (*As)[FP] = reinterpret_cast<float (*)[FP]>(smem), (*Bs)[FP] = As + FK;
  constexpr int U = FK / 8;   // values per thread and operand
  const int tx = threadIdx.x & 31, ty = threadIdx.x >> 5;
  const int kq = threadIdx.x >> 6, r4 = 4 * ((threadIdx.x >> 3) & 7), c4 = 4 * (threadIdx.x & 7);
  float ra[U], rb[U], o[4][4] = {};
  // a thread's values: along the operand's contiguous index tx (+ 32), along the other ty + 8 i
  auto fetch = [&](int kb) {
#pragma unroll
    for (int i = 0; i < U; ++i) {
      const int m = m0 + (AM ? tx : ty + 8 * (i & 3)), ka = kb + (AM ? ty + 8 * i : tx + 32 * (i >> 2));
      ra[i] = m < M && ka < k1 ? fa(m, ka) : 0.f;
      const int n = n0 + (BN ? tx : ty + 8 * (i & 3)), kk = kb + (BN ? ty + 8 * i : tx + 32 * (i >> 2));
      rb[i] = n < N && kk < k1 ? fb(kk, n) : 0.f;
    }
  };
  fetch(k0);
#pragma unroll 1
  for (int kb = k0; kb < k1; kb += FK) {
#pragma unroll
    for (int i = 0; i < U; ++i) {
      if (AM) As[ty + 8 * i][tx] = ra[i]; else As[tx + 32 * (i >> 2)][ty + 8 * (i & 3)] = ra[i];
      if (BN) Bs[ty + 8 * i][tx] = rb[i]; else Bs[tx + 32 * (i >> 2)][ty + 8 * (i & 3)] = rb[i];
    }
    __syncthreads();
    if (kb + FK < k1) fetch(kb + FK);
#pragma unroll 4
    for (int k = kq; k < FK; k += 4) {
      const float4 a = *reinterpret_cast<const float4*>(&As[k][r4]), b = *reinterpret_cast<const float4*>(&Bs[k][c4]);
      const float av[4] = {a.x, a.y, a.z, a.w}, bv[4] = {b.x, b.y, b.z, b.w};
#pragma unroll
      for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) o[i][j] = fmaf(av[i], bv[j], o[i][j]);
    }
    __syncthreads();
  }
  float (*Q)[FT][FP] = reinterpret_cast<float (*)[FT][FP]>(smem);   // [quarter][m][n]: 4 x 32 rows, as many as A and B have
#pragma unroll
  for (int i = 0; i < 4; ++i) *reinterpret_cast<float4*>(&Q[kq][r4 + i][c4]) = make_float4(o[i][0], o[i][1], o[i][2], o[i][3]);
  __syncthreads();
#pragma unroll
  for (int i = 0; i < 4; ++i) acc[i] += (Q[0][ty + 8 * i][tx] + Q[1][ty + 8 * i][tx]) + (Q[2][ty + 8 * i][tx] + Q[3][ty + 8 * i][tx]);
}
__host__ __device__ inline int up_div(int a, int b) { return (a + b - 1) / b; }

__global__ void __launch_bounds__(256) fold_weights_kernel(const FoldArgs f) {
  __shared__ __align__(16) float smem[2 * FK * FP];
  __shared__ float s_cq[256], s_phi[256];
  const int tx = threadIdx.x & 31, ty = threadIdx.x >> 5;
  const int d = f.d;
  float acc[4] = {0.f, 0.f, 0.f, 0.f};
  int b = blockIdx.x;
  if (b < f.seg[1]) {   // wA | wAp | cA of one head: [ldz, 2 d + 1]
    const int nm = up_div(f.ldz, FT), nn = up_div(2 * d + 1, FT);
    const int h = b / (nm * nn), t = b - h * nm * nn;
    const int m0 = (t / nn) * FT, n0 = (t % nn) * FT;
    if (n0 + FT > 2 * d) {   // the tile with the column of constants: cq = W_q,phi Phi(0) + b_q, eight lanes per row
      for (int j = threadIdx.x; j < d; j += blockDim.x) s_phi[j] = time_encode(0.f, f.time_b[j], 0.f);
      __syncthreads();
      const int l8 = threadIdx.x & 7;
      for (int e0 = 0; e0 < f.dh; e0 += 32) {
        const int e = e0 + (threadIdx.x >> 3);
        float s = 0.f;
        if (e < f.dh) {
          // (sixteen loads under way whatever d is: a loop unrolled by 16 left all 13 rounds of d = 100 to its remainder, a round
          // trip each: 15.2 us instead of 11.5 with the launch, d = 100 and 172 features)
          const float* row = f.wq + (int64_t)(h * f.dh + e) * 2 * d + d;
          for (int j0 = l8; j0 < d; j0 += 128) {
            float v[16];
#pragma unroll
            for (int i = 0; i < 16; ++i) v[i] = j0 + 8 * i < d ? __ldg(row + j0 + 8 * i) : 0.f;
#pragma unroll
            for (int i = 0; i < 16; ++i)
              if (j0 + 8 * i < d) s = fmaf(v[i], s_phi[j0 + 8 * i], s);
          }
        }
        for (int o = 4; o > 0; o >>= 1) s += __shfl_xor_sync(FULL, s, o);
        if (l8 == 0 && e < f.dh) {
          s += f.bq[h * f.dh + e];
          s_cq[e] = s;
          if (m0 == 0) f.cq[h * f.dh + e] = s;
        }
      }
      __syncthreads();
    }
    fold_tile<true, true>(
        smem, acc, m0, f.ldz, n0, 2 * d + 1, 0, f.dh,
        [&](int m, int k) { const int c = z_col(f, m); return c < 0 ? 0.f : __ldg(f.wk + (int64_t)(h * f.dh + k) * f.dkv + c); },
        [&](int k, int n) { return n < 2 * d ? __ldg(f.wq + (int64_t)(h * f.dh + k) * 2 * d + n) : s_cq[k]; });
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const int m = m0 + ty + 8 * i, n = n0 + tx;
      if (m >= f.ldz || n > 2 * d) continue;
      const float v = acc[i] * f.scale;
      const int64_t row = (int64_t)h * f.ldz + m;
      if (n < d) f.wA[row * d + n] = v;
      else if (n < 2 * d) f.wAp[row * d + n - d] = v;
      else f.cA[row] = v;
    }
  } else if (b < f.seg[2]) {   // wB's block of one head: [d, ldz]
    b -= f.seg[1];
    const int nm = up_div(d, FT), nn = up_div(f.ldz, FT);
    const int h = b / (nm * nn), t = b - h * nm * nn;
    const int m0 = (t / nn) * FT, n0 = (t % nn) * FT;
    fold_tile<false, true>(
        smem, acc, m0, d, n0, f.ldz, 0, f.dh, [&](int m, int k) { return __ldg(f.wo + (int64_t)m * 2 * d + h * f.dh + k); },
        [&](int k, int n) { const int c = z_col(f, n); return c < 0 ? 0.f : __ldg(f.wv + (int64_t)(h * f.dh + k) * f.dkv + c); });
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const int m = m0 + ty + 8 * i, n = n0 + tx;
      if (m < d && n < f.ldz) f.wB[(int64_t)m * f.ldc + h * f.ldz + n] = acc[i];
    }
  } else {   // wB's last columns: W_o,m and, for the column that says whether the root has a slot, W_o,a b_v
    const int m = (b - f.seg[2]) * 8 + ty;
    if (m >= d) return;
    const float* row = f.wo + (int64_t)m * 2 * d;
    float* out = f.wB + (int64_t)m * f.ldc + f.H * f.ldz;
    float s = 0.f;
#pragma unroll 4
    for (int j = tx; j < d; j += 32) {
      out[j] = __ldg(row + d + j);
      s = fmaf(__ldg(row + j), __ldg(f.bv + j), s);
    }
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(FULL, s, o);
    if (tx == 0) out[d] = s;
  }
}

// From the gradients of wB and wA to those of the model's matrices.  s = row d of T is the gradient of cA.  The gradient
// of b_k is zero: its effect on the logits is the same for all slots of a root.  The attention backward's per-block time-
// encoder sums are added up here too.
constexpr int FOLD_K = 64;   // contraction length per block of the two products over a head's ldz columns (added atomically)
constexpr int TG_ROWS = 32;   // per-block sums added by one block
__global__ void __launch_bounds__(256) unfold_grads_kernel(const FoldArgs f) {
  __shared__ __align__(16) float smem[2 * FK * FP];
  const int tx = threadIdx.x & 31, ty = threadIdx.x >> 5;
  const int d = f.d, HL = f.H * f.ldz, nk = up_div(f.ldz + 1, FOLD_K);
  float acc[4] = {0.f, 0.f, 0.f, 0.f};
  int b = blockIdx.x;
  link_release();
  if (b < f.seg[1]) {   // dW_v | db_v of one head: [dh, ldz + 1], over the d outputs
    const int nm = up_div(f.dh, FT), nn = up_div(f.ldz + 1, FT);
    const int h = b / (nm * nn), t = b - h * nm * nn;
    const int m0 = (t / nn) * FT, n0 = (t % nn) * FT;
    fold_tile<true, true>(
        smem, acc, m0, f.dh, n0, f.ldz + 1, 0, d, [&](int m, int k) { return __ldg(f.wo + (int64_t)k * 2 * d + h * f.dh + m); },
        [&](int k, int n) { return __ldg(f.dOut + (int64_t)k * f.ldc + (n < f.ldz ? h * f.ldz + n : HL + d)); });
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const int m = m0 + ty + 8 * i, n = n0 + tx;
      if (m >= f.dh || n > f.ldz) continue;
      if (n == f.ldz) { f.g_bv[h * f.dh + m] = acc[i]; continue; }
      const int c = z_col(f, n);
      if (c >= 0) f.g_wv[(int64_t)(h * f.dh + m) * f.dkv + c] = acc[i];
    }
  } else if (b < f.seg[2]) {   // dW_k of one head: [dh, ldz], over the d memory columns of the query and its constant
    b -= f.seg[1];
    const int nm = up_div(f.dh, FT), nn = up_div(f.ldz, FT);
    const int h = b / (nm * nn), t = b - h * nm * nn;
    const int m0 = (t / nn) * FT, n0 = (t % nn) * FT;
    fold_tile<false, true>(
        smem, acc, m0, f.dh, n0, f.ldz, 0, d + 1,
        [&](int m, int k) { return k < d ? __ldg(f.wq + (int64_t)(h * f.dh + m) * 2 * d + k) : __ldg(f.cq + h * f.dh + m); },
        [&](int k, int n) { return __ldg(f.T + (int64_t)k * HL + h * f.ldz + n); });
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const int m = m0 + ty + 8 * i, n = n0 + tx;
      if (m >= f.dh || n >= f.ldz) continue;
      const int c = z_col(f, n);
      if (c >= 0) f.g_wk[(int64_t)(h * f.dh + m) * f.dkv + c] = acc[i] * f.scale;
    }
  } else if (b < f.seg[3]) {   // dW_o's attention columns of one head: [d, dh], over the head's ldz columns and b_v
    b -= f.seg[2];
    const int nm = up_div(d, FT), nn = up_div(f.dh, FT);
    const int h = b / (nm * nn * nk), t = b - h * nm * nn * nk;
    const int kb = t / (nm * nn), u = t - kb * nm * nn;
    const int m0 = (u / nn) * FT, n0 = (u % nn) * FT;
    const int k0 = kb * FOLD_K, k1 = min(f.ldz + 1, k0 + FOLD_K);
    fold_tile<false, false>(
        smem, acc, m0, d, n0, f.dh, k0, k1,
        [&](int m, int k) { return __ldg(f.dOut + (int64_t)m * f.ldc + (k < f.ldz ? h * f.ldz + k : HL + d)); },
        [&](int k, int n) {
          if (k == f.ldz) return __ldg(f.bv + h * f.dh + n);
          const int c = z_col(f, k);
          return c < 0 ? 0.f : __ldg(f.wv + (int64_t)(h * f.dh + n) * f.dkv + c);
        });
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const int m = m0 + ty + 8 * i, n = n0 + tx;
      if (m < d && n < f.dh) atomicAdd(f.g_wo + (int64_t)m * 2 * d + h * f.dh + n, acc[i]);
    }
  } else if (b < f.seg[4]) {   // dW_q | db_q of one head: [dh, 2 d + 1], over the head's ldz columns
    b -= f.seg[3];
    const int nm = up_div(f.dh, FT), nn = up_div(2 * d + 1, FT);
    const int h = b / (nm * nn * nk), t = b - h * nm * nn * nk;
    const int kb = t / (nm * nn), u = t - kb * nm * nn;
    const int m0 = (u / nn) * FT, n0 = (u % nn) * FT;
    const int k0 = kb * FOLD_K, k1 = min(f.ldz, k0 + FOLD_K);
    fold_tile<false, false>(
        smem, acc, m0, f.dh, n0, 2 * d + 1, k0, k1,
        [&](int m, int k) { const int c = z_col(f, k); return c < 0 ? 0.f : __ldg(f.wk + (int64_t)(h * f.dh + m) * f.dkv + c); },
        [&](int k, int n) {
          const float* col = f.T + h * f.ldz + k;
          if (n < d) return __ldg(col + (int64_t)n * HL);
          const float s = __ldg(col + (int64_t)d * HL);
          return n < 2 * d ? s * time_encode(0.f, __ldg(f.time_b + n - d), 0.f) : s;
        });
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const int m = m0 + ty + 8 * i, n = n0 + tx;
      if (m >= f.dh || n > 2 * d) continue;
      if (n < 2 * d) atomicAdd(f.g_wq + (int64_t)(h * f.dh + m) * 2 * d + n, acc[i] * f.scale);
      else atomicAdd(f.g_bq + h * f.dh + m, acc[i] * f.scale);
    }
  } else if (b < f.seg[5]) {   // the roots' own encoding Phi(0): d/db = -sin(b) times the gradient of Phi(0), 32 rows of wAp per block
    const int c0 = (b - f.seg[4]) * 32, c1 = min(HL, c0 + 32);
    for (int j = threadIdx.x; j < d; j += blockDim.x) {
      float g = 0.f;
#pragma unroll 8
      for (int c = c0; c < c1; ++c) g = fmaf(__ldg(f.T + (int64_t)d * HL + c), __ldg(f.wAp + (int64_t)c * d + j), g);
      const double t = -(double)sinf(f.time_b[j]) * (double)g;
      if (t != 0.0) atomicAdd(f.tg + d + j, t);
    }
  } else if (b < f.seg[6]) {   // time-encoder sums of TG_ROWS blocks of the attention backward
    const int r0 = (b - f.seg[5]) * TG_ROWS, r1 = min(f.parts, r0 + TG_ROWS);
    for (int e = threadIdx.x; e < 2 * d; e += blockDim.x) {
      double t = 0.0;
#pragma unroll 8
      for (int r = r0; r < r1; ++r) t += __ldg(f.tg_part + (int64_t)r * 2 * d + e);
      if (t != 0.0) atomicAdd(f.tg + e, t);
    }
  } else {   // dW_o's memory columns
    const int m = (b - f.seg[6]) * 8 + ty;
    if (m >= d) return;
    for (int j = tx; j < d; j += 32) f.g_wo[(int64_t)m * 2 * d + d + j] = __ldg(f.dOut + (int64_t)m * f.ldc + HL + j);
  }
}

FoldArgs fold_args(tgnn_ctx* ctx) {
  const tgnn_config& c = ctx->cfg;
  const ParamLayout& L = ctx->L;
  Workspace& w = ctx->ws;
  float *P = ctx->params, *G = w.grads;
  FoldArgs f = {};
  f.d = c.d; f.de = c.d_e; f.H = c.heads; f.dh = c.d / c.heads; f.dkv = (int)L.dkv; f.ldz = ctx->ldz; f.ldc = ctx->ldc;
  f.scale = (float)(1.0 / sqrt((double)f.dh));
  f.time_b = P + L.time_b; f.wq = P + L.wq; f.bq = P + L.bq; f.wk = P + L.wk; f.wv = P + L.wv; f.bv = P + L.bv; f.wo = P + L.wo;
  f.wA = w.wA; f.wAp = w.wAp; f.cA = w.cA; f.cq = w.cq; f.wB = w.wB; f.dOut = w.dOut; f.T = w.dT;
  f.g_wq = G + L.wq; f.g_bq = G + L.bq; f.g_wk = G + L.wk; f.g_wv = G + L.wv; f.g_bv = G + L.bv; f.g_wo = G + L.wo;
  f.tg = w.tg_acc; f.tg_part = w.tg_part;
  return f;
}

AttnArgs attn_args(tgnn_ctx* ctx, const int32_t* nodes, const double* times, int n, const int32_t* nbr, const int32_t* eid,
                   const double* ts, const int32_t* cnt) {
  const tgnn_config& c = ctx->cfg;
  Workspace& w = ctx->ws;
  AttnArgs a = {};
  a.memory = ctx->memory; a.efeat = ctx->efeat;
  a.time_w = ctx->params + ctx->L.time_w; a.time_b = ctx->params + ctx->L.time_b;
  a.nodes = nodes; a.nbr = nbr; a.eid = eid; a.cnt = cnt; a.times = times; a.ts = ts;
  a.n = n; a.d = c.d; a.de = c.d_e; a.k = c.k; a.H = c.heads; a.ldz = ctx->ldz; a.ldc = ctx->ldc;
  a.N = c.num_nodes; a.E = ctx->num_events; a.status = w.status;
  a.qp = w.qp; a.prob = w.alpha; a.cat = w.cat; a.dcat = w.dcat; a.ldd = c.heads * ctx->ldz + c.d; a.dqp = w.dqp;
  a.dMemU = w.dMemU; a.upd_rows = ctx->copies.rows; a.copy_mask = ctx->copies.n - 1; a.tg_part = w.tg_part;
  return a;
}

// Two heads per warp share a slot's gathered row; an odd number of heads takes them one by one.  Tables that are not aligned
// to pieces of memory columns or pairs of feature columns (odd) are read by one kernel for all shapes.
bool odd_tables(const tgnn_ctx* ctx) {
  const tgnn_config& c = ctx->cfg;
  return ((uintptr_t)ctx->memory & 15) != 0 || (c.d_e > 0 && c.feat_dtype == TGNN_F32 && ((uintptr_t)ctx->efeat & 7) != 0);
}
int heads_per_warp(const tgnn_config& c, bool odd) { return c.heads % 2 == 0 && !odd ? 2 : 1; }
int slots_per_batch(const tgnn_config& c, bool odd) {
  if (c.d > 128 || heads_per_warp(c, odd) != 2) return 10;
  return c.k <= 5 ? 5 : c.k > 10 && c.k <= 16 ? 16 : 10;
}
AttnKernel pick_kernel(const tgnn_config& c, bool odd, bool bwd) {
  const int de = c.d_e;
  const bool bf16 = c.feat_dtype == TGNN_BF16;
  if (odd) return attn_kernel_words(de, bf16, bwd);
  if (heads_per_warp(c, odd) == 1) return c.d <= 128 ? attn_kernel<1, 10, true, 1>(de, bf16, bwd) : attn_kernel<1, 10, true, 2>(de, bf16, bwd);
  if (c.d > 128) return attn_kernel<2, 10, true, 2>(de, bf16, bwd);
  if (slots_per_batch(c, odd) == 16) return attn_kernel<2, 16, false, 1>(de, bf16, bwd);
  if (c.k > 10) return attn_kernel<2, 10, true, 1>(de, bf16, bwd);
  return slots_per_batch(c, odd) == 5 ? attn_kernel<2, 5, false, 1>(de, bf16, bwd) : attn_kernel<2, 10, false, 1>(de, bf16, bwd);
}
size_t attn_smem(const tgnn_config& c, bool odd) {
  const int words = slots_per_batch(c, odd) * staged_words(c.d, c.d_e, c.feat_dtype == TGNN_BF16 ? X_BF16 : X_F32);
  return (size_t)words * 4;
}
int attn_grid(const tgnn_ctx* ctx, int n, bool bwd) {
  const bool odd = odd_tables(ctx);
  const int items = n * (ctx->cfg.heads / heads_per_warp(ctx->cfg, odd));
  const int cap = 148 * ctx->attn_warps[odd][bwd];
  return items < cap ? items : cap;
}

// (of a warp, spread evenly where the warps do not fill the machine; 2 KB: more than the kernels' static scratch)
size_t attn_share(const tgnn_ctx* ctx, int n, bool bwd) {
  const bool odd = odd_tables(ctx);
  const int grid = attn_grid(ctx, n, bwd);
  const size_t need = attn_smem(ctx->cfg, odd);
  return grid < 148 * ctx->attn_warps[odd][bwd] ? even_share(grid, need, 2048, 48 * 1024) : need;
}

}  // namespace

// The query-side form keeps at most two pieces of four memory columns and four pairs of feature columns per lane (d and d_e
// up to 256).  Its cost grows with the number of heads (2 multiply-adds per head, slot and column, and root rows of
// heads x columns), where projecting every slot's key and value (k_embed.cu) does not: beyond eight heads that form is kept.
bool attn_query_side(const tgnn_config& c) { return c.model == TGNN_MODEL_TGN && c.heads <= 8 && c.d_e <= 256; }

// How many warps of the two kernels fit an SM.  The workspace has room for the time-encoder sums of as many backward warps as
// fit with aligned tables, asked for when the context is created; for other tables (whose kernel is only looked up when one
// of them is bound) no more are launched.
int attn_setup(tgnn_ctx* ctx) {
  const bool odd = odd_tables(ctx);
  if (ctx->attn_warps[odd][1] > 0) return TGNN_OK;
  for (int bwd = 0; bwd < 2; ++bwd) {
    AttnKernel k = pick_kernel(ctx->cfg, odd, bwd != 0);
    int warps = 0;
    // (the limit is a property of the kernel, not of the context: one value, the most that any shape needs)
    if (cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, 48 * 1024) != cudaSuccess ||
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&warps, k, 32, attn_smem(ctx->cfg, odd)) != cudaSuccess || warps < 1) {
      cudaGetLastError();
      return TGNN_ECUDA;
    }
    ctx->attn_warps[odd][bwd] = odd && bwd && warps > ctx->attn_warps[0][1] ? ctx->attn_warps[0][1] : warps;
  }
  return TGNN_OK;
}

int launch_fold_weights(tgnn_ctx* ctx, cudaStream_t s) {
  FoldArgs f = fold_args(ctx);
  f.seg[1] = f.H * up_div(f.ldz, FT) * up_div(2 * f.d + 1, FT);
  f.seg[2] = f.seg[1] + f.H * up_div(f.d, FT) * up_div(f.ldz, FT);
  {
    KernelScope scope__(ctx, "fold_weights", s);
    fold_weights_kernel<<<f.seg[2] + up_div(f.d, 8), 256, 0, s>>>(f);
  }
  TGNN_LAUNCH_OK(ctx, "fold_weights");
  return TGNN_OK;
}

// of_out: what follows from the gradient of wB and the attention backward (dW_v, dW_o, the time encoder); otherwise what follows from
// that of wA (dW_k, dW_q), which is ready later.
int launch_unfold_grads(tgnn_ctx* ctx, bool of_out, cudaStream_t s) {
  FoldArgs f = fold_args(ctx);
  const int nk = up_div(f.ldz + 1, FOLD_K);
  f.parts = attn_grid(ctx, ctx->e_n, true);
  const int o = of_out ? 1 : 0, t = 1 - o;   // (segments of the other part are empty)
  f.seg[1] = o * f.H * up_div(f.dh, FT) * up_div(f.ldz + 1, FT);
  f.seg[2] = f.seg[1] + t * f.H * up_div(f.dh, FT) * up_div(f.ldz, FT);
  f.seg[3] = f.seg[2] + o * f.H * up_div(f.d, FT) * up_div(f.dh, FT) * nk;
  f.seg[4] = f.seg[3] + t * f.H * up_div(f.dh, FT) * up_div(2 * f.d + 1, FT) * nk;
  f.seg[5] = f.seg[4] + t * up_div(f.H * f.ldz, 32);
  f.seg[6] = f.seg[5] + o * up_div(f.parts, TG_ROWS);
  {
    KernelScope scope__(ctx, "unfold_grads", s);
    unfold_grads_kernel<<<f.seg[6] + o * up_div(f.d, 8), 256, 0, s>>>(f);
  }
  TGNN_LAUNCH_OK(ctx, "unfold_grads");
  return TGNN_OK;
}

int launch_attn_fwd(tgnn_ctx* ctx, const int32_t* nodes, const double* times, int n, const int32_t* nbr, const int32_t* eid,
                    const double* ts, const int32_t* cnt, cudaStream_t s) {
  const AttnArgs a = attn_args(ctx, nodes, times, n, nbr, eid, ts, cnt);
  {
    KernelScope scope__(ctx, "attention_fwd", s);
    const bool odd = odd_tables(ctx);
    launch_link(ctx, pick_kernel(ctx->cfg, odd, false), dim3(attn_grid(ctx, n, false)), dim3(32), attn_share(ctx, n, false), s, 1, a);
  }
  TGNN_LAUNCH_OK(ctx, "attention_fwd");
  return TGNN_OK;
}

int launch_attn_bwd(tgnn_ctx* ctx, bool have_update, cudaStream_t s) {
  AttnArgs a = attn_args(ctx, ctx->e_nodes, ctx->e_times, ctx->e_n, ctx->e_nbr, ctx->e_eid, ctx->e_ts, ctx->e_cnt);
  a.node2slot = have_update ? ctx->ws.node2slot : nullptr;
  {
    KernelScope scope__(ctx, "attention_bwd", s);
    const bool odd = odd_tables(ctx);
    launch_link(ctx, pick_kernel(ctx->cfg, odd, true), dim3(attn_grid(ctx, a.n, true)), dim3(32), attn_share(ctx, a.n, true), s, 1, a);
  }
  TGNN_LAUNCH_OK(ctx, "attention_bwd");
  return TGNN_OK;
}

}  // namespace tgnn
