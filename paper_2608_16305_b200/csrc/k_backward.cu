// Step (6): masked link-prediction loss (Eq. 13), exact backward of steps (4)-(5),
// gradient norm g_r and the Adam update.
#include "tgnn_internal.cuh"
#include "tgnn_device.cuh"

namespace tgnn {
namespace {

constexpr unsigned FULL = 0xffffffffu;

// cat1[p] = [h_src || h_dst] for p < nq (positive pairs), [h_src || h_neg] for p >= nq.
__global__ void __launch_bounds__(256) head_gather_kernel(const float* __restrict__ h, int nq, int d,
                                                          float* __restrict__ cat1) {
  const int64_t total = (int64_t)2 * nq * 2 * d;
  for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < total; e += (int64_t)gridDim.x * blockDim.x) {
    const int p = (int)(e / (2 * d)), q = (int)(e % (2 * d));
    const int j = p < nq ? p : p - nq;
    const int row = q < d ? j : (p < nq ? nq + j : 2 * nq + j);
    cat1[e] = h[(int64_t)row * d + (q < d ? q : q - d)];
  }
}

// One warp per target event: both scores, the event's loss term, d loss / d score, then
// hid1 is overwritten by d loss / d pre1.  Accumulates dw_2, db_2 and the loss.
__global__ void __launch_bounds__(256) head_loss_kernel(float* __restrict__ hid1, const float* __restrict__ w2,
                                                        const float* __restrict__ b2,
                                                        const uint8_t* __restrict__ loss_mask, int nq, int d,
                                                        float* __restrict__ g_w2, float* __restrict__ g_b2,
                                                        float* __restrict__ loss_acc, uint8_t* __restrict__ hid_gate) {
  extern __shared__ float s_gw2[];  // [d]
  __shared__ float s_msum;
  __shared__ float s_gb2, s_loss;
  const int lane = threadIdx.x & 31;
  for (int q = threadIdx.x; q < d; q += blockDim.x) s_gw2[q] = 0.f;
  if (threadIdx.x == 0) { s_msum = 0.f; s_gb2 = 0.f; s_loss = 0.f; }
  __syncthreads();
  {  // every block counts the whole mask (a few KB)
    int c = 0;
    for (int j = threadIdx.x; j < nq; j += blockDim.x) c += loss_mask ? (loss_mask[j] != 0) : 1;
    for (int o = 16; o > 0; o >>= 1) c += __shfl_xor_sync(FULL, c, o);
    if (lane == 0 && c) atomicAdd(&s_msum, (float)c);
  }
  __syncthreads();
  const float msum = s_msum;
  const int warps = (gridDim.x * blockDim.x) >> 5;
  for (int j = (blockIdx.x * blockDim.x + threadIdx.x) >> 5; j < nq; j += warps) {
    const float m = (loss_mask ? (loss_mask[j] != 0) : 1) ? 1.f : 0.f;
    const float wj = msum > 0.f ? m / msum : 0.f;
    float* hp = hid1 + (int64_t)j * d;
    float* hn = hid1 + (int64_t)(nq + j) * d;
    float sp = 0.f, sn = 0.f;
    for (int q = lane; q < d; q += 32) {
      sp = fmaf(w2[q], hp[q], sp);
      sn = fmaf(w2[q], hn[q], sn);
    }
    for (int o = 16; o > 0; o >>= 1) {
      sp += __shfl_xor_sync(FULL, sp, o);
      sn += __shfl_xor_sync(FULL, sn, o);
    }
    sp += b2[0];
    sn += b2[0];
    const float dsp = wj != 0.f ? -wj * sigmoidf_(-sp) : 0.f;   // (an event without weight leaves nothing, whatever its score)
    const float dsn = wj != 0.f ? wj * sigmoidf_(sn) : 0.f;
    if (lane == 0 && wj != 0.f) {
      atomicAdd(&s_loss, wj * (softplusf_(-sp) + softplusf_(sn)));
      atomicAdd(&s_gb2, dsp + dsn);
    }
    for (int q = lane; q < d; q += 32) {
      const float a = hp[q], b = hn[q];
      if (wj != 0.f) atomicAdd(&s_gw2[q], dsp * a + dsn * b);
      hp[q] = a > 0.f ? dsp * w2[q] : 0.f;
      hn[q] = b > 0.f ? dsn * w2[q] : 0.f;
      hid_gate[(int64_t)j * d + q] = a > 0.f;
      hid_gate[(int64_t)(nq + j) * d + q] = b > 0.f;
    }
  }
  __syncthreads();
  for (int q = threadIdx.x; q < d; q += blockDim.x)
    if (s_gw2[q] != 0.f) atomicAdd(&g_w2[q], s_gw2[q]);
  if (threadIdx.x == 0) {
    if (s_gb2 != 0.f) atomicAdd(g_b2, s_gb2);
    if (s_loss != 0.f) atomicAdd(loss_acc, s_loss);
  }
}

// d loss / d pre_o = ReLU'(h) * d loss / d h, where dh collects the head's input gradients.
__global__ void __launch_bounds__(256) dh_kernel(const float* __restrict__ dcat1, const float* __restrict__ h, int nq,
                                                 int d, float* __restrict__ dpre_o, int relu_out) {
  const int64_t total = (int64_t)3 * nq * d;
  for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < total; e += (int64_t)gridDim.x * blockDim.x) {
    const int i = (int)(e / d), q = (int)(e % d);
    float g;
    if (i < nq)
      g = dcat1[(int64_t)i * 2 * d + q] + dcat1[(int64_t)(nq + i) * 2 * d + q];
    else if (i < 2 * nq)
      g = dcat1[(int64_t)(i - nq) * 2 * d + d + q];
    else
      g = dcat1[(int64_t)(i - nq) * 2 * d + d + q];
    dpre_o[e] = (!relu_out || h[e] > 0.f) ? g : 0.f;
  }
}

// The whole link-prediction head for EV target events (2 EV pairs: positive, negative) in one block: gather [h_a || h_b],
// hidden layer, scores, the masked loss (Eq. 13), and the backward pass down to d loss / d pre_o of the 3 EV embedding
// rows involved.  Also leaves what the leaves of the chain need: cat1 and d loss / d pre1 (for dW_1, db_1), the hidden
// gates, and the sums for dw_2, db_2 and the loss.  Rows of hsT: sources (and a row of zeros if EV is odd), destinations, negatives.
// relu_out: the embedding rows are outputs of a ReLU layer (attention model) and dpre_o is masked by it; otherwise
// dpre_o is the plain gradient with respect to the embedding rows.
// With a few events per SM there is nothing to hide a round trip behind, and the multiply-adds are few: what bounds the kernel
// is the number of instructions around them and the chain of its phases.  So
//   W_1 does not go through shared memory: every element is used by one thread, for all rows at once, and read where
//   neighbouring lanes read neighbouring words, a few steps ahead (W_1 transposed in the forward sweep, prepared beside the chain);
//   a lane owns four hidden units, then four input columns: eight multiply-adds of pairs per 16-byte load from shared memory
//   (a unit per lane, 1 024 threads: 19.7 us, bound by these loads; two, 512 threads: 21.3, by instructions around them);
//   the contraction is cut into as many slices as the warps make, which shared memory adds up;
//   loops are not unrolled where it does not pay: an instruction that runs once comes from L2 (unrolled throughout, 25 us).
// Two blocks fit an SM, but share its issue slots: the events per block are those that leave the fewest blocks on the fullest SM.
// 600 events, d = 100: 13.5 us (18.4 with W_1 in shared memory and two teams of 512 threads);
// 1 237 events, d = 128: 23.8 (37).
constexpr int HR_THREADS = 256, HR_WARPS = HR_THREADS / 32;
__host__ __device__ inline int hr_slices(int cols) { return HR_WARPS / ((cols / 4 + 31) / 32); }   // contraction slices when a lane has four columns
template <int EV>
struct HeadRows {
  static constexpr int EVP = (EV + 1) & ~1, R = EVP + 2 * EV, P = 2 * EV;    // rows of hsT, pairs
  // the shared arrays in words, each from a 16-byte boundary (d is a multiple of 4)
  static __host__ __device__ int up4(int x) { return (x + 3) & ~3; }
  static __host__ __device__ int rows(int d) { return up4(R * (d + 1)); }
  static __host__ __device__ int pairs(int d) { return up4(P * (d + 1)); }
  static size_t smem(int d) {
    const int fwd = hr_slices(d) * R * d, bwd = hr_slices(2 * d) * P * 2 * d;
    return (size_t)(rows(d) + pairs(d) + P * d + 2 * d + (fwd > bwd ? fwd : bwd)) * sizeof(float);
  }
};
inline int head_rows_events(int n_q) {
  int best = 4, least = 1 << 30;
  for (const int ev : {2, 4, 5, 6}) {   // (a block takes as long as 8 events more)
    const int cost = ((n_q + ev - 1) / ev + 147) / 148 * (8 + ev);
    if (cost < least) { least = cost; best = ev; }
  }
  return best;
}
__device__ __forceinline__ float4 ldg4(const float* p, bool vec) {
  if (vec) return __ldg(reinterpret_cast<const float4*>(p));
  return make_float4(__ldg(p), __ldg(p + 1), __ldg(p + 2), __ldg(p + 3));
}
__device__ __forceinline__ float4 add4(const float4& a, const float4& b) { return make_float4(a.x + b.x, a.y + b.y, a.z + b.z, a.w + b.w); }
// acc[i][r] += x[i] * v[2 r], v[2 r + 1] for N pairs of rows in shared memory (W: 16-byte aligned)
template <bool W, int N>
__device__ __forceinline__ void fma_rows(f32x2 (&acc)[4][N], const float4& x, const float* v) {
  const f32x2 xs[4] = {pack2(x.x, x.x), pack2(x.y, x.y), pack2(x.z, x.z), pack2(x.w, x.w)};
  f32x2 q[N];
#pragma unroll
  for (int r = 0; r < N; r += 2) {
    if (W && r + 1 < N) {
      const ulonglong2 t = *reinterpret_cast<const ulonglong2*>(v + 2 * r);
      q[r] = t.x; q[r + 1] = t.y;
    } else {
      q[r] = *reinterpret_cast<const f32x2*>(v + 2 * r);
      if (r + 1 < N) q[r + 1] = *reinterpret_cast<const f32x2*>(v + 2 * r + 2);
    }
  }
#pragma unroll
  for (int r = 0; r < N; ++r)
#pragma unroll
    for (int i = 0; i < 4; ++i) acc[i][r] = fma2(xs[i], q[r], acc[i][r]);
}
// the sums of four neighbouring columns, a row of out (pitch words) per row
template <int N>
__device__ __forceinline__ void store_rows(float* out, int pitch, const f32x2 (&acc)[4][N]) {
#pragma unroll
  for (int r = 0; r < N; ++r) {
    float4 lo, hi;
    unpack2(acc[0][r], lo.x, hi.x); unpack2(acc[1][r], lo.y, hi.y); unpack2(acc[2][r], lo.z, hi.z); unpack2(acc[3][r], lo.w, hi.w);
    *reinterpret_cast<float4*>(out + 2 * r * pitch) = lo;
    *reinterpret_cast<float4*>(out + (2 * r + 1) * pitch) = hi;
  }
}

template <int EV>
__global__ void __launch_bounds__(HR_THREADS, 2) head_rows_kernel(const float* __restrict__ h, const float* __restrict__ W1,
                                                                  const float* __restrict__ WT,
                                                                  const float* __restrict__ b1, const float* __restrict__ w2,
                                                                  const float* __restrict__ b2,
                                                                  const uint8_t* __restrict__ loss_mask, int nq, int d,
                                                                  float* __restrict__ cat1, float* __restrict__ dpre1,
                                                                  uint8_t* __restrict__ hid_gate, float* __restrict__ dpre_o,
                                                                  float* __restrict__ g_w2, float* __restrict__ g_b2,
                                                                  float* __restrict__ loss_acc, int relu_out) {
  using HR = HeadRows<EV>;
  constexpr int EVP = HR::EVP, R = HR::R, P = HR::P, T = HR_THREADS, FD = EV > 5 ? 2 : 3, BD = 5;   // FD, BD: pieces of W_1 in flight per lane and half
  constexpr bool WR = R % 4 == 0 && EVP % 4 == 0, WP = P % 4 == 0;
  extern __shared__ __align__(16) float sm[];
  __shared__ float s_msum, s_ds[P], s_loss[P];
  const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5, d4 = d >> 2;
  const int S = hr_slices(d), JS = hr_slices(2 * d);
  float* hsT = sm;                     // [d + 1][R] embedding rows, transposed, and a row of zeros (the pad row's values reach no result)
  float* dh1T = hsT + HR::rows(d);     // [d + 1][P] d loss / d pre1, and a row of zeros
  float* actT = dh1T + HR::pairs(d);   // [d][P] hidden units of the pairs
  float* b1s = actT + P * d;           // [d]
  float* w2s = b1s + d;                // [d]
  float* red = w2s + d;                // [slice][row][hidden unit], then [slice][pair][column]
  const float4 none = make_float4(0.f, 0.f, 0.f, 0.f);
  const int zero = link_wait(), ev0 = blockIdx.x * EV + zero;
  link_release();
  WT += zero;   // (written within the step, as h is)
  // forward: four hidden units from j on and a slice of the columns, of both halves of W_1.  A piece is asked for where the one
  // before it in the same registers has been used: no moves, which would wait for it.
  const int HW = (d4 + 31) >> 5, fs = wid / HW, j = 4 * (32 * (wid - fs * HW) + lane);   // (WT's rows are d words: d is a multiple of 4)
  const bool fwd = fs < S && j < d;
  const int c0 = fwd ? d * fs / S : 0, c1 = fwd ? d * (fs + 1) / S : 0;
  const float *wpa = WT + c0 * d + j, *wpo = wpa + d * d;
  float4 xa[FD], xo[FD];   // source half, other half
  const auto ask = [&](int c, int u) {
    xa[u] = xo[u] = none;
    if (c < c1) { xa[u] = __ldg(reinterpret_cast<const float4*>(wpa)); xo[u] = __ldg(reinterpret_cast<const float4*>(wpo)); }
    wpa += d; wpo += d;
  };
#pragma unroll
  for (int u = 0; u < FD; ++u) ask(c0 + u, u);
  const bool hvec = ((uintptr_t)h & 15) == 0;
#pragma unroll 1
  for (int e = tid; e < 3 * EV * d4; e += T) {
    const int r = e / d4, q = 4 * (e - r * d4);
    const int blk = r / EV, ev = ev0 + r - blk * EV;
    float4 v = none;
    if (ev < nq) {
      v = ldg4(h + ((int64_t)blk * nq + ev) * d + q, hvec);
      float* o = cat1 + (int64_t)(blk == 2 ? nq + ev : ev) * 2 * d + (blk == 0 ? 0 : d) + q;
      *reinterpret_cast<float4*>(o) = v;
      if (blk == 0) *reinterpret_cast<float4*>(o + (int64_t)nq * 2 * d) = v;
    }
    float* t = hsT + q * R + r + (blk > 0 ? EVP - EV : 0);
    t[0] = v.x; t[R] = v.y; t[2 * R] = v.z; t[3 * R] = v.w;
    if (EVP > EV && r == 0) { t[EV] = 0.f; t[R + EV] = 0.f; t[2 * R + EV] = 0.f; t[3 * R + EV] = 0.f; }
  }
  if (tid < d) { b1s[tid] = __ldg(b1 + tid); w2s[tid] = __ldg(w2 + tid); }   // (d <= 256)
  if (tid < R) hsT[d * R + tid] = 0.f;
  if (tid < P) dh1T[d * P + tid] = 0.f;
  if (tid == 0) s_msum = loss_mask ? 0.f : (float)nq;
  __syncthreads();
  if (loss_mask) {  // every block counts the whole mask (a few KB)
    int c = 0;
#pragma unroll 4
    for (int i = tid; i < nq; i += T) c += loss_mask[i] != 0;
    c = __reduce_add_sync(FULL, c);
    if (lane == 0 && c) atomicAdd(&s_msum, (float)c);   // (whole numbers below 2^24: exact in any order)
  }
  {  // hidden layer: the source rows serve the positive and the negative pair of their event, so their part is formed once
    f32x2 as[4][EVP / 2] = {}, ao[4][EV] = {};
#pragma unroll 1
    for (int c = c0; c < c1; c += FD)
#pragma unroll
      for (int u = 0; u < FD; ++u) {
        const float* hp = hsT + (c + u < c1 ? c + u : d) * R;
        fma_rows<WR>(as, xa[u], hp);
        fma_rows<WR>(ao, xo[u], hp + EVP);
        ask(c + FD + u, u);
      }
    if (fwd) {
      store_rows(red + fs * R * d + j, d, as);
      store_rows(red + (fs * R + EVP) * d + j, d, ao);
    }
  }
  // backward: four input columns from c2 on and a slice of the hidden units
  const int CW = (2 * d4 + 31) >> 5, bs = wid / CW, c2 = 4 * (32 * (wid - bs * CW) + lane);
  const bool bwd = bs < JS && c2 < 2 * d, wvec = ((uintptr_t)W1 & 15) == 0;
  const int j0 = bwd ? d * bs / JS : 0, j1 = bwd ? d * (bs + 1) / JS : 0;
  const float* wc = W1 + (int64_t)j0 * 2 * d + c2;
  float4 xb[BD];
  const auto ask1 = [&](int i, int u) {
    xb[u] = i < j1 ? ldg4(wc, wvec) : none;
    wc += 2 * d;
  };
#pragma unroll
  for (int u = 0; u < BD; ++u) ask1(j0 + u, u);
  __syncthreads();
  // hidden units of the pairs: the sums over the slices, bias, ReLU
#pragma unroll 1
  for (int e = tid; e < P * d4; e += T) {
    const int p = e / d4, q = 4 * (e - p * d4);
    const float *rs = red + (p < EV ? p : p - EV) * d + q, *ro = red + (EVP + p) * d + q;   // the pair's second row: destination or negative
    float4 x = none, y = none;
#pragma unroll 4
    for (int z = 0; z < S; ++z) {
      x = add4(x, *reinterpret_cast<const float4*>(rs + z * R * d));
      y = add4(y, *reinterpret_cast<const float4*>(ro + z * R * d));
    }
    x = add4(add4(x, y), *reinterpret_cast<const float4*>(b1s + q));
    float* t = actT + q * P + p;
    t[0] = fmaxf(x.x, 0.f); t[P] = fmaxf(x.y, 0.f); t[2 * P] = fmaxf(x.z, 0.f); t[3 * P] = fmaxf(x.w, 0.f);
  }
  __syncthreads();
#pragma unroll 1
  for (int p = wid; p < P; p += HR_WARPS) {   // scores and loss terms: one warp per pair
    const float msum = s_msum;
    const int half = p / EV, ev = ev0 + p - half * EV;
    const float m = ev < nq && (loss_mask ? (loss_mask[ev] != 0) : true) ? 1.f : 0.f;
    float sc = 0.f;
#pragma unroll 1
    for (int q = lane; q < d; q += 32) sc = fmaf(w2s[q], actT[q * P + p], sc);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) sc += __shfl_xor_sync(FULL, sc, o);
    sc += __ldg(b2);
    const float wj = msum > 0.f ? m / msum : 0.f;
    const float z = half == 0 ? -sc : sc;
    if (lane == 0) {
      s_ds[p] = wj != 0.f ? (half == 0 ? -wj : wj) * sigmoidf_(z) : 0.f;   // (an event without weight leaves nothing, whatever its score)
      s_loss[p] = wj != 0.f ? wj * softplusf_(z) : 0.f;
    }
  }
  __syncthreads();
  // d loss / d pre1, and the block's share of dw_2, db_2 and the loss
#pragma unroll 1
  for (int e = tid; e < P * d4; e += T) {
    const int p = e / d4, q = 4 * (e - p * d4), half = p / EV, ev = ev0 + p - half * EV;
    const float* t = actT + q * P + p;
    const float ds = s_ds[p];
    const float4 w = *reinterpret_cast<const float4*>(w2s + q);
    const bool b0 = t[0] > 0.f, g1 = t[P] > 0.f, g2 = t[2 * P] > 0.f, g3 = t[3 * P] > 0.f;
    const float4 v = make_float4(b0 ? ds * w.x : 0.f, g1 ? ds * w.y : 0.f, g2 ? ds * w.z : 0.f, g3 ? ds * w.w : 0.f);
    float* o = dh1T + q * P + p;
    o[0] = v.x; o[P] = v.y; o[2 * P] = v.z; o[3 * P] = v.w;
    if (ev < nq) {
      const int64_t at = ((int64_t)half * nq + ev) * d + q;
      *reinterpret_cast<float4*>(dpre1 + at) = v;
      *reinterpret_cast<uchar4*>(hid_gate + at) = make_uchar4(b0, g1, g2, g3);
    }
  }
  if (tid < d) {
    float t = 0.f;
#pragma unroll
    for (int p = 0; p < P; ++p) t += s_ds[p] != 0.f ? s_ds[p] * actT[tid * P + p] : 0.f;   // (events without weight are left out whatever their rows hold)
    if (t != 0.f) atomicAdd(&g_w2[tid], t);
  }
  if (tid == T - 1) {
    float l = 0.f, g = 0.f;
#pragma unroll
    for (int p = 0; p < P; ++p) { l += s_loss[p]; g += s_ds[p]; }
    if (g != 0.f) atomicAdd(g_b2, g);
    if (l != 0.f) atomicAdd(loss_acc, l);
  }
  __syncthreads();
  {  // input gradient of four columns of [h_a || h_b] for all pairs
    f32x2 acc[4][P / 2] = {};
#pragma unroll 1
    for (int i = j0; i < j1; i += BD)
#pragma unroll
      for (int u = 0; u < BD; ++u) {
        fma_rows<WP>(acc, xb[u], dh1T + (i + u < j1 ? i + u : d) * P);
        ask1(i + BD + u, u);
      }
    if (bwd) store_rows(red + bs * P * 2 * d + c2, 2 * d, acc);
  }
  __syncthreads();
  // the pairs folded into the embedding rows (a source row collects its positive and its negative pair)
#pragma unroll 1
  for (int e = tid; e < 3 * EV * d4; e += T) {
    const int r = e / d4, q = 4 * (e - r * d4);
    const int blk = r / EV, e4 = r - blk * EV, ev = ev0 + e4;
    if (ev >= nq) continue;
    const float* rz = red + (blk == 2 ? EV + e4 : e4) * 2 * d + (blk == 0 ? 0 : d) + q;
    const int step = blk == 0 ? EV * 2 * d : P * 2 * d, n = blk == 0 ? 2 * JS : JS;   // (the two pairs of a source row are half a slice apart)
    float4 g = none;
#pragma unroll 4
    for (int z = 0; z < n; ++z) g = add4(g, *reinterpret_cast<const float4*>(rz + z * step));
    if (relu_out) {
      const float* t = hsT + q * R + r + (blk > 0 ? EVP - EV : 0);
      g = make_float4(t[0] > 0.f ? g.x : 0.f, t[R] > 0.f ? g.y : 0.f, t[2 * R] > 0.f ? g.z : 0.f, t[3 * R] > 0.f ? g.w : 0.f);
    }
    *reinterpret_cast<float4*>(dpre_o + ((int64_t)blk * nq + ev) * d + q) = g;
  }
}

// W_1 [d][2d] -> WT[c2][j] = W_1[j][c2] (row pitch ldw): both halves transposed, the layout head_tile_kernel keeps in
// shared memory.  A warp owns four hidden units, its lanes walk the columns.
__global__ void __launch_bounds__(256) prep_head_wt_kernel(const float* __restrict__ W1, int d, int ldw, float* __restrict__ WT) {
  const int lane = threadIdx.x & 31, wid = (blockIdx.x * blockDim.x + threadIdx.x) >> 5, nw = (gridDim.x * blockDim.x) >> 5;
  for (int j4 = wid; j4 < (d >> 2); j4 += nw) {
    const float* w0 = W1 + (int64_t)(4 * j4) * 2 * d;
    for (int c2 = lane; c2 < 2 * d; c2 += 32) {
      float4 v;
      v.x = __ldg(w0 + c2); v.y = __ldg(w0 + 2 * d + c2); v.z = __ldg(w0 + 4 * d + c2); v.w = __ldg(w0 + 6 * d + c2);
      *reinterpret_cast<float4*>(WT + (size_t)c2 * ldw + 4 * j4) = v;
    }
  }
}

// The same head on tiles of TE events per block with register-blocked products (the form used when the model's
// width allows: d a multiple of 4 and both halves of W_1, transposed, fit in shared memory beside the tile).
// Rows of a tile: [0, TE) sources, [TE, 2TE) destinations, [2TE, 3TE) negatives; pairs: [0, TE) positive, [TE, 2TE)
// negative.  Shared memory, all c-major / j-major so that the inner loops read 16 bytes per operand:
//   WaT[c][j] = W_1[j][c], WbT[c][j] = W_1[j][d + c]   (pitch LDW)
//   HT[c][r]   embedding rows, transposed             (pitch RP)
//   PT[j][r]   W_1a h_r (sources) or W_1b h_r         (pitch RP)
//   D1T[j][p]  d loss / d pre1, transposed            (pitch PP)
// Hidden layer: a thread owns a 4 x 4 block of (hidden unit, row) and walks the d input columns (two 16-byte loads
// per 16 FMAs).  Input gradient: a thread owns 4 events x {positive, negative} x 4 input columns and walks the hidden
// units four at a time; it holds both pairs of its two events, so the source rows' two contributions meet in
// registers.  Scores: a lane per pair over slices of the hidden units, then a thread per hidden unit over the pairs (a warp per pair with its
// lanes over the units met four banks of shared memory, took three rounds and added up by atomics there: 14 000 of the kernel's
// 61 000 cycles).  4 000 events, step of the large workload: 405 -> 396 us with this and the rows loaded at once.
template <int TE>
struct HeadTile {
  // (pitches: odd multiples of four words, so that lanes that walk the columns meet eight banks, not four)
  static constexpr int ROWS = 3 * TE, PAIRS = 2 * TE, RP = 4 * ((ROWS / 4) | 1), PP = 4 * ((PAIRS / 4) | 1);
  static constexpr int THREADS = 832;   // 26 warps: the products' loops wait on shared-memory loads, and more warps hide that
  static constexpr int SLICES = THREADS / 64;   // of the hidden units, for the scores: a lane per pair
  static __host__ __device__ int ldw(int d) { return (d + 3) & ~3; }
  static __host__ __device__ size_t smem_floats(int d) { return (size_t)2 * d * ldw(d) + (size_t)2 * d * RP + (size_t)d * PP + 3 * (size_t)ldw(d) + SLICES * 64; }
};

template <int TE>
__global__ void __launch_bounds__(HeadTile<TE>::THREADS) head_tile_kernel(const float* __restrict__ h, const float* __restrict__ WT,
                                                                        const float* __restrict__ b1, const float* __restrict__ w2,
                                                                        const float* __restrict__ b2,
                                                                        const uint8_t* __restrict__ loss_mask, int nq, int d,
                                                                        float* __restrict__ cat1, float* __restrict__ dpre1,
                                                                        uint8_t* __restrict__ hid_gate, float* __restrict__ dpre_o,
                                                                        float* __restrict__ g_w2, float* __restrict__ g_b2,
                                                                        float* __restrict__ loss_acc, int relu_out) {
  using HT_ = HeadTile<TE>;
  constexpr int ROWS = HT_::ROWS, PAIRS = HT_::PAIRS, RP = HT_::RP, PP = HT_::PP, T = HT_::THREADS;
  extern __shared__ __align__(16) float sm[];
  __shared__ float s_msum, s_gb2, s_loss, s_ds[PAIRS], s_lp[PAIRS];
  const int LDW = HT_::ldw(d);
  const int tid = threadIdx.x, lane = tid & 31;
  float* WaT = sm;
  float* WbT = WaT + (size_t)d * LDW;
  float* HTs = WbT + (size_t)d * LDW;
  float* PTs = HTs + (size_t)d * RP;
  float* D1T = PTs + (size_t)d * RP;
  float* b1s = D1T + (size_t)d * PP;
  float* w2s = b1s + LDW;
  float* gw2 = w2s + LDW;
  float* part = gw2 + LDW;   // [SLICES][64]
  const bool hvec = ((uintptr_t)h & 15) == 0;
  const int zero = link_wait(), first = blockIdx.x + zero;
  link_release();
  WT += zero;   // (written within the step, as h is)
  {  // both transposed halves of W_1 (prepared once per step in this layout): a straight 16-byte copy
    const int n4 = (2 * d * LDW) >> 2;
    const float4* src = reinterpret_cast<const float4*>(WT);
    float4* dst = reinterpret_cast<float4*>(WaT);
    for (int i = tid; i < n4; i += T) dst[i] = __ldg(src + i);
  }
  for (int q = tid; q < d; q += T) { b1s[q] = b1[q]; w2s[q] = w2[q]; gw2[q] = 0.f; }
  if (tid == 0) { s_msum = 0.f; s_gb2 = 0.f; s_loss = 0.f; }
  __syncthreads();
  {  // every block counts the whole mask (a few KB)
    int c = 0;
    for (int j = tid; j < nq; j += T) c += loss_mask ? (loss_mask[j] != 0) : 1;
    for (int o = 16; o > 0; o >>= 1) c += __shfl_xor_sync(FULL, c, o);
    if (lane == 0 && c) atomicAdd(&s_msum, (float)c);
  }
  __syncthreads();
  const float msum = s_msum;
  const float bias2 = b2[0];
  const int tiles = (nq + TE - 1) / TE;
  for (int tile = first; tile < tiles; tile += gridDim.x) {
    const int ev0 = tile * TE;
    // ---- embedding rows -> HT (transposed) and cat1: all of a thread's loads before its first store ----
    {
      constexpr int V = 4;
      const int d4 = d >> 2, total = ROWS * d4;
#pragma unroll 1
      for (int e0 = tid; e0 < total; e0 += V * T) {
        float4 v[V];
#pragma unroll
        for (int u = 0; u < V; ++u) {
          const int e = e0 + u * T, r = e / d4, blk = r / TE, ev = ev0 + r - blk * TE;   // (TE is a compile-time constant)
          v[u] = e < total && ev < nq ? ldg4(h + ((int64_t)blk * nq + ev) * d + 4 * (e - r * d4), hvec) : make_float4(0.f, 0.f, 0.f, 0.f);
        }
#pragma unroll
        for (int u = 0; u < V; ++u) {
          const int e = e0 + u * T, r = e / d4, blk = r / TE, ev = ev0 + r - blk * TE, c = 4 * (e - r * d4);
          if (e >= total) break;
          if (ev < nq) {   // sources go to two rows
            float* o = cat1 + (int64_t)(blk == 2 ? nq + ev : ev) * 2 * d + (blk == 0 ? 0 : d) + c;
            *reinterpret_cast<float4*>(o) = v[u];
            if (blk == 0) *reinterpret_cast<float4*>(o + (int64_t)nq * 2 * d) = v[u];
          }
          float* t = HTs + c * RP + r;
          t[0] = v[u].x; t[RP] = v[u].y; t[2 * RP] = v[u].z; t[3 * RP] = v[u].w;
        }
      }
    }
    __syncthreads();
    // ---- hidden layer: PT[j][r] = sum_c W[j][c] h_r[c] ----
    {
      const int ntj = d >> 2, ntr = ROWS >> 2;
      for (int t = tid; t < ntj * ntr; t += T) {
        const int tj = t % ntj, tr = t / ntj;
        const float* Wp = (4 * tr < TE ? WaT : WbT) + 4 * tj;   // (TE is a multiple of 4: a row block lies in one part)
        const float* Hp = HTs + 4 * tr;
        float acc[4][4];
#pragma unroll
        for (int a = 0; a < 4; ++a)
#pragma unroll
          for (int b = 0; b < 4; ++b) acc[a][b] = 0.f;
#pragma unroll 4
        for (int c = 0; c < d; ++c) {
          const float4 wv = *reinterpret_cast<const float4*>(Wp + (size_t)c * LDW);
          const float4 hv = *reinterpret_cast<const float4*>(Hp + c * RP);
          const float wj[4] = {wv.x, wv.y, wv.z, wv.w};
          const float hr[4] = {hv.x, hv.y, hv.z, hv.w};
#pragma unroll
          for (int a = 0; a < 4; ++a)
#pragma unroll
            for (int b = 0; b < 4; ++b) acc[a][b] = fmaf(wj[a], hr[b], acc[a][b]);
        }
#pragma unroll
        for (int a = 0; a < 4; ++a)
          *reinterpret_cast<float4*>(PTs + (4 * tj + a) * RP + 4 * tr) = make_float4(acc[a][0], acc[a][1], acc[a][2], acc[a][3]);
      }
    }
    __syncthreads();
    // ---- scores: a lane per pair (neighbouring lanes, neighbouring words), the hidden units in slices ----
    {
      const int p = tid & 63, sl = tid >> 6;
      if (p < PAIRS) {
        const float *ps = PTs + (p < TE ? p : p - TE), *po = PTs + TE + p;   // source; destination or negative
        float sc = 0.f;
#pragma unroll 4
        for (int q = d * sl / HT_::SLICES; q < d * (sl + 1) / HT_::SLICES; ++q) sc = fmaf(w2s[q], fmaxf(ps[q * RP] + po[q * RP] + b1s[q], 0.f), sc);
        part[sl * 64 + p] = sc;
      }
    }
    __syncthreads();
    if (tid < PAIRS) {
      const int half = tid / TE, ev = ev0 + tid - half * TE;
      float sc = bias2;
#pragma unroll
      for (int z = 0; z < HT_::SLICES; ++z) sc += part[z * 64 + tid];
      const float m = ev < nq && (loss_mask ? (loss_mask[ev] != 0) : true) ? 1.f : 0.f;
      const float wj = msum > 0.f ? m / msum : 0.f;
      const float z = half == 0 ? -sc : sc;
      s_ds[tid] = wj != 0.f ? (half == 0 ? -wj : wj) * sigmoidf_(z) : 0.f;   // (an event without weight leaves nothing, whatever its score)
      s_lp[tid] = wj != 0.f ? wj * softplusf_(z) : 0.f;
    }
    __syncthreads();
    // ---- d loss / d pre1 and the gates: a thread keeps its hidden unit and walks the pairs; dw_2, db_2 and the loss on the way ----
    {
      const int DT = (d + 31) & ~31, grp = tid / DT, q = tid - grp * DT, ngrp = T / DT;
      if (q < d && grp < ngrp) {
        const float b = b1s[q], w = w2s[q];
        float gw = 0.f;
#pragma unroll 2
        for (int p = grp; p < PAIRS; p += ngrp) {
          const int half = p / TE, e = p - half * TE, ev = ev0 + e;
          const float a = fmaxf(PTs[q * RP + e] + PTs[q * RP + TE + p] + b, 0.f), ds = s_ds[p], dv = a > 0.f ? ds * w : 0.f;
          if (ds != 0.f) gw = fmaf(ds, a, gw);   // (events without weight are left out whatever their rows hold)
          D1T[q * PP + p] = dv;
          if (ev < nq) {
            const int64_t o = ((int64_t)half * nq + ev) * d + q;
            dpre1[o] = dv;
            hid_gate[o] = a > 0.f;
          }
        }
        if (gw != 0.f) atomicAdd(&gw2[q], gw);
      }
      if (tid == T - 1) {
        float l = 0.f, g = 0.f;
        for (int p = 0; p < PAIRS; ++p) { l += s_lp[p]; g += s_ds[p]; }
        s_loss += l; s_gb2 += g;
      }
    }
    __syncthreads();
    // ---- input gradient: dC[p][c2] = sum_j dh1[p][j] W_1[j][c2], both pairs of 2 events x 4 columns per thread ----
    {
      const int ntp = TE >> 1, ntc = (2 * d) >> 2;
      for (int t = tid; t < ntp * ntc; t += T) {
        const int tp = t % ntp, tc = t / ntp;
        const int c2 = 4 * tc;
        const bool lower = c2 < d;
        const float* Wp = lower ? WaT + (size_t)c2 * LDW : WbT + (size_t)(c2 - d) * LDW;
        const float* Dp = D1T + 2 * tp;
        float aP[2][4], aN[2][4];   // [event][column]
#pragma unroll
        for (int a = 0; a < 2; ++a)
#pragma unroll
          for (int b = 0; b < 4; ++b) { aP[a][b] = 0.f; aN[a][b] = 0.f; }
        for (int j0 = 0; j0 < d; j0 += 4) {
          float4 w4[4];
#pragma unroll
          for (int i = 0; i < 4; ++i) w4[i] = *reinterpret_cast<const float4*>(Wp + (size_t)i * LDW + j0);
#pragma unroll
          for (int jj = 0; jj < 4; ++jj) {
            const float2 dp = *reinterpret_cast<const float2*>(Dp + (j0 + jj) * PP);
            const float2 dn = *reinterpret_cast<const float2*>(Dp + (j0 + jj) * PP + TE);
            const float de[2] = {dp.x, dp.y};
            const float dm[2] = {dn.x, dn.y};
#pragma unroll
            for (int i = 0; i < 4; ++i) {
              const float wv = jj == 0 ? w4[i].x : (jj == 1 ? w4[i].y : (jj == 2 ? w4[i].z : w4[i].w));
#pragma unroll
              for (int e = 0; e < 2; ++e) {
                aP[e][i] = fmaf(de[e], wv, aP[e][i]);
                aN[e][i] = fmaf(dm[e], wv, aN[e][i]);
              }
            }
          }
        }
#pragma unroll
        for (int e = 0; e < 2; ++e) {
          const int el = 2 * tp + e, ev = ev0 + el;
          if (ev >= nq) continue;
          if (lower) {   // source rows collect their positive and their negative pair
            float o[4];
#pragma unroll
            for (int i = 0; i < 4; ++i)
              o[i] = (!relu_out || HTs[(c2 + i) * RP + el] > 0.f) ? aP[e][i] + aN[e][i] : 0.f;
            *reinterpret_cast<float4*>(dpre_o + (int64_t)ev * d + c2) = make_float4(o[0], o[1], o[2], o[3]);
          } else {
            const int cc = c2 - d;
            float o[4], n[4];
#pragma unroll
            for (int i = 0; i < 4; ++i) {
              o[i] = (!relu_out || HTs[(cc + i) * RP + TE + el] > 0.f) ? aP[e][i] : 0.f;
              n[i] = (!relu_out || HTs[(cc + i) * RP + 2 * TE + el] > 0.f) ? aN[e][i] : 0.f;
            }
            *reinterpret_cast<float4*>(dpre_o + ((int64_t)nq + ev) * d + cc) = make_float4(o[0], o[1], o[2], o[3]);
            *reinterpret_cast<float4*>(dpre_o + ((int64_t)2 * nq + ev) * d + cc) = make_float4(n[0], n[1], n[2], n[3]);
          }
        }
      }
    }
    __syncthreads();
  }
  for (int q = tid; q < d; q += T)
    if (gw2[q] != 0.f) atomicAdd(&g_w2[q], gw2[q]);
  if (tid == 0) {
    if (s_gb2 != 0.f) atomicAdd(g_b2, s_gb2);
    if (s_loss != 0.f) atomicAdd(loss_acc, s_loss);
  }
}

// One warp per root: backward of the weighted sum, the softmax and the scaled dot products, on the
// root's K | V rows staged in shared memory.  Lane p < H*k owns the (head, slot) pair p for the
// probability and logit gradients; afterwards the lanes own columns and write dQ and the dK | dV rows.
// SPLIT: the key/value gradient rows are written as two fp16 planes (hi, lo; row pitch ld_s, plane_s elements
// apart), multiplied by the power of two gscale so that they sit inside fp16's range, for the split products that
// consume them (which divide it out again), instead of as fp32 rows.
template <bool SPLIT>
__global__ void __launch_bounds__(256) attention_bwd_kernel(const float* __restrict__ Q, const float* __restrict__ KV,
                                                            const float* __restrict__ alpha,
                                                            const float* __restrict__ dcat_o,
                                                            const int32_t* __restrict__ cnt, int n, int d, int H, int k,
                                                            float* __restrict__ dQ, float* __restrict__ dKV,
                                                            __nv_bfloat16* __restrict__ dkv_hi, int64_t plane_s, int ld_s,
                                                            float gscale) {
  extern __shared__ __align__(16) float sm[];
  const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5;
  const int i = (int)((blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5);
  if (i >= n) return;
  float* Ks = sm + wib * attn_warp_floats(d, H, k);
  float* Vs = Ks + k * d;
  float* Qs = Vs + k * d;
  float* das = Qs + d;       // d loss / d a
  float* al = das + d;       // probabilities
  float* dal = al + H * k;   // d loss / d probability
  float* dl = dal + H * k;   // d loss / d logit, already scaled
  const int dh = d / H;
  const int c = max(0, min(cnt[i], k));
  const float scale = rsqrtf((float)dh);
  attn_stage_issue(Ks, Vs, Qs, Q, KV, i, c, d, k, lane);
  {
    const float* g = dcat_o + (int64_t)i * 2 * d;
    for (int e = lane; e < (d >> 2); e += 32) cp_async16(das + 4 * e, g + 4 * e);
    for (int p = lane; p < H * k; p += 32) al[p] = alpha[(int64_t)i * H * k + p];
  }
  attn_stage_wait();
  for (int p = lane; p < H * k; p += 32) {
    const int h = p / k, s = p - h * k;
    float a = 0.f;
    if (s < c) {
      const float* vr = Vs + s * d + h * dh;
      const float* gr = das + h * dh;
      for (int e = 0; e < dh; ++e) a = fmaf(gr[e], vr[e], a);
    }
    dal[p] = a;
  }
  __syncwarp();
  for (int p = lane; p < H * k; p += 32) {
    const int h = p / k, s = p - h * k;
    float g = 0.f;
    if (s < c) {
      float dot = 0.f;
      for (int t = 0; t < c; ++t) dot = fmaf(al[h * k + t], dal[h * k + t], dot);
      g = al[p] * (dal[p] - dot) * scale;
    }
    dl[p] = g;
  }
  __syncwarp();
  if (!SPLIT) {
    for (int e = lane; e < d; e += 32) {
      const int h = e / dh;
      const float qe = Qs[e], dae = das[e];
      float dq = 0.f;
      for (int s = 0; s < k; ++s) {
        float* row = dKV + ((int64_t)i * k + s) * 2 * d;
        if (s < c) {
          const float g = dl[h * k + s];
          dq = fmaf(g, Ks[s * d + e], dq);
          row[e] = g * qe;
          row[d + e] = al[h * k + s] * dae;
        } else {
          row[e] = 0.f;
          row[d + e] = 0.f;
        }
      }
      dQ[(int64_t)i * d + e] = dq;
    }
  } else {
    // a lane owns two neighbouring columns (d is even): each (hi, lo) pair goes out as one 32-bit word per plane
    for (int e = 2 * lane; e < d; e += 64) {
      const int h0 = e / dh, h1 = (e + 1) / dh;
      const float q0 = Qs[e], q1 = Qs[e + 1], a0 = das[e], a1 = das[e + 1];
      float dq0 = 0.f, dq1 = 0.f;
      for (int s = 0; s < k; ++s) {
        uint32_t* hi = reinterpret_cast<uint32_t*>(dkv_hi + ((int64_t)i * k + s) * ld_s);
        uint32_t* lo = reinterpret_cast<uint32_t*>(dkv_hi + plane_s + ((int64_t)i * k + s) * ld_s);
        uint32_t kh = 0u, kl = 0u, vh = 0u, vl = 0u;
        if (s < c) {
          const float g0 = dl[h0 * k + s], g1 = dl[h1 * k + s];
          dq0 = fmaf(g0, Ks[s * d + e], dq0);
          dq1 = fmaf(g1, Ks[s * d + e + 1], dq1);
          split_f16_pair(g0 * q0 * gscale, g1 * q1 * gscale, &kh, &kl);
          split_f16_pair(al[h0 * k + s] * a0 * gscale, al[h1 * k + s] * a1 * gscale, &vh, &vl);
        }
        hi[e >> 1] = kh; lo[e >> 1] = kl;
        hi[(d + e) >> 1] = vh; lo[(d + e) >> 1] = vl;
      }
      dQ[(int64_t)i * d + e] = dq0;
      dQ[(int64_t)i * d + e + 1] = dq1;
    }
  }
}

// The split form of the kernel above for compile-time shapes (D columns, H heads, KS slots; D / H even, H * KS <= 32,
// D <= 128).  The generic kernel is bound by instruction issue (2 800 instructions per root: loop control, scalar
// shared-memory loads, 32-bit plane stores); here the dot products read pairs of columns, a lane owns four
// neighbouring columns of the key / value gradient rows and writes them as one 64-bit word per plane and row.  Every
// sum keeps the generic kernel's order of operations.
template <int D, int H, int KS>
__global__ void __launch_bounds__(256) attention_bwd_fixed_kernel(const float* __restrict__ Q, const float* __restrict__ KV,
                                                                  const float* __restrict__ alpha,
                                                                  const float* __restrict__ dcat_o,
                                                                  const int32_t* __restrict__ cnt, int n,
                                                                  float* __restrict__ dQ, __nv_bfloat16* __restrict__ dkv_hi,
                                                                  int64_t plane_s, int ld_s, float gscale) {
  constexpr int DH = D / H, D4 = D / 4, P = H * KS;
  static_assert(D % 4 == 0 && DH % 2 == 0 && P <= 32 && D4 <= 32, "shape not covered by the fixed kernel");
  extern __shared__ __align__(16) float sm[];
  const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5;
  const int i = (int)((blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5);
  if (i >= n) return;
  float* Ks = sm + wib * attn_warp_floats(D, H, KS);
  float* Vs = Ks + KS * D;
  float* Qs = Vs + KS * D;
  float* das = Qs + D;       // d loss / d a
  float* al = das + D;       // probabilities
  float* dal = al + P;       // d loss / d probability
  float* dl = dal + P;       // d loss / d logit, already scaled
  const int c = max(0, min(cnt[i], KS));
  const float scale = rsqrtf((float)DH);
  {
    const float* q = Q + (int64_t)i * D;
    const float* g = dcat_o + (int64_t)i * 2 * D;
    if (lane < D4) {
      cp_async16(Qs + 4 * lane, q + 4 * lane);
      cp_async16(das + 4 * lane, g + 4 * lane);
    }
    // lane l < D / 4 copies chunk l of every valid row's K half and V half: constant offsets from two pointers
    const float* kv = KV + (int64_t)i * KS * 2 * D + 4 * lane;
    float* kd = Ks + 4 * lane;
    if (lane < D4) {
#pragma unroll
      for (int t = 0; t < KS; ++t) {
        if (t < c) {
          cp_async16(kd + t * D, kv + t * 2 * D);
          cp_async16(kd + (KS + t) * D, kv + t * 2 * D + D);   // (Vs = Ks + KS * D)
        }
      }
    }
    if (lane < P) al[lane] = alpha[(int64_t)i * P + lane];
  }
  attn_stage_wait();
  const int h = lane / KS, sl = lane - h * KS;
  const bool live = lane < P && sl < c;
  float a = 0.f;
  if (live) {
    const float2* vr = reinterpret_cast<const float2*>(Vs + sl * D + h * DH);
    const float2* gr = reinterpret_cast<const float2*>(das + h * DH);
#pragma unroll
    for (int e = 0; e < DH / 2; ++e) {
      const float2 gv = gr[e], vv = vr[e];
      a = fmaf(gv.x, vv.x, a);
      a = fmaf(gv.y, vv.y, a);
    }
  }
  if (lane < P) dal[lane] = a;
  __syncwarp();
  float gl = 0.f;
  if (live) {
    float dot = 0.f;
#pragma unroll
    for (int t = 0; t < KS; ++t)
      if (t < c) dot = fmaf(al[h * KS + t], dal[h * KS + t], dot);
    gl = al[lane] * (a - dot) * scale;
  }
  if (lane < P) dl[lane] = gl;
  __syncwarp();
  if (lane < D4) {
    const int h0 = (4 * lane) / DH, h1 = (4 * lane + 2) / DH;   // columns 4l, 4l+1 share a head, and so do 4l+2, 4l+3
    const float4 q4 = *reinterpret_cast<const float4*>(Qs + 4 * lane);
    const float4 a4 = *reinterpret_cast<const float4*>(das + 4 * lane);
    float4 dq = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
    for (int t = 0; t < KS; ++t) {
      __nv_bfloat16* hi_row = dkv_hi + ((int64_t)i * KS + t) * ld_s + 4 * lane;
      __nv_bfloat16* lo_row = hi_row + plane_s;
      uint2 kh = make_uint2(0u, 0u), kl = kh, vh = kh, vl = kh;
      if (t < c) {
        const float g0 = dl[h0 * KS + t], g1 = dl[h1 * KS + t];
        const float p0 = al[h0 * KS + t], p1 = al[h1 * KS + t];
        const float4 kv4 = *reinterpret_cast<const float4*>(Ks + t * D + 4 * lane);
        dq.x = fmaf(g0, kv4.x, dq.x); dq.y = fmaf(g0, kv4.y, dq.y);
        dq.z = fmaf(g1, kv4.z, dq.z); dq.w = fmaf(g1, kv4.w, dq.w);
        split_f16_pair(g0 * q4.x * gscale, g0 * q4.y * gscale, &kh.x, &kl.x);
        split_f16_pair(g1 * q4.z * gscale, g1 * q4.w * gscale, &kh.y, &kl.y);
        split_f16_pair(p0 * a4.x * gscale, p0 * a4.y * gscale, &vh.x, &vl.x);
        split_f16_pair(p1 * a4.z * gscale, p1 * a4.w * gscale, &vh.y, &vl.y);
      }
      *reinterpret_cast<uint2*>(hi_row) = kh;
      *reinterpret_cast<uint2*>(lo_row) = kl;
      *reinterpret_cast<uint2*>(hi_row + D) = vh;
      *reinterpret_cast<uint2*>(lo_row + D) = vl;
    }
    *reinterpret_cast<float4*>(dQ + (int64_t)i * D + 4 * lane) = dq;
  }
}

// Gradient rows flowing into memory rows that the last memory update wrote: one warp per
// source row, added into dMemU[node2slot[node]].  Rows [0, n k): dZm with node = nbr (k = 0: none);
// rows [n k, n k + n): the root's own row, the sum of its rows in ra and rb.
__global__ void __launch_bounds__(256) scatter_dmem_kernel(const float* __restrict__ dZm, const float* __restrict__ ra, int64_t lda,
                                                           const float* __restrict__ rb, int64_t ldb,
                                                           const int32_t* __restrict__ nbr,
                                                           const int32_t* __restrict__ nodes, int n, int k, int d,
                                                           const int32_t* __restrict__ node2slot,
                                                           float* __restrict__ dMemU, int64_t N, int upd_rows, int copy_mask) {
  const int first = (int)((blockIdx.x * blockDim.x + threadIdx.x) >> 5) + link_wait();
  link_release();
  dMemU += (int64_t)(blockIdx.x & copy_mask) * upd_rows * d;   // (copies of the rows, against additions that wait for one another)
  const int lane = threadIdx.x & 31;
  const int warps = (gridDim.x * blockDim.x) >> 5;
  const int nb_rows = n * k;
  const int d4 = d >> 2;  // <= 64: at most two 16-byte pieces per lane
  for (int r = first; r < nb_rows + n; r += warps) {
    // the row's gradient is requested before it is known whether its node was updated (most were not):
    // the index chain node -> slot and the row loads overlap
    const bool isn = r < nb_rows;
    const int i = r - nb_rows;
    float4 g[2];
#pragma unroll
    for (int u = 0; u < 2; ++u) {
      const int q4 = lane + 32 * u;
      g[u] = make_float4(0.f, 0.f, 0.f, 0.f);
      if (q4 < d4) {
        if (isn) {
          g[u] = __ldg(reinterpret_cast<const float4*>(dZm + (int64_t)r * 2 * d) + q4);  // memory half of the row
        } else {
          const float4 a = __ldg(reinterpret_cast<const float4*>(ra + i * lda) + q4);
          const float4 b = __ldg(reinterpret_cast<const float4*>(rb + i * ldb) + q4);
          g[u] = make_float4(a.x + b.x, a.y + b.y, a.z + b.z, a.w + b.w);
        }
      }
    }
    const int node = isn ? nbr[r] : nodes[i];
    if (node < 0 || node >= N) continue;   // (an id beyond the graph was reported by the forward pass)
    const int slot = node2slot[node];
    if (slot < 0 || slot >= upd_rows) continue;
    float4* out = reinterpret_cast<float4*>(dMemU + (int64_t)slot * d);
#pragma unroll
    for (int u = 0; u < 2; ++u) {
      const int q4 = lane + 32 * u;
      if (q4 < d4) atomicAdd(out + q4, g[u]);
    }
  }
}

// The same scatter for batches in which many rows hit few nodes (hub nodes: tens of thousands of rows onto one
// updated row serialise on its atomics).  A block takes SC_ROWS consecutive rows.  One thread per row first
// resolves row -> node -> slot and files the row under one of SC_WAYS lists (a list belongs to the first slot that
// claims it by compare-and-swap; a row whose list belongs to another slot goes to a list of singles).  The lists
// are then laid end to end, so that rows of one slot are neighbours, and every warp walks an equal share of that
// sequence, 6 / U row loads in flight: it sums in registers while the slot stays the same and adds the sum to
// dMemU when it changes.  Rows whose node was not updated are never read.
constexpr int SC_ROWS = 256, SC_WAYS = 32;  // 256 rows, 256 threads: the whole batch is one wave of blocks
template <int U>  // 16-byte pieces of a row per lane: 1 (d <= 128) or 2
__global__ void __launch_bounds__(256, 5) scatter_dmem_cached_kernel(const float* __restrict__ dZm,
                                                                     const float* __restrict__ ra, int64_t lda,
                                                                     const float* __restrict__ rb, int64_t ldb,
                                                                     const int32_t* __restrict__ nbr,
                                                                     const int32_t* __restrict__ nodes, int n, int k, int d,
                                                                     const int32_t* __restrict__ node2slot,
                                                                     float* __restrict__ dMemU, int64_t N, int upd_rows) {
  static_assert(SC_WAYS == 32, "one lane per list in the offset scan");
  static_assert(SC_ROWS == 256, "one thread per row, row numbers kept in a byte");
  __shared__ int s_id[SC_WAYS], s_cnt[SC_WAYS + 1], s_off[SC_WAYS + 1], s_slot[SC_ROWS];
  __shared__ unsigned char s_seq[SC_ROWS];
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  const int nb_rows = n * k, total = nb_rows + n;
  const int d4 = d >> 2;  // <= 32 U
  const int r_base = blockIdx.x * SC_ROWS;
  if (threadIdx.x < SC_WAYS) s_id[threadIdx.x] = -1;
  if (threadIdx.x <= SC_WAYS) s_cnt[threadIdx.x] = 0;  // (entry SC_WAYS: the singles)
  __syncthreads();
  int way = -1, pos = 0;
  if (r_base + threadIdx.x < total) {
    const int r = r_base + threadIdx.x;
    const int node = r < nb_rows ? nbr[r] : nodes[r - nb_rows];
    int slot = -1;
    if (node >= 0 && node < N) slot = node2slot[node];  // (an id beyond the graph was reported by the forward pass)
    if (slot >= upd_rows) slot = -1;
    s_slot[threadIdx.x] = slot;
    if (slot >= 0) {
      way = slot % SC_WAYS;
      const int owner = atomicCAS(&s_id[way], -1, slot);
      if (owner != -1 && owner != slot) way = SC_WAYS;
      pos = atomicAdd(&s_cnt[way], 1);
    }
  }
  __syncthreads();
  if (wid == 0) {  // exclusive scan of the list lengths
    const int c = s_cnt[lane];
    int incl = c;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int t = __shfl_up_sync(FULL, incl, o);
      if (lane >= o) incl += t;
    }
    s_off[lane] = incl - c;
    if (lane == 31) s_off[SC_WAYS] = incl;
  }
  __syncthreads();
  if (way >= 0) s_seq[s_off[way] + pos] = (unsigned char)threadIdx.x;
  __syncthreads();
  const int n_live = s_off[SC_WAYS] + s_cnt[SC_WAYS];
  const int share = (n_live + 7) >> 3;
  const int e_end = min(n_live, (wid + 1) * share);
  constexpr int V = 6 / U;  // (48 registers: five blocks share an SM, or fewer beside a persistent product)
  int cur = -1;
  float4 acc[U];
#pragma unroll
  for (int u = 0; u < U; ++u) acc[u] = make_float4(0.f, 0.f, 0.f, 0.f);
  auto flush = [&]() {
    if (cur < 0) return;
    float4* out = reinterpret_cast<float4*>(dMemU + (int64_t)cur * d);
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const int q4 = lane + 32 * u;
      if (q4 < d4) atomicAdd(out + q4, acc[u]);
      acc[u] = make_float4(0.f, 0.f, 0.f, 0.f);
    }
  };
  for (int e = wid * share; e < e_end; e += V) {
    float4 g[V][U];
    int t[V];
#pragma unroll
    for (int v = 0; v < V; ++v) {
      t[v] = e + v < e_end ? (int)s_seq[e + v] : -1;
      if (t[v] < 0) continue;
      const int r = r_base + t[v];
#pragma unroll
      for (int u = 0; u < U; ++u) {
        const int q4 = lane + 32 * u;
        g[v][u] = make_float4(0.f, 0.f, 0.f, 0.f);
        if (q4 < d4) {
          if (r < nb_rows) {
            g[v][u] = __ldg(reinterpret_cast<const float4*>(dZm + (int64_t)r * 2 * d) + q4);  // memory half of the row
          } else {
            const int i = r - nb_rows;
            const float4 a = __ldg(reinterpret_cast<const float4*>(ra + i * lda) + q4);
            const float4 b = __ldg(reinterpret_cast<const float4*>(rb + i * ldb) + q4);
            g[v][u] = make_float4(a.x + b.x, a.y + b.y, a.z + b.z, a.w + b.w);
          }
        }
      }
    }
#pragma unroll
    for (int v = 0; v < V; ++v) {
      if (t[v] < 0) continue;  // (uniform over the warp)
      const int slot = s_slot[t[v]];
      if (slot != cur) { flush(); cur = slot; }
#pragma unroll
      for (int u = 0; u < U; ++u) {
        acc[u].x += g[v][u].x; acc[u].y += g[v][u].y; acc[u].z += g[v][u].z; acc[u].w += g[v][u].w;
      }
    }
  }
  flush();
}

// Slot rows of large inputs in which many rows hit few nodes (small node set, large batch) are summed per block: the hub rows
// would serialise on their atomics.  Below four rows per node, and for the roots' rows alone (k = 0), the plain form with its
// copies is as fast or faster (12 000 roots, 2 000 nodes: 9.5 us, per block 26.6).
inline bool scatter_by_block(const tgnn_ctx* ctx, int n, int k) { return k > 0 && (int64_t)n * k + n >= 4 * ctx->cfg.num_nodes; }
inline void scatter_rows(tgnn_ctx* ctx, const float* dZm, const float* ra, int64_t lda, const float* rb, int64_t ldb, int n, int k,
                         cudaStream_t s) {
  const int d = ctx->cfg.d;
  const int64_t rows = (int64_t)n * k + n, N = ctx->cfg.num_nodes;
  Workspace& w = ctx->ws;
  const GradCopies& cp = ctx->copies;
  if (!scatter_by_block(ctx, n, k))
    launch_link(ctx, scatter_dmem_kernel, dim3((unsigned)((rows + 7) / 8)), dim3(256), 0, s, 1, dZm, ra, lda, rb, ldb, ctx->e_nbr, ctx->e_nodes, n, k, d,
                w.node2slot, w.dMemU, N, cp.rows, cp.n - 1);
  else if (d <= 128)
    scatter_dmem_cached_kernel<1><<<(int)((rows + SC_ROWS - 1) / SC_ROWS), 256, 0, s>>>(dZm, ra, lda, rb, ldb, ctx->e_nbr, ctx->e_nodes, n, k, d,
                                                                                       w.node2slot, w.dMemU, N, cp.rows);
  else
    scatter_dmem_cached_kernel<2><<<(int)((rows + SC_ROWS - 1) / SC_ROWS), 256, 0, s>>>(dZm, ra, lda, rb, ldb, ctx->e_nbr, ctx->e_nodes, n, k, d,
                                                                                       w.node2slot, w.dMemU, N, cp.rows);
}

// Time-encoder gradient: G[r, col0 + c] is d loss / d Phi(dt_r)_c and S[r, c] = sin(arg) was kept by
// the forward pass (S == nullptr: every row has dt = 0, sin(arg) = sin(b_c)).
//   dw_c += -S dt_r G,   db_c += -S G
// The terms are large (dt reaches the time span of the stream) and cancel, so they are summed in
// fp64.  Block = 8 warps over rows_per_block rows; lanes own columns c = lane + 32 j; the warps' partial sums
// meet in shared memory and leave as one pair of fp64 atomics per block and column into acc[0:d]
// (dw) and acc[d:2d] (db).  Dynamic shared memory: 8 * 2 * d doubles.
constexpr int TG_MAXJ = 8;
// Rows per block: every block ends with one fp64 atomic per column onto the same 2d addresses, and those
// serialise, so the grid is kept to about two blocks per SM, as many as fit at once (rows per block a multiple
// of the 8 warps); inside a block each warp walks its rows three at a time so that their loads overlap.
constexpr int TG_U = 3;   // rows a warp has in flight (four spill at the 128 registers that let two blocks share an SM)
inline int tg_rows_per_block(int rows) {
  const int r = (rows + 295) / 296;
  return r < 8 ? 8 : (r + 7) / 8 * 8;
}
template <int V>  // 16-byte column pieces per lane: 1 (d <= 128: half the registers, four blocks share an SM) or 2
__global__ void __launch_bounds__(256, V == 1 ? 4 : 2) time_grad_kernel(const float* __restrict__ G, int64_t ldg, int col0,
                                                        const float* __restrict__ S, const float* __restrict__ dt,
                                                        int rows, const int32_t* __restrict__ dev_rows, int d,
                                                        const float* __restrict__ time_w,
                                                        const float* __restrict__ time_b, double* __restrict__ acc,
                                                        int rows_per_block) {
  extern __shared__ double s_part[];  // [8][2][d]
  const int r0 = blockIdx.x * rows_per_block + link_wait();
  link_release();
  const int R = dev_rows ? min(*dev_rows, rows) : rows;
  const int r1 = min(R, r0 + rows_per_block);
  if (r0 >= r1) return;
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  // a lane owns columns 4 (lane + 32 v) .. + 3, v < V (d <= 128 V): 128-bit loads of G and S (d, ldg and col0 are
  // multiples of 4 and the rows 16-byte aligned)
  // Sines: saved rows S; or (S null, dt given) recomputed from the row's dt exactly as the forward pass formed
  // them -- a row with dt < 0 is an empty slot and contributes nothing; or (both null) the constant sin(b) of dt = 0.
  double gw[V][4], gb[V][4];
  float4 sb[V], wv[V], bv[V];
  const bool recompute = S == nullptr && dt != nullptr;
#pragma unroll
  for (int v = 0; v < V; ++v) {
    const int c = 4 * (lane + 32 * v);
#pragma unroll
    for (int e = 0; e < 4; ++e) { gw[v][e] = 0.0; gb[v][e] = 0.0; }
    sb[v] = wv[v] = bv[v] = make_float4(0.f, 0.f, 0.f, 0.f);
    if (S == nullptr && c < d) {
      bv[v] = make_float4(time_b[c], time_b[c + 1], time_b[c + 2], time_b[c + 3]);
      if (recompute) wv[v] = make_float4(time_w[c], time_w[c + 1], time_w[c + 2], time_w[c + 3]);
      else sb[v] = make_float4(sinf(bv[v].x), sinf(bv[v].y), sinf(bv[v].z), sinf(bv[v].w));
    }
  }
  for (int rb = r0 + wid; rb < r1; rb += 8 * TG_U) {  // rows rb, rb + 8, ...: loads first, sums after
    float4 g[TG_U][V], sn[TG_U][V];
    float dtr[TG_U];
#pragma unroll
    for (int u = 0; u < TG_U; ++u) {
      const int r = rb + 8 * u;
      const bool in = r < r1;
      dtr[u] = (in && dt) ? dt[r] : 0.f;
#pragma unroll
      for (int v = 0; v < V; ++v) {
        const int c = 4 * (lane + 32 * v);
        const bool ok = in && c < d;
        g[u][v] = ok ? __ldg(reinterpret_cast<const float4*>(G + (int64_t)r * ldg + col0 + c)) : make_float4(0.f, 0.f, 0.f, 0.f);
        sn[u][v] = ok ? (S ? __ldg(reinterpret_cast<const float4*>(S + (int64_t)r * d + c)) : sb[v]) : make_float4(0.f, 0.f, 0.f, 0.f);
      }
    }
    if (recompute) {
#pragma unroll
      for (int u = 0; u < TG_U; ++u) {
        const bool live = rb + 8 * u < r1 && dtr[u] >= 0.f;
#pragma unroll
        for (int v = 0; v < V; ++v) {
          const int c = 4 * (lane + 32 * v);
          float4 q = make_float4(0.f, 0.f, 0.f, 0.f);
          if (live && c < d) {
            q.x = __sinf(reduce_two_pi(time_arg(wv[v].x, bv[v].x, dtr[u])));
            q.y = __sinf(reduce_two_pi(time_arg(wv[v].y, bv[v].y, dtr[u])));
            q.z = __sinf(reduce_two_pi(time_arg(wv[v].z, bv[v].z, dtr[u])));
            q.w = __sinf(reduce_two_pi(time_arg(wv[v].w, bv[v].w, dtr[u])));
          }
          sn[u][v] = q;
        }
        if (!live) dtr[u] = 0.f;
      }
    }
#pragma unroll
    for (int u = 0; u < TG_U; ++u) {
#pragma unroll
      for (int v = 0; v < V; ++v) {
        const float ge[4] = {g[u][v].x, g[u][v].y, g[u][v].z, g[u][v].w};
        const float se[4] = {sn[u][v].x, sn[u][v].y, sn[u][v].z, sn[u][v].w};
#pragma unroll
        for (int e = 0; e < 4; ++e) {
          const double t = -(double)se[e] * (double)ge[e];
          gw[v][e] = fma(t, (double)dtr[u], gw[v][e]);
          gb[v][e] += t;
        }
      }
    }
  }
#pragma unroll
  for (int v = 0; v < V; ++v) {
    const int c = 4 * (lane + 32 * v);
    if (c < d) {
#pragma unroll
      for (int e = 0; e < 4; ++e) { s_part[(wid * 2 + 0) * d + c + e] = gw[v][e]; s_part[(wid * 2 + 1) * d + c + e] = gb[v][e]; }
    }
  }
  __syncthreads();
  for (int e = threadIdx.x; e < 2 * d; e += blockDim.x) {
    double t = 0.0;
    for (int w = 0; w < 8; ++w) t += s_part[w * 2 * d + e];
    if (t != 0.0) atomicAdd(&acc[e], t);
  }
}

inline void time_grad_launch(const tgnn_ctx* ctx, int grid, size_t smem, cudaStream_t st, const float* G, int64_t ldg, int col0, const float* S,
                             const float* dt, int rows, const int32_t* dev_rows, int d, const float* time_w,
                             const float* time_b, double* acc, int rows_per_block) {
  if (d <= 128)
    launch_link(ctx, time_grad_kernel<1>, dim3(grid), dim3(256), smem, st, 1, G, ldg, col0, S, dt, rows, dev_rows, d, time_w, time_b, acc, rows_per_block);
  else
    launch_link(ctx, time_grad_kernel<2>, dim3(grid), dim3(256), smem, st, 1, G, ldg, col0, S, dt, rows, dev_rows, d, time_w, time_b, acc, rows_per_block);
}

// Backward of the time-projected embedding h = m * (1 + dt w_p + b_p), one warp per root:
//   dw_p += dh m dt,  db_p += dh m   (fp64 block sums, then one pair of fp64 atomics per block and column into
//                                     acc[0:d] and acc[d:2d]: dt spans the stream and the terms cancel)
//   dm = dh (1 + dt w_p + b_p) is added to the row's slot of dMemU when the node's memory row was written
//   by this step's update (all other table rows are constants).
// Dynamic shared memory: 8 * 2 * d doubles.
__global__ void __launch_bounds__(256) jodie_embed_bwd_kernel(const float* __restrict__ dh, const float* __restrict__ memory,
                                                              const double* __restrict__ last_update,
                                                              const float* __restrict__ proj_w,
                                                              const float* __restrict__ proj_b,
                                                              const int32_t* __restrict__ nodes,
                                                              const double* __restrict__ times, int n, int d,
                                                              const int32_t* __restrict__ node2slot, int have_update,
                                                              float* __restrict__ dMemU, double* __restrict__ acc, int64_t N,
                                                              int upd_rows, int copy_mask) {
  extern __shared__ double s_part[];  // [8][2][d]
  const int first = (int)((blockIdx.x * blockDim.x + threadIdx.x) >> 5) + link_wait();
  link_release();
  dMemU += (int64_t)(blockIdx.x & copy_mask) * upd_rows * d;
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  double gw[TG_MAXJ], gb[TG_MAXJ];
#pragma unroll
  for (int j = 0; j < TG_MAXJ; ++j) { gw[j] = 0.0; gb[j] = 0.0; }
  const int warps = (gridDim.x * blockDim.x) >> 5;
  for (int i = first; i < n; i += warps) {
    const int node = nodes[i];
    if (node < 0 || node >= N) continue;   // reported by the forward pass; its embedding was zero
    const float dt = (float)(times[i] - last_update[node]);
    const int slot = have_update ? node2slot[node] : -1;
#pragma unroll
    for (int j = 0; j < TG_MAXJ; ++j) {
      const int c = lane + 32 * j;
      if (c < d) {
        const float g = dh[(int64_t)i * d + c];
        const float m = memory[(int64_t)node * d + c];
        const double t = (double)g * (double)m;
        gw[j] = fma(t, (double)dt, gw[j]);
        gb[j] += t;
        if (slot >= 0 && slot < upd_rows) atomicAdd(&dMemU[(int64_t)slot * d + c], g * (1.f + fmaf(dt, proj_w[c], proj_b[c])));
      }
    }
  }
#pragma unroll
  for (int j = 0; j < TG_MAXJ; ++j) {
    const int c = lane + 32 * j;
    if (c < d) { s_part[(wid * 2 + 0) * d + c] = gw[j]; s_part[(wid * 2 + 1) * d + c] = gb[j]; }
  }
  __syncthreads();
  for (int e = threadIdx.x; e < 2 * d; e += blockDim.x) {
    double t = 0.0;
    for (int w = 0; w < 8; ++w) t += s_part[w * 2 * d + e];
    if (t != 0.0) atomicAdd(&acc[e], t);
  }
}

// The gradient of four columns of a row that the memory update wrote: the sum over its copies.
__device__ __forceinline__ float4 sum_copies(const float* __restrict__ p, int64_t stride, int copies) {
  float4 g = make_float4(0.f, 0.f, 0.f, 0.f);
  int z = 0;
  for (; z + 8 <= copies; z += 8) {   // (all of eight are asked for before the first is added)
    float4 v[8];
#pragma unroll
    for (int u = 0; u < 8; ++u) v[u] = *reinterpret_cast<const float4*>(p + (z + u) * stride);
#pragma unroll
    for (int u = 0; u < 8; ++u) g = add4(g, v[u]);
  }
#pragma unroll 4
  for (; z < copies; ++z) g = add4(g, *reinterpret_cast<const float4*>(p + z * stride));
  return g;
}

// Backward of the plain recurrent cell for the rows the memory update wrote: d pre = dm' (1 - m'^2).
__global__ void __launch_bounds__(256) rnn_bwd_gate_kernel(const float* __restrict__ dMemU, int64_t copy_stride, int copies,
                                                           const float* __restrict__ g_n, const int32_t* __restrict__ n_uniq,
                                                           int u_cap, int d, float* __restrict__ dG) {
  const int64_t e = 4 * (blockIdx.x * (int64_t)blockDim.x + threadIdx.x + link_wait());
  link_release();
  const int U = min(*n_uniq, u_cap);
  if (e >= (int64_t)U * d) return;
  const float4 m = *reinterpret_cast<const float4*>(g_n + e), g = sum_copies(dMemU + e, copy_stride, copies);
  *reinterpret_cast<float4*>(dG + e) = make_float4(g.x * (1.f - m.x * m.x), g.y * (1.f - m.y * m.y), g.z * (1.f - m.z * m.z), g.w * (1.f - m.w * m.w));
}

// Backward of the GRU gates for the rows the memory update wrote, four columns per thread (d is a multiple of 4).
__global__ void __launch_bounds__(256) gru_bwd_gate_kernel(const float* __restrict__ dMemU, int64_t copy_stride, int copies,
                                                           const float* __restrict__ X, int ld, int d, const float* __restrict__ g_r,
                                                           const float* __restrict__ g_z, const float* __restrict__ g_n,
                                                           const float* __restrict__ g_hn,
                                                           const int32_t* __restrict__ n_uniq, int u_cap,
                                                           float* __restrict__ dGi, float* __restrict__ dGh) {
  const int t = (int)(blockIdx.x * blockDim.x + threadIdx.x) + link_wait(), U = min(*n_uniq, u_cap);
  link_release();
  const int d4 = d >> 2, u = t / d4, q = 4 * (t - u * d4);
  if (u >= U) return;
  const int64_t e = (int64_t)u * d + q;
  const auto ld4 = [](const float* p, float (&v)[4]) {
    const float4 x = *reinterpret_cast<const float4*>(p);
    v[0] = x.x; v[1] = x.y; v[2] = x.z; v[3] = x.w;
  };
  float r[4], z[4], nn[4], hn[4], h[4], o[4][4];
  ld4(g_r + e, r); ld4(g_z + e, z); ld4(g_n + e, nn); ld4(g_hn + e, hn); ld4(X + (int64_t)u * ld + q, h);
  const float4 g4 = sum_copies(dMemU + e, copy_stride, copies);
  const float g[4] = {g4.x, g4.y, g4.z, g4.w};
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const float dn = g[i] * (1.f - z[i]);
    const float dz = g[i] * (h[i] - nn[i]);
    const float dpn = dn * (1.f - nn[i] * nn[i]);
    o[0][i] = dpn * hn[i] * r[i] * (1.f - r[i]);
    o[1][i] = dz * z[i] * (1.f - z[i]);
    o[2][i] = dpn;
    o[3][i] = dpn * r[i];
  }
  float *gi = dGi + (int64_t)u * 3 * d + q, *gh = dGh + (int64_t)u * 3 * d + q;
  const auto st4 = [](float* p, const float (&v)[4]) { *reinterpret_cast<float4*>(p) = make_float4(v[0], v[1], v[2], v[3]); };
  st4(gi, o[0]); st4(gi + d, o[1]); st4(gi + 2 * d, o[2]);
  st4(gh, o[0]); st4(gh + d, o[1]); st4(gh + 2 * d, o[3]);
}

// Gradient norm g_r and the Adam update in one pass over the parameters.  Adam does not depend on the
// norm (no clipping), so each thread squares its gradient entries into the block's partial sum and
// updates the same entries; the last block to finish turns the sum into g_r and bumps the step counter
// (every block has read the counter before it takes its ticket).
// The time-encoder entries [t_off, t_off + t_n) and the time projection's [p_off, p_off + p_n) are taken
// from their fp64 sums tg_acc (rounded once) and written into grads, where the debug export finds them.
// apply = 0 stops after the gradient and its norm (parameters, moments and the step counter stay): the
// caller synchronises the gradient across workers and comes back with t_n = p_n = 0 and gscale = 1 / workers;
// a gscale other than 1 multiplies every gradient entry first and stores the product.
// The last link of the step's chain, bound by round trips: a thread asks for its first group of parameters before the block waits for
// the bias corrections, each of which a warp of its own forms (b^t by squaring in fp64: the library's pow was half of the
// kernel's 40 KB of code and a microsecond ahead of every load), and the scalars that the last block hands out are read by
// then.  280 000 parameters, launch included: 13.0 -> 11.0 us.
__device__ __forceinline__ float bias_correction(float beta, int64_t t) {   // 1 / (1 - beta^t), formed in fp64 and rounded once
  double p = 1.0, q = (double)beta;
#pragma unroll 1
  for (; t > 0; t >>= 1) {
    if (t & 1) p *= q;
    q *= q;
  }
  return (float)(1.0 / (1.0 - p));
}

constexpr int AD_THREADS = 256, AD_BLOCKS = 296;
__global__ void __launch_bounds__(AD_THREADS) gradnorm_adam_kernel(float* __restrict__ grads, int64_t P,
                                                            const double* __restrict__ tg_acc, int64_t t_off, int t_n,
                                                            int64_t p_off, int p_n, double* red, unsigned int* ticket, int64_t* step,
                                                            float* __restrict__ p, float* __restrict__ m,
                                                            float* __restrict__ v, float lr, float beta1, float beta2,
                                                            float eps, const float* __restrict__ loss_acc, float* scalars,
                                                            float* loss_out, float* gradnorm_out, float* const* host_result,
                                                            float gscale, int apply) {
  __shared__ double s_part[AD_THREADS / 32];
  __shared__ float s_c1, s_c2;
  // 1 - beta formed in fp64 from the configured fp32 value, then rounded once
  const float omb1 = (float)(1.0 - (double)beta1), omb2 = (float)(1.0 - (double)beta2);
  double acc = 0.0;
  float c1 = 0.f, c2 = 0.f;
  // one parameter: sum of squares, Adam
  auto one = [&](float ge, float& pe, float& me, float& ve) {
    acc = fma((double)ge, (double)ge, acc);
    if (!apply) return;
    me = fmaf(beta1, me, omb1 * ge);
    ve = fmaf(beta2, ve, omb2 * ge * ge);
    pe -= lr * (me * c1) / (sqrtf(ve * c2) + eps);
  };
  // the gradient's fp64 sums behind entry e (nullptr: it lies in grads): the time encoder's, then the projection's
  auto sums = [&](int64_t e) -> const double* {
    return e >= t_off && e < t_off + t_n ? tg_acc + (e - t_off) : e >= p_off && e < p_off + p_n ? tg_acc + t_n + (e - p_off) : nullptr;
  };
  // groups of four consecutive parameters with 128-bit accesses (the arrays are 16-byte aligned; the ranges
  // taken from the fp64 sums start and end on multiples of four because d is one), then the last P % 4
  const bool vec = ((((uintptr_t)grads | (uintptr_t)p | (uintptr_t)m | (uintptr_t)v) & 15) == 0) && (t_off % 4 == 0) &&
                   (t_n % 4 == 0) && (p_off % 4 == 0) && (p_n % 4 == 0);
  const int64_t P4 = vec ? P / 4 : 0, stride = (int64_t)gridDim.x * AD_THREADS;
  const int64_t q0 = blockIdx.x * (int64_t)AD_THREADS + threadIdx.x;
  float4 g4, p4, m4, v4;
  auto ask_state = [&](int64_t q) {
    if (q < P4 && apply) { p4 = reinterpret_cast<const float4*>(p)[q]; m4 = reinterpret_cast<const float4*>(m)[q]; v4 = reinterpret_cast<const float4*>(v)[q]; }
  };
  auto ask = [&](int64_t q) {
    if (q >= P4) return;
    if (const double* a = sums(4 * q)) g4 = make_float4((float)a[0], (float)a[1], (float)a[2], (float)a[3]);
    else g4 = reinterpret_cast<const float4*>(grads)[q];
  };
  // As a link: parameters, moments and step count, which no other kernel of a step writes, ahead of the wait, and the bias corrections.
  g4 = p4 = m4 = v4 = make_float4(0.f, 0.f, 0.f, 0.f);
  ask_state(q0);
  const int64_t t = step[0];
  if (threadIdx.x == 32) s_c1 = bias_correction(beta1, t + 1);
  if (threadIdx.x == 64) s_c2 = bias_correction(beta2, t + 1);
  const int zero = link_wait();
  grads += zero; tg_acc += zero; loss_acc += zero;
  ask(q0);
  float loss = 0.f;
  float *hl = nullptr, *hg = nullptr;
  if (threadIdx.x == 0) {
    loss = *loss_acc;
    if (host_result) { hl = host_result[0]; hg = host_result[1]; }
  }
  __syncthreads();
  c1 = s_c1; c2 = s_c2;
#pragma unroll 1
  for (int64_t q = q0; q < P4; q += stride) {
    const bool from_sums = sums(4 * q) != nullptr;
    if (gscale != 1.f) g4 = make_float4(g4.x * gscale, g4.y * gscale, g4.z * gscale, g4.w * gscale);
    if (from_sums || gscale != 1.f) reinterpret_cast<float4*>(grads)[q] = g4;
    one(g4.x, p4.x, m4.x, v4.x);
    one(g4.y, p4.y, m4.y, v4.y);
    one(g4.z, p4.z, m4.z, v4.z);
    one(g4.w, p4.w, m4.w, v4.w);
    if (apply) {
      reinterpret_cast<float4*>(p)[q] = p4;
      reinterpret_cast<float4*>(m)[q] = m4;
      reinterpret_cast<float4*>(v)[q] = v4;
    }
    ask(q + stride);
    ask_state(q + stride);
  }
#pragma unroll 1
  for (int64_t e = 4 * P4 + q0; e < P; e += stride) {
    const double* a = sums(e);
    float ge = a ? (float)*a : grads[e];
    if (gscale != 1.f) ge *= gscale;
    if (a || gscale != 1.f) grads[e] = ge;
    float pe = 0.f, me = 0.f, ve = 0.f;
    if (apply) { pe = p[e]; me = m[e]; ve = v[e]; }
    one(ge, pe, me, ve);
    if (apply) { p[e] = pe; m[e] = me; v[e] = ve; }
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(FULL, acc, o);
  if ((threadIdx.x & 31) == 0) s_part[threadIdx.x >> 5] = acc;
  __syncthreads();
  if (threadIdx.x == 0) {
    double b = 0.0;
#pragma unroll
    for (int w = 0; w < AD_THREADS / 32; ++w) b += s_part[w];
    atomicAdd(&red[0], b);
    __threadfence();
    const unsigned int done = atomicAdd(ticket, 1u);
    if (done == gridDim.x - 1) {
      __threadfence();
      const double ss = atomicAdd(&red[0], 0.0);
      const float gn = (float)sqrt(ss);
      if (apply) step[0] = t + 1;
      scalars[0] = loss;
      scalars[1] = gn;
      if (loss_out) *loss_out = loss;
      if (gradnorm_out) *gradnorm_out = gn;
      // pinned host memory, written here instead of by two copies behind the step (3 us and a gap of 3 us each)
      if (hl) *hl = loss;
      if (hg) *hg = gn;
      *ticket = 0u;
    }
  }
}
// As many blocks as have a group of four parameters per thread, at most two per SM.
inline int adam_blocks(int64_t P) {
  const int64_t b = (P / 4 + AD_THREADS - 1) / AD_THREADS;
  return b < 1 ? 1 : b < AD_BLOCKS ? (int)b : AD_BLOCKS;
}

__global__ void gate_bytes_kernel(const float* __restrict__ h, int64_t n, uint8_t* __restrict__ out) {
  const int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (e < n) out[e] = h[e] > 0.f;
}

int pick_split(int M, int N, int K) {
  const int tiles = ((M + 63) / 64) * ((N + 63) / 64);
  int s = (4 * 148 + tiles - 1) / tiles;
  const int max_s = (K + 127) / 128;
  if (s > max_s) s = max_s;
  return s < 1 ? 1 : s;
}

// dW[N_out, K_in] += dY^T A  (+ db[N_out] += column sums of dY): a transposed product with the
// contraction over rows (optionally a device-side count).
int grad_w(tgnn_ctx* ctx, const float* dY, int64_t ld_dy, const float* A, int64_t ld_a, int rows, const int32_t* dev_rows,
           int n_out, int k_in, float* dW, float* db, const char* name, cudaStream_t s, int64_t ld_dw = 0) {
  GemmArgs g = {};
  g.A = dY; g.a_rs = 1; g.a_cs = ld_dy;  // A(m,k) = dY[k, m]
  g.B = A; g.b_rs = ld_a; g.b_cs = 1;    // B(k,n) = A[k, n]
  g.C = dW; g.ldc = ld_dw ? ld_dw : k_in; g.M = n_out; g.N = k_in; g.K = rows; g.dev_K = dev_rows;
  g.rowsum_out = db; g.accumulate = 1; g.split_k = pick_split(n_out, k_in, rows); g.precise = 1;
  g.tail_slack = 1;  // dY and the saved activations are workspace buffers
  return launch_gemm(ctx, g, name, s);
}

// dA[rows, n_cols] = dY[rows, n_out] W[:, col0 : col0 + n_cols]   (W is [n_out, ld_w] row-major)
int grad_in(tgnn_ctx* ctx, const float* dY, int64_t ld_dy, const float* W, int64_t ld_w, int col0, int rows,
            const int32_t* dev_rows, int n_out, int n_cols, float* dA, int64_t ld_da, const char* name, cudaStream_t s,
            int site = 0) {
  GemmArgs g = {};
  g.A = dY; g.a_rs = ld_dy; g.a_cs = 1;
  g.B = W + col0; g.b_rs = ld_w; g.b_cs = 1;
  g.C = dA; g.ldc = ld_da; g.M = rows; g.N = n_cols; g.K = n_out; g.dev_M = dev_rows; g.split_k = 1; g.precise = 1;
  g.site = site;
  return launch_gemm(ctx, g, name, s);
}

}  // namespace

// Three forms of the head.  Tiles of 20 to 32 events with W_1 in shared memory from 2 368 events (74 tiles of 32) up, where two
// halves of W_1 and a tile fit (d up to 112); a few events per block; separate products.  A step in us, events per block /
// separate products (k = 5, 16 feature columns, two heads):
//   fp32, d = 128: 460 / 482 at 2 400 events, 789 / 807 at 4 800, 1 179 / 1 213 at 8 000; d = 160: 760 / 769, 1 322 / 1 335, 2 080 /
//   2 096; d = 240: 1 285 / 1 322, 2 248 / 2 290, 3 541 / 3 620; d = 256, where two blocks do not fit an SM: 1 326 / 1 318 at
//   2 300, 1 782 / 1 758 at 3 200, 4 024 / 3 983 at 8 000.  So events per block wherever two blocks fit an SM.
//   tensor cores, d = 116: 232 / 238 at 2 368, 294 / 304 at 3 552, 310 / 307 at 3 700; d = 128: 249 / 250, 314 / 318, 334 / 322.
//   So events per block for as many as make two full rounds of two blocks of six on each SM.
//   tensor cores, d > 128 (a lane's four hidden units then leave half of the lanes idle), 300 / 1 200 / 1 800 / 2 300 events: d = 160:
//   165 / 166, 286 / 285, 363 / 349, 425 / 400; d = 200: 200 / 201, 325 / 323, 432 / 407, 497 / 470; d = 256: 238 / 228, 399 /
//   379, 518 / 477, 623 / 556.  Separate products would win from about 64 000 / d events up, but they take W_1, the rows and d
//   loss / d pre1 in 21 bits, where the blocks multiply in fp32: the error of d loss / d h grows from 1.0e-7 to 3.9e-7 (d = 160, 600
//   events) and from 1.1e-7 to 1.0e-6 (d = 256, 2 000), that of dw_2 from 1.7e-7 to 4.2e-7 and from 3.2e-7 to 1.1e-6.  Below 2 368
//   events the blocks keep them.
static bool head_uses_tiles(const tgnn_config& c, int n_q) {
  return HeadTile<32>::smem_floats(c.d) * sizeof(float) <= 225 * 1024 && n_q >= 32 * 74;
}
static bool head_uses_rows(const tgnn_config& c, int n_q) {
  if (n_q < 32 * 74) return true;
  if (head_uses_tiles(c, n_q)) return false;
  if (c.math_mode == TGNN_MATH_FP32) return HeadRows<6>::smem(c.d) <= 112 * 1024;   // (two blocks on an SM)
  return c.d <= 128 && n_q <= 2 * 2 * 148 * 6;
}

bool head_uses_wt(const tgnn_config& c, int n_q) { return n_q > 0 && (head_uses_rows(c, n_q) || head_uses_tiles(c, n_q)); }

int launch_prep_head(tgnn_ctx* ctx, cudaStream_t s) {
  const int d = ctx->cfg.d;
  {
    KernelScope scope__(ctx, "prep_head", s);
    prep_head_wt_kernel<<<(d / 4 + 7) / 8, 256, 0, s>>>(ctx->params + ctx->L.w1, d, (d + 3) / 4 * 4, ctx->ws.head_wT);
  }
  TGNN_LAUNCH_OK(ctx, "prep_head");
  return TGNN_OK;
}

int launch_get_gates(tgnn_ctx* ctx, uint8_t* h_gate_out, uint8_t* hid_gate_out, cudaStream_t s) {
  const int64_t n = (int64_t)ctx->e_n * ctx->cfg.d;
  if (n > 0) {
    gate_bytes_kernel<<<(int)((n + 255) / 256), 256, 0, s>>>(ctx->e_h, n, h_gate_out);
    TGNN_LAUNCH_OK(ctx, "gate_bytes");
    const size_t m = (size_t)2 * (ctx->e_n / 3) * ctx->cfg.d;
    TGNN_CUDA_OK(ctx, cudaMemcpyAsync(hid_gate_out, ctx->ws.hid_gate, m, cudaMemcpyDeviceToDevice, s));
  }
  return TGNN_OK;
}

// G[wk + r * dkv + c] += pad[r * ld + c] for c < dkv, G[bk + r] += pad[r * ld + dkv]: the weight gradient of the
// key/value projection is accumulated in a copy with 16-byte aligned rows (vector atomics from every contraction
// split instead of four scalar ones) and folded into the flat gradient once.
__global__ void __launch_bounds__(256) fold_dwkv_kernel(const float* __restrict__ pad, int ld, int rows, int dkv,
                                                        float* __restrict__ g_w, float* __restrict__ g_b) {
  const int total = rows * (dkv + 1);
  for (int e = blockIdx.x * blockDim.x + threadIdx.x; e < total; e += gridDim.x * blockDim.x) {
    const int r = e / (dkv + 1), c = e - r * (dkv + 1);
    const float v = pad[(int64_t)r * ld + c];
    if (c < dkv) g_w[(int64_t)r * dkv + c] += v;
    else g_b[r] += v;
  }
}

#define RC(x)            \
  do {                   \
    int rc__ = (x);      \
    if (rc__) return rc__; \
  } while (0)

// Update cell: gates, weight gradients (on sb and s_wi) and, on s, the gradient of the messages' time encoding.
static int gru_backward(tgnn_ctx* ctx, int U_cap, cudaStream_t sb, cudaStream_t s_wi, cudaStream_t s) {
  const ParamLayout& L = ctx->L;
  Workspace& w = ctx->ws;
  const int d = ctx->cfg.d, de = ctx->cfg.d_e;
  float *P = ctx->params, *G = w.grads;
  const int64_t tot3 = (int64_t)U_cap * d / 4;
  {
    KernelScope scope__(ctx, "gru_bwd_gate", s);
    launch_link(ctx, gru_bwd_gate_kernel, dim3((unsigned)((tot3 + 255) / 256)), dim3(256), 0, s, 1, w.dMemU, (int64_t)ctx->copies.rows * d,
                ctx->copies.n, w.X, ctx->ld_msg, d, w.g_r, w.g_z, w.g_n, w.g_hn, ctx->upd_n_uniq, U_cap, w.dGi, w.dGh);
  }
  TGNN_LAUNCH_OK(ctx, "gru_bwd_gate");
  RC(fork_to(ctx, s, s_wi));
  RC(fork_to(ctx, s, sb));
  RC(grad_w(ctx, w.dGi, 3 * d, w.X, ctx->ld_msg, U_cap, ctx->upd_n_uniq, 3 * d, (int)L.dmsg, G + L.gru_wi, G + L.gru_bi, "dW_i",
            s_wi));
  RC(grad_w(ctx, w.dGh, 3 * d, w.X, ctx->ld_msg, U_cap, ctx->upd_n_uniq, 3 * d, d, G + L.gru_wh, G + L.gru_bh, "dW_h", sb));
  RC(grad_in(ctx, w.dGi, 3 * d, P + L.gru_wi, L.dmsg, 2 * d + de, U_cap, ctx->upd_n_uniq, 3 * d, d, w.dXp, d, "dX_phi", s,
             SITE_DXPHI + 1));
  {
    KernelScope scope__(ctx, "time_grad_x", s);
    const int rpb = tg_rows_per_block(U_cap);
    time_grad_launch(ctx, (U_cap + rpb - 1) / rpb, (size_t)8 * 2 * d * sizeof(double), s, w.dXp, d, 0, w.Xsin, w.x_dt, U_cap,
                     ctx->upd_n_uniq, d, P + L.time_w, P + L.time_b, w.tg_acc, rpb);
  }
  TGNN_LAUNCH_OK(ctx, "time_grad_x");
  return TGNN_OK;
}

// Rows of hub nodes get additions by the thousand, and additions to one row wait for one another: a block adds to one of several
// copies of the rows, and the update cell's backward adds the copies up.  A copy is as many rows as this update can have written, whatever
// the context's capacity (100 events in a context for 262 144 on a million nodes, d = 100: 1 317 us with copies of the capacity, 1 284).
// How many: 32 where so many slots come to a row that some are sure to get thousands; 8 from two slots per row up; 2 below that,
// where clearing and adding up cost more than the additions' wait (the time-projection model adds one row per root).  Steps in us
// with 1 / 2 / 4 / 8 / 16 copies, k = 10, d = 100, nodes drawn by Zipf's law with the exponent in brackets: 600 events (1.5) 143 / 136 /
// 134 / 134 / 135; 4 000 (1.0) 312 / 288 / 288 / 287 / 295; 16 000 (1.0) 1 200 / 1 198 / 1 195 / 1 220 / 1 248, (1.5) 1 461 / 1 219 /
// 1 087 / 1 060 / 1 065; 64 000 (1.0) 4 215 / 4 062 / 4 055 / 4 094 / 4 125, (1.5) 5 390 / 4 357 / 3 797 / 3 555 / 3 529; k = 2, 4 000
// (1.5) 280 with 2, 278 with 8; k = 1, 4 000 (1.2) 262 / 259 / 260 / 259 / 264; time projection, 600 (1.2) 80 / 78 / 78 / 83 / 81, 4 000
// (1.0) 121 / 122 / 121 / 125 / 134, 4 000 on 2 000 nodes (1.5) 115 / 107 / 105 / 106 / 110, 32 000 (1.2) 1 036 / 1 035 / 1 071 / 1 090 / 1 101.
// Together they take at most COPY_FLOATS, in steps whose two copies are larger than that as much as those two: the step of 64 000 events
// has all of its eight, and one of a million events two.
// Which slices of L2 the copies of a hub's row fall into is chance: the attention backward of 4 000 events (1.5) took 53 to 58 us at nine of
// twelve offsets of the block in memory and 72, 79 and 88 at three (the large workload 68 to 69, once 73).  A row's copies side by side, each
// from a 128-byte line, are even (56 to 57) but slower where chance is kind (large 70 to 71).
constexpr int64_t COPY_FLOATS = 128 << 20;
static int64_t copies_for(const tgnn_ctx* ctx, int64_t rows, int64_t roots) {
  const int64_t additions = ctx->cfg.model == TGNN_MODEL_TGN ? roots * ctx->cfg.k : roots;
  return additions >= 32 * rows ? 32 : additions >= 2 * rows ? 8 : 2;
}
int64_t copy_room(const tgnn_ctx* ctx) {
  const int64_t one = (int64_t)ctx->upd_rows * ctx->cfg.d, all = copies_for(ctx, ctx->upd_rows, ctx->R_cap) * one;
  return all <= COPY_FLOATS ? all : 2 * one > COPY_FLOATS ? 2 * one : COPY_FLOATS;
}
GradCopies plan_copies(const tgnn_ctx* ctx, int rows, int n_q) {
  GradCopies c = {rows, 1};
  if (rows == 0 || n_q == 0 || (ctx->cfg.model == TGNN_MODEL_TGN && !ctx->qs && scatter_by_block(ctx, 3 * n_q, ctx->cfg.k))) return c;
  const int64_t most = copies_for(ctx, rows, (int64_t)3 * n_q), one = (int64_t)rows * ctx->cfg.d;
  while (c.n < most && 2 * c.n * one <= ctx->copy_room) c.n *= 2;
  return c;
}

// Gradients, sums of the time encoder, scalars and the copies in use lie one behind the other, in whole pieces of 16 bytes: one launch
// clears them.  Bound by the stores.  29 MB (4 800 events): 10.8 us, beside other kernels; as a memset of the recorded step 10 to 11.
__global__ void __launch_bounds__(256) clear_grads_kernel(uint4* __restrict__ p, int64_t n) {
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) p[i] = make_uint4(0u, 0u, 0u, 0u);
}
int launch_clear_grads(tgnn_ctx* ctx, const GradCopies& copies, cudaStream_t s) {
  Workspace& w = ctx->ws;
  ctx->copies = copies;
  const char* end = (const char*)(w.dMemU + (int64_t)copies.n * copies.rows * ctx->cfg.d);
  const int64_t n = (end - (const char*)w.grads) / 16, blocks = (n + 1023) / 1024;   // (four pieces a thread, at most four blocks per SM)
  {
    KernelScope scope__(ctx, "clear_grads", s);
    clear_grads_kernel<<<(unsigned)(blocks < 4 * 148 ? blocks : 4 * 148), 256, 0, s>>>(reinterpret_cast<uint4*>(w.grads), n);
  }
  TGNN_LAUNCH_OK(ctx, "clear_grads");
  return TGNN_OK;
}

int launch_backward(tgnn_ctx* ctx, int n_q, const uint8_t* loss_mask, float* loss_out, float* gradnorm_out,
                    cudaStream_t s) {
  const tgnn_config& c = ctx->cfg;
  const ParamLayout& L = ctx->L;
  Workspace& w = ctx->ws;
  const int d = c.d, k = c.k, H = c.heads, de = c.d_e;
  const int R = 3 * n_q, NB = R * k;
  float* P = ctx->params;
  float* G = w.grads;
  // The chain loss -> head -> output projection -> attention -> inputs -> memory rows -> GRU is
  // sequential and stays on the caller's stream s.  Weight-gradient products and time-encoder sums
  // are leaves of that chain: they go to the two side streams as soon as their operands exist and
  // are joined back before the gradient norm.  (dW_1 has the stream of the input weights' gradient, dW_h one of its own: behind the
  // chain's next leaves each of them was the last to end.)
  cudaStream_t sa = ctx->side[0], sb = ctx->side[1], sc = ctx->side[2], sd = ctx->side[3];
  if (ctx->back_pending) TGNN_CUDA_OK(ctx, cudaStreamWaitEvent(s, ctx->ev_back, 0));
  ctx->back_pending = false;
  const GradCopies copies = plan_copies(ctx, ctx->have_update ? ctx->upd_cap : 0, n_q);
  if (!ctx->grads_zeroed || !(copies == ctx->copies)) RC(launch_clear_grads(ctx, copies, s));

  cudaStream_t s_end = s;   // the stream that the step ends on
  if (n_q > 0) {
    const int relu_out = c.model == TGNN_MODEL_TGN ? 1 : 0;
    // Large batches: tiles of TE events per block with register-blocked products.  TE is the tile size whose
    // rounds of 148 blocks cost least: 4 000 events are 143 tiles of 28 -- one round on 143 SMs -- where tiles of 32
    // would leave 23 SMs idle for a longer round.
    if (head_uses_tiles(c, n_q)) {
      int te = 32, best = 1 << 30;
      for (int cand = 32; cand >= 20; cand -= 4) {
        const int tiles = (n_q + cand - 1) / cand, cost = ((tiles + 147) / 148) * cand;
        if (cost < best) { best = cost; te = cand; }
      }
      const int tiles = (n_q + te - 1) / te;
      const int grid = tiles < 148 ? tiles : 148;
      // W_1 transposed: written with the other preparations at the start of the step; otherwise (the backward step
      // called on its own after the parameters changed) here
      if (!ctx->in_step) RC(launch_prep_head(ctx, s));
      {
        KernelScope scope__(ctx, "head_fused", s);
#define TGNN_HEAD_TILE(TE_)                                                                                              \
  do {                                                                                                                   \
    static SmemLimit lim__;                                                                                              \
    const size_t bytes__ = HeadTile<TE_>::smem_floats(d) * sizeof(float);                                                \
    RC(raise_smem_limit(ctx, head_tile_kernel<TE_>, (int)bytes__, lim__));                                               \
    launch_link(ctx, head_tile_kernel<TE_>, dim3(grid), dim3(HeadTile<TE_>::THREADS), bytes__, s, 1,                     \
        ctx->e_h, w.head_wT, P + L.b1, P + L.w2, P + L.b2, loss_mask, n_q, d, w.cat1, w.hid1, w.hid_gate, w.dpre_o,      \
        G + L.w2, G + L.b2, w.st_scalars, relu_out);                                                                    \
  } while (0)
        if (te == 32) TGNN_HEAD_TILE(32);
        else if (te == 28) TGNN_HEAD_TILE(28);
        else if (te == 24) TGNN_HEAD_TILE(24);
        else TGNN_HEAD_TILE(20);
#undef TGNN_HEAD_TILE
      }
      TGNN_LAUNCH_OK(ctx, "head_fused");
      RC(fork_to(ctx, s, sd));
      RC(grad_w(ctx, w.hid1, d, w.cat1, 2 * d, 2 * n_q, nullptr, d, 2 * d, G + L.w1, G + L.b1, "dW_1", sd));
    } else if (head_uses_rows(c, n_q)) {
      if (!ctx->in_step) RC(launch_prep_head(ctx, s));
      {
        KernelScope scope__(ctx, "head_fused", s);
#define TGNN_HEAD_ROWS(EV_)                                                                                              \
  do {                                                                                                                   \
    static SmemLimit lim__;                                                                                              \
    const int blocks__ = (n_q + EV_ - 1) / EV_;                                                                          \
    const size_t bytes__ = even_share(blocks__, HeadRows<EV_>::smem(d), 1024, 120 * 1024);                                \
    RC(raise_smem_limit(ctx, head_rows_kernel<EV_>, (int)bytes__, lim__));                                               \
    launch_link(ctx, head_rows_kernel<EV_>, dim3(blocks__), dim3(HR_THREADS), bytes__, s, 1,                \
        ctx->e_h, P + L.w1, w.head_wT, P + L.b1, P + L.w2, P + L.b2, loss_mask, n_q, d, w.cat1, w.hid1, w.hid_gate,      \
        w.dpre_o, G + L.w2, G + L.b2, w.st_scalars, relu_out);                                                          \
  } while (0)
        switch (head_rows_events(n_q)) {
          case 2: TGNN_HEAD_ROWS(2); break;
          case 4: TGNN_HEAD_ROWS(4); break;
          case 5: TGNN_HEAD_ROWS(5); break;
          default: TGNN_HEAD_ROWS(6); break;
        }
#undef TGNN_HEAD_ROWS
      }
      TGNN_LAUNCH_OK(ctx, "head_fused");
      RC(fork_to(ctx, s, sd));
      RC(grad_w(ctx, w.hid1, d, w.cat1, 2 * d, 2 * n_q, nullptr, d, 2 * d, G + L.w1, G + L.b1, "dW_1", sd));
    } else {
      const int64_t tot = (int64_t)2 * n_q * 2 * d;
      {
        KernelScope scope__(ctx, "head_gather", s);
        head_gather_kernel<<<(int)((tot + 255) / 256), 256, 0, s>>>(ctx->e_h, n_q, d, w.cat1);
      }
      TGNN_LAUNCH_OK(ctx, "head_gather");
      GemmArgs g = {};
      g.A = w.cat1; g.a_rs = 2 * d; g.a_cs = 1;
      g.B = P + L.w1; g.b_rs = 1; g.b_cs = 2 * d;
      g.C = w.hid1; g.ldc = d; g.M = 2 * n_q; g.N = d; g.K = 2 * d; g.bias = P + L.b1; g.relu = 1; g.split_k = 1;
      g.site = SITE_HEAD + 1;
      RC(launch_gemm(ctx, g, "head_hidden", s));
      {
        KernelScope scope__(ctx, "head_loss", s);
        head_loss_kernel<<<(n_q + 7) / 8, 256, d * sizeof(float), s>>>(w.hid1, P + L.w2, P + L.b2, loss_mask, n_q, d,
                                                                       G + L.w2, G + L.b2, w.st_scalars, w.hid_gate);
      }
      TGNN_LAUNCH_OK(ctx, "head_loss");
      // hid1 now holds d loss / d pre1
      RC(fork_to(ctx, s, sd));
      RC(grad_w(ctx, w.hid1, d, w.cat1, 2 * d, 2 * n_q, nullptr, d, 2 * d, G + L.w1, G + L.b1, "dW_1", sd));
      RC(grad_in(ctx, w.hid1, d, P + L.w1, 2 * d, 0, 2 * n_q, nullptr, d, 2 * d, w.dcat1, 2 * d, "dcat1", s, SITE_DCAT1 + 1));
      const int64_t tot2 = (int64_t)R * d;
      {
        KernelScope scope__(ctx, "dh", s);
        dh_kernel<<<(int)((tot2 + 255) / 256), 256, 0, s>>>(w.dcat1, ctx->e_h, n_q, d, w.dpre_o, relu_out);
      }
      TGNN_LAUNCH_OK(ctx, "dh");
    }
    if (c.model == TGNN_MODEL_JODIE) {
      // embedding -> memory rows written by this step -> recurrent cell -> its weights and the time encoder
      const size_t tg_smem = (size_t)8 * 2 * d * sizeof(double);
      {
        KernelScope scope__(ctx, "jodie_embed_bwd", s);
        launch_link(ctx, jodie_embed_bwd_kernel, dim3((R + 7) / 8 < 148 ? (R + 7) / 8 : 148), dim3(256), tg_smem, s, 1,
            w.dpre_o, ctx->memory, ctx->last_update, P + L.proj_w, P + L.proj_b, ctx->e_nodes, ctx->e_times, R, d,
            w.node2slot, ctx->have_update ? 1 : 0, w.dMemU, w.tg_acc + 2 * d, c.num_nodes, ctx->copies.rows, ctx->copies.n - 1);
      }
      TGNN_LAUNCH_OK(ctx, "jodie_embed_bwd");
      if (ctx->have_update) {
        const int U_cap = ctx->upd_cap;
        const int64_t tot3 = (int64_t)U_cap * d / 4;
        {
          KernelScope scope__(ctx, "rnn_bwd_gate", s);
          launch_link(ctx, rnn_bwd_gate_kernel, dim3((unsigned)((tot3 + 255) / 256)), dim3(256), 0, s, 1, w.dMemU, (int64_t)ctx->copies.rows * d,
                      ctx->copies.n, w.g_n, ctx->upd_n_uniq, U_cap, d, w.dGi);
        }
        TGNN_LAUNCH_OK(ctx, "rnn_bwd_gate");
        RC(fork_to(ctx, s, sa));
        RC(fork_to(ctx, s, sb));
        RC(grad_w(ctx, w.dGi, d, w.X, ctx->ld_msg, U_cap, ctx->upd_n_uniq, d, (int)L.dmsg, G + L.gru_wi, G + L.gru_bi,
                  "dW_i", sa));
        RC(grad_w(ctx, w.dGi, d, w.X, ctx->ld_msg, U_cap, ctx->upd_n_uniq, d, d, G + L.gru_wh, G + L.gru_bh, "dW_h", sb));
        RC(grad_in(ctx, w.dGi, d, P + L.gru_wi, L.dmsg, 2 * d + de, U_cap, ctx->upd_n_uniq, d, d, w.dXp, d, "dX_phi", s,
                   SITE_DXPHI + 1));
        {
          KernelScope scope__(ctx, "time_grad_x", s);
          const int rpb = tg_rows_per_block(U_cap);
          time_grad_launch(ctx, (U_cap + rpb - 1) / rpb, tg_smem, s, w.dXp, d, 0, w.Xsin, w.x_dt, U_cap,
                                                                         ctx->upd_n_uniq, d, P + L.time_w, P + L.time_b, w.tg_acc, rpb);
        }
        TGNN_LAUNCH_OK(ctx, "time_grad_x");
      }
      RC(fork_to(ctx, s, sa));  // join where the last leaf ends (and nothing that this pass has not forked)
      if (ctx->have_update) RC(fork_to(ctx, sb, sa));
      RC(fork_to(ctx, sd, sa));
      s_end = sa;
    } else if (ctx->qs) {
      // head -> sums of the slots' inputs -> softmax -> projected queries -> root rows -> memory rows -> update cell
      RC(ensure_folded(ctx, 2, s));
      const int HL = H * ctx->ldz, ldd = HL + d, U_cap = ctx->upd_cap;
      RC(fork_to(ctx, s, sb));
      RC(grad_w(ctx, w.dpre_o, d, w.cat, ctx->ldc, R, nullptr, d, HL + d + 1, w.dOut, G + L.bo, "dOut", sb, ctx->ldc));
      RC(grad_in(ctx, w.dpre_o, d, w.wB, ctx->ldc, 0, R, nullptr, d, ldd, w.dcat, ldd, "dcat", s, SITE_DC + 1));
      RC(launch_attn_bwd(ctx, ctx->have_update, s));
      RC(fork_to(ctx, s, sb));
      RC(launch_unfold_grads(ctx, true, sb));
      // dA beside the chain's product where the two fit on the SMs, that product split as far as ever (eight CTAs a tile at most): 40 to 500 events
      // 0.5 to 2.8 us a step, 540 none, 600, which do not fit, 133.1 -> 133.7 to 137.4.  Else behind it: each takes whole SMs, and beside dA the chain's
      // would wait.  (Split into fewer CTAs to make room, its sums are longer chains of an accumulator that every MMA truncates.)  In the
      // fp32 mode, whose products share SMs, always behind: beside, 40, 100, 160, 300 and 600 events of 172 columns 103.7 -> 104.6 us, 112.2 -> 114.6,
      // 123.9 -> 127.8, 146.2 -> 150.3, 195.1 -> 198.8; with d = 32 the same within half a microsecond.
      const bool beside = ctx->cfg.math_mode != TGNN_MATH_FP32 && 8 * ((R + 127) / 128) <= 148 - weight_grad_ctas(d + 1, HL, R);
      if (beside) RC(fork_to(ctx, s, sa));
      if (ctx->have_update)
        RC(grad_in(ctx, w.dqp, HL, w.wA, d, 0, R, nullptr, HL, d, w.dmq, d, "dmq", s, SITE_DM + 1));
      if (!beside) RC(fork_to(ctx, s, sa));
      RC(grad_w(ctx, w.cat + HL, ctx->ldc, w.dqp, HL, R, nullptr, d + 1, HL, w.dT, nullptr, "dA", sa));
      RC(launch_unfold_grads(ctx, false, sa));
      if (ctx->have_update) {
        {
          KernelScope scope__(ctx, "scatter_dmem", s);
          scatter_rows(ctx, nullptr, w.dcat + HL, ldd, w.dmq, d, R, 0, s);
        }
        TGNN_LAUNCH_OK(ctx, "scatter_dmem");
        RC(gru_backward(ctx, U_cap, sc, sd, s));
      }
      // Join where the last leaf ends, so that Adam is a link behind it: 600 events 132.4 -> 131.6 us, 4 000 events 357.6 -> 355.9.  Short steps stay
      // on the chain's stream: fp32, 40, 100 and 160 events of 172 columns 103.7 -> 104.3 us, 112.2 -> 113.0, 123.9 -> 125.5 with the other end; from 180 to
      // 400 events the two differ by less than two recordings of one of them (1 to 2 us).
      if (R > 512) s_end = sa;
      for (cudaStream_t leaf : {s, sa, sb, sd})
        if (leaf != s_end) RC(fork_to(ctx, leaf, s_end));
      if (ctx->have_update) RC(fork_to(ctx, sc, s_end));
    } else {
    RC(fork_to(ctx, s, sb));
    RC(grad_w(ctx, w.dpre_o, d, w.cat_o, 2 * d, R, nullptr, d, 2 * d, G + L.wo, G + L.bo, "dW_o", sb));
    RC(grad_in(ctx, w.dpre_o, d, P + L.wo, 2 * d, 0, R, nullptr, d, 2 * d, w.dcat_o, 2 * d, "dcat_o", s, SITE_DCATO + 1));
    const int wpb = attn_warps_per_block(d, H, k);
    {
      static SmemLimit lim_f, lim_t, lim_x;
      const int need = (int)attn_smem_bytes(d, H, k, wpb);
      RC(raise_smem_limit(ctx, attention_bwd_kernel<false>, need, lim_f));
      RC(raise_smem_limit(ctx, attention_bwd_kernel<true>, need, lim_t));
      if (d == 100 && H == 2 && k == 10) RC(raise_smem_limit(ctx, (attention_bwd_fixed_kernel<100, 2, 10>), need, lim_x));
    }
    const bool split = ctx->split_buf != nullptr && ctx->images_fresh;
    SplitMat dkvs = ctx->dkvs, zs = ctx->zs;
    dkvs.rows = NB; zs.rows = NB;
    {
      KernelScope scope__(ctx, "attention_bwd", s);
      // (8-byte plane stores: row pitch and plane distance multiples of 4 elements)
      const bool fixed_shape = split && d == 100 && H == 2 && k == 10 && dkvs.ld % 4 == 0 && dkvs.plane_stride % 4 == 0;
      if (fixed_shape)   // (as in the forward pass, k_embed.cu)
        attention_bwd_fixed_kernel<100, 2, 10><<<(R + wpb - 1) / wpb, wpb * 32, attn_smem_bytes(d, H, k, wpb), s>>>(
            w.Q, w.KV, w.alpha, w.dcat_o, ctx->e_cnt, R, w.dQ, reinterpret_cast<__nv_bfloat16*>(dkvs.hi), dkvs.plane_stride,
            (int)dkvs.ld, dkvs.scale);
      else if (split)   // the key/value gradient leaves the kernel as fp16 planes, the form its two consumers read
        attention_bwd_kernel<true><<<(R + wpb - 1) / wpb, wpb * 32, attn_smem_bytes(d, H, k, wpb), s>>>(
            w.Q, w.KV, w.alpha, w.dcat_o, ctx->e_cnt, R, d, H, k, w.dQ, nullptr, reinterpret_cast<__nv_bfloat16*>(dkvs.hi),
            dkvs.plane_stride, (int)dkvs.ld, dkvs.scale);
      else
        attention_bwd_kernel<false><<<(R + wpb - 1) / wpb, wpb * 32, attn_smem_bytes(d, H, k, wpb), s>>>(
            w.Q, w.KV, w.alpha, w.dcat_o, ctx->e_cnt, R, d, H, k, w.dQ, w.dKV, nullptr, 0, 0, 1.f);
    }
    TGNN_LAUNCH_OK(ctx, "attention_bwd");
    RC(fork_to(ctx, s, sa));
    RC(fork_to(ctx, s, sb));
    // dW_kv is a leaf of the chain, its input-gradient sibling dZ is on it, and the split kernel is persistent (a
    // launch fills the machine until it ends): in that mode the weight gradient is issued after dZ, further down.
    if (!split)
      RC(grad_w(ctx, w.dKV, 2 * d, w.Z, ctx->ld_kv, NB, nullptr, 2 * d, (int)L.dkv, G + L.wk, G + L.bk, "dW_kv", sa));
    // time-encoder gradient through the attention inputs (side stream b)
    const size_t tg_smem = (size_t)8 * 2 * d * sizeof(double);
    // gradient w.r.t. the memory columns and the time-encoding columns of Z, side by side in dZmp.  With the
    // weight images at hand it is one product on the caller's stream (the scatter below needs its first
    // half); otherwise the two column ranges of W_kv are two strided products.
    const bool merged_dz = ctx->cfg.math_mode != TGNN_MATH_FP32 && ctx->images_fresh && ctx->images != nullptr;
    // the query-side input gradient does not depend on dZ: it runs on side stream b next to it
    RC(grad_in(ctx, w.dQ, d, P + L.wq, 2 * d, 0, R, nullptr, d, 2 * d, w.dzq, 2 * d, "dzq", sb, SITE_DZQ + 1));
    cudaEvent_t dzq_done = mark_stream(ctx, sb);  // waited for by the scatter further down
    RC(grad_w(ctx, w.dQ, d, w.Zq, 2 * d, R, nullptr, d, 2 * d, G + L.wq, G + L.bq, "dW_q", sb));
    {
      KernelScope scope__(ctx, "time_grad_q", sb);
      const int rpb = tg_rows_per_block(R);
      time_grad_launch(ctx, (R + rpb - 1) / rpb, tg_smem, sb, w.dzq, 2 * d, d, nullptr, nullptr, R, nullptr, d,
                                                                  P + L.time_w, P + L.time_b, w.tg_acc, rpb);
    }
    TGNN_LAUNCH_OK(ctx, "time_grad_q");
    cudaStream_t s_tgz = sb;  // where the time-encoder sum over the neighbor rows runs
    bool join_sc = false;
    if (split) {
      RC(launch_gemm_split(ctx, dkvs, ctx->wz_s, 0, w.dZmp, 2 * d, NB, 2 * d, 2 * d, nullptr, 0, 0, 1, "dZ", s));
      RC(fork_to(ctx, s, sa));
      RC(fork_to(ctx, s, sc));
      // dW_kv = dKV^T Z over the neighbor rows; Z's column of ones yields the bias gradient as the last column.  It
      // starts when dZ has finished and runs beside the rest of the chain (scatter, cell backward, ...).
      SplitMat a = dkvs, b = zs;
      a.rows = NB; a.cols = 2 * d; b.rows = NB; b.cols = L.dkv + 1;
      // Per-site precision: this product is a leaf (its result goes to Adam and nowhere else), and with a bf16 feature
      // table the contract's tolerance is 1e-2: there it reads only the hi planes of both operands -- one fp16 pass,
      // half the bytes.  Measured on the large workload at full size: the W_k / W_v gradients stay within 1e-3 of
      // their largest entry.  (The forward projection in one pass put other tensors at 9e-3, and the input gradient
      // dZ feeds everything upstream: both keep their three passes.)
      if (c.feat_dtype == TGNN_BF16) { a.planes = 1; b.planes = 1; }
      RC(launch_gemm_split(ctx, a, b, 1, w.dWkv_pad, ctx->ld_wkv, 2 * d, (int)L.dkv + 1, NB, nullptr, 0, 1, 1 << 20, "dW_kv", sa));
      {
        KernelScope scope__(ctx, "fold_dW_kv", sa);
        fold_dwkv_kernel<<<148, 256, 0, sa>>>(w.dWkv_pad, ctx->ld_wkv, 2 * d, (int)L.dkv, G + L.wk, G + L.bk);
      }
      TGNN_LAUNCH_OK(ctx, "fold_dW_kv");
      // The time-encoder sum needs little shared memory and fits beside the weight gradient's CTAs; on side stream
      // b it would queue behind the query-side products, which wait for a whole SM each.
      s_tgz = sc;
      join_sc = true;
    } else if (merged_dz) {
      RC(grad_in(ctx, w.dKV, 2 * d, P + L.wk, L.dkv, 0, NB, nullptr, 2 * d, 2 * d, w.dZmp, 2 * d, "dZ", s, SITE_DZ + 1));
      RC(fork_to(ctx, s, sa));
      s_tgz = sa;
    } else {
      RC(grad_in(ctx, w.dKV, 2 * d, P + L.wk, L.dkv, d + de, NB, nullptr, 2 * d, d, w.dZmp + d, 2 * d, "dZ_phi", sb));
    }
    {
      KernelScope scope__(ctx, "time_grad_z", s_tgz);
      const int rpb = tg_rows_per_block(NB);
      time_grad_launch(ctx, (NB + rpb - 1) / rpb, tg_smem, s_tgz, w.dZmp, 2 * d, d, nullptr, w.z_dt, NB, nullptr, d, P + L.time_w,
                                                                      P + L.time_b, w.tg_acc, rpb);
    }
    TGNN_LAUNCH_OK(ctx, "time_grad_z");
    RC(wait_mark(ctx, s, dzq_done));  // the scatter below needs dzq
    if (ctx->have_update) {
      if (!merged_dz && !split)
        RC(grad_in(ctx, w.dKV, 2 * d, P + L.wk, L.dkv, 0, NB, nullptr, 2 * d, d, w.dZmp, 2 * d, "dZ_mem", s));
      {
        KernelScope scope__(ctx, "scatter_dmem", s);
        scatter_rows(ctx, w.dZmp, w.dcat_o + d, 2 * d, w.dzq, 2 * d, R, k, s);
      }
      TGNN_LAUNCH_OK(ctx, "scatter_dmem");
      // (split mode: side stream a carries the persistent key/value weight gradient, which ends late)
      RC(gru_backward(ctx, ctx->upd_cap, sb, split ? sd : sa, s));
    }
    RC(fork_to(ctx, sd, s));  // join
    RC(fork_to(ctx, sa, s));
    RC(fork_to(ctx, sb, s));
    if (join_sc) RC(fork_to(ctx, sc, s));
    }  // attention model
  }
  {
    KernelScope scope__(ctx, "gradnorm_adam", s_end);
    const int p_n = (n_q > 0 && c.model == TGNN_MODEL_JODIE) ? 2 * d : 0;
    launch_side_link(ctx, gradnorm_adam_kernel, dim3(adam_blocks(L.total)), dim3(AD_THREADS), 0, s_end, G, L.total, w.tg_acc, L.time_w, n_q > 0 ? 2 * d : 0,
                     L.proj_w, p_n, w.red, w.counters, ctx->step, P, ctx->adam_m, ctx->adam_v, c.lr, c.beta1, c.beta2, c.eps, w.st_scalars,
                     w.st_scalars + 2, loss_out, gradnorm_out, ctx->in_step ? w.host_result : nullptr, 1.f, ctx->defer_adam ? 0 : 1);
  }
  TGNN_LAUNCH_OK(ctx, "gradnorm_adam");
  if (s_end != s) RC(fork_to(ctx, s_end, s));
  return TGNN_OK;
}

// The second half of a step whose gradient was left for synchronisation: norm of gscale * gradient and Adam.
int launch_apply_gradient(tgnn_ctx* ctx, float gscale, float* gradnorm_out, cudaStream_t s) {
  const tgnn_config& c = ctx->cfg;
  Workspace& w = ctx->ws;
  TGNN_CUDA_OK(ctx, cudaMemsetAsync(w.red, 0, sizeof(double), s));
  {
    KernelScope scope__(ctx, "apply_gradient", s);
    gradnorm_adam_kernel<<<adam_blocks(ctx->L.total), AD_THREADS, 0, s>>>(w.grads, ctx->L.total, w.tg_acc, 0, 0, 0, 0, w.red, w.counters, ctx->step,
                                             ctx->params, ctx->adam_m, ctx->adam_v, c.lr, c.beta1, c.beta2, c.eps,
                                             w.st_scalars, w.st_scalars + 2, nullptr, gradnorm_out, nullptr, gscale, 1);
  }
  TGNN_LAUNCH_OK(ctx, "apply_gradient");
  return TGNN_OK;
}

}  // namespace tgnn
