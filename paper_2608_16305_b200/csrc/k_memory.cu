// Memory path: Message of Eq. 1 (step 2) and Update of Eq. 2 as a GRU cell with
// scatter write-back (step 4).
#include "tgnn_internal.cuh"
#include "tgnn_device.cuh"

namespace tgnn {
namespace {

// Writes one message row [m_self || m_other || x || Phi(dt)] (dm floats) with the lanes of a warp.
__device__ __forceinline__ void write_message_row(float* __restrict__ row, const float* __restrict__ memory,
                                                  const void* __restrict__ efeat, int feat_bf16,
                                                  const float* __restrict__ time_w, const float* __restrict__ time_b,
                                                  int d, int de, int self, int other, int eid, float dtf, int lane,
                                                  float* __restrict__ sin_row) {
  warp_copy_f32(row, memory + (int64_t)self * d, d, lane);
  warp_copy_f32(row + d, memory + (int64_t)other * d, d, lane);
  warp_copy_feat(row + 2 * d, efeat, feat_bf16, eid, de, lane);
  float* phi = row + 2 * d + de;
  if (sin_row == nullptr) {
    for (int q = lane; q < d; q += 32) phi[q] = time_encode(time_w[q], time_b[q], dtf);
  } else {
    for (int q = lane; q < d; q += 32) time_encode_sc(time_w[q], time_b[q], dtf, &phi[q], &sin_row[q]);
  }
}

// Only the nodes that the messages go to, a thread per event (the rows are then gathered for the winners alone).  One warp per
// message, 32 of them one after another, took 15.7 us for 720 events; 2.1 us now.
__global__ void __launch_bounds__(256) message_nodes_kernel(const int32_t* __restrict__ src, const int32_t* __restrict__ dst,
                                                            const int32_t* __restrict__ eid, const uint8_t* __restrict__ keep, int n,
                                                            int de, int64_t N, int64_t E, int32_t* status,
                                                            int32_t* __restrict__ msg_node_out) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  const int a = src[i], b = dst[i], e = eid[i];
  // an event naming a node or a feature row that does not exist is reported and sends no message
  const bool kept = (keep == nullptr || keep[i] != 0) && (index_ok(a, N, status) & index_ok(b, N, status) & (de == 0 || index_ok(e, E, status)));
  msg_node_out[2 * i] = kept ? a : -1;
  msg_node_out[2 * i + 1] = kept ? b : -1;
}

// One warp per message j = 2i + role.
__global__ void __launch_bounds__(256) build_messages_kernel(const float* __restrict__ memory,
                                                             const double* __restrict__ last_update,
                                                             const void* __restrict__ efeat, int feat_bf16,
                                                             const float* __restrict__ time_w,
                                                             const float* __restrict__ time_b, int d, int de,
                                                             const int32_t* __restrict__ src,
                                                             const int32_t* __restrict__ dst, const double* __restrict__ t,
                                                             const int32_t* __restrict__ eid,
                                                             const uint8_t* __restrict__ keep, int n, int64_t N, int64_t E,
                                                             int32_t* status, float* __restrict__ msg_out,
                                                             int32_t* __restrict__ msg_node_out) {
  const int lane = threadIdx.x & 31;
  const int warps = (gridDim.x * blockDim.x) >> 5;
  const int dm = 3 * d + de;
  for (int j = (blockIdx.x * blockDim.x + threadIdx.x) >> 5; j < 2 * n; j += warps) {
    const int i = j >> 1, role = j & 1;
    bool kept = keep == nullptr || keep[i] != 0;
    const int self = role ? dst[i] : src[i];
    const int other = role ? src[i] : dst[i];
    // an event naming a node or a feature row that does not exist is reported and sends no message
    if (kept) {
      int32_t* st = lane == 0 ? status : nullptr;
      kept = index_ok(self, N, st) & index_ok(other, N, st) & (de == 0 || index_ok(eid[i], E, st));
    }
    if (lane == 0) msg_node_out[j] = kept ? self : -1;
    float* row = msg_out + (int64_t)j * dm;
    if (!kept) {
      for (int q = lane; q < dm; q += 32) row[q] = 0.f;
      continue;
    }
    const float dtf = (float)(t[i] - last_update[self]);
    write_message_row(row, memory, efeat, feat_bf16, time_w, time_b, d, de, self, other, eid[i], dtf, lane, nullptr);
  }
}

// One warp per unique node u: the winner's message row into X (leading dimension ld), its dt and timestamp.
__global__ void __launch_bounds__(256) gather_winner_kernel(const float* __restrict__ memory,
                                                            const double* __restrict__ last_update,
                                                            const void* __restrict__ efeat, int feat_bf16,
                                                            const float* __restrict__ time_w,
                                                            const float* __restrict__ time_b, int d, int de,
                                                            const int32_t* __restrict__ src, const int32_t* __restrict__ dst,
                                                            const double* __restrict__ t, const int32_t* __restrict__ eid,
                                                            const float* __restrict__ msg, const int32_t* __restrict__ uniq,
                                                            const int32_t* __restrict__ winner,
                                                            const int32_t* __restrict__ n_uniq, int u_cap, int n_msg, int64_t N,
                                                            int64_t E, int32_t* status, int ld,
                                                            float* __restrict__ X, float* __restrict__ x_dt,
                                                            float* __restrict__ Xsin, double* __restrict__ win_t) {
  const int lane = threadIdx.x & 31;
  const int warps = (gridDim.x * blockDim.x) >> 5;
  const int zero = link_wait(), first = (int)((blockIdx.x * blockDim.x + threadIdx.x) >> 5) + zero;
  link_release();
  n_uniq += zero;   // (the kernel before has written it)
  if (blockIdx.x == 0 && threadIdx.x == 0) index_ok(*n_uniq, (long long)u_cap + 1, status);   // a count beyond the capacity
  const int U = max(0, min(*n_uniq, u_cap));
  const int dm = 3 * d + de;
  for (int u = first; u < U; u += warps) {
    float* row = X + (int64_t)u * ld;
    float* sin_row = Xsin + (int64_t)u * d;
    int32_t* st = lane == 0 ? status : nullptr;
    const int j = winner[u];
    bool good = index_ok(j, n_msg, st);
    const int i = good ? j >> 1 : 0, role = j & 1;
    const int self = good ? (role ? dst[i] : src[i]) : 0;
    const int other = good ? (role ? src[i] : dst[i]) : 0;
    good = good && index_ok(self, N, st) && index_ok(other, N, st) && (de == 0 || msg != nullptr || index_ok(eid[i], E, st));
    if (!good) {   // reported; the row is zero and the node's update starts from a zero message
      for (int q = lane; q < ld; q += 32) row[q] = 0.f;
      for (int q = lane; q < d; q += 32) sin_row[q] = 0.f;
      if (lane == 0) { x_dt[u] = 0.f; win_t[u] = 0.0; }
      continue;
    }
    const double ti = t[i];
    const float dtf = (float)(ti - last_update[self]);
    if (msg != nullptr) {
      warp_copy_f32(row, msg + (int64_t)j * dm, dm, lane);
      for (int q = lane; q < d; q += 32) sin_row[q] = sinf(time_arg(time_w[q], time_b[q], dtf));
    } else {
      write_message_row(row, memory, efeat, feat_bf16, time_w, time_b, d, de, self, other, eid[i], dtf, lane, sin_row);
    }
    for (int q = dm + lane; q < ld; q += 32) row[q] = 0.f;
    if (lane == 0) { x_dt[u] = dtf; win_t[u] = ti; }
  }
}

// Gates of the GRU cell and write-back, four columns per thread (d is a multiple of 4; only the table may start anywhere).
// Gi = W_i x + b_i, Gh = W_h h + b_h are given.
__global__ void __launch_bounds__(256) gru_gate_kernel(const float* __restrict__ Gi, const float* __restrict__ Gh,
                                                       const float* __restrict__ X, int ld, int d,
                                                       const int32_t* __restrict__ uniq, const double* __restrict__ win_t,
                                                       const int32_t* __restrict__ n_uniq, int u_cap,
                                                       float* __restrict__ g_r, float* __restrict__ g_z,
                                                       float* __restrict__ g_n, float* __restrict__ g_hn,
                                                       float* __restrict__ memory, double* __restrict__ last_update,
                                                       int64_t N, int32_t* status) {
  const int d4 = d >> 2, t = (int)(blockIdx.x * blockDim.x + threadIdx.x) + link_wait(), u = t / d4, q = 4 * (t - u * d4);
  link_release();
  if (u >= u_cap) return;
  const float *gi = Gi + (int64_t)u * 3 * d + q, *gh = Gh + (int64_t)u * 3 * d + q;
  const auto ld4 = [](const float* p, float (&v)[4]) {
    const float4 x = *reinterpret_cast<const float4*>(p);
    v[0] = x.x; v[1] = x.y; v[2] = x.z; v[3] = x.w;
  };
  // (asked for before it is known how many rows there are: rows beyond hold what an earlier step left there)
  float ir[4], iz[4], in[4], hr[4], hz[4], hn[4], h[4];
  ld4(gi, ir); ld4(gi + d, iz); ld4(gi + 2 * d, in); ld4(gh, hr); ld4(gh + d, hz); ld4(gh + 2 * d, hn); ld4(X + (int64_t)u * ld + q, h);
  const int node = uniq[u];
  const double tw = win_t[u];
  if (u >= min(*n_uniq, u_cap)) return;
  float r[4], z[4], n[4], o[4];
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    r[i] = sigmoidf_(ir[i] + hr[i]);
    z[i] = sigmoidf_(iz[i] + hz[i]);
    n[i] = tanhf(fmaf(r[i], hn[i], in[i]));
    o[i] = fmaf(z[i], h[i] - n[i], n[i]);  // (1 - z) n + z h
  }
  const int64_t e = (int64_t)u * d + q;
  const auto st4 = [](float* p, const float (&v)[4]) { *reinterpret_cast<float4*>(p) = make_float4(v[0], v[1], v[2], v[3]); };
  st4(g_r + e, r); st4(g_z + e, z); st4(g_n + e, n); st4(g_hn + e, hn);
  if (!index_ok(node, N, q == 0 ? status : nullptr)) return;   // reported, nothing written
  float* row = memory + (int64_t)node * d + q;
  if (((uintptr_t)memory & 15) == 0) st4(row, o);
  else {
#pragma unroll
    for (int i = 0; i < 4; ++i) row[i] = o[i];
  }
  if (q == 0) last_update[node] = tw;
}

// The plain recurrent cell and write-back: m' = tanh(Gi + Gh) with Gi = W_i x + b_i, Gh = W_h h + b_h
// (row pitch d).  The new row is kept in g_n for the backward pass (d tanh = 1 - m'^2).
__global__ void __launch_bounds__(256) rnn_gate_kernel(const float* __restrict__ Gi, const float* __restrict__ Gh, int d,
                                                       const int32_t* __restrict__ uniq, const double* __restrict__ win_t,
                                                       const int32_t* __restrict__ n_uniq, int u_cap,
                                                       float* __restrict__ g_n, float* __restrict__ memory,
                                                       double* __restrict__ last_update, int64_t N, int32_t* status) {
  const int64_t first = blockIdx.x * (int64_t)blockDim.x + threadIdx.x + link_wait();
  link_release();
  const int U = max(0, min(*n_uniq, u_cap));
  const int64_t total = (int64_t)U * d;
  for (int64_t e = first; e < total; e += (int64_t)gridDim.x * blockDim.x) {
    const int u = (int)(e / d), q = (int)(e % d);
    const float hnew = tanhf(Gi[e] + Gh[e]);
    g_n[e] = hnew;
    const int node = uniq[u];
    if (!index_ok(node, N, q == 0 ? status : nullptr)) continue;
    memory[(int64_t)node * d + q] = hnew;
    if (q == 0) last_update[node] = win_t[u];
  }
}

}  // namespace

int launch_build_messages(tgnn_ctx* ctx, const int32_t* src, const int32_t* dst, const double* t, const int32_t* eid,
                          const uint8_t* keep, int n, float* msg_out, int32_t* msg_node_out, cudaStream_t s) {
  if (n == 0) return TGNN_OK;
  const tgnn_config& c = ctx->cfg;
  {
    KernelScope scope__(ctx, "build_messages", s);
    if (msg_out == nullptr)
      message_nodes_kernel<<<(n + 255) / 256, 256, 0, s>>>(src, dst, eid, keep, n, c.d_e, c.num_nodes, ctx->num_events, ctx->ws.status,
                                                           msg_node_out);
    else
      build_messages_kernel<<<(2 * n + 7) / 8, 256, 0, s>>>(ctx->memory, ctx->last_update, ctx->efeat, c.feat_dtype == TGNN_BF16,
                                                            ctx->params + ctx->L.time_w, ctx->params + ctx->L.time_b, c.d, c.d_e, src,
                                                            dst, t, eid, keep, n, c.num_nodes, ctx->num_events, ctx->ws.status, msg_out,
                                                            msg_node_out);
  }
  TGNN_LAUNCH_OK(ctx, "build_messages");
  return TGNN_OK;
}

int launch_memory_update(tgnn_ctx* ctx, const float* msg, const int32_t* uniq, const int32_t* winner,
                         const int32_t* n_uniq, cudaStream_t s) {
  const tgnn_config& c = ctx->cfg;
  const ParamLayout& L = ctx->L;
  Workspace& w = ctx->ws;
  const int d = c.d, U_cap = min(ctx->upd_rows, 2 * ctx->m_n);
  const int gd = (int)L.gates * d;  // rows of the cell's matrices: 3d (GRU) or d (plain cell)
  if (U_cap == 0) return TGNN_OK;
  {
    KernelScope scope__(ctx, "gather_winner", s);
    launch_link_event(ctx, false, ctx->in_step ? ctx->ev_beside : nullptr, gather_winner_kernel, dim3((U_cap + 7) / 8), dim3(256), 0, s, 1, ctx->memory, ctx->last_update, ctx->efeat,
                                                         c.feat_dtype == TGNN_BF16, ctx->params + L.time_w,
                                                         ctx->params + L.time_b, d, c.d_e, ctx->m_src, ctx->m_dst, ctx->m_t,
                                                         ctx->m_eid, msg, uniq, winner, n_uniq, U_cap, 2 * ctx->m_n, c.num_nodes,
                                                         ctx->num_events, w.status, ctx->ld_msg, w.X, w.x_dt, w.Xsin, w.win_t);
  }
  TGNN_LAUNCH_OK(ctx, "gather_winner");
  GemmArgs g = {};
  g.A = w.X; g.a_rs = ctx->ld_msg; g.a_cs = 1;
  g.B = ctx->params + L.gru_wi; g.b_rs = 1; g.b_cs = L.dmsg;  // B(k,n) = W_i[n,k]
  g.C = w.Gi; g.ldc = gd; g.M = U_cap; g.N = gd; g.K = (int)L.dmsg; g.dev_M = n_uniq;
  g.bias = ctx->params + L.gru_bi;
  g.split_k = 1; g.site = SITE_GI + 1;
  // The call on its own takes the parameters as it finds them: the images of the cell's two matrices are written first.  (Without
  // them the input product ran 16 us for 720 events, through registers into a cleared Gi; 11 with them, 3 of them the images.)
  const bool alone = ctx->images != nullptr && !ctx->images_fresh;
  if (alone) {
    const int rc = launch_prep_cell(ctx, s);
    if (rc) return rc;
  }
  int rc = fork_to(ctx, s, ctx->side[0]);  // the hidden-state product runs beside the input product
  if (rc) return rc;
  if (alone) ctx->images_fresh = true;     // (of these two products' matrices, for these two products)
  rc = launch_gemm(ctx, g, "gru_gi", s);
  if (!rc) {
    g.B = ctx->params + L.gru_wh; g.b_cs = d; g.C = w.Gh; g.K = d; g.bias = ctx->params + L.gru_bh;
    g.site = SITE_GH + 1;
    rc = launch_gemm(ctx, g, "gru_gh", ctx->side[0]);
  }
  if (alone) ctx->images_fresh = false;
  if (rc) return rc;
  rc = fork_to(ctx, ctx->side[0], s);
  if (rc) return rc;
  const int64_t total = (int64_t)U_cap * d;
  if (c.model == TGNN_MODEL_JODIE) {
    {
      KernelScope scope__(ctx, "rnn_gate", s);
      launch_link(ctx, rnn_gate_kernel, dim3((unsigned)((total + 255) / 256)), dim3(256), 0, s, 1, w.Gi, w.Gh, d, uniq, w.win_t, n_uniq, U_cap, w.g_n,
                                                                 ctx->memory, ctx->last_update, c.num_nodes, w.status);
    }
    TGNN_LAUNCH_OK(ctx, "rnn_gate");
    return TGNN_OK;
  }
  {
    KernelScope scope__(ctx, "gru_gate", s);
    launch_link(ctx, gru_gate_kernel, dim3((unsigned)((total / 4 + 255) / 256)), dim3(256), 0, s, 1, w.Gi, w.Gh, w.X, ctx->ld_msg, d, uniq, w.win_t, n_uniq,
                                                               U_cap, w.g_r, w.g_z, w.g_n, w.g_hn, ctx->memory,
                                                               ctx->last_update, c.num_nodes, w.status);
  }
  TGNN_LAUNCH_OK(ctx, "gru_gate");
  return TGNN_OK;
}

}  // namespace tgnn
