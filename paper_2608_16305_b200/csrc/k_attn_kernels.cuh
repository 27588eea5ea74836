// Kernels of the attention on the query side (see k_attn.cu for the algebra).  A row z lies as [memory (d) | time encoding (d) |
// features (d_e) | padding to 4]: ldz columns.
#pragma once
#include "k_attn.cuh"

namespace tgnn {
namespace {

constexpr unsigned FULL = 0xffffffffu;

// Four columns as two pairs.
struct P4 {
  f32x2 a, b;
};
__device__ __forceinline__ P4 ld4(const void* p) {
  const ulonglong2 v = __ldg(reinterpret_cast<const ulonglong2*>(p));
  return P4{v.x, v.y};
}
__device__ __forceinline__ P4 ld4s(const float* p) {   // shared memory
  const ulonglong2 v = *reinterpret_cast<const ulonglong2*>(p);
  return P4{v.x, v.y};
}
__device__ __forceinline__ void st4(float* p, const P4& v) { *reinterpret_cast<ulonglong2*>(p) = make_ulonglong2(v.a, v.b); }
__device__ __forceinline__ void axpy(P4& y, f32x2 s, const P4& x) { y.a = fma2(s, x.a, y.a); y.b = fma2(s, x.b, y.b); }
__device__ __forceinline__ f32x2 dot2(const P4& x, const P4& y, f32x2 t) { return fma2(x.b, y.b, fma2(x.a, y.a, t)); }
__device__ __forceinline__ float sum2(f32x2 v) {
  float lo, hi;
  unpack2(v, lo, hi);
  return lo + hi;
}
__device__ __forceinline__ float4 as_float4(const P4& v) {
  float4 r;
  unpack2(v.a, r.x, r.y); unpack2(v.b, r.z, r.w);
  return r;
}
__device__ __forceinline__ P4 cos4(const P4& r) {
  const float4 x = as_float4(r);
  return P4{pack2(__cosf(x.x), __cosf(x.y)), pack2(__cosf(x.z), __cosf(x.w))};
}

// A pair of feature columns as it lies in memory.
template <int XM> struct RawPair { typedef f32x2 T; };
template <> struct RawPair<X_BF16> { typedef uint32_t T; };
template <> struct RawPair<X_BF16_SINGLE> { typedef uint32_t T; };
template <int B>
__device__ __forceinline__ void copy_async(uint32_t smem, const char* p) {
  // (through L1: a hub's row is asked for by every SM all the time, and one L2 slice would have to serve it)
  asm volatile("cp.async.ca.shared.global [%0], [%1], %2;" ::"r"(smem), "l"(p), "n"(B) : "memory");
}
template <int XM>
__device__ __forceinline__ void copy_pair(uint32_t smem, const char* p) {
  if constexpr (is_bf16(XM)) copy_async<4>(smem, p);
  else if constexpr (XM == X_F32) copy_async<8>(smem, p);
  else { copy_async<4>(smem, p); copy_async<4>(smem + 4, p + 4); }
}
template <int XM>
__device__ __forceinline__ void copy_piece(uint32_t smem, const char* p) {
  if constexpr (is_single(XM)) {
#pragma unroll
    for (int e = 0; e < 4; ++e) copy_async<4>(smem + 4 * e, p + 4 * e);
  } else {
    copy_async<16>(smem, p);
  }
}
template <int XM>
__device__ __forceinline__ P4 ld_piece(const char* p) {
  if constexpr (is_single(XM)) {
    const float* f = reinterpret_cast<const float*>(p);
    return P4{pack2(__ldg(f), __ldg(f + 1)), pack2(__ldg(f + 2), __ldg(f + 3))};
  } else {
    return ld4(p);
  }
}
__device__ __forceinline__ f32x2 widen(uint32_t w) { return pack2(__uint_as_float(w << 16), __uint_as_float(w & 0xffff0000u)); }
__device__ __forceinline__ f32x2 widen(f32x2 v) { return v; }

// Sums of NV <= 32 values over the 32 lanes of a warp, lane l < NV returning the sum of value l: each step exchanges half
// of what is left instead of running one butterfly per value.
template <int NV, int O>
__device__ __forceinline__ void reduce_step(float* v, int lane) {
  const bool up = (lane & O) != 0;
#pragma unroll
  for (int i = 0; i < O; ++i) {
    if (i + O < NV) {
      const float give = up ? v[i] : v[i + O], keep = up ? v[i + O] : v[i];
      v[i] = keep + __shfl_xor_sync(FULL, give, O);
    } else if (i < NV) {
      v[i] += __shfl_xor_sync(FULL, v[i], O);
    }
  }
}
template <int NV>
__device__ __forceinline__ float reduce_transposed(float (&v)[NV], int lane) {
  static_assert(NV <= 32 && NV >= 1, "one value per lane");
  reduce_step<NV, 16>(v, lane);
  reduce_step<(NV < 16 ? NV : 16), 8>(v, lane);
  reduce_step<(NV < 8 ? NV : 8), 4>(v, lane);
  reduce_step<(NV < 4 ? NV : 4), 2>(v, lane);
  reduce_step<(NV < 2 ? NV : 2), 1>(v, lane);
  return v[0];
}
__device__ __forceinline__ bool bit(unsigned m, int i) { return i < 32 && ((m >> i) & 1u) != 0u; }

// What a warp has to know of a root before it can ask for rows, one slot per lane: fetched one item ahead of its use.
struct Item {
  int node, eid, cnt, root;
  float dt;
};
__device__ __forceinline__ Item fetch_item(const AttnArgs& a, int i, int lane) {
  Item it{-1, -1, 0, -1, 0.f};
  if (i < a.n) {
    it.cnt = __ldg(a.cnt + i);
    it.root = __ldg(a.nodes + i);
    if (lane < a.k) {
      const int64_t o = (int64_t)i * a.k + lane;
      it.node = __ldg(a.nbr + o);
      it.eid = __ldg(a.eid + o);
      it.dt = (float)(__ldg(a.times + i) - __ldg(a.ts + o));
    }
  }
  return it;
}
// The slots that hold a row: slots at and beyond the count do not, nor do slots naming a node or a feature row that does
// not exist (reported).  Those read the rows of the root's first slot that does, with no weight: a row of another root
// would hand this one its infinities and NaN all the same.
__device__ __forceinline__ unsigned valid_slots(const AttnArgs& a, Item& it, int c, int lane, int32_t* status) {
  const bool ok = lane < c && it.node >= 0 && (index_ok(it.node, a.N, status) & (a.de == 0 || index_ok(it.eid, a.E, status)));
  const unsigned held = __ballot_sync(FULL, ok);
  const int first = held != 0u ? __ffs(held) - 1 : 0;   // (no slot at all: nothing is read)
  const int node = __shfl_sync(FULL, it.node, first), eid = __shfl_sync(FULL, it.eid, first);
  const float dt = __shfl_sync(FULL, it.dt, first);
  if (!ok) { it.node = node; it.eid = eid; it.dt = dt; }
  return held;
}
__device__ __forceinline__ const char* row_at(const char* base, unsigned row, unsigned pitch) {
  unsigned long long p;
  asm("mad.wide.u32 %0, %1, %2, %3;" : "=l"(p) : "r"(row), "r"(pitch), "l"(base));
  return reinterpret_cast<const char*>(p);
}

// How a warp covers a row: JD pieces of four columns per lane of the memory and of the encoding, PX pairs of feature
// columns.  A lane past the end of a part repeats the part's last piece with zero factors and stores nothing, so that all
// of it is straight-line code.
template <int JD, int PX, int XM>
struct Cols {
  static constexpr int PXA = PX > 0 ? PX : 1;
  int lane;
  bool has[JD], hasx[PXA];
  int col[JD], pcol[PXA];    // first column of a piece in its d-wide part; of a pair in the row
  const char* mbase[JD];     // piece j of row 0 of the memory table, pair j of row 0 of the feature table
  const char* xbase[PXA];
  int xoff[PXA];             // byte offset of pair j in a raw feature row
  P4 w[JD], b[JD];           // the encoder's frequencies and phases
  __device__ __forceinline__ Cols(const AttnArgs& a) {
    lane = threadIdx.x & 31;
    const int d4 = a.d >> 2, x2 = a.de >> 1;
#pragma unroll
    for (int j = 0; j < JD; ++j) {
      const int ch = min(lane + 32 * j, d4 - 1);
      has[j] = lane + 32 * j < d4;
      col[j] = 4 * ch;
      mbase[j] = reinterpret_cast<const char*>(a.memory) + 16 * ch;
      const float *pw = a.time_w + 4 * ch, *pb = a.time_b + 4 * ch;
      w[j] = P4{pack2(pw[0], pw[1]), pack2(pw[2], pw[3])};
      b[j] = P4{pack2(pb[0], pb[1]), pack2(pb[2], pb[3])};
    }
#pragma unroll
    for (int j = 0; j < PX; ++j) {
      const int ch = min(lane + 32 * j, x2 - 1);
      hasx[j] = lane + 32 * j < x2;
      pcol[j] = 2 * a.d + 2 * ch;
      xoff[j] = pair_bytes(XM) * ch;
      xbase[j] = reinterpret_cast<const char*>(a.efeat) + xoff[j];
    }
  }
  __device__ __forceinline__ P4 angle(int j, float dt) const {
    const f32x2 dt2 = pack2(dt, dt);
    return P4{reduce_two_pi2(fma2(w[j].a, dt2, b[j].a)), reduce_two_pi2(fma2(w[j].b, dt2, b[j].b))};
  }
};

// A lane's columns of a global row of ldz columns (zeros where the lane repeats another's).
template <int JD, int PX>
struct Vec {
  P4 m[JD], p[JD];
  f32x2 x[PX > 0 ? PX : 1];
  template <int XM>
  __device__ __forceinline__ void load(const Cols<JD, PX, XM>& c, const float* row, int d) {
#pragma unroll
    for (int j = 0; j < JD; ++j) {
      m[j] = ld4(row + c.col[j]);
      p[j] = ld4(row + d + c.col[j]);
      if (!c.has[j]) m[j] = p[j] = P4{0ull, 0ull};
    }
#pragma unroll
    for (int j = 0; j < PX; ++j) {
      x[j] = __ldg(reinterpret_cast<const f32x2*>(row + c.pcol[j]));
      if (!c.hasx[j]) x[j] = 0ull;
    }
  }
  template <int XM>
  __device__ __forceinline__ void store(const Cols<JD, PX, XM>& c, float* row, int d, int pad_col) const {
#pragma unroll
    for (int j = 0; j < JD; ++j)
      if (c.has[j]) { st4(row + c.col[j], m[j]); st4(row + d + c.col[j], p[j]); }
#pragma unroll
    for (int j = 0; j < PX; ++j)
      if (c.hasx[j]) *reinterpret_cast<f32x2*>(row + c.pcol[j]) = x[j];
    if (pad_col >= 0 && c.lane == 0) *reinterpret_cast<f32x2*>(row + pad_col) = 0ull;   // two columns of padding
  }
  __device__ __forceinline__ void clear() {
#pragma unroll
    for (int j = 0; j < JD; ++j) m[j] = p[j] = P4{0ull, 0ull};
#pragma unroll
    for (int j = 0; j < PX; ++j) x[j] = 0ull;
  }
  __device__ __forceinline__ void scale(f32x2 s) {
#pragma unroll
    for (int j = 0; j < JD; ++j) {
      m[j] = P4{mul2(m[j].a, s), mul2(m[j].b, s)};
      p[j] = P4{mul2(p[j].a, s), mul2(p[j].b, s)};
    }
#pragma unroll
    for (int j = 0; j < PX; ++j) x[j] = mul2(x[j], s);
  }
};

// A warp's scratch in shared memory: per slot of the batch the weights of the HU heads and, in the backward pass, their
// gradients, each twice (the two halves of a pair); the logits of all slots of the root.
template <int HU, int SB>
struct Scratch {
  alignas(16) f32x2 wgt[SB][HU];
  alignas(16) f32x2 dl[SB][HU];
  float lg[HU][40];
  float part[HU][SB];
};
template <int HU>
__device__ __forceinline__ void lds_heads(f32x2 (&w)[HU], const f32x2 (&row)[HU]) {
  if constexpr (HU == 2) {
    const ulonglong2 v = *reinterpret_cast<const ulonglong2*>(&row[0]);
    w[0] = v.x; w[1] = v.y;
  } else {
    w[0] = row[0];
  }
}
// Asks for the memory and feature columns of slots s0 .. s0 + SB - 1, all of them before any is used: asynchronous copies
// into the warp's staging rows, which need no registers for what is on the way.
template <int JD, int PX, int XM, int SB>
__device__ __forceinline__ void stage_rows(const AttnArgs& a, const Cols<JD, PX, XM>& c, const Item& it, int s0, uint32_t rows, int rw) {
  const unsigned ms = 4u * a.d, xs = (unsigned)(pair_bytes(XM) / 2) * a.de;
#pragma unroll
  for (int s = 0; s < SB; ++s) {
    const unsigned node = __shfl_sync(FULL, it.node, s0 + s);
#pragma unroll
    for (int j = 0; j < JD; ++j) copy_piece<XM>(rows + 4 * (s * rw + c.col[j]), row_at(c.mbase[j], node, ms));
    if (PX > 0) {
      const unsigned e = __shfl_sync(FULL, it.eid, s0 + s);
#pragma unroll
      for (int j = 0; j < PX; ++j) copy_pair<XM>(rows + 4 * (s * rw + 2 * a.d) + c.xoff[j], row_at(c.xbase[j], e, xs));
    }
  }
}
template <int JD, int PX, int XM>
__device__ __forceinline__ f32x2 staged_pair(const Cols<JD, PX, XM>& c, const float* row, int d, int j) {
  return widen(*reinterpret_cast<const typename RawPair<XM>::T*>(reinterpret_cast<const char*>(row + 2 * d) + c.xoff[j]));
}

// Forward.  A warp per root and HU heads, walking the items in strides of the grid.  It streams the root's slots SB at a
// time: asks for all their rows, encodes their time differences while those are on the way, forms the logits (one
// transposed warp reduction for all heads and slots of the batch), and adds the weighted rows to its sums, rescaling them
// when a later batch raises the maximum.  Between the two uses the rows wait in shared memory.
// What bounds it is instruction issue and the latency of the gathers (memory rows from L2, feature rows from HBM): hence
// pairs of columns per instruction, no branches and no address arithmetic per piece, and as many warps as the staged rows
// allow.
template <int HU, int SB, bool MULTI, int JD, int PX, int XM>   // MULTI: more than one batch (k > SB)
__global__ void __launch_bounds__(32, JD == 2 ? 8 : (MULTI || SB > 10 ? 12 : 16)) attn_fwd_kernel(const AttnArgs a) {
  constexpr int NV = HU * SB;
  extern __shared__ __align__(16) float s_rows[];   // [SB][staged_words]
  __shared__ Scratch<HU, SB> ws;
  const int first = blockIdx.x + link_wait();
  link_release();
  const Cols<JD, PX, XM> c(a);
  const int lane = c.lane, d = a.d, rw = staged_words(d, a.de, XM), pad = (a.de & 3) ? 2 * d + a.de : -1;
  const uint32_t rows = (uint32_t)__cvta_generic_to_shared(s_rows);
  const int NU = a.H / HU, items = a.n * NU;
  const int lh = min(lane / SB, HU - 1), ls = lane - lh * SB;   // the (head, slot) of the batch whose logit this lane receives
  int t = first, i = t / NU, u = t - i * NU;
  Item nx = fetch_item(a, t < items ? i : a.n, lane);
  while (t < items) {
    Item it = nx;
    const int n = max(0, min(it.cnt, a.k));
    const unsigned ok = valid_slots(a, it, n, lane, a.status);
    const float* qrow = a.qp + ((int64_t)i * a.H + u * HU) * a.ldz;
    float* crow = a.cat + (int64_t)i * a.ldc;
    float* prow = a.prob + ((int64_t)i * a.H + u * HU) * a.k;
    const int tn = t + gridDim.x, in = tn / NU, un = tn - in * NU;
    const bool root_ok = index_ok(it.root, a.N, lane == 0 ? a.status : nullptr);
    P4 own[JD];
    Vec<JD, PX> acc[HU];
    if (MULTI || ok == 0u) {
#pragma unroll
      for (int h = 0; h < HU; ++h) acc[h].clear();
    }
    float mx = -INFINITY, den = 0.f;   // of this lane's head
    for (int s0 = 0; ok != 0u && s0 < n; s0 += SB) {
      stage_rows<JD, PX, XM, SB>(a, c, it, s0, rows, rw);
      Vec<JD, PX> q[HU];
#pragma unroll
      for (int h = 0; h < HU; ++h) q[h].load(c, qrow + h * a.ldz, d);
      if (s0 == 0) nx = fetch_item(a, tn < items ? in : a.n, lane);
      float v[NV];
#pragma unroll
      for (int s = 0; s < SB; ++s) {   // the encodings, while the rows are on the way
        const float dt = __shfl_sync(FULL, it.dt, s0 + s);
        f32x2 x[HU];
#pragma unroll
        for (int h = 0; h < HU; ++h) x[h] = 0ull;
#pragma unroll
        for (int j = 0; j < JD; ++j) {
          const P4 zp = cos4(c.angle(j, dt));
          st4(s_rows + s * rw + d + c.col[j], zp);
#pragma unroll
          for (int h = 0; h < HU; ++h) x[h] = dot2(zp, q[h].p[j], x[h]);
        }
#pragma unroll
        for (int h = 0; h < HU; ++h) v[h * SB + s] = sum2(x[h]);
      }
      cp_async_wait_all();
      __syncwarp();
#pragma unroll
      for (int s = 0; s < SB; ++s) {
        const float* row = s_rows + s * rw;
        f32x2 x[HU];
#pragma unroll
        for (int h = 0; h < HU; ++h) x[h] = 0ull;
#pragma unroll
        for (int j = 0; j < JD; ++j) {
          const P4 zm = ld4s(row + c.col[j]);
#pragma unroll
          for (int h = 0; h < HU; ++h) x[h] = dot2(zm, q[h].m[j], x[h]);
        }
#pragma unroll
        for (int j = 0; j < PX; ++j) {
          const f32x2 zx = staged_pair<JD, PX, XM>(c, row, d, j);
#pragma unroll
          for (int h = 0; h < HU; ++h) x[h] = fma2(zx, q[h].x[j], x[h]);
        }
#pragma unroll
        for (int h = 0; h < HU; ++h) v[h * SB + s] += sum2(x[h]);
        if (s & 1) asm volatile("" ::: "memory");   // (two slots' loads ahead are enough; more would cost registers)
      }
      if (s0 == 0) {
#pragma unroll
        for (int j = 0; j < JD; ++j) own[j] = ld_piece<XM>(row_at(c.mbase[j], root_ok ? it.root : 0, 4u * d));
      }
      const float dots = reduce_transposed<NV>(v, lane);
      const bool live = lane < NV && s0 + ls < n, holds = live && bit(ok, s0 + ls);
      const float lg = holds ? dots : 0.f;   // (a slot that holds no row because its record is bad keeps its share of the weights)
      if (live) ws.lg[lh][s0 + ls] = lg;
      __syncwarp();
      float nm = mx;
#pragma unroll
      for (int s = 0; s < SB; ++s)
        if (s0 + s < n) nm = fmaxf(nm, ws.lg[lh][s0 + s]);
      // (a batch may hold nothing but logits of minus infinity: they weigh nothing then, unless all of the root's do)
      const float ref = nm == -INFINITY && MULTI ? 0.f : nm;
      const float e = live ? expf(lg - ref) : 0.f, eh = holds ? e : 0.f;
      const float grow = expf(mx - ref);   // (0 in the first batch)
      if (lane < NV) { ws.wgt[ls][lh] = pack2(eh, eh); ws.dl[ls][lh] = pack2(e, e); }
      __syncwarp();
      float sum = 0.f;
#pragma unroll
      for (int s = 0; s < SB; ++s) sum += __uint_as_float((unsigned)ws.dl[s][lh]);
      den = fmaf(den, grow, sum);
      mx = nm;
      if (MULTI && s0 > 0) {
#pragma unroll
        for (int h = 0; h < HU; ++h) {
          const float g = __shfl_sync(FULL, grow, h * SB);
          acc[h].scale(pack2(g, g));
        }
      }
      if (!MULTI) {
#pragma unroll
        for (int h = 0; h < HU; ++h) acc[h].clear();
      }
#pragma unroll
      for (int s = 0; s < SB; ++s) {
        const float* row = s_rows + s * rw;
        f32x2 w[HU];
        lds_heads<HU>(w, ws.wgt[s]);
#pragma unroll
        for (int j = 0; j < JD; ++j) {
          const P4 zm = ld4s(row + c.col[j]), zp = ld4s(row + d + c.col[j]);
#pragma unroll
          for (int h = 0; h < HU; ++h) { axpy(acc[h].m[j], w[h], zm); axpy(acc[h].p[j], w[h], zp); }
        }
#pragma unroll
        for (int j = 0; j < PX; ++j) {
          const f32x2 zx = staged_pair<JD, PX, XM>(c, row, d, j);
#pragma unroll
          for (int h = 0; h < HU; ++h) acc[h].x[j] = fma2(w[h], zx, acc[h].x[j]);
        }
      }
      __syncwarp();   // the staged rows and the scratch are free again
      if (!MULTI) break;
    }
    if (ok == 0u) {
      nx = fetch_item(a, tn < items ? in : a.n, lane);
#pragma unroll
      for (int j = 0; j < JD; ++j) own[j] = ld_piece<XM>(row_at(c.mbase[j], root_ok ? it.root : 0, 4u * d));
    }
    if (u == 0) {   // the root's own row, and whether it has a slot
#pragma unroll
      for (int j = 0; j < JD; ++j)
        if (c.has[j]) st4(crow + a.H * a.ldz + c.col[j], root_ok ? own[j] : P4{0ull, 0ull});
      if (lane == 0) crow[a.H * a.ldz + d] = n > 0 ? 1.f : 0.f;
    }
#pragma unroll
    for (int h = 0; h < HU; ++h) {
      const float mh = __shfl_sync(FULL, mx, h * SB), inv = 1.f / __shfl_sync(FULL, den, h * SB);
      if (lane < a.k) prow[h * a.k + lane] = lane < n ? (ok != 0u ? expf(ws.lg[h][lane] - mh) * inv : 1.f / (float)n) : 0.f;
      acc[h].scale(ok != 0u ? pack2(inv, inv) : 0ull);
      acc[h].store(c, crow + (u * HU + h) * a.ldz, d, pad);
    }
    __syncwarp();
    t = tn; i = in; u = un;
  }
}

// Backward: from dzbar the gradient of each slot's weight and from there
//   dp_hs = z_s . dzbar_h,   dl_hs = p_hs (dp_hs - sum_t p_ht dp_ht),
//   dqp_h = sum_s dl_hs z_s,   dz_s = sum_h p_hs dzbar_h + dl_hs qp_h.
// (The sum over t from the same dp: the logit gradients of a root then add up to zero to rounding of that sum alone, and a
// single slot's is exactly zero.  zbar_h . dzbar_h in its place carries a residue, which slots years back multiply by dt.)
// Of dz the memory columns are added to the rows that this step's memory update wrote and the encoding columns to the time
// encoder's fp64 sums; the feature columns lead nowhere.  The rows are gathered and encoded a second time rather than
// kept.  Rows of hub nodes come by the thousand, and additions to one row wait for one another: so there are several copies
// of those rows, a block adds to one of them, and the update cell's backward adds the copies up.  (12 000 roots, us with the launch, 186
// bf16 feature columns and 17 000 nodes / none and 2 000 nodes with hubs: one copy 134 / 283; 2: 84 / 223; 4: 70 / 129; 8: 69 / 78; 16: 69 /
// 69; 32: 69 / 51.  A cache of four rows in each warp's shared memory in front of one copy: 97 / 90.)
template <int HU, int SB, bool MULTI, int JD, int PX, int XM>
__global__ void __launch_bounds__(32, JD == 2 ? 8 : 12) attn_bwd_kernel(const AttnArgs a) {
  constexpr int NV = HU * SB;
  extern __shared__ __align__(16) float s_rows[];   // [SB][staged_words] (angles instead of encodings)
  __shared__ Scratch<HU, SB> ws;
  const int first = blockIdx.x + link_wait();
  link_release();
  const Cols<JD, PX, XM> c(a);
  const int lane = c.lane, d = a.d, rw = staged_words(d, a.de, XM), pad = (a.de & 3) ? 2 * d + a.de : -1;
  const uint32_t rows = (uint32_t)__cvta_generic_to_shared(s_rows);
  float* upd_rows = a.dMemU + (int64_t)(blockIdx.x & a.copy_mask) * a.upd_rows * d;
  const int NU = a.H / HU, items = a.n * NU;
  const int lh = min(lane / SB, HU - 1), ls = lane - lh * SB;
  double gw[JD][4], gb[JD][4];
#pragma unroll
  for (int j = 0; j < JD; ++j)
#pragma unroll
    for (int e = 0; e < 4; ++e) { gw[j][e] = 0.0; gb[j][e] = 0.0; }
  int t = first, i = t / NU, u = t - i * NU;
  Item nx = fetch_item(a, t < items ? i : a.n, lane);
  while (t < items) {
    Item it = nx;
    const int n = max(0, min(it.cnt, a.k));
    const unsigned ok = valid_slots(a, it, n, lane, nullptr);
    int my_slot = a.node2slot != nullptr && bit(ok, lane) ? __ldg(a.node2slot + it.node) : -1;
    if (my_slot >= a.upd_rows) my_slot = -1;   // (a reduction of more nodes since the memory update)
    const float* qrow = a.qp + ((int64_t)i * a.H + u * HU) * a.ldz;
    const float* grow = a.dcat + (int64_t)i * a.ldd + u * HU * a.ldz;
    const float* prow = a.prob + ((int64_t)i * a.H + u * HU + lh) * a.k;
    float* drow = a.dqp + ((int64_t)i * a.H + u * HU) * a.ldz;
    const int tn = t + gridDim.x, in = tn / NU, un = tn - in * NU;
    Vec<JD, PX> acc[HU];
    if (MULTI || ok == 0u) {
#pragma unroll
      for (int h = 0; h < HU; ++h) acc[h].clear();
    }
    float dp = 0.f, pd = 0.f;   // of this lane's (head, slot); sum of p dp over its slots of all batches
    for (int s0 = 0; ok != 0u && s0 < n; s0 += SB) {
      const float p = lane < NV && bit(ok, s0 + ls) ? __ldg(prow + s0 + ls) : 0.f;
      stage_rows<JD, PX, XM, SB>(a, c, it, s0, rows, rw);
      float v[NV];
      Vec<JD, PX> g[HU];
#pragma unroll
      for (int h = 0; h < HU; ++h) g[h].load(c, grow + h * a.ldz, d);
      if (s0 == 0) {   // (wanted further down, where nothing else would hide the round trip: 73 -> 70 us for 12 000 roots)
#pragma unroll
        for (int h = 0; h < HU; ++h)
#pragma unroll
          for (int j = 0; j < JD; ++j) {
            asm volatile("prefetch.global.L1 [%0];" ::"l"(qrow + h * a.ldz + c.col[j]));
            asm volatile("prefetch.global.L1 [%0];" ::"l"(qrow + h * a.ldz + d + c.col[j]));
          }
      }
      if (s0 == 0) nx = fetch_item(a, tn < items ? in : a.n, lane);
#pragma unroll
      for (int s = 0; s < SB; ++s) {   // the encodings, while the rows are on the way (their angles are kept)
        const float dt = __shfl_sync(FULL, it.dt, s0 + s);
        f32x2 x[HU];
#pragma unroll
        for (int h = 0; h < HU; ++h) x[h] = 0ull;
#pragma unroll
        for (int j = 0; j < JD; ++j) {
          const P4 an = c.angle(j, dt), zp = cos4(an);
          st4(s_rows + s * rw + d + c.col[j], an);
#pragma unroll
          for (int h = 0; h < HU; ++h) x[h] = dot2(zp, g[h].p[j], x[h]);
        }
#pragma unroll
        for (int h = 0; h < HU; ++h) v[h * SB + s] = sum2(x[h]);
      }
      cp_async_wait_all();
      __syncwarp();
#pragma unroll
      for (int s = 0; s < SB; ++s) {
        const float* row = s_rows + s * rw;
        f32x2 x[HU];
#pragma unroll
        for (int h = 0; h < HU; ++h) x[h] = 0ull;
#pragma unroll
        for (int j = 0; j < JD; ++j) {
          const P4 zm = ld4s(row + c.col[j]);
#pragma unroll
          for (int h = 0; h < HU; ++h) x[h] = dot2(zm, g[h].m[j], x[h]);
        }
#pragma unroll
        for (int j = 0; j < PX; ++j) {
          const f32x2 zx = staged_pair<JD, PX, XM>(c, row, d, j);
#pragma unroll
          for (int h = 0; h < HU; ++h) x[h] = fma2(zx, g[h].x[j], x[h]);
        }
#pragma unroll
        for (int h = 0; h < HU; ++h) v[h * SB + s] += sum2(x[h]);
        if (s & 1) asm volatile("" ::: "memory");
      }
      dp = reduce_transposed<NV>(v, lane);
      pd = fmaf(p, dp, pd);
      if (MULTI && lane < NV) ws.lg[lh][s0 + ls] = dp;
      if (!MULTI) break;
      __syncwarp();   // the staged rows are free again
    }
    if (lane < NV) ws.part[lh][ls] = pd;
    __syncwarp();
    float dsum = 0.f;
#pragma unroll
    for (int s = 0; s < SB; ++s) dsum += ws.part[lh][s];
    const int last = n > 0 ? (n - 1) / SB * SB : 0;
    for (int s0 = MULTI ? last : 0; ok != 0u && s0 >= 0; s0 -= SB) {   // the last batch first: its rows are still there
      if (MULTI && s0 != last) {
        stage_rows<JD, PX, XM, SB>(a, c, it, s0, rows, rw);
#pragma unroll
        for (int s = 0; s < SB; ++s) {
          const float dt = __shfl_sync(FULL, it.dt, s0 + s);
#pragma unroll
          for (int j = 0; j < JD; ++j) st4(s_rows + s * rw + d + c.col[j], c.angle(j, dt));
        }
        cp_async_wait_all();
        __syncwarp();
      }
      const float p = lane < NV && bit(ok, s0 + ls) ? __ldg(prow + s0 + ls) : 0.f;
      if (MULTI && lane < NV) dp = ws.lg[lh][s0 + ls];
      const float dl = p * (dp - dsum);
      if (lane < NV) { ws.wgt[ls][lh] = pack2(p, p); ws.dl[ls][lh] = pack2(dl, dl); }
      __syncwarp();
      if (!MULTI) {
#pragma unroll
        for (int h = 0; h < HU; ++h) acc[h].clear();
      }
      // feature columns: only the projected query's gradient
#pragma unroll
      for (int s = 0; s < SB; ++s) {
        f32x2 wl[HU];
        lds_heads<HU>(wl, ws.dl[s]);
#pragma unroll
        for (int j = 0; j < PX; ++j) {
          const f32x2 zx = staged_pair<JD, PX, XM>(c, s_rows + s * rw, d, j);
#pragma unroll
          for (int h = 0; h < HU; ++h) acc[h].x[j] = fma2(wl[h], zx, acc[h].x[j]);
        }
      }
      const unsigned upd = __ballot_sync(FULL, my_slot >= 0);   // slots whose node's row this step has written
#pragma unroll
      for (int j = 0; j < JD; ++j) {
        P4 gm[HU], gp[HU], qm[HU], qp[HU];
#pragma unroll
        for (int h = 0; h < HU; ++h) {
          gm[h] = ld4(grow + h * a.ldz + c.col[j]); gp[h] = ld4(grow + h * a.ldz + d + c.col[j]);
          qm[h] = ld4(qrow + h * a.ldz + c.col[j]); qp[h] = ld4(qrow + h * a.ldz + d + c.col[j]);
        }
#pragma unroll
        for (int s = 0; s < SB; ++s) {
          const float* row = s_rows + s * rw;
          const P4 zm = ld4s(row + c.col[j]), an = ld4s(row + d + c.col[j]), zp = cos4(an);
          f32x2 wp[HU], wl[HU];
          lds_heads<HU>(wp, ws.wgt[s]);
          lds_heads<HU>(wl, ws.dl[s]);
          P4 gz = {0ull, 0ull};
#pragma unroll
          for (int h = 0; h < HU; ++h) {
            axpy(acc[h].m[j], wl[h], zm);
            axpy(acc[h].p[j], wl[h], zp);
            axpy(gz, wp[h], gp[h]);
            axpy(gz, wl[h], qp[h]);
          }
          const float4 r = as_float4(an), ge = as_float4(gz);
          const float se[4] = {__sinf(r.x), __sinf(r.y), __sinf(r.z), __sinf(r.w)}, gf[4] = {ge.x, ge.y, ge.z, ge.w};
          const double dt = (double)__shfl_sync(FULL, it.dt, s0 + s);
#pragma unroll
          for (int e = 0; e < 4; ++e) {
            const double x = (double)se[e] * (double)gf[e];
            gw[j][e] = fma(x, dt, gw[j][e]);
            gb[j][e] += x;
          }
          if (!bit(upd, s0 + s)) continue;   // (uniform over the warp)
          const int slot = __shfl_sync(FULL, my_slot, s0 + s);
          P4 gm_s = {0ull, 0ull};
#pragma unroll
          for (int h = 0; h < HU; ++h) { axpy(gm_s, wp[h], gm[h]); axpy(gm_s, wl[h], qm[h]); }
          if (c.has[j]) atomicAdd(reinterpret_cast<float4*>(upd_rows + (int64_t)slot * d + c.col[j]), as_float4(gm_s));
        }
      }
      __syncwarp();
      if (!MULTI) break;
    }
    if (ok == 0u) nx = fetch_item(a, tn < items ? in : a.n, lane);
#pragma unroll
    for (int h = 0; h < HU; ++h) acc[h].store(c, drow + h * a.ldz, d, pad);
    t = tn; i = in; u = un;
  }
  double* part = a.tg_part + (int64_t)blockIdx.x * 2 * d;
#pragma unroll
  for (int j = 0; j < JD; ++j)
    if (c.has[j]) {
#pragma unroll
      for (int e = 0; e < 4; ++e) { part[c.col[j] + e] = -gw[j][e]; part[d + c.col[j] + e] = -gb[j][e]; }
    }
}

template <int HU, int SB, bool MULTI, int JD, int PX, int XM>
AttnKernel pick_dir(bool bwd) { return bwd ? attn_bwd_kernel<HU, SB, MULTI, JD, PX, XM> : attn_fwd_kernel<HU, SB, MULTI, JD, PX, XM>; }
template <int HU, int SB, bool MULTI, int JD, int XM>
AttnKernel pick_pairs(int de, bool bwd) {
  if constexpr (JD == 1 && HU == 2) {
    if (de <= 64) return pick_dir<HU, SB, MULTI, JD, 1, XM>(bwd);
    if (de > 128 && de <= 192) return pick_dir<HU, SB, MULTI, JD, 3, XM>(bwd);
  }
  return de <= 128 ? pick_dir<HU, SB, MULTI, JD, 2, XM>(bwd) : pick_dir<HU, SB, MULTI, JD, 4, XM>(bwd);
}

}  // namespace

template <int HU, int SB, bool MULTI, int JD>
AttnKernel attn_kernel(int de, bool bf16, bool bwd) {
  if (de == 0) return pick_dir<HU, SB, MULTI, JD, 0, X_F32>(bwd);
  return bf16 ? pick_pairs<HU, SB, MULTI, JD, X_BF16>(de, bwd) : pick_pairs<HU, SB, MULTI, JD, X_F32>(de, bwd);
}

}  // namespace tgnn
