// Dense projections on the 5th-generation tensor cores (TGNN_MATH_TF32).
//
// One CTA computes a 128 x BN tile of C = A B over a range of the contraction
// (split-K across blockIdx.z) with tcgen05.mma.kind::tf32: fp32 operands rounded to
// TF32 (round-to-nearest, by the producer warps, so there is no truncation bias),
// fp32 accumulation in tensor memory.  With `precise` set every operand is split into
// a TF32 head and a TF32 tail (x = hi + lo) and three MMAs (lo*hi, hi*lo, hi*hi) give
// close to fp32 accuracy; the gradient products, whose terms cancel, use it.
//
// Warp roles:
//   G producer groups of 4 warps.  Group g fills the stages of contraction blocks
//     i = g, g + G, ...: global -> registers (all 128-bit loads of a block issued before
//     the first use) -> round to TF32 -> shared memory in the swizzled canonical layout
//     the MMA descriptors expect.  Several blocks are therefore in flight at once.
//     Afterwards all groups run the epilogue (tcgen05.ld of the 32 TMEM lanes their warp
//     may touch, bias / ReLU / store or atomic accumulate), sharing the columns.
//   1 MMA warp: allocates tensor memory; one lane issues the MMAs and commits.
//   1 issuing warp, where activations come as tiles of 16 columns beside a prepared weight image: it asks for both, the groups
//     only write the tails.
// A ring of (A tile, B tile) stages is handed over through mbarriers: full[s] (128
// producer arrivals) and empty[s] (tcgen05.commit).  Every wait is bounded; on expiry
// the kernel records TGNN_ETIMEOUT in the status word, stops waiting, frees its tensor
// memory and returns.
//
// Operands may be K-major (contraction index contiguous) or MN-major (row/column index
// contiguous), so the forward projections (activations [M,K] x weights [N,K]), the
// input gradients (dY [M,N'] x W [N',K]) and the weight gradients (dY^T x A, contraction
// over rows) all run here without a transposed copy.
#include <cuda.h>

#include <cstdlib>

#include "tgnn_device.cuh"
#include "tgnn_images.cuh"
#include "tgnn_internal.cuh"
#include "tgnn_tensor_map.cuh"

namespace tgnn {
namespace {

constexpr int BM = 128;    // rows of C per CTA (UMMA M)
constexpr int BK = IMAGE_K;   // contraction elements per stage: one 128-byte swizzle row of fp32
constexpr int UMMA_K = 8;  // tf32
constexpr int GROUP = 128; // threads per producer group
constexpr int CL_MIN_K = 8 * 32;   // contraction from which a stored product is split over clusters
constexpr int EPI_PITCH = 36;  // floats between rows of an epilogue staging square (16-byte aligned, bank-staggered)
constexpr unsigned SPIN_LIMIT = 1u << 24;
constexpr unsigned FULL = 0xffffffffu;

struct TcArgs {
  const float* A; int64_t lda; int a_major;
  const float* B; int64_t ldb; int b_major;
  float* C; int64_t ldc;
  int M, N, K;
  const int32_t* dev_M;
  const int32_t* dev_K;
  const float* bias;
  float* rowsum_out;
  int relu, accumulate, split_k;
  int in_cluster;      // the split_k CTAs of a tile are a cluster and add up their accumulators in shared memory
  int32_t* status;
  // B operand prepared as shared-memory images (see WeightSite): image of n-tile x, contraction block
  // kb at b_image + x * b_tile_stride + kb * (COPIES * B_BYTES); nullptr: B goes through registers
  const unsigned char* b_image;
  int64_t b_tile_stride;
  // Row-indirect leading columns of a K-major A: A(m, k) for k < a_tab_cols is a_tab[a_idx[m] * a_tab_cols + k]
  // (zero if a_idx[m] < 0) instead of A[m * lda + k]; nullptr: plain A.  Lets the key/value projection
  // read the neighbors' memory rows straight from the table.
  const int32_t* a_idx;
  const float* a_tab;
  int a_tab_cols;
  int64_t a_tab_rows;
  // K-major A as a tiled tensor map (box 32 x 128, 128-byte swizzle; TMA == 3: 16 x 128, 64-byte swizzle): the tensor-memory-access unit brings
  // whole activation tiles into shared memory; a_tma = 0: A goes through registers
  int a_tma;
  CUtensorMap a_map;
  // both operands MN-major (weight gradients): A and B as four-dimensional views of their row-major matrices
  // whose boxes land in the operand tiles' atom layout (see encode_mn_map); b_box_atoms = 32-column atoms per B box
  CUtensorMap b_map;
  int b_box_atoms;
  CUtensorMap c_map;   // gemm_short_kernel: C in boxes of 32 x 32, 128-byte swizzle
};

template <int BN_T, bool PRECISE, int TMA = 0>
struct Cfg {
  // Contraction rows per block: 16 where both operands arrive as tiles and are split (weight gradients), so that four or six
  // stages fit: a tile takes 2 000 cycles to come and 700 to be used by the tensor core (rows of 32 in two stages: 2 900 cycles
  // per 32 rows of 128 x 224, 1 350 of them the tensor core's).  100 x 877 x 12 000: 38.4 -> 32.8 us.
  // 16 too for stored products with a prepared weight image (TMA == 3): seven stages, so that a CTA of a split contraction has all of its
  // loads under way at once, and a warp that does nothing but ask for them.  What bounds those, by clock stamps of a CTA in a plain step: of the 15 100
  // cycles of 1 800 x 845 x 100 (8 CTAs per tile) 1 600 are set-up that the predecessor hides in part, 800 the wait, 2 500 until the first block is there
  // and split, 2 800 the products, 2 100 until the accumulators lie in shared memory and the cluster is ready, 3 300 its sum's copies, 1 900 adding, storing
  // and the last barrier.  12 000 x 877 x 100, not split: 446 cycles per 16 columns, 384 of which are the two products' (256 and 128 columns) on
  // a tensor core of 2 048 tf32 multiply-adds a cycle.  Against rows of 32 in three stages and a cluster's sum through loads of the others' memory:
  // 1 800 events 18 200 -> 14 000 cycles of a CTA, steps of 600 events 144.9 -> 143.2 us, of 4 000 events 368.8 -> 363.9, 259.7 -> 256.7.
  static constexpr int KB = TMA >= 2 ? 16 : BK;
  static constexpr int STAGES = TMA == 3 ? (BN_T > 128 ? 4 : 7) : TMA == 2 ? (BN_T > 128 ? 4 : 6) : PRECISE ? (BN_T > 128 ? 2 : 3) : 4;
  // A group's consecutive blocks must not be more than one use of a stage apart (the waits tell phases apart
  // by parity only), so there are never more groups than stages.
  static constexpr int GROUPS = TMA >= 2 ? 4 : STAGES < 3 ? STAGES : 3;
  static_assert(GROUPS <= STAGES, "a producer group may not lap a stage");
  static constexpr int THREADS = GROUPS * GROUP + (TMA == 3 ? 64 : 32);
  static constexpr int A_BYTES = BM * KB * 4, B_BYTES = BN_T * KB * 4;
  static constexpr int COPIES = PRECISE ? 2 : 1;  // head (+ tail) copy of each operand tile
  static constexpr int STAGE_BYTES = COPIES * (A_BYTES + B_BYTES);
  static constexpr int SMEM = 1024 + STAGES * STAGE_BYTES;
  // The corrections (tail x head, head x tail) have an accumulator of their own, added in the epilogue: the tensor core truncates
  // at the accumulator's last bit with every MMA, and a long contraction on one accumulator lost what the tails had saved.
  static constexpr uint32_t ACC_COLS = BN_T <= 128 ? 128 : 256, TMEM_COLS = (PRECISE ? 2 : 1) * ACC_COLS;
  static_assert(SMEM <= 227 * 1024, "shared memory budget");
};

__device__ __forceinline__ uint32_t smem_u32(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }

__device__ __forceinline__ void mbar_init(uint32_t bar, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(count) : "memory");
}
__device__ __forceinline__ void mbar_arrive(uint32_t bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(bar) : "memory");
}
// Bounded wait on a phase parity.  Returns false if the limit was reached.
__device__ __forceinline__ bool mbar_wait(uint32_t bar, uint32_t parity) {
  for (unsigned it = 0; it < SPIN_LIMIT; ++it) {
    uint32_t done;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(done)
        : "r"(bar), "r"(parity)
        : "memory");
    if (done) return true;
  }
  return false;
}

// Loads and stores are volatile asm so that the compiler keeps every load of a block ahead of
// the first store (it otherwise sinks each load next to its use and serialises the round trips).
__device__ __forceinline__ float4 ldg_v4(const float* p) {
  float4 v;
  asm volatile("ld.global.nc.v4.f32 {%0,%1,%2,%3}, [%4];" : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w) : "l"(p));
  return v;
}
__device__ __forceinline__ float ldg_f(const float* p) {
  float v;
  asm volatile("ld.global.nc.f32 %0, [%1];" : "=f"(v) : "l"(p));
  return v;
}
__device__ __forceinline__ void sts_v4(uint32_t addr, uint32_t a, uint32_t b, uint32_t c, uint32_t d) {
  asm volatile("st.shared.v4.b32 [%0], {%1,%2,%3,%4};" ::"r"(addr), "r"(a), "r"(b), "r"(c), "r"(d) : "memory");
}
__device__ __forceinline__ float4 lds_v4(uint32_t addr) {
  float4 v;
  asm volatile("ld.shared.v4.f32 {%0,%1,%2,%3}, [%4];" : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w) : "r"(addr) : "memory");
  return v;
}
// One 16-byte chunk of an operand tile.  Single pass: the values rounded to TF32.  Split: the values as they
// are in the head copy -- the tensor core reads sign, exponent and the upper 10 mantissa bits of a tf32
// operand and ignores the 13 bits below, so the head it sees is the value truncated -- and the exact
// remainder (the part it ignores) in the tail copy, of which it again sees the upper bits.  Head + tail then
// carry 21 mantissa bits; truncation's bias is in the tail's dropped bits only (2^-21 relative).
__device__ __forceinline__ uint32_t tf32_remainder(float x) {
  return __float_as_uint(x - __uint_as_float(__float_as_uint(x) & 0xffffe000u));
}
template <bool PRECISE>
__device__ __forceinline__ void store_chunk(uint32_t addr, uint32_t tail_offset, const float4& v) {
  if (PRECISE) {
    sts_v4(addr, __float_as_uint(v.x), __float_as_uint(v.y), __float_as_uint(v.z), __float_as_uint(v.w));
    sts_v4(addr + tail_offset, tf32_remainder(v.x), tf32_remainder(v.y), tf32_remainder(v.z), tf32_remainder(v.w));
  } else {
    sts_v4(addr, to_tf32(v.x), to_tf32(v.y), to_tf32(v.z), to_tf32(v.w));
  }
}

// A chunk that a TMA copy left in the head tile as plain fp32 stays there as the head; only its tail is written.
__device__ __forceinline__ void store_tail_of_raw(uint32_t tail_addr, const float4& v) {
  sts_v4(tail_addr, tf32_remainder(v.x), tf32_remainder(v.y), tf32_remainder(v.z), tf32_remainder(v.w));
}

// 64-bit shared-memory matrix descriptor.  layout: 2 = 128-byte swizzle on 16-byte chunks (K-major
// operands), 1 = 128-byte swizzle with a 32-byte base (the only layout for MN-major 32-bit operands).
__device__ __forceinline__ uint64_t make_desc(uint32_t saddr, uint32_t lbo_bytes, uint32_t sbo_bytes, uint32_t layout) {
  uint64_t d = 0;
  d |= (uint64_t)((saddr >> 4) & 0x3FFF);
  d |= (uint64_t)((lbo_bytes >> 4) & 0x3FFF) << 16;
  d |= (uint64_t)((sbo_bytes >> 4) & 0x3FFF) << 32;
  d |= (uint64_t)1 << 46;  // descriptor version for this architecture
  d |= (uint64_t)layout << 61;
  return d;
}

// One producer group (128 threads, index t) fills one operand tile for contraction block [k0, k0+32).
//   K-major:  rows [r0, r0 + rows_t) x 32 k; row r lives at (r/8)*1024 + (r%8)*128, its 16-byte
//             chunk c at position c ^ (r%8).
//   MN-major: 32 k-rows x rows_t (MN) values in atoms of 4 k-rows x 32 values (512 B); k-row kk, MN
//             atom a, chunk c lives at (kk/4)*(atoms*512) + a*512 + (kk%4)*128 + ((c ^ 2*(kk%4))*16):
//             the swizzle exchanges 32-byte pairs of chunks (address bits 5-6 ^= bits 7-8).
// rows_t is a multiple of 32 (MN-major) or of 8 (K-major); chunks outside the valid range are zero.
// The tile is filled in two steps so that a producer can have the loads of its next block in flight
// while it waits for a free stage and stores the current one.
// FAST (every chunk is wholly inside or wholly outside the operand, pointers 16-byte aligned): the
// loads are unconditional -- an out-of-range chunk reads the operand's first chunk instead and is
// zeroed at store time from the returned mask -- so nothing between the loads depends on a loaded
// value and all of a block's round trips overlap.  Otherwise chunks are read element by element
// under their bounds checks.
template <int ROWS_MAX, bool FAST>
__device__ __forceinline__ uint32_t load_regs(float4 (&v)[ROWS_MAX * 8 / GROUP], const float* __restrict__ P, int64_t ld,
                                              int major, int r0, int R, int rows_t, int k0, int k1, bool vec, int t,
                                              const int32_t* tab_row = nullptr, const float* __restrict__ tab = nullptr,
                                              int tab_cols = 0) {
  constexpr int ITERS = ROWS_MAX * 8 / GROUP;
  uint32_t mask = 0;
  if (major == MAJOR_K) {
#pragma unroll
    for (int i = 0; i < ITERS; ++i) {
      const int idx = t + i * GROUP;
      const int r = idx >> 3, c = idx & 7;
      const int gr = r0 + r, gk = k0 + 4 * c;
      bool valid = r < rows_t && gr < R && gk < k1;
      const float* p = P + (int64_t)gr * ld + gk;
      if (tab_row != nullptr && gk < tab_cols) {  // tab_cols is a multiple of 4: the chunk is all table or all A
        valid = valid && tab_row[i] >= 0;
        p = tab + (int64_t)tab_row[i] * tab_cols + gk;
      }
      if (FAST) {
        v[i] = ldg_v4(valid ? p : P);
        mask |= (valid ? 1u : 0u) << i;
      } else {
        v[i] = make_float4(0.f, 0.f, 0.f, 0.f);
        if (valid) {
          if (vec && gk + 3 < k1) {
            v[i] = ldg_v4(p);
          } else {
            v[i].x = ldg_f(p);
            if (gk + 1 < k1) v[i].y = ldg_f(p + 1);
            if (gk + 2 < k1) v[i].z = ldg_f(p + 2);
            if (gk + 3 < k1) v[i].w = ldg_f(p + 3);
          }
        }
      }
    }
  } else {
    const int cpr = rows_t >> 2;  // 16-byte chunks per k-row (multiple of 8)
#pragma unroll
    for (int i = 0; i < ITERS; ++i) {
      const int idx = t + i * GROUP;
      const int kk = idx / cpr, cm = idx - kk * cpr;
      const int gk = k0 + kk, gr = r0 + 4 * cm;
      const bool valid = kk < BK && gk < k1 && gr < R;
      const float* p = P + (int64_t)gk * ld + gr;
      if (FAST) {
        v[i] = ldg_v4(valid ? p : P);
        mask |= (valid ? 1u : 0u) << i;
      } else {
        v[i] = make_float4(0.f, 0.f, 0.f, 0.f);
        if (valid) {
          if (vec && gr + 3 < R) {
            v[i] = ldg_v4(p);
          } else {
            v[i].x = ldg_f(p);
            if (gr + 1 < R) v[i].y = ldg_f(p + 1);
            if (gr + 2 < R) v[i].z = ldg_f(p + 2);
            if (gr + 3 < R) v[i].w = ldg_f(p + 3);
          }
        }
      }
    }
  }
  return FAST ? mask : 0xffffffffu;
}

template <int ROWS_MAX, bool PRECISE>
__device__ __forceinline__ void store_regs(const float4 (&v)[ROWS_MAX * 8 / GROUP], uint32_t mask, uint32_t tile,
                                           uint32_t tail_offset, int major, int rows_t, int t, float4* rowsum) {
  constexpr int ITERS = ROWS_MAX * 8 / GROUP;
  if (major == MAJOR_K) {
#pragma unroll
    for (int i = 0; i < ITERS; ++i) {
      const int idx = t + i * GROUP;
      const int r = idx >> 3, c = idx & 7;
      const float4 x = (mask >> i) & 1u ? v[i] : make_float4(0.f, 0.f, 0.f, 0.f);
      if (r < rows_t) store_chunk<PRECISE>(tile + (r >> 3) * 1024 + (r & 7) * 128 + ((c ^ (r & 7)) << 4), tail_offset, x);
    }
  } else {
    const int cpr = rows_t >> 2;
    const int atoms = rows_t >> 5;
#pragma unroll
    for (int i = 0; i < ITERS; ++i) {
      const int idx = t + i * GROUP;
      const int kk = idx / cpr, cm = idx - kk * cpr;
      if (kk < BK) {
        const int a = cm >> 3, c = cm & 7;
        const float4 x = (mask >> i) & 1u ? v[i] : make_float4(0.f, 0.f, 0.f, 0.f);
        store_chunk<PRECISE>(tile + (kk >> 2) * (atoms * 512) + a * 512 + (kk & 3) * 128 + ((c ^ ((kk & 3) << 1)) << 4),
                             tail_offset, x);
        if (rowsum && rows_t == BM) {  // cm == t % 32 for every i: per-thread sums of 4 rows of C
          rowsum->x += x.x; rowsum->y += x.y; rowsum->z += x.z; rowsum->w += x.w;
        }
      }
    }
  }
}

template <int ROWS_MAX, bool PRECISE, bool FAST>
__device__ __forceinline__ void load_tile(uint32_t tile, uint32_t tail_offset, const float* __restrict__ P, int64_t ld,
                                          int major, int r0, int R, int rows_t, int k0, int k1, bool vec, int t,
                                          float4* rowsum) {
  float4 v[ROWS_MAX * 8 / GROUP];
  const uint32_t mask = load_regs<ROWS_MAX, FAST>(v, P, ld, major, r0, R, rows_t, k0, k1, vec, t);
  store_regs<ROWS_MAX, PRECISE>(v, mask, tile, tail_offset, major, rows_t, t, rowsum);
}

// One thread of the warp, chosen once.  The issuing code below runs in all lanes with only these instructions predicated: inside
// a divergent branch every descriptor would be moved to the uniform registers that the MMA takes it from, eight moves for
// each MMA, which took longer than the MMA.
__device__ __forceinline__ uint32_t elect_one() {
  uint32_t e;
  asm volatile("{\n\t.reg .pred p;\n\telect.sync _|p, 0xffffffff;\n\tselp.u32 %0, 1, 0, p;\n\t}" : "=r"(e));
  return e;
}
__device__ __forceinline__ void mma_tf32(uint32_t tmem, uint64_t da, uint64_t db, uint32_t idesc, uint32_t acc, uint32_t elected) {
  asm volatile(
      "{\n\t.reg .pred p, q;\n\t"
      "setp.ne.b32 p, %4, 0;\n\t"
      "setp.ne.b32 q, %5, 0;\n\t"
      "@q tcgen05.mma.cta_group::1.kind::tf32 [%0], %1, %2, %3, p;\n\t}"
      ::"r"(tmem), "l"(da), "l"(db), "r"(idesc), "r"(acc), "r"(elected)
      : "memory");
}
// 32 columns of an accumulator, a row per lane (complete after tcgen05.wait::ld).
__device__ __forceinline__ void tmem_ld32(uint32_t (&r)[32], uint32_t taddr) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x32.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,"
      "%16,%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31}, [%32];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]),
        "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]), "=r"(r[16]),
        "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]), "=r"(r[24]),
        "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
      : "r"(taddr));
}
__device__ __forceinline__ void tmem_ld16(uint32_t (&r)[16], uint32_t taddr) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]),
        "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
      : "r"(taddr));
}
// The same with the descriptors' low words, which hold the address: the high words stay where they are.
__device__ __forceinline__ void mma_tf32(uint32_t tmem, uint32_t a_lo, uint32_t a_hi, uint32_t b_lo, uint32_t b_hi, uint32_t idesc, uint32_t acc,
                                         uint32_t elected) {
  asm volatile(
      "{\n\t.reg .pred p, q;\n\t.reg .b64 a, b;\n\t"
      "setp.ne.b32 p, %6, 0;\n\t"
      "setp.ne.b32 q, %7, 0;\n\t"
      "mov.b64 a, {%1, %2};\n\tmov.b64 b, {%3, %4};\n\t"
      "@q tcgen05.mma.cta_group::1.kind::tf32 [%0], a, b, %5, p;\n\t}"
      ::"r"(tmem), "r"(a_lo), "r"(a_hi), "r"(b_lo), "r"(b_hi), "r"(idesc), "r"(acc), "r"(elected)
      : "memory");
}
// The barrier gets an arrival once the MMAs issued so far have completed.
__device__ __forceinline__ void mma_commit(uint32_t bar, uint32_t elected) {
  asm volatile(
      "{\n\t.reg .pred q;\n\t"
      "setp.ne.b32 q, %1, 0;\n\t"
      "@q tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];\n\t}"
      ::"r"(bar), "r"(elected)
      : "memory");
}

// grid: (n tiles, m tiles, split_k).  Dynamic shared memory: Cfg::SMEM bytes.
template <int BN_T, bool PRECISE, bool FAST, int TMA>
__global__ void __launch_bounds__(Cfg<BN_T, PRECISE, TMA>::THREADS, 1) gemm_tf32_kernel(const __grid_constant__ TcArgs g) {
  using C_ = Cfg<BN_T, PRECISE, TMA>;
  constexpr int STAGES = C_::STAGES, GROUPS = C_::GROUPS, THREADS = C_::THREADS, KB = C_::KB;
  constexpr int MMA_WARP = GROUPS * 4;
  extern __shared__ unsigned char smem_raw[];
  __shared__ __align__(8) uint64_t s_full[STAGES], s_empty[STAGES], s_accum, s_raw[STAGES], s_recv;
  __shared__ uint32_t s_tmem;
  __shared__ int s_abort;
  __shared__ float s_rowsum[BM];
  __shared__ __align__(16) float s_bias[BN_T];

  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int m0 = blockIdx.y * BM;
  const int bn = min(BN_T, ((g.N + gridDim.x - 1) / gridDim.x + 31) / 32 * 32);  // columns per n-tile
  const int n0 = blockIdx.x * bn;
  if (m0 >= g.M || n0 >= g.N) return;
  const int n_valid = min(bn, g.N - n0);
  // MMA N: multiple of 16; MN-major B tiles are loaded in whole 32-column atoms
  const int n_mma = (n_valid + 15) / 16 * 16;
  const int b_rows = TMA == 2 ? g.b_box_atoms * 32  // the tile's layout is the box's, whatever part of it is valid
                              : (g.b_major == MAJOR_MN ? (n_valid + 31) / 32 * 32 : (n_mma + 7) / 8 * 8);
  // Heads and tails of a prepared weight tile of up to 128 columns lie side by side along N, and so do the two accumulators: the
  // heads of A go through the tensor core once for both.  Three products per step read 128 x 8 of A and of B from shared
  // memory each, more than it delivers; two products read a sixth less (12 000 x 100 x 501, launch included: 21.7 -> 20.1 us;
  // 12 000 x 100 x 877: 31.0 -> 29.9).
  // The CTAs of a cluster add up their accumulators: each owns a slice of the tile's rows.  An accumulator lies in the idle pipeline memory, rows
  // of an odd number of 16-byte pieces (no bank conflicts), the other CTAs' parts of the own slice behind it.
  const bool in_cluster = BN_T <= 128 && g.in_cluster;
  const int c4 = (n_valid + 3) >> 2, cl_pitch = 16 * (c4 | 1), cl_rank = blockIdx.z;
  const auto slice = [&](int z) { return z * BM / g.split_k; };   // first row of CTA z's
  const int cl_most = (BM + g.split_k - 1) / g.split_k;           // rows of the largest
  const bool joint = PRECISE && BN_T == 128 && g.b_image != nullptr;
  const uint32_t corr = joint ? (uint32_t)b_rows : C_::ACC_COLS;   // first column of the corrections
  unsigned char* smem = reinterpret_cast<unsigned char*>(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
  const uint32_t smem_base = smem_u32(smem);

  if (tid == 0) {
    for (int s = 0; s < STAGES; ++s) {
      mbar_init(smem_u32(&s_full[s]), TMA == 3 ? GROUP / 32 : GROUP + (g.b_image ? 1 : 0));
      mbar_init(smem_u32(&s_empty[s]), 1);
    }
    mbar_init(smem_u32(&s_accum), 1);
    mbar_init(smem_u32(&s_recv), 1);
    for (int r = 0; r < STAGES; ++r) mbar_init(smem_u32(&s_raw[r]), 1);
    s_abort = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (tid < BM) s_rowsum[tid] = 0.f;
  // (The bias is a parameter or was folded ahead of the kernel that this one follows: asked for here, in shared memory before the epilogue.)
  const float my_bias = g.bias != nullptr && tid < n_valid ? __ldg(g.bias + n0 + tid) : 0.f;
  if (warp == MMA_WARP) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&s_tmem)),
                 "r"(C_::TMEM_COLS)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  const uint32_t tmem = s_tmem;
  // TMA == 3: half a block of the weight image into stage s, heads and tails, and the block of A behind them on the same barrier.
  const uint32_t half_bytes = TMA == 3 ? (uint32_t)(b_rows / 32 * 2048) : 0;   // of heads, or of tails
  const auto ask_weights = [&](int kb, int s) {
    constexpr uint32_t image = C_::COPIES * BN_T * BK * 4;   // a block of 32 contraction rows
    const uint32_t bar = smem_u32(&s_raw[s]), dst = smem_base + s * C_::STAGE_BYTES + C_::COPIES * C_::A_BYTES;
    const unsigned char* src = g.b_image + blockIdx.x * g.b_tile_stride + (int64_t)(kb >> 1) * image + (joint ? 2 : 1) * (kb & 1) * half_bytes;
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"((uint32_t)C_::A_BYTES + 2 * half_bytes) : "memory");
    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
                 ::"r"(dst), "l"(src), "r"((joint ? 2 : 1) * half_bytes), "r"(bar)
                 : "memory");
    if (!joint)
      asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
                   ::"r"(dst + C_::B_BYTES), "l"(src + image / 2), "r"(half_bytes), "r"(bar)
                   : "memory");
  };
  const auto ask_rows = [&](int kb, int s) {
    asm volatile("cp.async.bulk.tensor.2d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3}], [%4];"
                 ::"r"(smem_base + s * C_::STAGE_BYTES), "l"(&g.a_map), "r"(kb * KB), "r"(m0), "r"(smem_u32(&s_raw[s]))
                 : "memory");
  };
  // The first stages are asked for by a warp each (a copy takes 200 cycles to issue), their weights ahead of the wait where the rows are counted on
  // the host: the images are written ahead of the kernel that this one follows.
  const int first = TMA == 3 && warp < STAGES && lane == 0 ? warp : -1;
  const auto has_block = [&](int i) {   // (TMA == 3: the contraction's length is known on the host)
    const int total = (g.K + KB - 1) / KB, per = (total + g.split_k - 1) / g.split_k;
    return i < min(per, total - (int)blockIdx.z * per) ? (int)blockIdx.z * per + i : -1;
  };
  const int first_kb = first >= 0 ? has_block(first) : -1;
  if (first_kb >= 0 && g.dev_M == nullptr) ask_weights(first_kb, first);
  if (TMA == 3 && tid == 32 * (MMA_WARP + 1)) asm volatile("prefetch.tensormap [%0];" ::"l"(&g.a_map) : "memory");
  link_wait();
  const int M = g.dev_M ? min(*g.dev_M, g.M) : g.M;
  const int K = g.dev_K ? min(*g.dev_K, g.K) : g.K;
  const int nkb_total = (K + KB - 1) / KB;
  const int per = (nkb_total + g.split_k - 1) / g.split_k;
  const int kb0 = blockIdx.z * per, kb1 = min(nkb_total, kb0 + per);
  const int nkb = kb1 - kb0;
  if (m0 >= M || nkb <= 0) {  // nothing to contract: store mode still owes bias (+ReLU)
    if (m0 < M && !g.accumulate && blockIdx.z == 0) {
      for (int e = tid; e < BM * n_valid; e += THREADS) {
        const int r = e / n_valid, c = e - r * n_valid;
        if (m0 + r < M) {
          float v = g.bias ? g.bias[n0 + c] : 0.f;
          if (g.relu) v = fmaxf(v, 0.f);
          g.C[(int64_t)(m0 + r) * g.ldc + n0 + c] = v;
        }
      }
    }
    if (warp == MMA_WARP)
      asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(C_::TMEM_COLS) : "memory");
    return;
  }

  if (first_kb >= 0) {
    if (g.dev_M != nullptr) ask_weights(first_kb, first);
    ask_rows(first_kb, first);
  }
  if (warp < MMA_WARP) {
    // ------------------------------------------------------------ producers
    const int grp = warp >> 2, t = tid & (GROUP - 1);
    const bool a_vec = (((uintptr_t)g.A & 15) == 0) && (g.lda % 4 == 0);
    const bool b_vec = (((uintptr_t)g.B & 15) == 0) && (g.ldb % 4 == 0);
    const bool want_rowsum = g.rowsum_out != nullptr && blockIdx.x == 0 && g.a_major == MAJOR_MN;
    float4 rs = make_float4(0.f, 0.f, 0.f, 0.f);
    int rs_row = 4 * (t & 31);   // first of the 4 rows of C whose sums of A the thread has in rs
    const int k_end = min(K, kb1 * BK);
    bool ok = true;
    // The A registers of the group's next block are loaded before it waits for the current stage,
    // so that round trip overlaps the wait, the stores and the MMAs of the blocks in between.
    float4 va[BM * 8 / GROUP], vn[BM * 8 / GROUP];
    int32_t tab_row[BM * 8 / GROUP];  // table row of each of the thread's A rows (row-indirect mode)
    const int32_t* trp = nullptr;
    if (g.a_idx != nullptr && g.a_major == MAJOR_K) {
#pragma unroll
      for (int q = 0; q < BM * 8 / GROUP; ++q) {
        const int gr = m0 + ((t + q * GROUP) >> 3);
        const int ti = gr < M ? g.a_idx[gr] : -1;
        tab_row[q] = ti < g.a_tab_rows ? ti : -1;   // an index beyond the table reads as a zero row
      }
      trp = tab_row;
    }
    uint32_t ma = 0, mn = 0;
    // The B tile of block i into stage s: one bulk asynchronous copy of the prepared image (head and tail);
    // it signals full[s] itself.
    auto b_image_copy = [&](int i, int s, uint32_t b_tile) {
      constexpr uint32_t bytes = C_::COPIES * C_::B_BYTES;
      const unsigned char* src = g.b_image + blockIdx.x * g.b_tile_stride + (int64_t)(kb0 + i) * bytes;
      const uint32_t bar = smem_u32(&s_full[s]);
      asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes) : "memory");
      asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
                   ::"r"(b_tile), "l"(src), "r"(bytes), "r"(bar)
                   : "memory");
    };
    if constexpr (TMA == 3) {
      // Activations and weights arrive by the issuing warp below, 16 contraction columns at a time (rows of 64 bytes, 64-byte swizzle):
      // the groups only write the tails, in the order of the tile's bytes.
      for (int i = grp; i < nkb; i += GROUPS) {
        const int s = i % STAGES;
        // (A stage's uses fall to different groups.  One that came here before the stage's use before had landed would take the barrier's
        // parity for that of its own block, and mark a stage that holds nothing: so the use before has to have been read first.)
        if (i >= STAGES) ok = mbar_wait(smem_u32(&s_empty[s]), ((i / STAGES) - 1) & 1);
        if (ok) ok = mbar_wait(smem_u32(&s_raw[s]), (i / STAGES) & 1);
        if (!ok) break;
        const uint32_t a_tile = smem_base + s * C_::STAGE_BYTES + 16 * t;
        constexpr int V = BM * KB / 4 / GROUP;
        float4 x[V];
#pragma unroll
        for (int q = 0; q < V; ++q) x[q] = lds_v4(a_tile + 16 * q * GROUP);
#pragma unroll
        for (int q = 0; q < V; ++q) store_tail_of_raw(a_tile + C_::A_BYTES + 16 * q * GROUP, x[q]);
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
        __syncwarp();
        if (lane == 0) mbar_arrive(smem_u32(&s_full[s]));
      }
    } else if constexpr (TMA == 2) {
      // Weight gradients: both operands are transposed views (contraction over rows).  One thread asks for the
      // block's two boxes -- KB contraction rows x 128 (A) or KB x b_rows (B) values, delivered as atoms of
      // 4 rows x 32 values with the 32-byte swizzle, i.e. in the operand tiles' own layout -- and when they have
      // landed every thread rounds / splits its own chunks in place.  Values beyond the matrix edge inside the
      // last atom are whatever follows in memory: they only reach rows / columns of C that are never stored.
      static_assert(PRECISE, "weight gradients are always split");
      rs_row = (t >> 5) * 32 + 4 * ((t & 7) ^ (((t >> 3) & 3) << 1));
      const uint32_t b_bytes = (uint32_t)b_rows * KB * 4;
      for (int i = grp; i < nkb; i += GROUPS) {
        const int s = i % STAGES;
        if (i >= STAGES) {
          ok = mbar_wait(smem_u32(&s_empty[s]), ((i / STAGES) - 1) & 1);
          if (!ok) break;
        }
        const uint32_t a_tile = smem_base + s * C_::STAGE_BYTES;
        const uint32_t b_tile = a_tile + C_::COPIES * C_::A_BYTES;
        const uint32_t raw_bar = smem_u32(&s_raw[s]);
        if (t == 0) {
          asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(raw_bar), "r"((uint32_t)C_::A_BYTES + b_bytes)
                       : "memory");
          asm volatile(
              "cp.async.bulk.tensor.4d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4, %5}], [%6];"
              ::"r"(a_tile), "l"(&g.a_map), "r"(0), "r"(0), "r"(m0 >> 5), "r"((kb0 + i) * (KB / 4)), "r"(raw_bar)
              : "memory");
          asm volatile(
              "cp.async.bulk.tensor.4d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4, %5}], [%6];"
              ::"r"(b_tile), "l"(&g.b_map), "r"(0), "r"(0), "r"(n0 >> 5), "r"((kb0 + i) * (KB / 4)), "r"(raw_bar)
              : "memory");
        }
        ok = mbar_wait(raw_bar, (i / STAGES) & 1);
        if (!ok) break;
        // Tails: the tiles are walked in the order of their bytes, which needs no coordinates -- a thread's A chunks all hold
        // the same columns (rs_row), of rows 4 q + (t / 8) % 4.  (Finding each chunk's row and column cost a division per
        // chunk and 3.3 us per block of 256 columns.)
        const int left = K - (kb0 + i) * KB;
        if (left >= KB) {
          constexpr int V = BM * KB / 4 / GROUP;   // chunks in flight per thread: all loads of a batch before its stores
          float4 x[V];
#pragma unroll
          for (int q = 0; q < V; ++q) x[q] = lds_v4(a_tile + 16 * (t + q * GROUP));
#pragma unroll
          for (int q = 0; q < V; ++q) {
            store_tail_of_raw(a_tile + C_::A_BYTES + 16 * (t + q * GROUP), x[q]);
            if (want_rowsum) { rs.x += x[q].x; rs.y += x[q].y; rs.z += x[q].z; rs.w += x[q].w; }
          }
          for (int i0 = t; i0 < b_rows * (KB / 4); i0 += V * GROUP) {   // (b_rows is a multiple of 32: whole warps take part or do not)
#pragma unroll
            for (int q = 0; q < V; ++q)
              if (i0 + q * GROUP < b_rows * (KB / 4)) x[q] = lds_v4(b_tile + 16 * (i0 + q * GROUP));
#pragma unroll
            for (int q = 0; q < V; ++q)
              if (i0 + q * GROUP < b_rows * (KB / 4)) store_tail_of_raw(b_tile + C_::B_BYTES + 16 * (i0 + q * GROUP), x[q]);
          }
        } else {   // the last block of the contraction: rows beyond it are whatever follows in memory
          for (int q = 0; q < BM * KB / 4 / GROUP; ++q) {
            const uint32_t addr = a_tile + 16 * (t + q * GROUP);
            float4 x = make_float4(0.f, 0.f, 0.f, 0.f);
            if (4 * q + ((t >> 3) & 3) < left) x = lds_v4(addr);
            else sts_v4(addr, 0u, 0u, 0u, 0u);
            store_tail_of_raw(addr + C_::A_BYTES, x);
            if (want_rowsum) { rs.x += x.x; rs.y += x.y; rs.z += x.z; rs.w += x.w; }
          }
          for (int idx = t; idx < b_rows * (KB / 4); idx += GROUP) {
            const uint32_t addr = b_tile + 16 * idx;
            float4 x = make_float4(0.f, 0.f, 0.f, 0.f);
            if (4 * (idx / b_rows) + ((idx >> 3) & 3) < left) x = lds_v4(addr);
            else sts_v4(addr, 0u, 0u, 0u, 0u);
            store_tail_of_raw(addr + C_::B_BYTES, x);
          }
        }
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
        mbar_arrive(smem_u32(&s_full[s]));
      }
    } else if constexpr (TMA == 1) {
      // A arrives as whole tiles: once the stage is free, one thread of the group asks the tensor-memory-access
      // unit for block i (box 32 x 128 at column k, row m0; rows and columns outside the matrix come back as
      // zeros) straight into the stage's head tile, already in its 128-byte-swizzled layout.  When the tile
      // has landed every thread rounds its own chunks in place and writes their tails -- shared memory to
      // shared memory, no thread touches another's chunk.  Blocks that overlap the row-indirect columns still
      // go through registers from global memory.
      auto by_tma = [&](int i) { return !(g.a_idx != nullptr && (kb0 + i) * BK < g.a_tab_cols); };
      for (int i = grp; i < nkb; i += GROUPS) {
        const int s = i % STAGES;
        const bool tile = by_tma(i);
        if (!tile)
          ma = load_regs<BM, FAST>(va, g.A, g.lda, g.a_major, m0, M, BM, (kb0 + i) * BK, k_end, a_vec, t, trp, g.a_tab,
                                   g.a_tab_cols);
        if (i >= STAGES) {
          ok = mbar_wait(smem_u32(&s_empty[s]), ((i / STAGES) - 1) & 1);
          if (!ok) break;
        }
        const uint32_t a_tile = smem_base + s * C_::STAGE_BYTES;
        const uint32_t b_tile = a_tile + C_::COPIES * C_::A_BYTES;
        const uint32_t raw_bar = smem_u32(&s_raw[s]);
        if (t == 0) {
          if (tile) {
            asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(raw_bar), "r"((uint32_t)C_::A_BYTES)
                         : "memory");
            asm volatile(
                "cp.async.bulk.tensor.2d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3}], [%4];"
                ::"r"(a_tile), "l"(&g.a_map), "r"((kb0 + i) * BK), "r"(m0), "r"(raw_bar)
                : "memory");
          }
          b_image_copy(i, s, b_tile);
        }
        if (tile) {
          int before = 0;  // tile blocks that used this stage (and its tile barrier) before block i: the phase
          for (int j = s; j < i; j += STAGES) before += by_tma(j) ? 1 : 0;
          ok = mbar_wait(raw_bar, before & 1);
          if (!ok) break;
#pragma unroll
          for (int q = 0; q < BM * 8 / GROUP; ++q) {
            const int idx = t + q * GROUP, r = idx >> 3, c = idx & 7;
            const uint32_t addr = a_tile + r * 128 + ((c ^ (r & 7)) << 4);
            asm volatile("ld.shared.v4.f32 {%0,%1,%2,%3}, [%4];"
                         : "=f"(va[q].x), "=f"(va[q].y), "=f"(va[q].z), "=f"(va[q].w) : "r"(addr) : "memory");
          }
          ma = 0xffffffffu;
        }
        if (tile && PRECISE) {  // the landed values stay in place as heads
#pragma unroll
          for (int q = 0; q < BM * 8 / GROUP; ++q) {
            const int idx = t + q * GROUP, r = idx >> 3, c = idx & 7;
            store_tail_of_raw(a_tile + C_::A_BYTES + r * 128 + ((c ^ (r & 7)) << 4), va[q]);
          }
        } else {
          store_regs<BM, PRECISE>(va, ma, a_tile, C_::A_BYTES, MAJOR_K, BM, t, nullptr);
        }
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
        mbar_arrive(smem_u32(&s_full[s]));
      }
    } else {
    if (grp < nkb)
      ma = load_regs<BM, FAST>(va, g.A, g.lda, g.a_major, m0, M, BM, (kb0 + grp) * BK, k_end, a_vec, t, trp, g.a_tab,
                               g.a_tab_cols);
    for (int i = grp; i < nkb; i += GROUPS) {
      const int s = i % STAGES;
      if (i + GROUPS < nkb)
        mn = load_regs<BM, FAST>(vn, g.A, g.lda, g.a_major, m0, M, BM, (kb0 + i + GROUPS) * BK, k_end, a_vec, t, trp,
                                 g.a_tab, g.a_tab_cols);
      if (i >= STAGES) {
        ok = mbar_wait(smem_u32(&s_empty[s]), ((i / STAGES) - 1) & 1);
        if (!ok) break;
      }
      const uint32_t a_tile = smem_base + s * C_::STAGE_BYTES;
      const uint32_t b_tile = a_tile + C_::COPIES * C_::A_BYTES;
      const int k0 = (kb0 + i) * BK;
      if (g.b_image != nullptr && t == 0) b_image_copy(i, s, b_tile);
      store_regs<BM, PRECISE>(va, ma, a_tile, C_::A_BYTES, g.a_major, BM, t, want_rowsum ? &rs : nullptr);
      if (g.b_image == nullptr)
        load_tile<BN_T, PRECISE, FAST>(b_tile, C_::B_BYTES, g.B, g.ldb, g.b_major, n0, g.N, b_rows, k0, k_end, b_vec, t, nullptr);
      asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
      mbar_arrive(smem_u32(&s_full[s]));
#pragma unroll
      for (int q = 0; q < BM * 8 / GROUP; ++q) va[q] = vn[q];
      ma = mn;
    }
    }
    if (!ok) { s_abort = 1; atomicCAS(g.status, 0, TGNN_ETIMEOUT); }
    if (want_rowsum) {
      const int r = rs_row;
      atomicAdd(&s_rowsum[r], rs.x); atomicAdd(&s_rowsum[r + 1], rs.y);
      atomicAdd(&s_rowsum[r + 2], rs.z); atomicAdd(&s_rowsum[r + 3], rs.w);
    }
    // ------------------------------------------------------------ epilogue
    if (ok) ok = mbar_wait(smem_u32(&s_accum), 0);
    if (!ok) { s_abort = 1; atomicCAS(g.status, 0, TGNN_ETIMEOUT); }
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    if (in_cluster) {   // (the pipeline memory is idle: the others may write into it)
      if (tid == 0)
        asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;"
                     ::"r"(smem_u32(&s_recv)), "r"((uint32_t)((g.split_k - 1) * (slice(cl_rank + 1) - slice(cl_rank)) * cl_pitch)) : "memory");
      __syncwarp();
      asm volatile("barrier.cluster.arrive.relaxed.aligned;" ::: "memory");
    }
    if (tid < BN_T) s_bias[tid] = my_bias;
    asm volatile("bar.sync 1, %0;" ::"n"(GROUPS * GROUP) : "memory");  // all producers: s_rowsum and s_bias complete
    if (want_rowsum && tid < BM && m0 + tid < M && s_rowsum[tid] != 0.f) atomicAdd(&g.rowsum_out[m0 + tid], s_rowsum[tid]);
    if (__all_sync(FULL, ok && !s_abort)) {  // warp-uniform: the TMEM loads are warp-collective
      // Each warp moves 32 rows x 32 columns at a time: TMEM -> registers (one row per lane) -> its
      // own staging square in the now idle pipeline memory -> global, re-read so that 8 lanes cover
      // 128 contiguous bytes of one row of C (whole sectors per request; a lane-per-row store would
      // touch 32 rows with 16 bytes each).
      const int q4 = warp & 3;  // the TMEM lane quarter this warp may access
      const uint32_t taddr = tmem + ((uint32_t)(q4 * 32) << 16);
      if (in_cluster) {   // the whole accumulator into the idle pipeline memory, a lane per row
        const uint32_t part = smem_base + (q4 * 32 + lane) * cl_pitch;
        for (int c0 = grp * 16; c0 < n_valid; c0 += GROUPS * 16) {
          uint32_t r[16], r2[16];
          tmem_ld16(r, taddr + (uint32_t)c0);
          if (PRECISE) tmem_ld16(r2, taddr + corr + (uint32_t)c0);
          asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
          if (PRECISE) {
#pragma unroll
            for (int q = 0; q < 16; ++q) r[q] = __float_as_uint(__uint_as_float(r[q]) + __uint_as_float(r2[q]));
          }
#pragma unroll
          for (int q = 0; q < 4; ++q)
            if ((c0 >> 2) + q < c4) sts_v4(part + 4 * c0 + 16 * q, r[4 * q], r[4 * q + 1], r[4 * q + 2], r[4 * q + 3]);
        }
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");   // (read by bulk copies)
      } else {
      float* stg = reinterpret_cast<float*>(smem) + warp * (32 * EPI_PITCH);
      const bool c_vec = (((uintptr_t)g.C & 15) == 0) && (g.ldc % 4 == 0);
      const int sub = lane >> 3, ch = lane & 7;
      for (int c0 = grp * 32; c0 < n_valid; c0 += GROUPS * 32) {
        uint32_t r[32], r2[32];
        tmem_ld32(r, taddr + (uint32_t)c0);
        if (PRECISE) tmem_ld32(r2, taddr + corr + (uint32_t)c0);
        asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
        if (PRECISE) {
#pragma unroll
          for (int q = 0; q < 32; ++q) r[q] = __float_as_uint(__uint_as_float(r[q]) + __uint_as_float(r2[q]));
        }
#pragma unroll
        for (int q = 0; q < 8; ++q)
          *reinterpret_cast<uint4*>(stg + lane * EPI_PITCH + 4 * q) = make_uint4(r[4 * q], r[4 * q + 1], r[4 * q + 2], r[4 * q + 3]);
        __syncwarp();
        const int col = c0 + 4 * ch;  // first of this lane's 4 columns, relative to the tile
        const float4 b4 = blockIdx.z == 0 ? *reinterpret_cast<const float4*>(s_bias + col) : make_float4(0.f, 0.f, 0.f, 0.f);
        const bool full4 = col + 3 < n_valid;
#pragma unroll
        for (int j = 0; j < 8; ++j) {
          const int rr = j * 4 + sub;
          const int row = m0 + q4 * 32 + rr;
          float4 v = *reinterpret_cast<const float4*>(stg + rr * EPI_PITCH + 4 * ch);
          if (row < M && col < n_valid) {
            v.x += b4.x; v.y += b4.y; v.z += b4.z; v.w += b4.w;
            float* cp = g.C + (int64_t)row * g.ldc + n0 + col;
            if (g.accumulate) {
              if (full4 && c_vec) {
                atomicAdd(reinterpret_cast<float4*>(cp), v);
              } else {
                atomicAdd(cp, v.x);
                if (col + 1 < n_valid) atomicAdd(cp + 1, v.y);
                if (col + 2 < n_valid) atomicAdd(cp + 2, v.z);
                if (col + 3 < n_valid) atomicAdd(cp + 3, v.w);
              }
            } else {
              if (g.relu) { v.x = fmaxf(v.x, 0.f); v.y = fmaxf(v.y, 0.f); v.z = fmaxf(v.z, 0.f); v.w = fmaxf(v.w, 0.f); }
              if (full4 && c_vec) {
                *reinterpret_cast<float4*>(cp) = v;
              } else {
                cp[0] = v.x;
                if (col + 1 < n_valid) cp[1] = v.y;
                if (col + 2 < n_valid) cp[2] = v.z;
                if (col + 3 < n_valid) cp[3] = v.w;
              }
            }
          }
        }
        __syncwarp();
      }
      }
    }
  } else if (TMA == 3 && warp > MMA_WARP) {
    // ------------------------------------------------------------ issuing warp: everything a stage holds, as soon as it is free again
    if (lane == 0) {
      bool ok = true;
      int i = STAGES, s = 0, ph = 0;   // ph: parity of the stage's last release
      for (; i < nkb; ++i) {
        ok = mbar_wait(smem_u32(&s_empty[s]), ph);
        if (!ok) break;
        ask_weights(kb0 + i, s);
        ask_rows(kb0 + i, s);
        if (++s == STAGES) { s = 0; ph ^= 1; }
      }
      i = min(i, nkb);
      if (!ok) { s_abort = 1; atomicCAS(g.status, 0, TGNN_ETIMEOUT); }
      for (int q = 1; q <= STAGES && q <= i; ++q)   // what was asked for has landed before the CTA goes
        mbar_wait(smem_u32(&s_raw[(i - q) % STAGES]), ((i - q) / STAGES) & 1);
    }
    __syncwarp();
    if (in_cluster) asm volatile("barrier.cluster.arrive.relaxed.aligned;" ::: "memory");
  } else {
    // ------------------------------------------------------------ MMA issuer
    // instruction descriptor: D fp32, A/B tf32, majors, N >> 3, M >> 4
    const uint32_t idesc = (1u << 4) | (2u << 7) | (2u << 10) | ((uint32_t)g.a_major << 15) | ((uint32_t)g.b_major << 16) |
                           ((uint32_t)(n_mma >> 3) << 17) | ((uint32_t)(BM >> 4) << 24);
    // K-major: 8-row x 128 B atoms 1024 B apart (SBO); one MMA advances 32 B inside the swizzle row.
    // MN-major: 4-k-row atoms of 512 B; MN atoms 512 B apart (LBO), k-groups atoms*512 B apart (SBO); one MMA consumes
    // two k-groups.
    // (One thread issues everything: descriptors are a base and an increment, not built for each MMA.)
    const int b_atoms = (b_rows >> 5) << (joint ? 1 : 0);   // atoms per group of 4 k-rows, tails included if joint
    const uint32_t b_smem = smem_base + C_::COPIES * C_::A_BYTES;
    const uint64_t a_desc = TMA == 3 ? make_desc(smem_base, 16, 512, 4) : g.a_major == MAJOR_K ? make_desc(smem_base, 16, 1024, 2) : make_desc(smem_base, 512, (BM / 32) * 512, 1);
    const uint64_t b_desc = g.b_major == MAJOR_K ? make_desc(b_smem, 16, 1024, 2) : make_desc(b_smem, 512, b_atoms * 512, 1);
    const uint32_t a_step = g.a_major == MAJOR_K ? 2 : (BM / 32) * 64, b_step = g.b_major == MAJOR_K ? 2 : b_atoms * 64;
    const uint32_t idesc2 = (idesc & ~(0x3fu << 17)) | ((corr + b_rows) >> 3) << 17;
    const uint32_t elected = elect_one();
    bool ok = true;
    if constexpr (TMA == 3 && BN_T == 128) {
      // (Counters and 32-bit sums: with the descriptors built from the block's number, issuing half a block took 550 cycles, 420 now; the
      // tensor core needs 370 for it.)
      const uint32_t a0 = (uint32_t)a_desc, ah = (uint32_t)(a_desc >> 32), b0 = (uint32_t)b_desc, bh = (uint32_t)(b_desc >> 32), tc = tmem + corr;
      uint32_t a = a0, b = b0, more = 0, ph = 0;
      int s = 0;
#pragma unroll 1
      for (int i = 0; i < nkb; ++i) {
        ok = mbar_wait(smem_u32(s_full) + 8 * s, ph);
        if (!ok) break;
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        mma_tf32(tmem, a, ah, b, bh, idesc2, more, elected);                                      // head(A) * [head(B) | tail(B)]
        mma_tf32(tc, a + (C_::A_BYTES >> 4), ah, b, bh, idesc, 1u, elected);                      // tail(A) * head(B)
        mma_tf32(tmem, a + 2, ah, b + b_step, bh, idesc2, 1u, elected);
        mma_tf32(tc, a + (C_::A_BYTES >> 4) + 2, ah, b + b_step, bh, idesc, 1u, elected);
        mma_commit(smem_u32(s_empty) + 8 * s, elected);   // frees the stage once the MMAs that read it have completed
        more = 1;
        a += C_::STAGE_BYTES >> 4; b += C_::STAGE_BYTES >> 4;
        if (++s == STAGES) { s = 0; ph ^= 1; a = a0; b = b0; }
      }
    } else {
      for (int i = 0; i < nkb && ok; ++i) {
        const int s = i % STAGES;
        ok = mbar_wait(smem_u32(&s_full[s]), (i / STAGES) & 1);
        if (!ok) break;
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        const uint64_t da = a_desc + ((s * C_::STAGE_BYTES) >> 4), db = b_desc + ((s * C_::STAGE_BYTES) >> 4);
  #pragma unroll
        for (int k = 0; k < KB / UMMA_K; ++k) {
          const uint32_t first = (i > 0 || k > 0) ? 1u : 0u;
          if (PRECISE && joint) {
            mma_tf32(tmem, da + k * a_step, db + k * b_step, idesc2, first, elected);                                  // head(A) * [head(B) | tail(B)]
            mma_tf32(tmem + corr, da + (C_::A_BYTES >> 4) + k * a_step, db + k * b_step, idesc, 1u, elected);          // tail(A) * head(B)
          } else if (PRECISE) {
            mma_tf32(tmem + C_::ACC_COLS, da + (C_::A_BYTES >> 4) + k * a_step, db + k * b_step, idesc, first, elected);  // tail(A) * head(B)
            mma_tf32(tmem + C_::ACC_COLS, da + k * a_step, db + (C_::B_BYTES >> 4) + k * b_step, idesc, 1u, elected);     // head(A) * tail(B)
            mma_tf32(tmem, da + k * a_step, db + k * b_step, idesc, first, elected);                          // head(A) * head(B)
          } else {
            mma_tf32(tmem, da + k * a_step, db + k * b_step, idesc, first, elected);
          }
        }
        // frees the stage for the producers once the MMAs that read it have completed
        mma_commit(smem_u32(&s_empty[s]), elected);
      }
    }
    link_release();
    if (ok) mma_commit(smem_u32(&s_accum), elected);
    else if (lane == 0) { s_abort = 1; atomicCAS(g.status, 0, TGNN_ETIMEOUT); }
    __syncwarp();
    if (in_cluster) asm volatile("barrier.cluster.arrive.relaxed.aligned;" ::: "memory");
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  if (warp == MMA_WARP) {
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(C_::TMEM_COLS) : "memory");
  }
  if (in_cluster) {
    // Every CTA sends the slices of its accumulator to their owners, one bulk copy each, adds up its own and stores it (all of them get
    // here: every wait above is bounded).  Loads of the others' shared memory in their place, all eight of a thread under way at once, ran at 10
    // bytes a cycle and took 4 500 cycles for 45 KB.  (Nothing is handed over by the barriers themselves, which say that a CTA's memory is idle
    // and that its part has come: relaxed, a release costs 900 cycles each time.)
    const int S = g.split_k, r0 = slice(cl_rank), rows = slice(cl_rank + 1) - r0;
    const uint32_t recv = smem_base + BM * cl_pitch;
    asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
    if (tid < S && tid != cl_rank) {
      const int z = tid, first = slice(z);
      uint32_t to, bar;
      asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(to) : "r"(recv + (cl_rank < z ? cl_rank : cl_rank - 1) * cl_most * cl_pitch), "r"(z));
      asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(bar) : "r"(smem_u32(&s_recv)), "r"(z));
      asm volatile("cp.async.bulk.shared::cluster.shared::cta.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
                   ::"r"(to), "r"(smem_base + first * cl_pitch), "r"((uint32_t)((slice(z + 1) - first) * cl_pitch)), "r"(bar)
                   : "memory");
    }
    __syncwarp();
    const int cl_row = tid / c4, cl_col = 4 * (tid - cl_row * c4), cl_step = THREADS / c4, cl_rest = 4 * (THREADS - cl_step * c4);   // the thread's pieces of the slice
    const bool landed = mbar_wait(smem_u32(&s_recv), 0);
    if (!landed) atomicCAS(g.status, 0, TGNN_ETIMEOUT);
    __syncwarp();
    asm volatile("barrier.cluster.arrive.relaxed.aligned;" ::: "memory");   // (what was sent to this CTA is here)
    const bool c_vec = (((uintptr_t)g.C & 15) == 0) && (g.ldc % 4 == 0);
    if (landed && !s_abort)
#pragma unroll 1
      for (int row = cl_row, col = cl_col; row < rows; row += cl_step, col += cl_rest) {
        if (col >= 4 * c4) { col -= 4 * c4; if (++row >= rows) break; }
        if (m0 + r0 + row >= M) break;
        const uint32_t own = smem_base + (r0 + row) * cl_pitch + 4 * col;
        uint32_t at = recv + row * cl_pitch + 4 * col;
        float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll 4
        for (int z = 0; z < S; ++z) {
          const float4 x = lds_v4(z == cl_rank ? own : at);
          if (z != cl_rank) at += cl_most * cl_pitch;
          v.x += x.x; v.y += x.y; v.z += x.z; v.w += x.w;
        }
        const float4 b = *reinterpret_cast<const float4*>(s_bias + col);
        float o[4] = {v.x + b.x, v.y + b.y, v.z + b.z, v.w + b.w};
        if (g.relu) {
#pragma unroll
          for (int q = 0; q < 4; ++q) o[q] = fmaxf(o[q], 0.f);
        }
        float* cp = g.C + (int64_t)(m0 + r0 + row) * g.ldc + n0 + col;
        if (c_vec && col + 3 < n_valid) *reinterpret_cast<float4*>(cp) = make_float4(o[0], o[1], o[2], o[3]);
        else {
#pragma unroll
          for (int q = 0; q < 4; ++q)
            if (col + q < n_valid) cp[q] = o[q];
        }
      }
    asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");   // (and what this CTA has sent is there: its memory may go)
  }
}

// ---- short contractions (K <= 128) ------------------------------------------------------------------------------
// A stored product with a prepared weight image whose contraction fits shared memory whole: the projected queries, the
// gradient of the attention's output inputs, the update cell's hidden gates.  With 4 contraction blocks there is nothing
// for a ring of stages to hide behind: gemm_tf32_kernel spends its time on set-up, on splitting the same rows of A again for
// every tile of columns, and on a store that nothing overlaps.  Here a CTA splits its 128 rows of A once and walks a range
// of column tiles with them: one warp brings weight blocks (up to four stages), one issues the MMAs into two accumulators in turn,
// and eight warps store one accumulator while the other fills.  What bounds it is the weight traffic (64 KB of heads and
// tails per 64 columns' worth of MMAs) and the store.
// 12 000 x 772 x 100 (projected queries): 46 us on the general kernel, 28 us here.
// The corrections have accumulators of their own here too: with one for all three products, 48 MMAs at K = 128 truncated at its
// last bit, a bias of 1.6e-6 of sums of positive terms (fp32 FMA tiles: 1e-7); 16 do now, 5.3e-7.  Times are the same.
constexpr int SHORT_NKB = 4, SHORT_BN = 128, SHORT_STAGES = 4, SHORT_WORKERS = 8, SHORT_STG_BYTES = 32 * 128;
constexpr int SHORT_THREADS = 32 * (SHORT_WORKERS + 2);
constexpr uint32_t SHORT_ACC = 2 * SHORT_BN, SHORT_TMEM = 2 * SHORT_ACC;   // an accumulator and its corrections; two of them in turn
constexpr int SHORT_A_BYTES = 2 * BM * 128, SHORT_B_BYTES = 2 * SHORT_BN * 128;   // heads and tails of one contraction block
constexpr int SHORT_TAIL_BYTES = 2 * BM * 32;   // the last block of A when it has at most 8 columns: one MMA step, rows of 32 bytes
__host__ __device__ inline bool short_tail(int K) { return K % BK != 0 && K % BK <= UMMA_K; }
__host__ __device__ inline int short_a_bytes(int K) {
  return short_tail(K) ? K / BK * SHORT_A_BYTES + SHORT_TAIL_BYTES : (K + BK - 1) / BK * SHORT_A_BYTES;
}
inline int short_smem(int K, int stages) {
  return 1024 + short_a_bytes(K) + stages * SHORT_B_BYTES + SHORT_WORKERS * SHORT_STG_BYTES;
}
inline int short_stages(int K) {   // as many as fit: a weight block takes three times as long to come as to be used
  int s = SHORT_STAGES;
  while (s > 2 && short_smem(K, s) > 226 * 1024) --s;
  return s;
}

// A last block of A of at most 8 columns is the operand of one MMA step: rows of 32 bytes, groups of 8 rows 256 bytes apart, the
// two 16-byte chunks of a row exchanged in rows 4 to 7 of a group (32-byte swizzle).
// grid: (groups of column tiles, m tiles).  bn: columns per tile, per: tiles per CTA.
__global__ void __launch_bounds__(SHORT_THREADS, 1) gemm_short_kernel(const __grid_constant__ TcArgs g, int n_tiles, int bn, int per, int stages) {
  extern __shared__ unsigned char smem_raw[];
  __shared__ __align__(8) uint64_t s_a, s_bfull[SHORT_STAGES], s_bempty[SHORT_STAGES], s_acc[2], s_accfree[2];
  __shared__ uint32_t s_tmem;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int m0 = blockIdx.y * BM, t0 = blockIdx.x * per, nt = min(per, n_tiles - t0);
  if (m0 >= g.M || nt <= 0) return;
  const int nkb = (g.K + BK - 1) / BK;
  unsigned char* smem = reinterpret_cast<unsigned char*>(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
  const uint32_t a_base = smem_u32(smem), b_base = a_base + short_a_bytes(g.K);
  const bool tail = short_tail(g.K);
  if (tid == 0) {
    mbar_init(smem_u32(&s_a), SHORT_WORKERS);
    for (int i = 0; i < SHORT_STAGES; ++i) { mbar_init(smem_u32(&s_bfull[i]), 1); mbar_init(smem_u32(&s_bempty[i]), 1); }
    for (int i = 0; i < 2; ++i) { mbar_init(smem_u32(&s_acc[i]), 1); mbar_init(smem_u32(&s_accfree[i]), SHORT_WORKERS); }
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == SHORT_WORKERS) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&s_tmem)), "r"(SHORT_TMEM) : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  const uint32_t tmem = s_tmem;
  const auto valid_cols = [&](int it) { return min(bn, g.N - (t0 + it) * bn); };
  // block kb of column tile it into stage s: heads and tails of the contraction rows that it uses, the first of the block's bytes
  const auto ask_weights = [&](int it, int kb, int s) {
    const uint32_t bytes = (uint32_t)((valid_cols(it) + 31) / 32 * 2048 * (min(BK, g.K - kb * BK + UMMA_K - 1) / UMMA_K)), bar = smem_u32(s_bfull) + 8 * s;
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes) : "memory");
    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
                 ::"r"(b_base + s * SHORT_B_BYTES), "l"(g.b_image + (t0 + it) * g.b_tile_stride + (int64_t)kb * SHORT_B_BYTES), "r"(bytes), "r"(bar)
                 : "memory");
  };
  // The first stages' weights are asked for by a warp each (a copy takes 200 cycles to issue), where the rows are counted on the host ahead of
  // the wait: images are written ahead of the kernel that this one follows, and so are the row numbers of a table.
  const bool asks = lane == 0 && warp < stages && warp < nt * nkb;
  if (asks && g.dev_M == nullptr) ask_weights(warp / nkb, warp % nkb, warp);
  int row = -1;   // of the table or of A (an index beyond the table reads as a zero row)
  if (warp < SHORT_WORKERS && lane < BM / SHORT_WORKERS) {
    const int r = m0 + warp * (BM / SHORT_WORKERS) + lane;
    if (r < g.M) row = g.a_idx != nullptr ? g.a_idx[r] : r;
    if (g.a_idx != nullptr && row >= g.a_tab_rows) row = -1;
  }
  link_wait();
  const int M = g.dev_M ? min(*g.dev_M, g.M) : g.M;
  if (m0 >= M) {
    if (warp == SHORT_WORKERS)
      asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(SHORT_TMEM) : "memory");
    return;
  }
  if (asks && g.dev_M != nullptr) ask_weights(warp / nkb, warp % nkb, warp);
  bool ok = true;

  if (warp < SHORT_WORKERS) {
    // A warp copies 16 rows of A, a lane one 16-byte chunk of each, straight to where the MMA reads them (the raw values
    // are the heads), and writes the tails of its own chunks.  Two short loops: straight-line code of this length ran at the
    // pace of its instruction fetches, 7 us.
    const int grp = warp >> 2, r0 = warp * (BM / SHORT_WORKERS), c4 = g.K >> 2, kb = lane >> 3;
    const bool in_tail = tail && kb == nkb - 1, used = lane < ((c4 + 1) & ~1);   // (an MMA step takes two chunks)
    const uint32_t blk = a_base + kb * SHORT_A_BYTES, lo = in_tail ? BM * 32 : BM * 128;
    const auto chunk = [&](int r) {
      return blk + (in_tail ? r * 32 + ((((lane & 7) ^ (r >> 2)) & 1) << 4) : r * 128 + (((lane & 7) ^ (r & 7)) << 4));
    };
    const float* base = g.a_idx != nullptr ? g.a_tab : g.A;
    const int64_t pitch = g.a_idx != nullptr ? g.a_tab_cols : g.lda;
    if (m0 + r0 + lane >= M) row = -1;
#pragma unroll 1
    for (int i = 0; i < BM / SHORT_WORKERS; i += 4) {   // (four at a time: shuffles and addresses of a single row would wait for one another)
      int src[4];
#pragma unroll
      for (int u = 0; u < 4; ++u) src[u] = __shfl_sync(FULL, row, i + u);
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        const bool there = src[u] >= 0 && lane < c4;
        const float* p = there ? base + src[u] * pitch + 4 * lane : base;
        if (used)
          asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(chunk(r0 + i + u)), "l"(p), "r"(there ? 16 : 0) : "memory");
      }
    }
    asm volatile("cp.async.wait_all;" ::: "memory");
    if (used) {
#pragma unroll 1
      for (int i = 0; i < BM / SHORT_WORKERS; i += 4) {
        float4 x[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) x[u] = lds_v4(chunk(r0 + i + u));
#pragma unroll
        for (int u = 0; u < 4; ++u) store_tail_of_raw(chunk(r0 + i + u) + lo, x[u]);
      }
    }
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    __syncwarp();
    if (lane == 0) mbar_arrive(smem_u32(&s_a));
    // store: a warp takes its quarter of the rows and every other 32 columns of the tile; a lane has a row, puts it into the
    // warp's staging square (rows of 128 bytes, chunks swizzled) and one lane hands the square to the tensor-memory-access
    // unit, which leaves out what lies beyond the matrix
    const uint32_t stg = b_base + stages * SHORT_B_BYTES + warp * SHORT_STG_BYTES;
    const int q4 = warp & 3, row0 = m0 + q4 * 32;
    for (int it = 0; it < nt; ++it) {
      const int buf = it & 1, n0 = (t0 + it) * bn, n_valid = valid_cols(it);
      float next_bias = g.bias != nullptr && n0 + grp * 32 + lane < g.N ? __ldg(g.bias + n0 + grp * 32 + lane) : 0.f;   // (ahead of the accumulator)
      ok = mbar_wait(smem_u32(&s_acc[buf]), (it >> 1) & 1);
      if (!__all_sync(FULL, ok)) { ok = false; break; }
      asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
      const uint32_t taddr = tmem + buf * SHORT_ACC + ((uint32_t)(q4 * 32) << 16), corr = (uint32_t)((n_valid + 31) / 32 * 32);
      for (int c0 = grp * 32; c0 < n_valid; c0 += 64) {
        uint32_t r[32], r2[32];
        tmem_ld32(r, taddr + (uint32_t)c0);
        tmem_ld32(r2, taddr + corr + (uint32_t)c0);
        const float bias = next_bias;
        if (g.bias != nullptr && n0 + c0 + 64 + lane < g.N) next_bias = __ldg(g.bias + n0 + c0 + 64 + lane);
        if (lane == 0) asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory");   // the square has been read out
        asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
        __syncwarp();
        float v[32];
#pragma unroll
        for (int e = 0; e < 32; ++e) v[e] = __uint_as_float(r[e]) + __uint_as_float(r2[e]);
        if (g.bias != nullptr) {
#pragma unroll
          for (int e = 0; e < 32; ++e) v[e] += __shfl_sync(FULL, bias, e);
        }
        if (g.relu) {
#pragma unroll
          for (int e = 0; e < 32; ++e) v[e] = fmaxf(v[e], 0.f);
        }
#pragma unroll
        for (int q = 0; q < 8; ++q)
          sts_v4(stg + lane * 128 + ((q ^ (lane & 7)) << 4), __float_as_uint(v[4 * q]), __float_as_uint(v[4 * q + 1]),
                 __float_as_uint(v[4 * q + 2]), __float_as_uint(v[4 * q + 3]));
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
        __syncwarp();
        if (lane == 0 && row0 < M) {
          asm volatile("cp.async.bulk.tensor.2d.global.shared::cta.bulk_group [%0, {%1, %2}], [%3];"
                       ::"l"(&g.c_map), "r"(n0 + c0), "r"(row0), "r"(stg)
                       : "memory");
          asm volatile("cp.async.bulk.commit_group;" ::: "memory");
        }
      }
      asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
      __syncwarp();
      if (lane == 0) mbar_arrive(smem_u32(&s_accfree[buf]));
    }
    if (lane == 0) asm volatile("cp.async.bulk.wait_group 0;" ::: "memory");
  } else if (warp == SHORT_WORKERS) {
    // MMA issuer (counters and the descriptors' low words: remainders and 64-bit sums for each block take longer than its products)
    const uint32_t elected = elect_one();
    const uint64_t a_desc = make_desc(a_base, 16, 1024, 2), at_desc = make_desc(a_base, 16, 256, 6);
    const uint32_t idesc0 = (1u << 4) | (2u << 7) | (2u << 10) | ((uint32_t)MAJOR_MN << 16) | ((uint32_t)(BM >> 4) << 24);
    int s = 0;
    uint32_t ring_ph = 0;
    ok = mbar_wait(smem_u32(&s_a), 0);
#pragma unroll 1
    for (int it = 0; it < nt && ok; ++it) {
      const int buf = it & 1, n_valid = valid_cols(it), b_atoms = (n_valid + 31) / 32;
      // (one N for heads and tails side by side, one for the heads alone)
      const uint32_t idesc = idesc0 | (uint32_t)((n_valid + 15) / 16 * 2) << 17, idesc2 = idesc0 | (uint32_t)(b_atoms * 8) << 17;
      const uint64_t b_desc = make_desc(b_base, 512, 2 * b_atoms * 512, 1);
      const uint32_t b_step = b_atoms * 128, d = tmem + buf * SHORT_ACC, dc = d + b_atoms * 32, b_lo = (uint32_t)b_desc, b_hi = (uint32_t)(b_desc >> 32);
      if (it >= 2) ok = mbar_wait(smem_u32(&s_accfree[buf]), ((it >> 1) - 1) & 1);
#pragma unroll 1
      for (int kb = 0; kb < nkb && ok; ++kb) {
        ok = mbar_wait(smem_u32(s_bfull) + 8 * s, ring_ph);
        if (!ok) break;
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        const bool last = tail && kb == nkb - 1;
        const uint32_t a = (uint32_t)(last ? at_desc : a_desc) + ((kb * SHORT_A_BYTES) >> 4), ah = (uint32_t)((last ? at_desc : a_desc) >> 32);
        const uint32_t al = a + ((last ? BM * 32 : BM * 128) >> 4), b = b_lo + ((s * SHORT_B_BYTES) >> 4);
        const int steps = min(BK, g.K - kb * BK + UMMA_K - 1) / UMMA_K;
#pragma unroll
        for (int q = 0; q < BK / UMMA_K; ++q)
          if (q < steps) {
            mma_tf32(d, a + 2 * q, ah, b + q * b_step, b_hi, idesc2, kb > 0 || q > 0 ? 1u : 0u, elected);   // head(A) * [head(B) | tail(B)]
            mma_tf32(dc, al + 2 * q, ah, b + q * b_step, b_hi, idesc, 1u, elected);                         // tail(A) * head(B)
          }
        mma_commit(smem_u32(s_bempty) + 8 * s, elected);
        if (++s == stages) { s = 0; ring_ph ^= 1; }
      }
      if (ok) mma_commit(smem_u32(&s_acc[buf]), elected);
      __syncwarp();
    }
    link_release();
  } else if (lane == 0) {
    // weight blocks behind the first of every stage
    const int total = nt * nkb;
    int i = min(stages, total), it = i / nkb, kb = i - it * nkb, s = 0, ph = 0;
    for (; i < total; ++i) {
      ok = mbar_wait(smem_u32(s_bempty) + 8 * s, ph);
      if (!ok) break;
      ask_weights(it, kb, s);
      if (++kb == nkb) { kb = 0; ++it; }
      if (++s == stages) { s = 0; ph ^= 1; }
    }
    for (int q = 0; q < stages && q < i; ++q)   // what was asked for has landed before the CTA goes
      mbar_wait(smem_u32(&s_bfull[(i - 1 - q) % stages]), ((i - 1 - q) / stages) & 1);
  }
  if (!ok) atomicCAS(g.status, 0, TGNN_ETIMEOUT);
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  if (warp == SHORT_WORKERS) {
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(SHORT_TMEM) : "memory");
  }
}

// n-tiles of at most 256 columns, balanced, in whole 32-column atoms; narrower tiles (down to 64
// columns) when a store-mode product would otherwise occupy only a few SMs.
void tile_plan(int M, int N, bool split_accumulate, int* n_tiles, int* bn, int widest = 256) {
  int nt = (N + widest - 1) / widest;
  const int m_tiles = (M + BM - 1) / BM;
  // (only while the narrower tiles still make one wave of CTAs: a CTA takes a whole SM)
  if (!split_accumulate)
    while (m_tiles * (nt + 1) <= 148 && ((N + nt - 1) / nt + 31) / 32 * 32 > 64) ++nt;
  *bn = ((N + nt - 1) / nt + 31) / 32 * 32;
  *n_tiles = (N + *bn - 1) / *bn;   // (rounded up to whole atoms, fewer tiles may do: none is empty)
}

// Writes the B-operand images of the weight sites from `first` on.  One thread per 16-byte chunk.
__global__ void __launch_bounds__(256) prep_weights_kernel(const WeightSite* __restrict__ sites,
                                                           const float* __restrict__ params,
                                                           const char* __restrict__ arena, int first,
                                                           unsigned char* __restrict__ images) {
  const WeightSite st = sites[first + blockIdx.y];
  const int idx = (int)(blockIdx.x * blockDim.x + threadIdx.x);
  if (idx >= st.chunks) return;
  write_image_chunk(st, first >= SITE_FOLDED ? reinterpret_cast<const float*>(arena + st.w_off) : params + st.w_off, images, idx);
}

// Parts of the contraction of a weight gradient (a leaf of the backward chain, run on a side stream).  The
// CTAs fill about half the machine, with >= 4 blocks of work each: the chain's own kernels keep the other
// half, and fewer, longer CTAs pay the per-CTA set-up and the atomic epilogue less often.  Measured on
// the wiki-shaped step: 148 CTAs 253.7 us, 74 CTAs 246.2 us; the batch-4000 workloads gain 1 - 3 %.
// Not fewer parts than that where the tiles are few: every MMA truncates the accumulator at its last bit, so a part's error grows with its length.
// 100 x 200 over 8 000 rows against fp64 (normal operands, 2-norm): 63 parts 6.4e-7, 15 parts 1.6e-6, with operands of one sign 9.5e-7 and 3.8e-6.
int weight_splits(int tiles, int K) {
  const int s = (74 + tiles - 1) / tiles, most = (K + 4 * BK - 1) / (4 * BK);
  return s < 1 ? 1 : s > most ? most : s;
}

template <int BN_T, bool PRECISE, bool FAST, int TMA>
int launch_tc(tgnn_ctx* ctx, const TcArgs& a, int n_tiles, const char* name, cudaStream_t s) {
  using C_ = Cfg<BN_T, PRECISE, TMA>;
  static SmemLimit smem_limit;   // one per template instance
  {
    const int rc = raise_smem_limit(ctx, gemm_tf32_kernel<BN_T, PRECISE, FAST, TMA>, C_::SMEM, smem_limit);
    if (rc) return rc;
  }
  dim3 grid(n_tiles, (a.M + BM - 1) / BM, a.split_k);
  {
    KernelScope scope__(ctx, name, s);
    launch_link(ctx, gemm_tf32_kernel<BN_T, PRECISE, FAST, TMA>, grid, dim3(C_::THREADS), C_::SMEM, s, a.in_cluster ? a.split_k : 1, a);
  }
  TGNN_LAUNCH_OK(ctx, name);
  return TGNN_OK;
}

// How many clusters of S CTAs of the kernel for K-major tiles run at once (a cluster stays inside a group of SMs, so this is less
// than their number by S).
template <bool PRECISE>
int clusters_at_once(int S) {
  struct Table {
    int n[9] = {};
    Table() {
      constexpr int TMA = PRECISE ? 3 : 1;
      const auto kernel = gemm_tf32_kernel<128, PRECISE, true, TMA>;
      using C_ = Cfg<128, PRECISE, TMA>;
      if (cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, C_::SMEM) != cudaSuccess) { cudaGetLastError(); return; }
      for (int s = 2; s <= 8; ++s) {
        cudaLaunchConfig_t cfg = {};
        cfg.gridDim = dim3(1, 1, s); cfg.blockDim = dim3(C_::THREADS); cfg.dynamicSmemBytes = C_::SMEM;
        cudaLaunchAttribute at;
        at.id = cudaLaunchAttributeClusterDimension;
        at.val.clusterDim.x = 1; at.val.clusterDim.y = 1; at.val.clusterDim.z = s;
        cfg.attrs = &at; cfg.numAttrs = 1;
        if (cudaOccupancyMaxActiveClusters(&n[s], kernel, &cfg) != cudaSuccess) { cudaGetLastError(); n[s] = 0; }
      }
    }
  };
  static const Table t;
  return t.n[S];
}

// Tiled tensor map of a row-major fp32 matrix [rows, cols] (row pitch ld floats): boxes of 32 columns x 128
// rows, 128-byte swizzle (of 16 columns: 64-byte swizzle), zeros outside.  Returns false if the encoder is unavailable or refuses the shape.
bool encode_a_map(CUtensorMap* map, const float* base, int64_t rows, int64_t cols, int64_t ld, int width = BK) {
  const TensorMapEncodeFn enc = tensor_map_encoder();
  if (!enc || rows <= 0 || cols <= 0) return false;
  const cuuint64_t dims[2] = {(cuuint64_t)cols, (cuuint64_t)rows};
  const cuuint64_t strides[1] = {(cuuint64_t)ld * sizeof(float)};
  const cuuint32_t box[2] = {(cuuint32_t)width, BM};
  const cuuint32_t elem[2] = {1, 1};
  return enc(map, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 2, const_cast<float*>(base), dims, strides, box, elem,
             CU_TENSOR_MAP_INTERLEAVE_NONE, width == BK ? CU_TENSOR_MAP_SWIZZLE_128B : CU_TENSOR_MAP_SWIZZLE_64B, CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
             CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}
// A row-major output of M x N, ld floats per row: box 32 x 32.
bool encode_c_map(CUtensorMap* map, float* base, int64_t M, int64_t N, int64_t ld) {
  const TensorMapEncodeFn enc = tensor_map_encoder();
  if (!enc || M <= 0 || N <= 0) return false;
  const cuuint64_t dims[2] = {(cuuint64_t)N, (cuuint64_t)M};
  const cuuint64_t strides[1] = {(cuuint64_t)ld * 4};
  const cuuint32_t box[2] = {32, 32}, elem[2] = {1, 1};
  return enc(map, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 2, base, dims, strides, box, elem, CU_TENSOR_MAP_INTERLEAVE_NONE,
             CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_128B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

}  // namespace

namespace {
// A row-major fp32 matrix [rows (contraction), cols] as the transposed operand of a product: a four-dimensional
// view (value within a 32-wide atom, row within a group of 4, atom, group) whose box of 32 x 4 x atoms x 4 lands
// in shared memory exactly as the MN-major operand tile is laid out: groups of 4 contraction rows, inside a group
// one 512-byte atom per 32 columns, 32-byte swizzle.  rows must be a multiple of 4; the last atom of a row may run
// past the row end (into the next row, or up to 124 bytes past the matrix).
bool encode_mn_map(CUtensorMap* map, const float* base, int64_t rows, int64_t cols, int64_t ld, int box_atoms) {
  const TensorMapEncodeFn enc = tensor_map_encoder();
  if (!enc || rows <= 0 || cols <= 0 || rows % 4 != 0 || box_atoms < 1 || box_atoms > 8) return false;
  const cuuint64_t dims[4] = {32, 4, (cuuint64_t)((cols + 31) / 32), (cuuint64_t)(rows / 4)};
  const cuuint64_t strides[3] = {(cuuint64_t)ld * 4, 128, (cuuint64_t)ld * 16};
  const cuuint32_t box[4] = {32, 4, (cuuint32_t)box_atoms, Cfg<256, true, 2>::KB / 4};
  const cuuint32_t elem[4] = {1, 1, 1, 1};
  return enc(map, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 4, const_cast<float*>(base), dims, strides, box, elem,
             CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B_ATOM_32B, CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
             CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}
}  // namespace

// Returns TGNN_OK after launching, or 1 if the product does not fit this kernel (caller falls back to the FMA tiles).
int launch_gemm_tf32(tgnn_ctx* ctx, const GemmArgs& g, const char* name, cudaStream_t s) {
  TcArgs a = {};
  if (g.a_cs == 1) { a.a_major = MAJOR_K; a.lda = g.a_rs; }
  else if (g.a_rs == 1) { a.a_major = MAJOR_MN; a.lda = g.a_cs; }
  else return 1;
  if (g.b_rs == 1) { a.b_major = MAJOR_K; a.ldb = g.b_cs; }
  else if (g.b_cs == 1) { a.b_major = MAJOR_MN; a.ldb = g.b_rs; }
  else return 1;
  if (g.rowsum_out && a.a_major != MAJOR_MN) return 1;
  a.A = g.A; a.B = g.B; a.C = g.C; a.ldc = g.ldc;
  a.M = g.M; a.N = g.N; a.K = g.K; a.dev_M = g.dev_M; a.dev_K = g.dev_K;
  a.bias = g.bias; a.rowsum_out = g.rowsum_out; a.relu = g.relu; a.accumulate = g.accumulate;
  a.status = ctx->ws.status;
  if (g.a_idx && a.a_major == MAJOR_K && g.a_tab_cols % 4 == 0 && (((uintptr_t)g.a_tab & 15) == 0)) {
    a.a_idx = g.a_idx; a.a_tab = g.a_tab; a.a_tab_cols = g.a_tab_cols;
    a.a_tab_rows = g.a_tab_rows > 0 ? g.a_tab_rows : ((int64_t)1 << 62);
  } else if (g.a_idx) {
    return 1;
  }
  int n_tiles, bn;
  bool precise = g.precise != 0;
  tile_plan(g.M, g.N, g.accumulate && g.split_k > 1, &n_tiles, &bn);
  if (g.site > 0 && ctx->images && (g.site > SITE_DC ? ctx->fold_fresh > 1 : g.site > SITE_FOLDED ? ctx->fold_fresh > 0 : ctx->images_fresh)) {  // B is a weight matrix whose images are up to date
    const WeightSite& st = ctx->sites[g.site - 1];
    n_tiles = st.n_tiles; bn = st.bn; precise = st.precise != 0;
    a.b_image = ctx->images + st.image_off;
    a.b_tile_stride = (int64_t)st.nkb * (st.precise ? 2 : 1) * st.bn_t * 128;
    a.b_major = st.major;
  }
  a.split_k = 1;
  if (g.accumulate && g.split_k > 1) a.split_k = weight_splits(n_tiles * ((g.M + BM - 1) / BM), g.K);
  // whole-chunk operands: 16-byte aligned rows, and the dimension the 16-byte chunks run along is a
  // multiple of 4 and known on the host
  // (An MN-major operand of a workspace buffer may end inside a chunk when its row pitch covers the chunk: the
  // values read past the end only reach rows or columns of C beyond M or N, which are not stored.)
  const bool slack = g.tail_slack != 0;
  const auto whole = [slack](const float* p, int64_t ld, int major, int k, const int* dev_k, int mn, const int* dev_mn) {
    if (((uintptr_t)p & 15) != 0 || ld % 4 != 0) return false;
    return major == MAJOR_K ? (k % 4 == 0 && dev_k == nullptr)
                            : ((mn % 4 == 0 || (slack && (mn + 3) / 4 * 4 <= ld)) && dev_mn == nullptr);
  };
  const bool fast = whole(a.A, a.lda, a.a_major, a.K, a.dev_K, a.M, a.dev_M) &&
                    (a.b_image != nullptr || whole(a.B, a.ldb, a.b_major, a.K, a.dev_K, a.N, nullptr));
  // activations as TMA tiles: K-major whole-chunk A beside a prepared weight image
  static const bool tma_off = getenv("TGNN_NO_TMA") != nullptr;  // debugging aid: activations through registers, plain stores
  // (tiles need 16-byte aligned rows only: a ragged contraction length is the tensor map's edge, filled with zeros)
  const auto aligned = [](const float* p, int64_t ld) { return ((uintptr_t)p & 15) == 0 && ld % 4 == 0; };
  // a short contraction: rows of A split once, column tiles walked with them; as many CTAs as there are SMs share them
  if (!tma_off && a.b_image != nullptr && precise && bn <= SHORT_BN && a.K <= SHORT_NKB * BK && a.a_major == MAJOR_K && !a.accumulate &&
      a.dev_K == nullptr && aligned(a.A, a.lda) && a.K % 4 == 0 && (a.a_idx == nullptr || a.a_tab_cols == a.K) && aligned(a.C, a.ldc) && encode_c_map(&a.c_map, a.C, a.M, a.N, a.ldc)) {
    const int m_tiles = (a.M + BM - 1) / BM, groups = m_tiles >= 148 ? 1 : 148 / m_tiles;
    const int per = (n_tiles + groups - 1) / groups, stages = short_stages(a.K), smem = short_smem(a.K, stages);
    static SmemLimit limit;
    const int rc = raise_smem_limit(ctx, gemm_short_kernel, 226 * 1024, limit);
    if (rc) return rc;
    const dim3 grid((n_tiles + per - 1) / per, m_tiles);
    {
      KernelScope scope__(ctx, name, s);
      launch_link(ctx, gemm_short_kernel, grid, dim3(SHORT_THREADS), smem, s, 1, a, n_tiles, bn, per, stages);
    }
    TGNN_LAUNCH_OK(ctx, name);
    return TGNN_OK;
  }
  const bool halves = precise && a.a_idx == nullptr;   // blocks of 16 columns
  if (!tma_off && aligned(a.A, a.lda) && a.dev_K == nullptr && a.a_major == MAJOR_K && a.b_image != nullptr &&
      encode_a_map(&a.a_map, a.A, a.M, a.K, a.lda, halves ? BK / 2 : BK)) {
    a.a_tma = 1;
    // A stored product of few tiles and a long contraction: split over the CTAs of a cluster, at least 96 columns each, into the
    // most parts of which all run at once.  A CTA takes 0.4 us per 32 columns: 27 blocks on each of 15 tiles took 20 us when it was 0.7,
    // 4 blocks on each of 105 CTAs and the sum 11 us.
    if (!a.accumulate && bn <= 128) {
      const int kb = halves ? BK / 2 : BK, tiles = n_tiles * ((a.M + BM - 1) / BM), nkb = (a.K + kb - 1) / kb;
      for (int S = 8; S > 1; --S) {
        const int per = (nkb + S - 1) / S;
        if (per * kb < 3 * BK || (nkb + per - 1) / per != S) continue;   // (no CTA without a block)
        if (tiles > (precise ? clusters_at_once<true>(S) : clusters_at_once<false>(S))) continue;
        a.split_k = S;
        a.in_cluster = 1;
        break;
      }
    }
    if (halves) {
      if (bn <= 128) return launch_tc<128, true, true, 3>(ctx, a, n_tiles, name, s);
      return launch_tc<256, true, true, 3>(ctx, a, n_tiles, name, s);
    }
    if (precise) {
      if (bn <= 128) return launch_tc<128, true, true, 1>(ctx, a, n_tiles, name, s);
      return launch_tc<256, true, true, 1>(ctx, a, n_tiles, name, s);
    }
    if (bn <= 128) return launch_tc<128, false, true, 1>(ctx, a, n_tiles, name, s);
    return launch_tc<256, false, true, 1>(ctx, a, n_tiles, name, s);
  }
  // weight gradients: both operands transposed, the contraction in groups of 4 rows.  (Workspace matrices may be read past
  // their last row, inside the arena; the kernel takes rows beyond the contraction, whose length may be on the device, as zeros.)
  const int k4 = (a.K + 3) / 4 * 4;
  if (!tma_off && aligned(a.A, a.lda) && aligned(a.B, a.ldb) && precise && a.a_major == MAJOR_MN && a.b_major == MAJOR_MN &&
      a.b_image == nullptr && (g.tail_slack || (a.dev_K == nullptr && a.K % 4 == 0)) && bn % 32 == 0 &&
      (g.tail_slack || ((a.M + 31) / 32 * 32 <= a.lda && (a.N + 31) / 32 * 32 <= a.ldb)) &&  // no read past a caller's matrix
      encode_mn_map(&a.a_map, a.A, k4, a.M, a.lda, BM / 32) && encode_mn_map(&a.b_map, a.B, k4, a.N, a.ldb, bn / 32)) {
    a.a_tma = 2;
    a.b_box_atoms = bn / 32;
    if (bn <= 128) return launch_tc<128, true, true, 2>(ctx, a, n_tiles, name, s);
    return launch_tc<256, true, true, 2>(ctx, a, n_tiles, name, s);
  }
  const int sel = (precise ? 4 : 0) | (bn <= 128 ? 0 : 2) | (fast ? 1 : 0);
  switch (sel) {
    case 0: return launch_tc<128, false, false, 0>(ctx, a, n_tiles, name, s);
    case 1: return launch_tc<128, false, true, 0>(ctx, a, n_tiles, name, s);
    case 2: return launch_tc<256, false, false, 0>(ctx, a, n_tiles, name, s);
    case 3: return launch_tc<256, false, true, 0>(ctx, a, n_tiles, name, s);
    case 4: return launch_tc<128, true, false, 0>(ctx, a, n_tiles, name, s);
    case 5: return launch_tc<128, true, true, 0>(ctx, a, n_tiles, name, s);
    case 6: return launch_tc<256, true, false, 0>(ctx, a, n_tiles, name, s);
    default: return launch_tc<256, true, true, 0>(ctx, a, n_tiles, name, s);
  }
}

}  // namespace tgnn

namespace tgnn {

int weight_grad_ctas(int M, int N, int K) {
  int n_tiles, bn;
  tile_plan(M, N, true, &n_tiles, &bn);
  const int tiles = n_tiles * ((M + BM - 1) / BM);
  return tiles * weight_splits(tiles, K);
}

size_t plan_weight_sites(tgnn_ctx* ctx) {
  const ParamLayout& L = ctx->L;
  const int d = (int)L.d, de = (int)L.de;
  const bool all_precise = ctx->cfg.math_mode != TGNN_MATH_TF32_FAST;
  struct Def { int id; int64_t w_off, ld; int major, N, K, col0, n_split, col1, M_cap, split_acc, grad; };
  const int U = ctx->upd_rows, R = ctx->R_cap, NB = ctx->NB_cap, Q2 = 2 * ctx->nq_cap;
  const int gd = (int)L.gates * d;              // rows of the update cell's matrices
  // the attention block is empty for the time-projection model; with the attention on the query side its products are
  // those with the folded weights
  const int att = L.wo > L.wq && !ctx->qs ? 1 : 0, qs = ctx->qs ? 1 : 0;
  const int HL = ctx->cfg.heads * ctx->ldz;
  const int64_t oA = (const char*)ctx->ws.wA - (const char*)ctx->arena, oB = (const char*)ctx->ws.wB - (const char*)ctx->arena;
  const Def defs[SITE_COUNT] = {
      {SITE_GI, L.gru_wi, L.dmsg, MAJOR_K, gd, (int)L.dmsg, 0, 0, 0, U, 0, 0},
      {SITE_GH, L.gru_wh, d, MAJOR_K, gd, d, 0, 0, 0, U, 0, 0},
      {SITE_KV, L.wk, L.dkv, MAJOR_K, att * 2 * d, (int)L.dkv, 0, 0, 0, NB, 0, 0},
      {SITE_Q, L.wq, 2 * d, MAJOR_K, att * d, 2 * d, 0, 0, 0, R, 0, 0},
      {SITE_OUT, L.wo, 2 * d, MAJOR_K, att * d, 2 * d, 0, 0, 0, R, 0, 0},
      {SITE_HEAD, L.w1, 2 * d, MAJOR_K, d, 2 * d, 0, 0, 0, Q2, 0, 0},
      {SITE_DCAT1, L.w1, 2 * d, MAJOR_MN, 2 * d, d, 0, 2 * d, 0, Q2, 0, 1},
      {SITE_DCATO, L.wo, 2 * d, MAJOR_MN, att * 2 * d, d, 0, 2 * d, 0, R, 0, 1},
      {SITE_DZQ, L.wq, 2 * d, MAJOR_MN, att * 2 * d, d, 0, 2 * d, 0, R, 0, 1},
      {SITE_DZ, L.wk, L.dkv, MAJOR_MN, att * 2 * d, 2 * d, 0, d, d + de, NB, 0, 1},
      {SITE_DXPHI, L.gru_wi, L.dmsg, MAJOR_MN, d, gd, 2 * d + de, d, 0, U, 0, 1},
      {SITE_QP, oA, d, MAJOR_K, qs * HL, d, 0, 0, 0, R, 0, 0},
      {SITE_OUTC, oB, ctx->ldc, MAJOR_K, qs * d, HL + d + 1, 0, 0, 0, R, 0, 0},
      {SITE_DC, oB, ctx->ldc, MAJOR_MN, qs * (HL + d), d, 0, HL + d, 0, R, 0, 1},
      {SITE_DM, oA, d, MAJOR_MN, qs * d, HL, 0, d, 0, R, 0, 1},
  };
  size_t off = 0;
  for (const Def& f : defs) {
    WeightSite& st = ctx->sites[f.id];
    if (f.N == 0) {  // a projection this model does not have: an empty image
      st = WeightSite{};
      st.image_off = (int64_t)off;
      continue;
    }
    st.w_off = f.w_off; st.ld = f.ld; st.major = f.major; st.N = f.N; st.K = f.K;
    st.col0 = f.col0; st.n_split = f.n_split; st.col1 = f.col1;
    st.precise = (all_precise || f.grad) ? 1 : 0;
    // short contractions: tiles of the width that gemm_short_kernel takes, MN-major (so that a last block of few rows is short)
    const bool brief = st.precise && f.K <= SHORT_NKB * BK;
    // (split: MN-major, so that half a block is contiguous)
    st.by_rows = st.precise && f.major == MAJOR_K;
    if (st.precise) st.major = MAJOR_MN;
    // (to be split over clusters: full-width tiles, the split fills the machine)
    const bool split = f.K >= CL_MIN_K && 2 * ((f.M_cap + BM - 1) / BM) <= 148;
    tile_plan(f.M_cap, f.N, split, &st.n_tiles, &st.bn, brief || split ? SHORT_BN : 256);
    st.bn_t = st.bn <= 128 ? 128 : 256;
    st.nkb = (f.K + BK - 1) / BK;
    st.image_off = (int64_t)off;
    st.chunks = (int64_t)st.n_tiles * st.nkb * st.bn_t * 8;
    off += (size_t)st.n_tiles * st.nkb * (st.precise ? 2 : 1) * st.bn_t * 128;
  }
  return off;
}

static int launch_images(tgnn_ctx* ctx, int first, int end, const char* name, cudaStream_t s) {
  int64_t mx = 0;
  for (int i = first; i < end; ++i) mx = ctx->sites[i].chunks > mx ? ctx->sites[i].chunks : mx;
  if (mx == 0) return TGNN_OK;
  dim3 grid((unsigned)((mx + 255) / 256), end - first);
  {
    KernelScope scope__(ctx, name, s);
    prep_weights_kernel<<<grid, 256, 0, s>>>(ctx->sites_dev, ctx->params, (const char*)ctx->arena, first, ctx->images);
  }
  TGNN_LAUNCH_OK(ctx, name);
  return TGNN_OK;
}

int launch_prep_cell(tgnn_ctx* ctx, cudaStream_t s) { return launch_images(ctx, SITE_GI, SITE_GH + 1, "prep_cell", s); }

int launch_prep_folded(tgnn_ctx* ctx, bool backward, cudaStream_t s) {
  if (!ctx->qs) return TGNN_OK;
  if (!backward) {
    const int rc = launch_fold_weights(ctx, s);
    if (rc) return rc;
  }
  if (!ctx->images) return TGNN_OK;
  return backward ? launch_images(ctx, SITE_DC, SITE_COUNT, "prep_folded_bwd", s) : launch_images(ctx, SITE_FOLDED, SITE_DC, "prep_folded", s);
}

int ensure_folded(tgnn_ctx* ctx, int parts, cudaStream_t s) {
  for (; ctx->fold_fresh < parts; ++ctx->fold_fresh) {
    const int rc = launch_prep_folded(ctx, ctx->fold_fresh == 1, s);
    if (rc) return rc;
  }
  return TGNN_OK;
}

}  // namespace tgnn
