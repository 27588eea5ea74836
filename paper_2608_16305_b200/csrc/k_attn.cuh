// The query-side attention's kernels as their launcher (k_attn.cu) sees them.
#pragma once
#include "tgnn_internal.cuh"
#include "tgnn_device.cuh"

namespace tgnn {

struct AttnArgs {
  const float* memory;
  const void* efeat;
  const float *time_w, *time_b;
  const int32_t *nodes, *nbr, *eid, *cnt;
  const double *times, *ts;
  int n, d, de, k, H, ldz, ldc;   // ldc: row pitch of cat
  int64_t N, E;
  int32_t* status;
  const float* qp;                // [n, H ldz]
  float* prob;                    // [n, H, k]
  float* cat;                     // [n, ldc]: zbar per head | m_root | 1 if the root has a slot
  // backward
  const float* dcat;              // [n, ldd]: gradient of cat's first H ldz + d columns
  int ldd;
  float* dqp;                     // [n, H ldz]
  const int32_t* node2slot;       // null: no memory update in this step
  float* dMemU;                   // [copies][upd_rows][d]: a block adds to one of the copies
  int upd_rows;                   // rows of a copy
  int copy_mask;                  // copies - 1
  double* tg_part;                // [blocks][2 d] time-encoder sums of each block
};

typedef void (*AttnKernel)(const AttnArgs);

// Memory rows are read as pieces of four columns, feature rows as pairs of columns (one 32-bit word of a bf16 table, 64 bits
// of an fp32 table); SINGLE: both word by word, for tables that are not aligned to that.  Raw: as they lie in memory.
enum { X_F32 = 0, X_F32_SINGLE = 1, X_BF16 = 2, X_BF16_SINGLE = 3 };
__host__ __device__ constexpr bool is_bf16(int XM) { return XM >= X_BF16; }
__host__ __device__ constexpr bool is_single(int XM) { return XM == X_F32_SINGLE || XM == X_BF16_SINGLE; }
__host__ __device__ constexpr int pair_bytes(int XM) { return XM >= X_BF16 ? 4 : 8; }
// Words of a staged slot row: memory, encoding, raw feature pairs.
__host__ __device__ inline int staged_words(int d, int de, int XM) { return 2 * d + (((de >> 1) * pair_bytes(XM) / 4 + 3) & ~3); }

// What the choices are worth (attention forward / backward of 12 000 roots, k = 10, d = 100, two heads, us):
// (backward: of a build with one copy of the updated rows' gradients behind a cache, 97; with several copies, k_attn_kernels.cuh, it is
// 69, and the lines on k = 11 to 16 are of that)
//   two heads per warp 52 / 90, one 103 / 163 (186 bf16 columns): the heads share a slot's gathered row;
//   slots in batches of 5 for k = 5: 34 / 57, of 10: 50 / 71: every loop runs over a whole batch;
//   slots in one batch of 16 for k = 11 to 16 instead of two of 10, the first of which the backward pass gathered twice: 49 / 80
//   and 58 / 85 (3 711 roots, k = 15, d = 128, 4 heads, 90 fp32 columns), 59 / 87 and 80 / 114 (9 000 roots, k = 15, d = 100, 186 bf16
//   columns), 14 / 17 and 16 / 21 (900 roots, d = 32); k = 11: 49 / 79 and 57 / 84;
//   feature columns in 3 pairs per lane for 129 to 192: 54 / 93, in 4: 71 / 103 (172 fp32 columns); in 1 pair up to 64:
//   37 / 87, in 2: 53 / 90 (64 fp32 columns).
// Registers: 128 forward and 168 backward at k <= 10 and d <= 128 (16 and 12 warps per SM), 168 both for more neighbors (at k = 11 to
// 16 the staged rows allow 7 to 12 warps) or one head, up to 255 for d > 128.  Most instances spill a few words (0 to 44 bytes of
// stores per thread at k <= 10 and up to three pairs, 84 with four); the forward for more than 16 neighbors, whose sums live beside the query row, spills 16 to
// 128 bytes up to two pairs, 250 at three and 460 at four, and its backward half of that.
//
// The forward or backward kernel for HU heads per warp, SB slots per batch (MULTI: k may exceed SB), JD pieces of four memory
// columns per lane and d_e feature columns.  108 kernels in all, of which a context takes two: they are spread over files
// (k_attn_*.cu), because a file's kernels are loaded together when the first of them is asked for.  In one file that took
// 21 ms of a process's first context.
template <int HU, int SB, bool MULTI, int JD>
AttnKernel attn_kernel(int de, bool bf16, bool bwd);
AttnKernel attn_kernel_words(int de, bool bf16, bool bwd);   // tables that are not aligned to its pieces: one head, any shape

}  // namespace tgnn
