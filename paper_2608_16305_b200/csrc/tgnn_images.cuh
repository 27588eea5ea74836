// Images of the weight matrices (WeightSite): what a chunk holds and where it lies.
#pragma once
#include "tgnn_internal.cuh"

namespace tgnn {

enum { MAJOR_K = 0, MAJOR_MN = 1 };
constexpr int IMAGE_K = 32;   // contraction elements per block of an image

// Round-to-nearest (ties away from zero) to the 10 mantissa bits of TF32: add half an ulp to the
// magnitude and clear the 13 low bits.  Same result as cvt.rna.tf32.f32 for finite inputs, but on
// the integer pipe at full rate (the conversion pipe would bound the producers).
__device__ __forceinline__ uint32_t to_tf32(float x) { return (__float_as_uint(x) + 0x1000u) & 0xffffe000u; }

// Chunk idx (16 bytes) of a site's images from the matrix W: the rounding / head-tail split and the swizzled placement that the
// tensor-core kernels expect of a B tile.
__device__ __forceinline__ void write_image_chunk(const WeightSite& st, const float* __restrict__ W, unsigned char* __restrict__ images, int idx) {
  const int per_tile_kb = st.bn_t * 8;  // logical chunks per (tile, k-block)
  const int tk = idx / per_tile_kb, cidx = idx - tk * per_tile_kb, tile = tk / st.nkb, kb = tk - tile * st.nkb;   // (32 bits: a site has at most a few million chunks)
  const int n0 = tile * st.bn;
  const int n_valid = min(st.bn, st.N - n0);
  const int n_mma = (n_valid + 15) / 16 * 16;
  const int copies = st.precise ? 2 : 1;
  const int b_bytes = st.bn_t * 128;
  unsigned char* img = images + st.image_off + ((int64_t)tile * st.nkb + kb) * copies * b_bytes;
  float v[4] = {0.f, 0.f, 0.f, 0.f};
  uint32_t off, tail = b_bytes;   // place of the chunk, distance of its tail
  if (st.major == MAJOR_K) {
    const int r = cidx >> 3, c = cidx & 7;
    const int n = n0 + r, k = kb * IMAGE_K + 4 * c;
    if (r < (n_mma + 7) / 8 * 8 && n < st.N)
      for (int e = 0; e < 4; ++e)
        if (k + e < st.K) v[e] = W[(int64_t)n * st.ld + k + e];
    off = (r >> 3) * 1024 + (r & 7) * 128 + ((c ^ (r & 7)) << 4);
  } else {
    const int b_rows = (n_valid + 31) / 32 * 32;
    const int cpr = b_rows >> 2, atoms = b_rows >> 5;
    // (neighbouring threads run along the matrix's rows: along k of one that is read as W[n * ld + k], 32 loads of a row each where
    // they would touch 32 rows)
    const int kk = st.by_rows ? cidx & (IMAGE_K - 1) : cidx / cpr, cm = st.by_rows ? cidx / IMAGE_K : cidx - kk * cpr;
    if (kk >= IMAGE_K || cm >= cpr) return;  // beyond the region this tile uses
    const int k = kb * IMAGE_K + kk;
    for (int e = 0; e < 4; ++e) {
      const int n = n0 + 4 * cm + e;
      if (k < st.K && n < st.N) {
        const int col = n < st.n_split ? st.col0 + n : st.col1 + (n - st.n_split);
        v[e] = st.by_rows ? W[(int64_t)n * st.ld + k] : W[(int64_t)k * st.ld + col];
      }
    }
    const int a = cm >> 3, c = cm & 7;
    const int joint = copies == 2 && st.bn_t == 128;   // the tails' atoms behind the heads' in every group of 4 k-rows
    if (joint) tail = atoms * 512;
    off = (kk >> 2) * ((atoms << joint) * 512) + a * 512 + (kk & 3) * 128 + ((c ^ ((kk & 3) << 1)) << 4);
  }
  const uint32_t h0 = to_tf32(v[0]), h1 = to_tf32(v[1]), h2 = to_tf32(v[2]), h3 = to_tf32(v[3]);
  *reinterpret_cast<uint4*>(img + off) = make_uint4(h0, h1, h2, h3);
  if (st.precise)
    *reinterpret_cast<uint4*>(img + tail + off) =
        make_uint4(to_tf32(v[0] - __uint_as_float(h0)), to_tf32(v[1] - __uint_as_float(h1)),
                   to_tf32(v[2] - __uint_as_float(h2)), to_tf32(v[3] - __uint_as_float(h3)));
}

}  // namespace tgnn
