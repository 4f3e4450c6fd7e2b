// Tensor maps of the z-passes' TMA-fed tiles, and the launch shapes that depend on one (host).
#pragma once
#include <cuda.h>
#include <cudaTypedefs.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <cstdint>

#include "gfp_kernels.cuh"

namespace gfp {

inline int round32(int x) { return ((x + 31) / 32) * 32; }

// cuTensorMapEncodeTiled from the driver (looked up once; null if unavailable).
inline PFN_cuTensorMapEncodeTiled_v12000 tensor_map_encoder() {
  static PFN_cuTensorMapEncodeTiled_v12000 fn = nullptr;
  static bool tried = false;
  if (!tried) {
    tried = true;
    void* p = nullptr;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault, &q) == cudaSuccess &&
        q == cudaDriverEntryPointSuccess)
      fn = reinterpret_cast<PFN_cuTensorMapEncodeTiled_v12000>(p);
  }
  return fn;
}

// Tensor map of a half spectrum (FP32 or FP64 complex) as reals {2P, n2, n3, 6} with z-tiles of
// `cols` columns x min(n3, 256) rows.  FP32 tiles of 8 columns (64-byte rows) use the 64-byte swizzle at the lengths whose
// z-pass reads it (pass_z_s_kernel, pass_z_l_kernel), all others none.  Returns false if the shape is not TMA-eligible.
inline bool encode_ztmap(CUtensorMap* m, const void* spec, const Dims& d, int cols, int real_bytes) {
  PFN_cuTensorMapEncodeTiled_v12000 enc = tensor_map_encoder();
  if (!enc || cols < 1 || (2 * cols * real_bytes) % 16 != 0 || ((uintptr_t)spec & 15) != 0) return false;
  const cuuint64_t es = (cuuint64_t)real_bytes;
  cuuint64_t dims[4] = {(cuuint64_t)(2 * d.P), (cuuint64_t)d.n2, (cuuint64_t)d.n3, 6};
  cuuint64_t strides[3] = {2 * (cuuint64_t)d.P * es, (cuuint64_t)d.n2 * 2 * d.P * es, (cuuint64_t)d.S * 2 * es};
  cuuint32_t box[4] = {(cuuint32_t)(2 * cols), 1, (cuuint32_t)std::min(d.n3, 256), 1};
  cuuint32_t estr[4] = {1, 1, 1, 1};
  const CUresult r = enc(m, real_bytes == 4 ? CU_TENSOR_MAP_DATA_TYPE_FLOAT32 : CU_TENSOR_MAP_DATA_TYPE_FLOAT64, 4,
                         const_cast<void*>(spec), dims, strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
                         (real_bytes == 4 && cz_swizzled(d.n3, cols)) ? CU_TENSOR_MAP_SWIZZLE_64B : CU_TENSOR_MAP_SWIZZLE_NONE,
                         CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
                         CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  return r == CUDA_SUCCESS;
}

// Recompute the thread counts and partial-sum count after a tile change.
inline void finalize_cfg(const Dims& d, LaunchCfg& c) {
  auto clampt = [](int t) { return std::min(512, std::max(64, round32(t))); };
  c.x_threads = clampt(3 * c.x_lines * d.n1 / 8);
  c.y_threads = clampt(c.y_cols * d.n2 / 8);
  c.z_threads = clampt(6 * c.z_cols * d.n3 / 8);
  c.z_blocks = ((d.n1h + c.z_cols - 1) / c.z_cols) * d.n2;
}

// Encode the tensor map of a launch configuration's z-tiles on `spec`, a grid's or a batch slot's spectrum; without one the pass
// takes the register-FFT kernel with ordinary loads, at a width that kernel has (FP32 tiles of 8 columns at 512 rows are
// the TMA-fed kernel's alone).
inline void attach_ztmap(LaunchCfg& lc, CUtensorMap* m, const void* spec, const Dims& d, bool mixed) {
  lc.ztmap = encode_ztmap(m, spec, d, lc.z_cols, mixed ? 4 : 8) ? m : nullptr;
  if (!lc.ztmap && mixed && d.n3 == 512 && lc.z_cols == 8) {
    lc.z_cols = 4;
    lc.z_tma = 0;
    finalize_cfg(d, lc);
  }
}

}  // namespace gfp
