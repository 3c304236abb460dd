// Instantiations of the fixed-point FP64 stencil (dslash_fx.cuh) and the
// conversion of links and clover blocks to its 64-bit integers.
#include <algorithm>

#include "dslash_fx.cuh"
#include "kernels.h"

namespace bridge {

#define BRIDGE_FX_CASES(X)                                                                                         \
  X(0, R_NONE) X(F_E_CLOV, R_NONE) X(F_SELF, R_NONE) X(F_SELF, R_DOT_A) X(F_SELF, R_TS) X(F_SELF, R_NORM)         \
  X(F_SELF | F_E_CLOV, R_NONE) X(F_SELF | F_E_CLOV, R_DOT_A) X(F_SELF | F_E_CLOV, R_TS)                           \
  X(F_SELF | F_E_CLOV, R_NORM) X(F_SELF | F_SELF_CLOV, R_NONE) X(F_AUX | F_SELF, R_NORM)                          \
  X(F_AUX | F_SELF | F_SELF_CLOV, R_NORM) X(F_SELF | F_G5, R_NONE)

bool fx_has(int flags, int red) {
#define BRIDGE_FX_HAS(FL, RD) \
  if (flags == (FL) && red == (RD)) return true;
  BRIDGE_FX_CASES(BRIDGE_FX_HAS)
#undef BRIDGE_FX_HAS
  return false;
}

bool launch_hop_fx(int flags, int red, const HopArgs& args, int block, cudaStream_t st, int* occ) {
  // at most a block for every 64 sites (the reduction slots every caller
  // provides); a shape that covers the lattice at the caller's block size
  // covers it here too
  HopArgs a = args;
  const long cover = ((long)a.g.vh + FX_SITES - 1) / FX_SITES;
  a.nblk = (int)((long)a.nblk * block >= (long)a.g.vh ? cover : std::min<long>(a.nblk, cover));
  const dim3 grid((unsigned)(a.nblk * a.nrhs));
#define BRIDGE_FX_LAUNCH(FL, RD)                                                                                   \
  if (flags == (FL) && red == (RD)) {                                                                               \
    /* one grid for both kernels: the order of a reduction does not depend on which of them runs */                 \
    if (occ)                                                                                                        \
      return cudaOccupancyMaxActiveBlocksPerMultiprocessor(occ, hop_kernel_fx<(FL), (RD), false>, FX_THREADS, 0) == \
             cudaSuccess;                                                                                           \
    if (a.fx == FX_RAW)                                                                                             \
      hop_kernel_fx<(FL), (RD), true><<<grid, FX_THREADS, 0, st>>>(a);                                              \
    else                                                                                                            \
      hop_kernel_fx<(FL), (RD), false><<<grid, FX_THREADS, 0, st>>>(a);                                             \
    return true;                                                                                                    \
  }
  BRIDGE_FX_CASES(BRIDGE_FX_LAUNCH)
#undef BRIDGE_FX_LAUNCH
  return false;
}

// FP64 half-lattice field -> its fixed-point form (layout: fx_block_bytes).
__global__ void __launch_bounds__(256) k_field_to_fx(const CopyArgs a) {
  const int rhs = blockIdx.x % a.nrhs;
  if (rhs_finished(a.red, rhs)) return;
  for (uint32_t ih = (uint32_t)(blockIdx.x / a.nrhs) * blockDim.x + threadIdx.x; ih < a.vh;
       ih += (uint32_t)a.nblk * blockDim.x) {
    cx<double> s[12];
    load_spinor<P_F64>(a.src + rhs * a.src_rs, a.vh, ih, s);
    fx_store(a.dst + rhs * a.dst_rs, a.vh, ih, s);
  }
}

void launch_field_to_fx(const CopyArgs& a, int block, cudaStream_t st) {
  k_field_to_fx<<<(unsigned)(a.nblk * a.nrhs), block, 0, st>>>(a);
}

// nb blocks of n double2 entries (block_bytes apart; the padding between them
// is not touched) of magnitude up to 2^e -> two limbs of each real.
__global__ void __launch_bounds__(256) k_to_fx(const char* src, char* dst, int nb, long n, long block_bytes, int e) {
  for (long k = (long)blockIdx.x * blockDim.x + threadIdx.x; k < nb * n; k += (long)gridDim.x * blockDim.x) {
    const long off = (k / n) * block_bytes + (k % n) * 16;
    const uint4 w = *reinterpret_cast<const uint4*>(src + off);
    const Fx2 r = fx_limbs_of(w.x, w.y, 1023 + e), i = fx_limbs_of(w.z, w.w, 1023 + e);
    *reinterpret_cast<uint4*>(dst + off) = make_uint4((uint32_t)r.l, (uint32_t)r.h, (uint32_t)i.l, (uint32_t)i.h);
  }
}

void launch_to_fx(const char* src, char* dst, int nb, long n, long block_bytes, int e, cudaStream_t st) {
  const long grid = std::min<long>((nb * n + 255) / 256, 152L * 64);
  k_to_fx<<<(unsigned)grid, 256, 0, st>>>(src, dst, nb, n, block_bytes, e);
}

}  // namespace bridge
