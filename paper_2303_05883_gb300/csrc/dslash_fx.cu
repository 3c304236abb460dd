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
#define BRIDGE_FX_LAUNCH(FL, RD)                                                                                  \
  if (flags == (FL) && red == (RD)) {                                                                             \
    if (occ)                                                                                                       \
      return cudaOccupancyMaxActiveBlocksPerMultiprocessor(occ, hop_kernel_fx<(FL), (RD)>, FX_THREADS, 0) ==  \
             cudaSuccess;                                                                                          \
    hop_kernel_fx<(FL), (RD)><<<grid, FX_THREADS, 0, st>>>(a);                                           \
    return true;                                                                                                   \
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
// is not touched) of magnitude up to 2^e -> two limbs of each real times
// 2^(60 - e); *top receives the largest high word met.
__global__ void __launch_bounds__(256) k_to_fx(const char* src, char* dst, int nb, long n, long block_bytes, int e,
                                               uint32_t* top) {
  uint32_t m = 0;
  for (long k = (long)blockIdx.x * blockDim.x + threadIdx.x; k < nb * n; k += (long)gridDim.x * blockDim.x) {
    const long off = (k / n) * block_bytes + (k % n) * 16;
    const uint4 w = *reinterpret_cast<const uint4*>(src + off);
    m = max(m, max(w.y & 0x7fffffffu, w.w & 0x7fffffffu));
    // 2^e, exponent 1023 + e, becomes the integer 2^60; larger entries are refused by the caller
    const int E = 1023 + e;
    Fx2 r = fx_split(fx_from_bits<8>(w.x, w.y, max(E, (int)((w.y >> 20) & 0x7ffu)), 0));
    Fx2 i = fx_split(fx_from_bits<8>(w.z, w.w, max(E, (int)((w.w >> 20) & 0x7ffu)), 0));
    // the stencil negates limbs: keep the low one off -2^31 (by one unit, 2^(e - 60))
    r.l = max(r.l, -0x7fffffff);
    i.l = max(i.l, -0x7fffffff);
    *reinterpret_cast<uint4*>(dst + off) = make_uint4((uint32_t)r.l, (uint32_t)r.h, (uint32_t)i.l, (uint32_t)i.h);
  }
#pragma unroll
  for (int off = 16; off > 0; off >>= 1) m = max(m, __shfl_xor_sync(0xffffffffu, m, off));
  if ((threadIdx.x & 31) == 0) atomicMax(top, m);
}

void launch_to_fx(const char* src, char* dst, int nb, long n, long block_bytes, int e, uint32_t* top, cudaStream_t st) {
  const long grid = std::min<long>((nb * n + 255) / 256, 152L * 64);
  k_to_fx<<<(unsigned)grid, 256, 0, st>>>(src, dst, nb, n, block_bytes, e, top);
}

}  // namespace bridge
