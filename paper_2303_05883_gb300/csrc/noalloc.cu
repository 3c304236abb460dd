// bridge_mult_Dhat_noalloc: the Schur operator applied without allocating
// any device memory during the call.
//
// Some callers cannot call cudaMalloc when they apply the operator: a host
// application that reserves all device memory up front for its own pool and
// forbids allocations afterwards, or a latency-critical loop in which
// cudaMalloc / cudaFree (which can synchronize the whole device) are not
// allowed.  This entry point serves them.  Its scratch -- the input, the odd
// intermediate and the output in the GPU site layout -- lives in one
// file-scope device array of fixed size that every GPU loading the library
// holds until the process exits.
//
// The computation is the same as bridge_mult_Dhat_dev: canonical FP64 in ->
// GPU layout, pass 1 (tmp_o = T_oo^-1 (-kappa H_oe in_e)), pass 2
// (out_e = in_e + kappa T_ee^-1 H_eo tmp_o), GPU layout -> canonical FP64.
#include <algorithm>
#include <cstring>
#include <mutex>

#include "host.h"

using namespace bridge;

namespace bridge {
extern std::atomic<long> g_launches;
}

// 64 MiB of scratch per device (three half-lattice fields of the chosen
// precision and nrhs must fit; see BRIDGE_NOALLOC_SCRATCH_BYTES in bridge.h).
static __device__ __align__(256) char g_dhat_scratch[BRIDGE_NOALLOC_SCRATCH_BYTES];

namespace {

constexpr int kMaxDevices = 64;
std::mutex g_scratch_mu;
char* g_scratch_ptr[kMaxDevices] = {};

// Device address of the scratch array on the current device (looked up once
// per device; the host-side name of the array is not a device address).
char* scratch_on_current_device() {
  int dev = 0;
  BR_CUDA(cudaGetDevice(&dev));
  BR_CHECK(dev >= 0 && dev < kMaxDevices, BRIDGE_ECUDA, "device index out of range");
  std::lock_guard<std::mutex> lk(g_scratch_mu);
  if (!g_scratch_ptr[dev]) {
    void* p = nullptr;
    cudaError_t e = cudaGetSymbolAddress(&p, g_dhat_scratch);
    if (e != cudaSuccess) {
      cudaGetLastError();
      throw Error{BRIDGE_ECUDA, std::string("cudaGetSymbolAddress of the scratch array: ") + cudaGetErrorString(e)};
    }
    g_scratch_ptr[dev] = static_cast<char*>(p);
  }
  return g_scratch_ptr[dev];
}

// Launch shape of a hop without touching the lattice's shape table: the tuned
// entry if one exists, else what an untuned launch takes.
LaunchShape shape_readonly(bridge_lattice_s* L, int prec, int flags, const HopArgs& a) {
  const std::string key = "hop/" + std::to_string(prec) + "/" + std::to_string(flags) + "/0/" +
                          std::to_string(L->dims[0]) + "x" + std::to_string(L->dims[1]) + "x" +
                          std::to_string(L->dims[2]) + "x" + std::to_string(L->dims[3]) + "/" + std::to_string(a.nrhs);
  LaunchShape s;
  bool found = false;
  {
    std::lock_guard<std::mutex> lk(L->tune_mu);
    auto it = L->tuned.find(key);
    if (it != L->tuned.end()) {
      s = it->second;
      found = true;
    }
  }
  if (!found) s = default_hop_shape(prec, flags, R_NONE, a, false);
  const long cover = (L->vh + s.block - 1) / s.block;
  if (s.nblk <= 0 || s.nblk > cover) s.nblk = (int)cover;
  return s;
}

// The clover set of this lattice for kcsw, if its inverse in precision prec
// was built before; nullptr otherwise (nothing is built here).
std::shared_ptr<CloverSet> existing_clover(bridge_lattice_s* L, double kcsw, int prec) {
  std::lock_guard<std::mutex> lk(L->clover_mu);
  for (auto& s : L->clovers)
    if (s->kcsw == kcsw) {
      std::lock_guard<std::mutex> lk2(s->mu);
      return s->Tinv[prec] ? s : nullptr;
    }
  return nullptr;
}

}  // namespace

extern "C" int bridge_mult_Dhat_noalloc(bridge_lattice L, const bridge_op* op, int prec, const double* in_dev,
                                        double* out_dev, int nrhs) {
  try {
    BR_CHECK(L != nullptr && op != nullptr, BRIDGE_EINVAL, "NULL argument");
    BR_CHECK(prec >= BRIDGE_F64 && prec <= BRIDGE_BF16, BRIDGE_EINVAL, "precision");
    BR_CHECK(op->kind == BRIDGE_WILSON || op->kind == BRIDGE_CLOVER, BRIDGE_EINVAL, "op.kind");
    for (int k = 0; k < 4; ++k) BR_CHECK(op->bc[k] == 1 || op->bc[k] == -1, BRIDGE_EINVAL, "op.bc must be +1 or -1");
    BR_CHECK(nrhs >= 0, BRIDGE_EINVAL, "nrhs < 0");
    if (nrhs == 0) return BRIDGE_OK;
    BR_CHECK(in_dev != nullptr && out_dev != nullptr, BRIDGE_EINVAL, "in/out is NULL");
    const long block = spinor_block_bytes(prec, L->vh);
    const long need = 3L * nrhs * block;
    BR_CHECK(need <= (long)BRIDGE_NOALLOC_SCRATCH_BYTES, BRIDGE_EINVAL,
             "lattice too large for the no-allocation scratch: needs " + std::to_string(need) + " bytes, maximum " +
                 std::to_string((long)BRIDGE_NOALLOC_SCRATCH_BYTES));
    std::lock_guard<std::mutex> lk(L->api_mu);
    BR_CHECK(L->have_gauge && L->gauge[prec], BRIDGE_ESTATE,
             "links in this precision not built yet: apply the operator once with bridge_mult_Dhat first");
    const bool clov = op_is_clover(*op);
    std::shared_ptr<CloverSet> set;
    if (clov) {
      set = existing_clover(L, op_kcsw(*op), prec);
      BR_CHECK(set != nullptr, BRIDGE_ESTATE,
               "clover term for this kappa*c_sw and precision not built yet: apply the operator once first");
    }
    char* scratch = scratch_on_current_device();
    char* f_in = scratch;                    // even, nrhs blocks
    char* f_tmp = scratch + nrhs * block;    // odd
    char* f_out = scratch + 2 * nrhs * block;  // even
    cudaStream_t st = L->stream;

    CopyArgs ca;
    std::memset(&ca, 0, sizeof(ca));
    ca.vh = (uint32_t)L->vh;
    ca.nrhs = nrhs;
    ca.g = L->g;
    ca.V = L->V;
    ca.nblk = (int)((L->vh + 255) / 256);
    ca.canon = in_dev;
    ca.canon_full = 0;
    ca.dst = f_in;
    ca.dst_rs = block;
    BR_CHECK(launch_canon_to_field(prec, ca, st), BRIDGE_EINVAL, "precision");

    HopArgs a;
    std::memset(&a, 0, sizeof(a));
    a.g = L->g;
    a.nrhs = nrhs;
    for (int k = 0; k < 4; ++k) a.bc[k] = op->bc[k];
    a.gauge = L->gauge[prec]->ptr;
    a.clovE = set ? set->Tinv[prec]->ptr : nullptr;
    const FxCopies none;  // FP64: without copies and scratch, to the same bits
    // pass 1: tmp_o = T_oo^-1 (-kappa H_oe in_e)
    const int f1 = clov ? F_E_CLOV : 0;
    a.out_parity = 1;
    a.beta = -op->kappa;
    a.out = f_tmp;
    a.out_rs = block;
    a.in = f_in;
    a.in_rs = block;
    if (prec == P_F64) set_fx_args(L, a, f1, R_NONE, set.get(), &none, nullptr, st);
    const LaunchShape s1 = shape_readonly(L, prec, f1, a);
    a.nblk = s1.nblk;
    BR_CHECK(launch_hop_any(prec, f1, R_NONE, a, s1.block, st, nullptr, launch_variant(s1)), BRIDGE_EINVAL, "hop variant");
    // pass 2: out_e = in_e + kappa T_ee^-1 H_eo tmp_o
    const int f2 = F_SELF | (clov ? F_E_CLOV : 0);
    a.out_parity = 0;
    a.beta = op->kappa;
    a.s1 = 1.0;
    a.out = f_out;
    a.in = f_tmp;
    a.self = f_in;
    a.self_rs = block;
    if (prec == P_F64) set_fx_args(L, a, f2, R_NONE, set.get(), &none, nullptr, st);
    const LaunchShape s2 = shape_readonly(L, prec, f2, a);
    a.nblk = s2.nblk;
    BR_CHECK(launch_hop_any(prec, f2, R_NONE, a, s2.block, st, nullptr, launch_variant(s2)), BRIDGE_EINVAL, "hop variant");

    ca.canon = nullptr;
    ca.dst = nullptr;
    ca.canon_out = out_dev;
    ca.src = f_out;
    ca.src_rs = block;
    BR_CHECK(launch_field_to_canon(prec, ca, st), BRIDGE_EINVAL, "precision");
    BR_CUDA(cudaGetLastError());
    g_launches.fetch_add(4);
  } catch (const Error& e) {
    set_error(e.code, e.msg);
    return e.code;
  }
  return BRIDGE_OK;
}
