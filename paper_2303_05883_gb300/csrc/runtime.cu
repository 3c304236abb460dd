// Host runtime: device buffers, fields, gauge and clover storage, operator
// application, launch statistics and launch shapes.
#include <algorithm>
#include <cmath>
#include <cstring>
#include <string>

#include "dslash_fx.cuh"
#include "host.h"

namespace bridge {

static thread_local std::string tl_last_error;
void set_error(int code, const std::string& msg) {
  (void)code;
  tl_last_error = msg;
}
const char* last_error_text() { return tl_last_error.c_str(); }

std::atomic<long> g_launches{0};
std::atomic<long> g_dev_allocs{0};

const char* kclass_name(int k) {
  static const char* names[K_NCLASS] = {"hop_deo",      "dirac_full",    "schur_pass1", "schur_pass2",
                                        "schur_pass2_alpha", "schur_pass2_omega", "evenodd_prep", "residual64",
                                        "blas_init",    "blas_s",        "blas_xr",     "blas_p",
                                        "convert",      "norm",          "clover_site", "setup",
                                        "dwf_mix",      "dwf_hop",       "dwf_schur_pass1", "dwf_schur_pass2",
                                        "dwf_schur_pass2_cg", "dwf_evenodd_prep", "dwf_residual64",
                                        "stag_hop",     "stag_pass1",    "stag_pass2",  "stag_vec",
                                        "stag_prep",    "stag_residual64",
                                        "mg_sap",       "mg_residual32", "mg_transfer", "mg_coarse",
                                        "mg_vec",       "mg_outer_dirac", "mg_setup"};
  return (k >= 0 && k < K_NCLASS) ? names[k] : "?";
}

// Keep freed stream-ordered memory in the pool (no release back to the
// driver between solves), once per device.
static void retain_pool_memory() {
  static std::mutex mu;
  static bool done[64] = {};
  int dev = 0;
  cudaGetDevice(&dev);
  std::lock_guard<std::mutex> lk(mu);
  if (dev < 0 || dev >= 64 || done[dev]) return;
  cudaMemPool_t pool;
  if (cudaDeviceGetDefaultMemPool(&pool, dev) == cudaSuccess) {
    uint64_t thr = ~0ull;
    cudaMemPoolSetAttribute(pool, cudaMemPoolAttrReleaseThreshold, &thr);
  }
  cudaGetLastError();
  done[dev] = true;
}

DevBuf::DevBuf(size_t n, cudaStream_t stream, bool stream_ordered) : st(stream), async(stream_ordered) {
  if (n == 0) return;
  cudaError_t e;
  if (async) {
    retain_pool_memory();
    e = cudaMallocAsync(reinterpret_cast<void**>(&ptr), n, st);
  } else {
    e = cudaMalloc(reinterpret_cast<void**>(&ptr), n);
  }
  if (e != cudaSuccess) {
    cudaGetLastError();
    ptr = nullptr;
    throw Error{BRIDGE_ENOMEM, "device allocation of " + std::to_string(n) + " bytes failed: " + cudaGetErrorString(e)};
  }
  bytes = n;
  g_dev_allocs.fetch_add(1);
}
DevBuf::~DevBuf() {
  if (!ptr) return;
  if (async)
    cudaFreeAsync(ptr, st);
  else
    cudaFree(ptr);
}

Field make_field(int prec, int subset, int nrhs, long vh, cudaStream_t st, bool stream_ordered, size_t at_least) {
  Field f;
  f.prec = prec;
  f.subset = subset;
  f.nrhs = nrhs;
  f.vh = vh;
  f.block = spinor_block_bytes(prec, vh);
  f.rs = (subset == BRIDGE_FULL ? 2 : 1) * f.block;
  f.buf = std::make_shared<DevBuf>(std::max((size_t)(f.rs * (nrhs > 0 ? nrhs : 1)), at_least), st, stream_ordered);
  return f;
}

int sm_count() {
  static int n = 0;
  if (n == 0) {
    int dev = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev);
    if (n <= 0) n = 1;
  }
  return n;
}

// ----------------------------------------------------------- statistics
void note_launch(bridge_lattice_s* L, int cls, double bytes, double flops, cudaStream_t st, bool begin) {
  Stats& S = L->stats;
  std::lock_guard<std::mutex> lk(S.mu);
  if (begin) {
    g_launches.fetch_add(1);
    S.k[cls].launches += 1;
    S.k[cls].bytes += bytes;
    S.k[cls].flops += flops;
    if (S.profiling) {
      Stats::Rec r;
      r.cls = cls;
      if (S.pool.size() < 2) {
        cudaEvent_t e;
        for (int i = 0; i < 64; ++i) {
          cudaEventCreate(&e);
          S.pool.push_back(e);
        }
      }
      r.a = S.pool.back();
      S.pool.pop_back();
      r.b = S.pool.back();
      S.pool.pop_back();
      cudaEventRecord(r.a, st);
      S.recs.push_back(r);
    }
  } else if (S.profiling && !S.recs.empty()) {
    cudaEventRecord(S.recs.back().b, st);
  }
}

static LaunchShape default_shape(int nrhs, const std::function<int(int)>& occ, int variant, bool cover_once) {
  LaunchShape s;
  s.variant = variant;
  s.block = variant == 4 && !cover_once ? 256 : 128;
  const int per_sm = occ ? occ(s.block) : 0;
  const long resident = (long)sm_count() * (per_sm > 0 ? per_sm : 4);
  const int groups = (nrhs + hop_variant_rpt(variant) - 1) / hop_variant_rpt(variant);
  s.nblk = variant == 4 && cover_once ? 0 : (int)std::max<long>(1, resident / std::max(1, groups));
  return s;
}

LaunchShape shape_for(bridge_lattice_s* L, const std::string& key, long vh, int nrhs,
                      const std::function<int(int)>& occ, int variant, bool cover_once) {
  std::lock_guard<std::mutex> lk(L->tune_mu);
  LaunchShape s;
  auto it = L->tuned.find(key);
  if (it != L->tuned.end()) {
    s = it->second;
  } else {
    s = default_shape(nrhs, occ, variant, cover_once);
    L->tuned[key] = s;
  }
  const long cover = (vh + s.block - 1) / s.block;
  if (s.nblk <= 0 || s.nblk > cover) s.nblk = (int)cover;
  return s;
}

void ensure_red_scratch(bridge_lattice_s* L, long n_partials, int nrhs) {
  size_t need = (size_t)n_partials * 4 * sizeof(double);
  if (!L->red_partials || L->red_partials->bytes < need) L->red_partials.reset(new DevBuf(need));
  size_t rneed = (size_t)(nrhs > 0 ? nrhs : 1) * 4 * sizeof(double);
  if (!L->red_result || L->red_result->bytes < rneed) L->red_result.reset(new DevBuf(rneed < 4096 ? 4096 : rneed));
  if (!L->red_counter) {
    L->red_counter.reset(new DevBuf(256));
    BR_CUDA(cudaMemsetAsync(L->red_counter->ptr, 0, 256, L->stream));
  }
}

// ------------------------------------------------------- gauge / clover
bool op_is_clover(const bridge_op& op) { return op.kind == BRIDGE_CLOVER && op.csw != 0.0 && op.kappa != 0.0; }
double op_kcsw(const bridge_op& op) { return op_is_clover(op) ? op.kappa * op.csw : 0.0; }

const char* gauge_ptr(bridge_lattice_s* L, int prec) {
  BR_CHECK(L->have_gauge, BRIDGE_ESTATE, "no gauge field uploaded");
  if (!L->gauge[prec]) {
    L->gauge[prec].reset(new DevBuf((size_t)(8 * link_block_bytes(prec, L->vh))));
    note_launch(L, K_SETUP, 0, 0, L->stream, true);
    BR_CHECK(launch_gauge_convert(prec, L->g, L->gauge[P_F64]->ptr, L->gauge[prec]->ptr, L->stream), BRIDGE_EINVAL,
             "gauge precision");
    note_launch(L, K_SETUP, 0, 0, L->stream, false);
    BR_CUDA(cudaGetLastError());
  }
  return L->gauge[prec]->ptr;
}

std::shared_ptr<CloverSet> clover_set(bridge_lattice_s* L, double kcsw) {
  BR_CHECK(L->have_gauge, BRIDGE_ESTATE, "no gauge field uploaded");
  std::lock_guard<std::mutex> lk(L->clover_mu);
  for (size_t i = 0; i < L->clovers.size(); ++i) {
    if (L->clovers[i]->kcsw == kcsw) {
      auto s = L->clovers[i];
      L->clovers.erase(L->clovers.begin() + i);
      L->clovers.insert(L->clovers.begin(), s);
      return s;
    }
  }
  auto s = std::make_shared<CloverSet>();
  s->kcsw = kcsw;
  const size_t n = (size_t)(2 * clover_block_bytes(P_F64, L->vh));
  s->T[P_F64].reset(new DevBuf(n + 256));  // (behind T: the largest entries met)
  s->Tinv[P_F64].reset(new DevBuf(n));
  uint32_t* top = reinterpret_cast<uint32_t*>(s->T[P_F64]->ptr + n);
  BR_CUDA(cudaMemsetAsync(top, 0, sizeof(s->top), L->stream));
  note_launch(L, K_SETUP, 0, 0, L->stream, true);
  launch_clover_build(L->g, L->gauge[P_F64]->ptr, kcsw, s->T[P_F64]->ptr, s->Tinv[P_F64]->ptr, top, L->stream);
  note_launch(L, K_SETUP, 0, 0, L->stream, false);
  BR_CUDA(cudaGetLastError());
  BR_CUDA(cudaMemcpyAsync(s->top, top, sizeof(s->top), cudaMemcpyDeviceToHost, L->stream));
  BR_CUDA(cudaStreamSynchronize(L->stream));
  L->clovers.insert(L->clovers.begin(), s);
  const size_t keep = 4;  // sets still used by a solve stay alive through its reference
  if (L->clovers.size() > keep) L->clovers.resize(keep);
  return s;
}

const char* clover_ptr(bridge_lattice_s* L, CloverSet& set, int prec, bool inverse) {
  std::lock_guard<std::mutex> lk(set.mu);
  std::unique_ptr<DevBuf>* arr = inverse ? set.Tinv : set.T;
  if (!arr[prec]) {
    arr[prec].reset(new DevBuf((size_t)(2 * clover_block_bytes(prec, L->vh))));
    note_launch(L, K_SETUP, 0, 0, L->stream, true);
    BR_CHECK(launch_clover_convert(prec, L->g, arr[P_F64]->ptr, arr[prec]->ptr, L->stream), BRIDGE_EINVAL,
             "clover precision");
    note_launch(L, K_SETUP, 0, 0, L->stream, false);
    BR_CUDA(cudaGetLastError());
  }
  return arr[prec]->ptr;
}

const char* clover_ptr(bridge_lattice_s* L, int prec, bool inverse, double kcsw) {
  auto s = clover_set(L, kcsw);
  return clover_ptr(L, *s, prec, inverse);
}

static bool capturing(cudaStream_t st) {
  cudaStreamCaptureStatus cap = cudaStreamCaptureStatusNone;
  const bool known = cudaStreamIsCapturing(st, &cap) == cudaSuccess;
  if (!known) cudaGetLastError();
  return !known || cap != cudaStreamCaptureStatusNone;
}

bool fx_fits(bridge_lattice_s* L, const CloverSet* set, int flags, int* eE, int* eM) {
  const int m = set ? fx_clov_exponent(set->top[0]) : 0, e = set ? fx_clov_exponent(set->top[1]) : 0;
  if (eM) *eM = m;
  if (eE) *eE = e;
  return L->gauge_top < FX_LINK_TOP && (!(flags & F_SELF_CLOV) || m) && (!(flags & F_E_CLOV) || e);
}

// Whether `bytes` may go to data that only makes things faster: at most an
// eighth of what is free, to leave the memory to the fields of a solve (up to
// 4 KB a site, seven link copies) where it is scarce.  What the library's pool
// holds unused is free.
static bool fx_room(size_t bytes, size_t keep_free) {
  int dev = 0;
  cudaMemPool_t pool;
  uint64_t held = 0, used = 0;
  if (cudaGetDevice(&dev) == cudaSuccess && cudaDeviceGetDefaultMemPool(&pool, dev) == cudaSuccess) {
    cudaMemPoolGetAttribute(pool, cudaMemPoolAttrReservedMemCurrent, &held);
    cudaMemPoolGetAttribute(pool, cudaMemPoolAttrUsedMemCurrent, &used);
  }
  cudaGetLastError();
  const size_t idle = held > used ? (size_t)(held - used) : 0;
  if (bytes <= idle / 8 && bytes + keep_free <= idle) return true;
  size_t free_b = 0, total_b = 0;
  BR_CUDA(cudaMemGetInfo(&free_b, &total_b));
  return bytes <= (free_b + idle) / 8 && bytes + keep_free <= free_b + idle;
}

// A buffer, from the pool in the order of the lattice stream if pooled, or null.
static std::unique_ptr<DevBuf> fx_buffer(bridge_lattice_s* L, size_t bytes, bool pooled, size_t keep_free = 0) {
  if (!fx_room(bytes, keep_free)) return nullptr;
  try {
    return std::unique_ptr<DevBuf>(new DevBuf(bytes, L->stream, pooled));
  } catch (const Error&) {
    return nullptr;
  }
}

// The copy is made on the lattice stream, which orders it after the FP64 data.
static void fx_convert(bridge_lattice_s* L, const char* src, char* dst, int nb, long block_bytes, long n, int e) {
  const double bytes = 2.0 * nb * block_bytes;
  note_launch(L, K_SETUP, bytes, 0, L->stream, true);
  launch_to_fx(src, dst, nb, n, block_bytes, e, L->stream);
  note_launch(L, K_SETUP, bytes, 0, L->stream, false);
  BR_CUDA(cudaGetLastError());
}

// (A clover set may outlive the stream of its lattice: its copies are not of
// the pool.)
static const char* fx_clover(bridge_lattice_s* L, CloverSet& set, bool inverse, size_t keep_free) {
  std::unique_ptr<DevBuf>& buf = set.fx[inverse];
  if (!buf) {
    const long cbb = clover_block_bytes(P_F64, L->vh);
    auto to = fx_buffer(L, (size_t)(2 * cbb), false, keep_free);
    if (!to) return nullptr;
    fx_convert(L, (inverse ? set.Tinv : set.T)[P_F64]->ptr, to->ptr, 2, cbb, 36 * L->vh, fx_clov_exponent(set.top[inverse]));
    buf = std::move(to);
  }
  return buf->ptr;
}

FxCopies fx_copies(bridge_lattice_s* L, CloverSet* set, int flags, size_t keep_free) {
  FxCopies c;
  if (capturing(L->stream)) return c;
  {
    std::lock_guard<std::mutex> lk(L->fx_mu);
    const long lbb = link_block_bytes(P_F64, L->vh);
    if (!L->gauge_fx) L->gauge_fx = fx_buffer(L, (size_t)(8 * lbb), true, keep_free);
    if (L->gauge_fx && !L->gauge_fx_made) {
      fx_convert(L, L->gauge[P_F64]->ptr, L->gauge_fx->ptr, 8, lbb, 9 * L->vh, 0);
      L->gauge_fx_made = true;
    }
    if (L->gauge_fx_made) c.U = L->gauge_fx->ptr;
  }
  if (!c.U || !(flags & (F_E_CLOV | F_SELF_CLOV))) return c;
  std::lock_guard<std::mutex> lk(set->mu);
  if (flags & F_SELF_CLOV) c.M = fx_clover(L, *set, false, keep_free);
  if (flags & F_E_CLOV) c.E = fx_clover(L, *set, true, keep_free);
  return c;
}

bool fx_release(bridge_lattice_s* L) {
  // (a stream in a capture cannot be waited for)
  if (L->in_flight.load() != 0 || capturing(L->stream)) return false;
  BR_CUDA(cudaStreamSynchronize(L->stream));
  bool any = L->fx_scratch || L->gauge_fx;
  L->fx_scratch.reset();
  {
    std::lock_guard<std::mutex> lk(L->fx_mu);
    L->gauge_fx.reset();
    L->gauge_fx_made = false;
  }
  std::lock_guard<std::mutex> lk(L->clover_mu);
  for (auto& s : L->clovers) {
    std::lock_guard<std::mutex> ls(s->mu);
    for (auto& b : s->fx) {
      any = any || b;
      b.reset();
    }
  }
  BR_CUDA(cudaStreamSynchronize(L->stream));
  return any;
}

char* fx_scratch(bridge_lattice_s* L, size_t need) {
  if (capturing(L->stream)) return nullptr;
  if (!L->fx_scratch || L->fx_scratch->bytes < need) {
    auto grown = fx_buffer(L, need, true);
    if (!grown) return nullptr;
    L->fx_scratch = std::move(grown);
  }
  return L->fx_scratch->ptr;
}

void set_fx_args(bridge_lattice_s* L, HopArgs& a, int flags, int red, CloverSet* set, const FxCopies* copies,
                 char* scratch, cudaStream_t st) {
  a.fx = FX_OFF;
  if (!fx_has(flags, red) || !fx_fits(L, set, flags, &a.eE_fx, &a.eM_fx)) return;
  a.eb_fx = a.beta != 0.0 && std::isfinite(a.beta) ? std::ilogb(a.beta) : -5000;
  a.fx = FX_RAW;
  const FxCopies c = copies ? *copies : st == L->stream ? fx_copies(L, set, flags) : FxCopies{};
  if (!c.U || ((flags & F_E_CLOV) && !c.E) || ((flags & F_SELF_CLOV) && !c.M)) return;
  if (!a.in_fx) {
    if (!scratch && st == L->stream) scratch = fx_scratch(L, (size_t)a.nrhs * fx_block_bytes(L->vh));
    if (!scratch) return;
    CopyArgs v;
    std::memset(&v, 0, sizeof(v));
    v.vh = (uint32_t)L->vh;
    v.nrhs = a.nrhs;
    v.nblk = (int)((L->vh + 255) / 256);
    v.src = a.in;
    v.src_rs = a.in_rs;
    v.dst = scratch;
    v.dst_rs = fx_block_bytes(L->vh);
    v.red = a.red;  // right-hand sides whose solve has ended are skipped
    const double bytes = (double)L->vh * a.nrhs * (192 + 196);
    note_launch(L, K_CONVERT, bytes, 0, st, true);
    launch_field_to_fx(v, 256, st);
    note_launch(L, K_CONVERT, bytes, 0, st, false);
    a.in_fx = scratch;
    a.in_fx_rs = v.dst_rs;
  }
  a.fx = FX_COPIES;
  a.gauge_fx = c.U;
  a.clovE_fx = c.E;
  a.clovM_fx = c.M;
}

// ------------------------------------------------------------ operators
static long spinor_site_bytes(int prec) { return prec == P_F64 ? 192 : prec == P_F32 ? 96 : 52; }
static long link_site_bytes(int prec) { return prec == P_F64 ? 144 : prec == P_F32 ? 48 : 24; }
static long clover_site_bytes(int prec) { return prec == P_F64 ? 576 : prec == P_F32 ? 288 : 144; }

HopCost hop_cost(int prec, int flags, int red) {
  const double S = (double)spinor_site_bytes(prec);
  double per_rhs = 2 * S;  // one input read, one output written
  if (flags & F_SELF) per_rhs += S;
  if (flags & F_AUX) per_rhs += S;
  if (red == R_DOT_A) per_rhs += S;
  double shared = 8.0 * link_site_bytes(prec);
  if (flags & F_E_CLOV) shared += clover_site_bytes(prec);
  if (flags & F_SELF_CLOV) shared += clover_site_bytes(prec);
  double fl = 1320 + 24;  // hop (8 projected hops) and the scale by beta
  if (flags & F_E_CLOV) fl += 504;
  if (flags & F_SELF_CLOV) fl += 504;
  if (flags & F_SELF) fl += 48;
  if (flags & F_AUX) fl += 48;
  if (red != R_NONE) fl += 48;
  return HopCost{per_rhs, shared, fl};
}

static int default_hop_variant(int prec, int flags, int red, long vh, int nrhs, bool mapped);

static std::string dims_key(const bridge_lattice_s* L) {
  return std::to_string(L->dims[0]) + "x" + std::to_string(L->dims[1]) + "x" + std::to_string(L->dims[2]) + "x" +
         std::to_string(L->dims[3]);
}

// Resident blocks per SM of an untuned launch, by its block size.
static std::function<int(int)> hop_occupancy(int prec, int flags, int red, const HopArgs& a, int variant) {
  return [=, &a](int block) {
    int n = 0;
    launch_hop_any(prec, flags, red, a, block, nullptr, &n, variant + (variant == 9 || variant == 10 ? HOP_TILE_WIDE : 0));
    return n;
  };
}

LaunchShape default_hop_shape(int prec, int flags, int red, const HopArgs& a, bool mapped) {
  const int variant = default_hop_variant(prec, flags, red, a.g.vh, a.nrhs, mapped);
  return default_shape(a.nrhs, hop_occupancy(prec, flags, red, a, variant), variant, red == R_NONE);
}

void run_hop(bridge_lattice_s* L, HopCall c, cudaStream_t st) {
  HopArgs a;
  std::memset(&a, 0, sizeof(a));
  a.g = L->g;
  a.out_parity = c.out_parity;
  a.nrhs = c.nrhs;
  a.beta = c.beta;
  a.s1 = c.s1;
  a.caux = c.caux;
  for (int k = 0; k < 4; ++k) a.bc[k] = (double)c.bc[k];
  a.out = c.out;
  a.out_rs = c.out_rs;
  a.in = c.in;
  a.in_rs = c.in_rs;
  a.self = c.self;
  a.self_rs = c.self_rs;
  a.aux = c.aux;
  a.aux_rs = c.aux_rs;
  a.avec = c.avec;
  a.avec_rs = c.avec_rs;
  a.gauge = gauge_ptr(L, c.prec);
  std::shared_ptr<CloverSet> keep;
  CloverSet* cs = c.clov;
  if (c.flags & (F_E_CLOV | F_SELF_CLOV)) {
    if (!cs) {
      keep = clover_set(L, c.kcsw);
      cs = keep.get();
    }
    a.clovE = (c.flags & F_E_CLOV) ? clover_ptr(L, *cs, c.prec, true) : nullptr;
    a.clovM = (c.flags & F_SELF_CLOV) ? clover_ptr(L, *cs, c.prec, false) : nullptr;
  }
  a.red = c.redargs;
  a.in_fx = c.in_fx;
  a.in_fx_rs = c.in_fx_rs;
  if (c.prec == P_F64 && !c.site_map) set_fx_args(L, a, c.flags, c.red, cs, c.fx, c.fx_scratch, st);
  const std::string key = "hop/" + std::to_string(c.prec) + "/" + std::to_string(c.flags) + "/" +
                          std::to_string(c.red) + "/" + dims_key(L) + "/" + std::to_string(c.nrhs);
  const int variant = default_hop_variant(c.prec, c.flags, c.red, L->vh, c.nrhs, c.site_map != nullptr);
  LaunchShape sh = shape_for(L, key, L->vh, c.nrhs, hop_occupancy(c.prec, c.flags, c.red, a, variant), variant,
                             c.red == R_NONE);
  a.nblk = sh.nblk;
  if (c.red != R_NONE && a.red.partials == nullptr) {
    // a fixed-point launch takes up to one block for 64 sites
    const long nb = a.fx != FX_OFF ? std::max<long>(sh.nblk, (L->vh + 63) / 64) : sh.nblk;
    ensure_red_scratch(L, nb * c.nrhs, c.nrhs);
    a.red.partials = reinterpret_cast<double*>(L->red_partials->ptr);
    a.red.counter = reinterpret_cast<unsigned*>(L->red_counter->ptr);
    a.red.result = reinterpret_cast<double*>(L->red_result->ptr);
    if (a.red.fin == FIN_NONE) a.red.fin = FIN_STORE;
  }
  const HopCost hc = hop_cost(c.prec, c.flags, c.red);
  a.site_map = c.site_map;
  a.n_map = c.n_map;
  const double bytes =
      c.count_work ? c.work_fraction * (double)L->vh * (hc.rhs_bytes * c.nrhs + hc.shared_bytes) : 0.0;
  const double flops = c.count_work ? c.work_fraction * (double)L->vh * c.nrhs * hc.rhs_flops : 0.0;
  note_launch(L, c.cls, bytes, flops, st, true);
  BR_CHECK(launch_hop_any(c.prec, c.flags, c.red, a, sh.block, st, nullptr, launch_variant(sh)), BRIDGE_EINVAL,
           "hop variant not instantiated");
  note_launch(L, c.cls, bytes, flops, st, false);
  BR_CUDA(cudaGetLastError());
}

char* fx_input(bridge_lattice_s* L, const bridge_op& op, int which, int nblocks) {
  std::shared_ptr<CloverSet> set;
  int flags = 0;
  if (op_is_clover(op) && (which == BRIDGE_APPLY_D || which == BRIDGE_APPLY_DHAT)) {
    set = clover_set(L, op_kcsw(op));
    flags = which == BRIDGE_APPLY_D ? F_SELF_CLOV : F_E_CLOV;
  }
  if (!fx_fits(L, set.get(), flags)) return nullptr;
  const FxCopies c = fx_copies(L, set.get(), flags);
  if (!c.U || ((flags & F_E_CLOV) && !c.E) || ((flags & F_SELF_CLOV) && !c.M)) return nullptr;
  return fx_scratch(L, (size_t)nblocks * fx_block_bytes(L->vh));
}

void apply_deo(bridge_lattice_s* L, const bridge_op& op, int q, const Field& out, const Field& in, cudaStream_t st) {
  HopCall c;
  c.prec = in.prec;
  c.flags = 0;
  c.cls = K_HOP;
  c.out_parity = q;
  c.nrhs = in.nrhs;
  c.beta = -op.kappa;
  for (int k = 0; k < 4; ++k) c.bc[k] = op.bc[k];
  c.out = out.ptr(q);
  c.out_rs = out.rs;
  c.in = in.ptr(1 - q);
  c.in_rs = in.rs;
  c.in_fx = in.fx_ptr(1 - q);
  c.in_fx_rs = in.fx_rs();
  run_hop(L, c, st);
}

void apply_d(bridge_lattice_s* L, const bridge_op& op, const Field& out, const Field& in, cudaStream_t st) {
  const bool clov = op_is_clover(op);
  for (int q = 0; q < 2; ++q) {
    HopCall c;
    c.prec = in.prec;
    c.flags = F_SELF | (clov ? F_SELF_CLOV : 0);
    c.cls = K_FULLD;
    c.out_parity = q;
    c.nrhs = in.nrhs;
    c.beta = -op.kappa;
    c.s1 = 1.0;
    c.kcsw = op_kcsw(op);
    for (int k = 0; k < 4; ++k) c.bc[k] = op.bc[k];
    c.out = out.ptr(q);
    c.out_rs = out.rs;
    c.in = in.ptr(1 - q);
    c.in_rs = in.rs;
    c.in_fx = in.fx_ptr(1 - q);
    c.in_fx_rs = in.fx_rs();
    c.self = in.ptr(q);
    c.self_rs = in.rs;
    run_hop(L, c, st);
  }
}

void apply_dhat(bridge_lattice_s* L, const bridge_op& op, const Field& out, const Field& in, const Field& tmp,
                cudaStream_t st) {
  const bool clov = op_is_clover(op);
  HopCall c;
  c.prec = in.prec;
  c.nrhs = in.nrhs;
  c.kcsw = op_kcsw(op);
  for (int k = 0; k < 4; ++k) c.bc[k] = op.bc[k];
  // pass 1: tmp_o = T_oo^-1 (-kappa H_oe in_e)
  c.flags = clov ? F_E_CLOV : 0;
  c.cls = K_DHAT1;
  c.out_parity = 1;
  c.beta = -op.kappa;
  c.out = tmp.ptr(1);
  c.out_rs = tmp.rs;
  c.in = in.ptr(0);
  c.in_rs = in.rs;
  c.in_fx = in.fx_ptr(0);
  c.in_fx_rs = in.fx_rs();
  run_hop(L, c, st);
  c.in_fx = nullptr;
  // pass 2: out_e = in_e - T_ee^-1 (-kappa H_eo tmp_o)
  c.flags = F_SELF | (clov ? F_E_CLOV : 0);
  c.cls = K_DHAT2;
  c.out_parity = 0;
  c.beta = op.kappa;
  c.s1 = 1.0;
  c.out = out.ptr(0);
  c.out_rs = out.rs;
  c.in = tmp.ptr(1);
  c.in_rs = tmp.rs;
  c.self = in.ptr(0);
  c.self_rs = in.rs;
  run_hop(L, c, st);
}

// ------------------------------------------------------------ layouts
static CopyArgs copy_args(bridge_lattice_s* L, const Field& f) {
  CopyArgs a;
  std::memset(&a, 0, sizeof(a));
  a.vh = (uint32_t)L->vh;
  a.nrhs = f.nrhs;
  a.g = L->g;
  a.V = L->V;
  const int block = 256;
  a.nblk = (int)((L->vh + block - 1) / block);
  return a;
}

void canon_to_field(bridge_lattice_s* L, const double* canon, const Field& f, cudaStream_t st, const int* mask,
                    long canon_rs) {
  CopyArgs a = copy_args(L, f);
  a.canon = canon;
  a.canon_rs = canon_rs / 2;
  a.canon_full = f.subset == BRIDGE_FULL;
  a.dst = f.ptr(a.canon_full ? 0 : f.subset);
  if (a.canon_full) a.dst2 = f.ptr(1);
  a.dst_rs = f.rs;
  a.fx = f.fx;
  a.fx2 = f.fx ? f.fx_ptr(1) : nullptr;
  a.fx_rs = f.fx_rs();
  a.mask = mask;
  const double sites = (double)(a.canon_full ? L->V : L->vh) * f.nrhs;
  const double bytes = sites * (192 + spinor_site_bytes(f.prec) + (f.fx ? 196 : 0));
  note_launch(L, K_CONVERT, bytes, 0, st, true);
  launch_canon_to_field(f.prec, a, st);
  note_launch(L, K_CONVERT, bytes, 0, st, false);
  BR_CUDA(cudaGetLastError());
}

void field_to_canon(bridge_lattice_s* L, const Field& f, double* canon, cudaStream_t st, long canon_rs) {
  CopyArgs a = copy_args(L, f);
  a.canon_out = canon;
  a.canon_rs = canon_rs / 2;
  a.canon_full = f.subset == BRIDGE_FULL;
  a.src = f.ptr(a.canon_full ? 0 : f.subset);
  if (a.canon_full) a.src2 = f.ptr(1);
  a.src_rs = f.rs;
  const double bytes = (double)(a.canon_full ? L->V : L->vh) * f.nrhs * (192 + spinor_site_bytes(f.prec));
  note_launch(L, K_CONVERT, bytes, 0, st, true);
  launch_field_to_canon(f.prec, a, st);
  note_launch(L, K_CONVERT, bytes, 0, st, false);
  BR_CUDA(cudaGetLastError());
}

void convert_field(bridge_lattice_s* L, const Field& src, const Field& dst, int parity, cudaStream_t st, const int* mask) {
  CopyArgs a = copy_args(L, src);
  a.src = src.ptr(parity);
  a.src_rs = src.rs;
  a.dst = dst.ptr(parity);
  a.dst_rs = dst.rs;
  a.mask = mask;
  const double bytes = (double)L->vh * src.nrhs * (spinor_site_bytes(src.prec) + spinor_site_bytes(dst.prec));
  note_launch(L, K_CONVERT, bytes, 0, st, true);
  launch_convert(src.prec, dst.prec, a, 256, st);
  note_launch(L, K_CONVERT, bytes, 0, st, false);
  BR_CUDA(cudaGetLastError());
}

void accumulate64(bridge_lattice_s* L, const Field& src, int sp, const Field& dst, int dp, cudaStream_t st,
                  const int* mask) {
  CopyArgs a = copy_args(L, src);
  a.src = src.ptr(sp);
  a.src_rs = src.rs;
  a.dst = dst.ptr(dp);
  a.dst_rs = dst.rs;
  a.mask = mask;
  const double bytes = (double)L->vh * src.nrhs * (spinor_site_bytes(src.prec) + 2 * 192);
  note_launch(L, K_CONVERT, bytes, (double)L->vh * src.nrhs * 24, st, true);
  launch_accumulate64(src.prec, a, 256, st);
  note_launch(L, K_CONVERT, bytes, 0, st, false);
  BR_CUDA(cudaGetLastError());
}

void norm2_field(bridge_lattice_s* L, const Field& f, int parity, RedArgs red, cudaStream_t st) {
  CopyArgs a = copy_args(L, f);
  a.src = f.ptr(parity);
  a.src_rs = f.rs;
  a.red = red;
  a.nblk = std::max(1, std::min(a.nblk, sm_count() * 8 / std::max(1, f.nrhs)));
  const double bytes = (double)L->vh * f.nrhs * spinor_site_bytes(f.prec);
  note_launch(L, K_NORM, bytes, (double)L->vh * f.nrhs * 48, st, true);
  launch_norm2(f.prec, a, 256, st);
  note_launch(L, K_NORM, bytes, 0, st, false);
  BR_CUDA(cudaGetLastError());
}

void clover_site(bridge_lattice_s* L, int prec, bool inverse, double kcsw, int parity, const Field& src, int sp,
                 const Field& dst, int dp, int nrhs, cudaStream_t st, CloverSet* set) {
  const char* cl = (set ? clover_ptr(L, *set, prec, inverse) : clover_ptr(L, prec, inverse, kcsw)) +
                   (long)parity * clover_block_bytes(prec, L->vh);
  CopyArgs a = copy_args(L, src);
  a.nrhs = nrhs;
  a.src = src.ptr(sp);
  a.src_rs = src.rs;
  a.dst = dst.ptr(dp);
  a.dst_rs = dst.rs;
  const double bytes = (double)L->vh * (nrhs * 2.0 * spinor_site_bytes(prec) + clover_site_bytes(prec));
  note_launch(L, K_CLOVER, bytes, (double)L->vh * nrhs * 504, st, true);
  launch_clover_site(prec, a, cl, 256, st);
  note_launch(L, K_CLOVER, bytes, 0, st, false);
  BR_CUDA(cudaGetLastError());
}

bool hop_has_variant(int prec, int flags, int red, int variant) {
#define BRIDGE_HOP_IS(FL, RD) || (flags == (FL) && red == (RD))
  const bool budget = false BRIDGE_HOP_BUDGET_CASES(BRIDGE_HOP_IS), apply = false BRIDGE_HOP_APPLY_CASES(BRIDGE_HOP_IS);
  const bool shared = false BRIDGE_HOP_SHARED_CASES(BRIDGE_HOP_IS), tile = false BRIDGE_HOP_TILE_CASES(BRIDGE_HOP_IS);
#undef BRIDGE_HOP_IS
  if (variant == 0) return true;
  if (prec == P_F64) return variant < 6 && budget;
  if (variant < 6) return budget || (variant == 4 && apply);
  if (variant < 9) return shared;
  if (variant < 11) return shared || tile;
  return shared && (prec == P_F16 || prec == P_BF16);
}

// The variant an untuned launch takes, by its working set (microseconds on a
// GB300, default persistent shape of variant 0 -> the variant; Schur pass 1 /
// pass 2 with a dot product):
//   * from 4 right-hand sides on 2^18 half-lattice sites, or 6 on 2^16, the
//     tile kernel, which loads, widens and scales each link and clover block
//     once for all of them: 24^3 x 48 F32 4 RHS 123 -> 113 / 189 -> 163, 12
//     RHS 332 -> 283 / 525 -> 388, F16 12 RHS 347 -> 246 / 424 -> 330 (variants 9
//     and 10; rounding as variant 0, as untuned launches do, four D^ on 12 RHS in
//     F16 take 2.9 ms with their conversions instead of 3.8); 16^3 x 32 6 RHS 39 -> 38 / 72 -> 68, but 4 RHS 27 -> 29 /
//     51 -> 53, and 12^3 x 16 12 RHS 17 -> 21 / 40 -> 58 (too few tiles for the
//     SMs).  Two tiles a barrier from 8 right-hand sides (195 against 208), one
//     below (157 against 170);
//   * fewer right-hand sides on 2^17 sites or more: at most 80 registers and
//     read-once operands past L1, 256-thread blocks (pass 2, 32^3 x 64: F32
//     186 -> 175, 3 RHS 429 -> 360, F16 136 -> 130); on 16^3 x 32 it is slower.
static int default_hop_variant(int prec, int flags, int red, long vh, int nrhs, bool mapped) {
  if (prec == P_F64 || mapped) return 0;
  const int per_block = (nrhs + (nrhs + 11) / 12 - 1) / ((nrhs + 11) / 12);  // right-hand sides of a tile block
  if (((per_block >= 4 && vh >= (1L << 18)) || (per_block >= 6 && vh >= (1L << 16))) &&
      hop_has_variant(prec, flags, red, 9))
    return per_block >= 8 ? 10 : 9;
  return vh >= (1L << 17) && (flags & F_AUX) == 0 && hop_has_variant(prec, flags, red, 4) ? 4 : 0;
}

bool launch_hop_any(int prec, int flags, int red, const HopArgs& a, int block, cudaStream_t st, int* occ,
                    int variant) {
  for (;;) {
    bool ok = false;
    switch (prec) {
      case P_F64: ok = launch_hop<P_F64>(flags, red, a, block, st, occ, variant); break;
      case P_F32: ok = launch_hop<P_F32>(flags, red, a, block, st, occ, variant); break;
      case P_F16: ok = launch_hop<P_F16>(flags, red, a, block, st, occ, variant); break;
      case P_BF16: ok = launch_hop<P_BF16>(flags, red, a, block, st, occ, variant); break;
    }
    if (ok || variant == 0) return ok;
    variant = 0;  // this kernel has no such variant (e.g. several RHS per thread in FP64)
  }
}

}  // namespace bridge
