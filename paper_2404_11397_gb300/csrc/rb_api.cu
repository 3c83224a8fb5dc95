// rb_api.cu -- the C ABI of librb (declared in include/rb.h): event build,
// batched likelihood / gradient calls, strain generation, diagnostics.
// Host code only orchestrates: every step of the computation runs in the
// kernels of rb_setup.cu, rb_loglike.cu and rb_summary.cu.
#include <algorithm>
#include <atomic>
#include <cmath>
#include <cstdarg>
#include <cstdio>
#include <cstddef>
#include <cstring>
#include <mutex>
#include <new>
#include <vector>

#include "rb.h"
#include "rb_api_internal.h"
#include "rb_internal.cuh"

namespace rb {

// ---- launchers defined in the kernel translation units ----
cudaError_t launch_ref_values(const double* theta_ref_dev, const EventConst& ec, RefValues* out, cudaStream_t s);
cudaError_t launch_setup(int mode, const double* theta, int64_t W, const EventConst& ec, const RefValues* ref,
                         void* ws, void* tan, bool grad, cudaStream_t s);
cudaError_t launch_rb_mixed(const EventDev& ev, const void* ws, const void* tan, int64_t W, double* logl,
                            double* grad, bool phase64, bool spread, cudaStream_t s, int n_sm, const MalaArgs* mala);
cudaError_t launch_rb_fused(const EventDev& ev, const EventConst& ec, const double* theta, int64_t W, double* logl,
                            double* grad, cudaStream_t s, int n_sm, const MalaArgs* mala, bool* done);
cudaError_t launch_rb_f64(const EventDev& ev, const void* ws, const void* tan, int64_t W, double* logl, double* grad,
                          cudaStream_t s, int n_sm, const MalaArgs* mala);
cudaError_t launch_bin_edges(double f_low, double f_high, double T, int64_t kmin, int64_t N, int B, int64_t* edges,
                             double* span, cudaStream_t s);
size_t bin_edges_agnostic_scratch_bytes(int64_t N);
size_t chunk_coef_bytes(int64_t N);
size_t mixed_smem_slot_bytes();
cudaError_t launch_chunk_coef(int64_t N, int D, const RefValues* ref, const void* cq, void* chunk_coef, cudaStream_t s);
cudaError_t launch_bin_edges_agnostic(const double* theta_ref_dev, double T, int64_t kmin, int64_t N, int B,
                                      int64_t* edges, double* span, void* scratch, cudaStream_t s);
cudaError_t launch_summary(const DataPtrs& in, int64_t kmin, int64_t N, double T, int D, int B,
                           const int64_t* edges, const RefValues* ref, const SummaryOut& so, double* h0_out,
                           cudaStream_t s);
cudaError_t launch_summary_stored(const DataPtrs& in, const double* h0, int64_t N, double T, int D, int B,
                                  const int64_t* edges, const SummaryOut& so, int n_parts, cudaStream_t s);
cudaError_t launch_summary_chunk64(const DataPtrs& in, double* h0_out, void* scratch, int64_t kmin, int64_t N, double T, int D,
                                   int B, const int64_t* edges, const RefValues* ref, const SummaryOut& so, int n_parts,
                                   cudaStream_t s);
cudaError_t launch_edge_tables(int64_t kmin, double T, int D, int B, int Ep, int Bp, const int64_t* edges,
                               float* tab32, size_t edge32_floats, double* tab64, double* inv_df, float* slot32,
                               int n_slots, cudaStream_t s);
cudaError_t launch_chunk_q(int64_t kmin, double T, int64_t N, void* cq, cudaStream_t s);
size_t chunk_q_bytes(int64_t N);
cudaError_t launch_strain(const RefValues* src, int64_t kmin, int64_t N, double T, double* h, cudaStream_t s);
cudaError_t launch_summary_parts(const void* w32, const float* is32, const int* exps, int64_t N, double T, int D, int B,
                                 const int64_t* edges, const RefValues* ref, const void* chunk_q, const void* recs,
                                 const SummaryOut& so, cudaStream_t s);
cudaError_t launch_ref_dd(const double* theta_ref_dev, const EventConst& ec, RefValues* out, SummarySync* base_reset,
                          cudaStream_t s);
cudaError_t launch_tangents(const double* theta, int64_t W, const EventConst& ec, void* tan, cudaStream_t s);
cudaError_t launch_data32(const DataPtrs& in, int64_t N, int D, void* w32, float* is32, int* exps, cudaStream_t s);
cudaError_t launch_pull32(const DataPtrs& src, int64_t N, int D, double* data, double* psd, void* w32, float* is32,
                          int* exps, int n_sm, cudaStream_t s);

// ---- diagnostics ----
static thread_local char g_err[512] = "no error";
static std::atomic<uint64_t> g_launches{0};
static thread_local uint64_t t_launches = 0;  // this thread's share: what a capture on it enqueued
static std::atomic<uint64_t> g_event_uid{0};

int set_error(int code, const char* fmt, ...) {
  va_list ap;
  va_start(ap, fmt);
  vsnprintf(g_err, sizeof(g_err), fmt, ap);
  va_end(ap);
  return code;
}
void count_launches(uint64_t n) {
  g_launches.fetch_add(n, std::memory_order_relaxed);
  t_launches += n;
}

int cuda_fail(cudaError_t e, const char* what) {
  if (e == cudaErrorMemoryAllocation) return set_error(RB_ENOMEM, "%s: %s", what, cudaGetErrorString(e));
  return set_error(RB_ECUDA, "%s: %s", what, cudaGetErrorString(e));
}

// Stream-ordered workspace allocations come from a memory pool owned by the
// library (one per device) that keeps up to 1 GiB of freed memory reserved.
// The device's default pool returns freed memory at every synchronisation,
// after which the next allocation maps it again: with a synchronising caller
// (the host-buffer entry points) that costs more than the kernels.
static cudaMemPool_t library_pool(int dev) {
  static std::mutex mu;
  static cudaMemPool_t pools[64] = {};
  static bool tried[64] = {};
  if (dev < 0 || dev >= 64) return nullptr;
  std::lock_guard<std::mutex> lk(mu);
  if (!tried[dev]) {
    tried[dev] = true;
    cudaMemPoolProps props = {};
    props.allocType = cudaMemAllocationTypePinned;
    props.location.type = cudaMemLocationTypeDevice;
    props.location.id = dev;
    cudaMemPool_t pool = nullptr;
    if (cudaMemPoolCreate(&pool, &props) == cudaSuccess) {
      uint64_t keep = 1ull << 30;
      if (cudaMemPoolSetAttribute(pool, cudaMemPoolAttrReleaseThreshold, &keep) == cudaSuccess) pools[dev] = pool;
      else cudaMemPoolDestroy(pool);
    } else {
      cudaGetLastError();  // fall back to the default pool
    }
  }
  return pools[dev];
}

cudaError_t ws_alloc(void** p, size_t bytes, cudaStream_t s) {
  int dev = 0;
  cudaError_t err = cudaGetDevice(&dev);
  if (err != cudaSuccess) return err;
  cudaMemPool_t pool = library_pool(dev);
  return pool ? cudaMallocFromPoolAsync(p, bytes, pool, s) : cudaMallocAsync(p, bytes, s);
}

int sm_count() {
  static std::once_flag once;
  static int n = 0;
  std::call_once(once, [] {
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess)
      n = 1;
  });
  return n;
}

// ---- site geometry (host) ----
static void arm_unit(double lat, double lon, double az, double a[3]) {
  const double n[3] = {-std::sin(lat) * std::cos(lon), -std::sin(lat) * std::sin(lon), std::cos(lat)};  // North
  const double e[3] = {-std::sin(lon), std::cos(lon), 0.0};                                            // East
  for (int i = 0; i < 3; ++i) a[i] = std::cos(az) * n[i] + std::sin(az) * e[i];
}

// v = out[0] + out[1] with two floats (hi = v rounded, lo = the rest rounded).
static void split_pair(double v, float* out) {
  out[0] = (float)v;
  out[1] = (float)(v - (double)out[0]);
}

DetGeom make_geom(double lat, double lon, double elev, double xaz, double yaz) {
  DetGeom g;
  double x[3], y[3];
  arm_unit(lat, lon, xaz, x);
  arm_unit(lat, lon, yaz, y);
  for (int i = 0; i < 3; ++i)
    for (int j = 0; j < 3; ++j) g.D[i][j] = 0.5 * (x[i] * x[j] - y[i] * y[j]);
  // WGS-84 geodetic -> Earth-fixed Cartesian
  const double a = 6378137.0, e2 = 6.69437999014e-3;
  const double s = std::sin(lat), c = std::cos(lat);
  const double Nr = a / std::sqrt(1.0 - e2 * s * s);
  g.r[0] = (Nr + elev) * c * std::cos(lon);
  g.r[1] = (Nr + elev) * c * std::sin(lon);
  g.r[2] = (Nr * (1.0 - e2) + elev) * s;
  for (int i = 0; i < 3; ++i) {
    split_pair(x[i], g.xa[i]);
    split_pair(y[i], g.ya[i]);
    split_pair(g.r[i] / kClight, g.rc[i]);
  }
  return g;
}

static bool theta_ok(const double* th) {
  for (int j = 0; j < kNPar; ++j)
    if (!std::isfinite(th[j])) return false;
  return th[0] > 0.0 && th[1] > 0.0 && th[1] <= 1.0 && th[6] > 0.0;
}

static int round_up(int x, int m) { return (x + m - 1) / m * m; }

}  // namespace rb

using namespace rb;

struct rb_event_s {
  rb::EventEntry e;
};

namespace rb {
const EventEntry* event_entry(::rb_event_s* ev) { return ev ? &ev->e : nullptr; }
}  // namespace rb

extern "C" {

int rb_abi_version(void) { return 2; }

#ifdef RB_BOUNDS_CHECK
extern "C" int rb_bounds_read_loglike(rb::BoundsRecord* out);
extern "C" int rb_bounds_read_summary(rb::BoundsRecord* out);
#endif

int rb_debug_bounds(int* site, long long* index, long long* limit) {
#ifdef RB_BOUNDS_CHECK
  int (*const readers[])(rb::BoundsRecord*) = {rb_bounds_read_loglike, rb_bounds_read_summary};
  long long total = 0;
  bool first = true;
  for (auto rd : readers) {
    rb::BoundsRecord r{};
    const int e = rd(&r);
    if (e != 0) return cuda_fail((cudaError_t)e, "rb_debug_bounds");
    if (r.count && first) {
      if (site) *site = r.site;
      if (index) *index = r.index;
      if (limit) *limit = r.limit;
      first = false;
    }
    total += r.count;
  }
  return (int)(total > 0x7fffffff ? 0x7fffffff : total);
#else
  (void)site;
  (void)index;
  (void)limit;
  return -1;
#endif
}

const char* rb_last_error(void) { return g_err; }

uint64_t rb_kernel_launch_count(void) { return g_launches.load(); }

const char* rb_strerror(int status) {
  switch (status) {
    case RB_OK: return "ok";
    case RB_PENDING: return "pending";
    case RB_EINVAL: return "invalid argument";
    case RB_ENOMEM: return "out of memory";
    case RB_ECUDA: return "CUDA error";
    case RB_ETIMEDOUT: return "timed out";
    case RB_EBUSY: return "busy: admission refused";
    case RB_ENOTFOUND: return "unknown ticket";
    case RB_ECLOSED: return "server closed";
    default: return "unknown status";
  }
}

// Split every bin into parts of at most kPartPoints grid points for the fast
// summary build (bin edges are final here; they do not change on a rebuild).
static int make_parts(EventEntry& e, cudaStream_t s) {
  const int B = e.n_bins;
  std::vector<int64_t> edges(B + 1);
  cudaError_t err = cudaMemcpyAsync(edges.data(), e.d_edges, sizeof(int64_t) * (B + 1), cudaMemcpyDeviceToHost, s);
  if (err == cudaSuccess) err = cudaStreamSynchronize(s);
  if (err != cudaSuccess) return cuda_fail(err, "rb_build_summary: read bin edges");
  std::vector<PartDesc> parts;
  for (int b = 0; b < B; ++b) {
    const int64_t k0 = edges[b], k1 = (b == B - 1) ? edges[b + 1] + 1 : edges[b + 1];
    const int np = (int)((k1 - k0 + kPartPoints - 1) / kPartPoints);
    const int first = (int)parts.size();
    for (int p = 0; p < np; ++p) {
      PartDesc d{};
      d.bin = b;
      d.start = (int)(k0 + (int64_t)p * kPartPoints);
      d.end = (int)std::min<int64_t>(k1, k0 + (int64_t)(p + 1) * kPartPoints);
      d.first = first;
      d.n_parts = np;
      parts.push_back(d);
    }
  }
  e.n_parts = (int)parts.size();
  const size_t pb = sizeof(PartDesc) * parts.size(), sb = sizeof(float) * 2 * 7 * kMaxDet * parts.size();
  if ((err = cudaMalloc((void**)&e.d_parts, pb)) != cudaSuccess) return cuda_fail(err, "parts");
  e.device_bytes += pb;
  if ((err = cudaMalloc((void**)&e.d_part_sums, sb)) != cudaSuccess) return cuda_fail(err, "part sums");
  e.device_bytes += sb;
  err = cudaMemcpyAsync(e.d_parts, parts.data(), pb, cudaMemcpyHostToDevice, s);
  if (err == cudaSuccess) err = cudaStreamSynchronize(s);  // `parts` is freed on return
  if (err != cudaSuccess) return cuda_fail(err, "upload parts");
  return RB_OK;
}

int rb_event_free(rb_event_t ev) {
  RB_NVTX("rb_event_free");
  if (!ev) return RB_OK;
  EventEntry& e = ev->e;
  cudaFree(e.d_edges);
  cudaFree(e.d_summ);
  cudaFree(e.d_tab32);
  cudaFree(e.d_slot32);
  cudaFree(e.d_tab64);
  cudaFree(e.d_ref);
  cudaFree(e.d_base);
  cudaFree(e.d_data);
  cudaFree(e.d_psd);
  cudaFree(e.d_theta_ref);
  cudaFree(e.d_chunkq);
  cudaFree(e.d_chunks);
  cudaFree(e.d_invdf);
  cudaFree(e.d_share);
  cudaFree(e.step_ws);
  for (int i = 0; i < e.n_step_ws_old; ++i) cudaFree(e.step_ws_old[i]);
  if (e.hg_exec) cudaGraphExecDestroy(e.hg_exec);
  if (e.hs_exec) cudaGraphExecDestroy(e.hs_exec);
  if (e.hg_stream) cudaStreamDestroy(e.hg_stream);
  cudaFree(e.hg_ws);
  if (e.ev_fork) cudaEventDestroy(e.ev_fork);
  if (e.ev_join) cudaEventDestroy(e.ev_join);
  if (e.ev_ref) cudaEventDestroy(e.ev_ref);
  if (e.ev_setup) cudaEventDestroy(e.ev_setup);
  if (e.ev_data) cudaEventDestroy(e.ev_data);
  if (e.ev_tan) cudaEventDestroy(e.ev_tan);
  if (e.tanst) cudaStreamDestroy(e.tanst);
  if (e.copy) cudaStreamDestroy(e.copy);
  if (e.side) cudaStreamDestroy(e.side);
  cudaFree(e.d_sync);
  cudaFree(e.d_w32);
  cudaFree(e.d_is32);
  cudaFree(e.d_wexp);
  cudaFree(e.d_parts);
  cudaFree(e.d_part_sums);
  cudaFree(e.d_h0);
  delete ev;
  return RB_OK;
}

// chunk_h0: h0 from Taylor chunks (rebuild_event), as the event that was saved had it.
static int build_event(const rb_event_desc* desc, rb_event_t* out, bool chunk_h0) {
  if (!desc || !out) return set_error(RB_EINVAL, "rb_build_summary: NULL descriptor or output");
  *out = nullptr;
  const int D = desc->n_det, B = desc->n_bins;
  if (D < 1 || D > RB_MAX_DET) return set_error(RB_EINVAL, "rb_build_summary: n_det=%d not in 1..%d", D, RB_MAX_DET);
  if (!(desc->T > 0.0) || !std::isfinite(desc->T) || !(desc->f_low > 0.0) || !(desc->f_high > desc->f_low) ||
      !std::isfinite(desc->f_high) || !std::isfinite(desc->gmst))
    return set_error(RB_EINVAL, "rb_build_summary: invalid T/f_low/f_high/gmst");
  const int64_t kmin = (int64_t)std::ceil(desc->f_low * desc->T - 1e-9);
  const int64_t kmax = (int64_t)std::floor(desc->f_high * desc->T + 1e-9);
  const int64_t N = kmax - kmin + 1;
  if (N < 2) return set_error(RB_EINVAL, "rb_build_summary: grid has %lld points", (long long)N);
  if (B < 1 || B > N - 1) return set_error(RB_EINVAL, "rb_build_summary: n_bins=%d not in 1..%lld", B, (long long)(N - 1));
  if ((int64_t)B + 1 > (int64_t)1 << 20) return set_error(RB_EINVAL, "rb_build_summary: too many bins");
  for (int d = 0; d < D; ++d)
    if (!desc->det[d].data || !desc->det[d].psd) return set_error(RB_EINVAL, "rb_build_summary: detector %d has NULL data/psd", d);
  if (!theta_ok(desc->theta_ref)) return set_error(RB_EINVAL, "rb_build_summary: unphysical theta_ref");
  if (desc->bin_scheme != RB_BINS_PN && desc->bin_scheme != RB_BINS_AGNOSTIC)
    return set_error(RB_EINVAL, "rb_build_summary: bin_scheme=%d is neither RB_BINS_PN nor RB_BINS_AGNOSTIC",
                     desc->bin_scheme);

  rb_event_t ev = new (std::nothrow) rb_event_s();
  if (!ev) return set_error(RB_ENOMEM, "rb_build_summary: host allocation");
  EventEntry& e = ev->e;
  cudaStream_t s = (cudaStream_t)desc->cuda_stream;
  e.uid = ++g_event_uid;
  e.n_det = D;
  e.n_bins = B;
  e.kmin = kmin;
  e.N = N;
  e.T = desc->T;
  e.f_low = desc->f_low;
  e.f_high = desc->f_high;
  e.gmst = desc->gmst;
  e.bin_scheme = desc->bin_scheme;
  std::memcpy(e.theta_ref, desc->theta_ref, sizeof(e.theta_ref));
  e.ec.n_det = D;
  e.ec.pad = 0;
  e.ec.gmst = desc->gmst;
  split_pair(desc->gmst, e.ec.gmst2);
  for (int d = 0; d < RB_MAX_DET; ++d) {
    if (d < D) {
      const rb_detector_desc& dd = desc->det[d];
      e.ec.det[d] = make_geom(dd.lat, dd.lon, dd.elev_m, dd.xarm_az, dd.yarm_az);
      const double row[5] = {dd.lat, dd.lon, dd.elev_m, dd.xarm_az, dd.yarm_az};
      std::memcpy(e.geom[d], row, sizeof(row));
    } else {
      std::memset(&e.ec.det[d], 0, sizeof(DetGeom));
    }
  }
  const int E = B + 1;
  const int Ep = round_up(E, 4), Bp = round_up(B, 4);
  const size_t edge32 = (size_t)4 * kEdgeQuads * Ep;
  const size_t tab32 = edge32 + (size_t)D * 6 * Bp;
  const size_t tab64 = (size_t)(kNBasis + 1) * Ep + (size_t)D * 6 * Bp;
  const int NS = slot_count(B);
  const size_t slot32 = (size_t)NS * (4 * (kNBasis + 1) + kSlotBinFloats * D);
  {
    // the batch kernels stage all edge and bin tables in shared memory
    int dev = 0, smem_max = 0;
    cudaError_t qerr = cudaGetDevice(&dev);
    if (qerr == cudaSuccess) qerr = cudaDeviceGetAttribute(&smem_max, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
    if (qerr != cudaSuccess) {
      delete ev;
      return cuda_fail(qerr, "rb_build_summary: device query");
    }
    // (plus the per-warp walker slots of the mixed kernel)
    const size_t need = std::max(slot32 * sizeof(float), (size_t)(kNBasis + 1) * Ep * sizeof(double) +
                                                             (size_t)D * 6 * Bp * sizeof(float)) +
                        mixed_smem_slot_bytes();
    if (need > (size_t)smem_max) {
      delete ev;
      return set_error(RB_EINVAL, "rb_build_summary: %d bins x %d detectors need %zu B of shared memory (max %d)",
                       B, D, need, smem_max);
    }
  }

  int rc = RB_OK;
  cudaError_t err;
  void* bins_scratch = nullptr;  // build-time only (agnostic bin placement)
  double* d_span = nullptr;
  do {
    struct { void** p; size_t n; const char* what; } allocs[] = {
        {(void**)&e.d_edges, sizeof(int64_t) * E, "edges"},
        {(void**)&e.d_summ, sizeof(double) * 6 * D * B, "summary"},
        {(void**)&e.d_tab32, sizeof(float) * tab32, "tab32"},
        {(void**)&e.d_slot32, sizeof(float) * slot32, "slot image"},
        {(void**)&e.d_tab64, sizeof(double) * tab64, "tab64"},
        {(void**)&e.d_ref, sizeof(RefValues), "ref"},
        {(void**)&e.d_base, sizeof(double), "base"},
        {(void**)&e.d_data, sizeof(double) * 2 * D * N, "strain"},
        {(void**)&e.d_psd, sizeof(double) * D * N, "psd"},
        {(void**)&e.d_h0, sizeof(double) * 2 * D * N, "stored fiducial waveform"},
        {(void**)&e.d_theta_ref, sizeof(double) * kNPar, "theta_ref"},
        {(void**)&e.d_chunkq, chunk_q_bytes(N), "chunk matrices"},
        {(void**)&e.d_chunks, chunk_coef_bytes(N), "chunk records"},
        {(void**)&e.d_invdf, sizeof(double) * B, "bin widths"},
        {(void**)&e.d_share, sizeof(double) * D * B, "base shares"},
        {(void**)&e.d_sync, offsetof(SummarySync, bin_parts_done) + sizeof(unsigned) * B, "build counters"},
        {(void**)&e.d_w32, sizeof(float) * 2 * D * N, "FP32 data copy"},
        {(void**)&e.d_is32, sizeof(float) * D * N, "FP32 inverse PSD copy"},
        {(void**)&e.d_wexp, sizeof(int) * 2 * kMaxDet, "FP32 copy scales"}};
    for (auto& a : allocs) {
      if ((err = cudaMalloc(a.p, a.n)) != cudaSuccess) { rc = cuda_fail(err, a.what); break; }
      e.device_bytes += a.n;
    }
    if (rc != RB_OK) break;
    if ((err = cudaStreamCreateWithFlags(&e.side, cudaStreamNonBlocking)) != cudaSuccess ||
        (err = cudaEventCreateWithFlags(&e.ev_fork, cudaEventDisableTiming)) != cudaSuccess ||
        (err = cudaEventCreateWithFlags(&e.ev_join, cudaEventDisableTiming)) != cudaSuccess ||
        (err = cudaEventCreateWithFlags(&e.ev_ref, cudaEventDisableTiming)) != cudaSuccess ||
        (err = cudaEventCreateWithFlags(&e.ev_setup, cudaEventDisableTiming)) != cudaSuccess) {
      rc = cuda_fail(err, "rebuild stream and events");
      break;
    }
    e.dev.n_det = D;
    e.dev.n_bins = B;
    e.dev.n_edges = E;
    e.dev.e_pad = Ep;
    e.dev.b_pad = Bp;
    e.dev.kmin = kmin;
    e.dev.n_freq = N;
    e.dev.T = e.T;
    e.dev.base_logl = e.d_base;
    e.dev.sync = e.d_sync;
    e.dev.share = e.d_share;
    e.dev.tab32 = e.d_tab32;
    e.dev.tab32_floats = tab32;
    e.dev.edge32_floats = edge32;
    e.dev.slot32 = e.d_slot32;
    e.dev.slot32_floats = slot32;
    e.dev.n_slots = NS;
    {
      // each |g_k| is largest at an end of the grid (the powers are monotonic,
      // |ln f| and |f^1/3 ln f| quasi-convex); 1 % added
      const double fe[2] = {(double)kmin / e.T, (double)(kmin + N - 1) / e.T};
      double gm[kNBasis + 1] = {};
      for (double f : fe) {
        const double lf = std::log(f), cf = std::cbrt(f);
        const double g[kNBasis + 1] = {std::pow(f, -5.0 / 3.0), 1.0 / f, std::pow(f, -2.0 / 3.0), 1.0 / cf, lf, cf,
                                       cf * lf, cf * cf, f * cf * cf, f * f * cf, f * kTwoPi};
        for (int k = 0; k <= kNBasis; ++k) gm[k] = std::max(gm[k], std::fabs(g[k]) / kTwoPi);
      }
      for (int k = 0; k <= kNBasis; ++k) e.dev.gmax[k] = (float)(1.01 * gm[k]);
    }
    e.dev.tab64 = e.d_tab64;
    e.dev.ref = e.d_ref;
    const cudaMemcpyKind kind = desc->data_on_device ? cudaMemcpyDeviceToDevice : cudaMemcpyHostToDevice;
    for (int d = 0; d < D && rc == RB_OK; ++d) {
      if ((err = cudaMemcpyAsync(e.d_data + 2 * (size_t)d * N, desc->det[d].data, sizeof(double) * 2 * N, kind, s)) != cudaSuccess) rc = cuda_fail(err, "copy strain");
      else if ((err = cudaMemcpyAsync(e.d_psd + (size_t)d * N, desc->det[d].psd, sizeof(double) * N, kind, s)) != cudaSuccess) rc = cuda_fail(err, "copy psd");
    }
    if (rc != RB_OK) break;
    if ((err = cudaMemcpyAsync(e.d_theta_ref, e.theta_ref, sizeof(double) * kNPar, cudaMemcpyHostToDevice, s)) != cudaSuccess) { rc = cuda_fail(err, "copy theta_ref"); break; }
    if ((err = cudaMemsetAsync(e.d_sync, 0, offsetof(SummarySync, bin_parts_done) + sizeof(unsigned) * B, s)) != cudaSuccess) { rc = cuda_fail(err, "zero counters"); break; }
    if ((err = cudaMalloc((void**)&d_span, sizeof(double))) != cudaSuccess) { rc = cuda_fail(err, "bin span"); break; }
    if (e.bin_scheme == RB_BINS_AGNOSTIC) {
      if ((err = cudaMalloc(&bins_scratch, bin_edges_agnostic_scratch_bytes(N))) != cudaSuccess) { rc = cuda_fail(err, "bin placement scratch"); break; }
      if ((err = launch_bin_edges_agnostic(e.d_theta_ref, e.T, kmin, N, B, e.d_edges, d_span, bins_scratch, s)) != cudaSuccess) { rc = cuda_fail(err, "agnostic bin edge kernels"); break; }
      count_launches(8);
    } else {
      if ((err = launch_bin_edges(e.f_low, e.f_high, e.T, kmin, N, B, e.d_edges, d_span, s)) != cudaSuccess) { rc = cuda_fail(err, "bin edge kernels"); break; }
    }
    if ((rc = make_parts(e, s)) != RB_OK) break;
    if ((err = launch_edge_tables(kmin, e.T, D, B, Ep, Bp, e.d_edges, e.d_tab32, edge32, e.d_tab64, e.d_invdf, e.d_slot32, NS, s)) != cudaSuccess) { rc = cuda_fail(err, "edge table kernel"); break; }
    if ((err = launch_chunk_q(kmin, e.T, N, e.d_chunkq, s)) != cudaSuccess) { rc = cuda_fail(err, "chunk matrix kernel"); break; }
    count_launches(4);
    if ((rc = rebuild_event(e, nullptr, RB_FP64, s, nullptr, chunk_h0)) != RB_OK) break;
    if ((err = cudaStreamSynchronize(s)) != cudaSuccess) { rc = cuda_fail(err, "build synchronise"); break; }
    double span = 0.0;
    if ((err = cudaMemcpy(&span, d_span, sizeof(double), cudaMemcpyDeviceToHost)) != cudaSuccess) { rc = cuda_fail(err, "read bin span"); break; }
    e.epsilon = span / (double)B;
  } while (false);
  if (bins_scratch || d_span) {
    cudaStreamSynchronize(s);
    cudaFree(bins_scratch);
    cudaFree(d_span);
  }
  if (rc != RB_OK) {
    cudaStreamSynchronize(s);
    rb_event_free(ev);
    return rc;
  }
  *out = ev;
  return RB_OK;
}

int rb_build_summary(const rb_event_desc* desc, rb_event_t* out) {
  RB_NVTX("rb_build_summary");
  return build_event(desc, out, false);
}

int rb_event_rebuild(rb_event_t ev, const double* theta_ref_host, const double* const* data, const double* const* psd,
                     int data_on_device, int mode, void* stream) {
  RB_NVTX("rb_event_rebuild");
  if (!ev) return set_error(RB_EINVAL, "rb_event_rebuild: NULL event");
  if (mode != RB_MIXED && mode != RB_FP64 && mode != RB_MIXED_F64PHASE) return set_error(RB_EINVAL, "rb_event_rebuild: bad mode %d", mode);
  EventEntry& e = ev->e;
  cudaStream_t s = (cudaStream_t)stream;
  cudaError_t err;
  if (theta_ref_host) {
    if (!theta_ok(theta_ref_host)) return set_error(RB_EINVAL, "rb_event_rebuild: unphysical theta_ref");
    std::memcpy(e.theta_ref, theta_ref_host, sizeof(e.theta_ref));
    e.h0_valid = false;  // the stored fiducial waveform belongs to the old theta_ref
    if ((err = cudaMemcpyAsync(e.d_theta_ref, theta_ref_host, sizeof(double) * kNPar, cudaMemcpyHostToDevice, s)) != cudaSuccess)
      return cuda_fail(err, "rb_event_rebuild: copy theta_ref");
  }
  DataPtrs in{};
  bool have = false;
  if (data || psd) {
    if (!data || !psd) return set_error(RB_EINVAL, "rb_event_rebuild: data and psd must both be given");
    for (int d = 0; d < e.n_det; ++d)
      if (!data[d] || !psd[d]) return set_error(RB_EINVAL, "rb_event_rebuild: detector %d has NULL data/psd", d);
    const int64_t N = e.N;
    if (data_on_device) {  // read in place, no copy
      for (int d = 0; d < e.n_det; ++d) {
        in.data[d] = data[d];
        in.psd[d] = psd[d];
      }
      have = true;
    } else {  // stage into the event's resident copy
      e.w32_resident = false;
      for (int d = 0; d < e.n_det; ++d) {
        if ((err = cudaMemcpyAsync(e.d_data + 2 * (size_t)d * N, data[d], sizeof(double) * 2 * N, cudaMemcpyHostToDevice, s)) != cudaSuccess)
          return cuda_fail(err, "rb_event_rebuild: copy strain");
        if ((err = cudaMemcpyAsync(e.d_psd + (size_t)d * N, psd[d], sizeof(double) * N, cudaMemcpyHostToDevice, s)) != cudaSuccess)
          return cuda_fail(err, "rb_event_rebuild: copy psd");
      }
    }
  }
  return rebuild_event(e, have ? &in : nullptr, mode, s, nullptr, theta_ref_host != nullptr);
}

void rb_set_trace_events(void* before_main, void* after_main) { set_trace_events(before_main, after_main); }

int rb_event_get_info(rb_event_t ev, rb_event_info* info) {
  RB_NVTX("rb_event_get_info");
  if (!ev || !info) return set_error(RB_EINVAL, "rb_event_get_info: NULL argument");
  const EventEntry& e = ev->e;
  info->n_det = e.n_det;
  info->n_bins = e.n_bins;
  info->kmin = e.kmin;
  info->n_freq = e.N;
  info->T = e.T;
  info->gmst = e.gmst;
  info->device_bytes = e.device_bytes;
  std::memcpy(info->theta_ref, e.theta_ref, sizeof(info->theta_ref));
  info->bin_scheme = e.bin_scheme;
  info->reserved = 0;
  info->epsilon = e.epsilon;
  // log L(theta_ref) as the kernels read it (event_base_logl): the fast build
  // leaves the fixed-point sum of the shares, the FP64 builds the value
  SummarySync hs{};
  cudaError_t err = cudaMemcpy(&hs, e.d_sync, offsetof(SummarySync, bin_parts_done), cudaMemcpyDeviceToHost);
  if (err == cudaSuccess) {
    if (hs.base_in_acc == 0u) {
      err = cudaMemcpy(&info->base_logl, e.d_base, sizeof(double), cudaMemcpyDeviceToHost);
    } else if (hs.overflow == 0u) {
      info->base_logl = (double)(long long)hs.base_acc * (1.0 / 4294967296.0);
    } else {
      std::vector<double> sh((size_t)e.n_det * e.n_bins);
      err = cudaMemcpy(sh.data(), e.d_share, sizeof(double) * sh.size(), cudaMemcpyDeviceToHost);
      double t = 0.0;
      for (double v : sh) t += v;
      info->base_logl = t;
    }
  }
  if (err != cudaSuccess) return cuda_fail(err, "rb_event_get_info: read base");
  return RB_OK;
}

// ---- event files: checkpoint and resume ----
namespace {
constexpr char kEventMagic[8] = {'R', 'B', 'E', 'V', 'E', 'N', 'T', '2'};
struct EventFileHeader {  // followed by strain [n_det][n_freq][2] and PSD [n_det][n_freq], FP64
  char magic[8];
  int32_t n_det, n_bins;
  int64_t n_freq;
  double T, f_low, f_high, gmst;
  double geom[RB_MAX_DET][5];
  double theta_ref[RB_NPAR];
  int32_t bin_scheme;
  int32_t chunk_h0;  // 1: the FP64 summary's h0 came from Taylor chunks (0 in files written before there was a choice)
};
}  // namespace

int rb_event_save(rb_event_t ev, const char* path) {
  RB_NVTX("rb_event_save");
  if (!ev || !path) return set_error(RB_EINVAL, "rb_event_save: NULL event or path");
  const EventEntry& e = ev->e;
  if (e.last_in_place)
    return set_error(RB_EINVAL, "rb_event_save: the last rebuild read caller data in place, which the event does not hold");
  EventFileHeader h{};
  std::memcpy(h.magic, kEventMagic, sizeof(h.magic));
  h.n_det = e.n_det;
  h.n_bins = e.n_bins;
  h.n_freq = e.N;
  h.T = e.T;
  h.f_low = e.f_low;
  h.f_high = e.f_high;
  h.gmst = e.gmst;
  std::memcpy(h.geom, e.geom, sizeof(h.geom));
  std::memcpy(h.theta_ref, e.theta_ref, sizeof(h.theta_ref));
  h.bin_scheme = e.bin_scheme;
  h.chunk_h0 = e.h0_valid && e.h0_chunks ? 1 : 0;
  const size_t nd = (size_t)2 * e.n_det * e.N, np = (size_t)e.n_det * e.N;
  std::vector<double> data(nd), psd(np);
  // the resident copy, after every call already issued on any stream
  cudaError_t err = cudaDeviceSynchronize();
  if (err == cudaSuccess) err = cudaMemcpy(data.data(), e.d_data, sizeof(double) * nd, cudaMemcpyDeviceToHost);
  if (err == cudaSuccess) err = cudaMemcpy(psd.data(), e.d_psd, sizeof(double) * np, cudaMemcpyDeviceToHost);
  if (err != cudaSuccess) return cuda_fail(err, "rb_event_save: read the resident data");
  FILE* f = std::fopen(path, "wb");
  if (!f) return set_error(RB_EINVAL, "rb_event_save: cannot open %s for writing", path);
  const bool ok = std::fwrite(&h, sizeof(h), 1, f) == 1 && std::fwrite(data.data(), sizeof(double), nd, f) == nd &&
                  std::fwrite(psd.data(), sizeof(double), np, f) == np;
  if (std::fclose(f) != 0 || !ok) return set_error(RB_EINVAL, "rb_event_save: write to %s failed", path);
  return RB_OK;
}

int rb_event_load(const char* path, void* stream, rb_event_t* out) {
  RB_NVTX("rb_event_load");
  if (!path || !out) return set_error(RB_EINVAL, "rb_event_load: NULL path or output");
  *out = nullptr;
  FILE* f = std::fopen(path, "rb");
  if (!f) return set_error(RB_EINVAL, "rb_event_load: cannot open %s", path);
  EventFileHeader h{};
  bool ok = std::fread(&h, sizeof(h), 1, f) == 1 && std::memcmp(h.magic, kEventMagic, sizeof(h.magic)) == 0 &&
            h.n_det >= 1 && h.n_det <= RB_MAX_DET && h.n_bins >= 1 && h.n_freq >= 2 && h.n_freq <= ((int64_t)1 << 31) &&
            h.T > 0.0 && std::isfinite(h.T) && h.f_high > h.f_low && h.f_low > 0.0;
  if (ok) {  // the grid the header's T and band define must be the one the arrays hold
    const int64_t kmin = (int64_t)std::ceil(h.f_low * h.T - 1e-9), kmax = (int64_t)std::floor(h.f_high * h.T + 1e-9);
    ok = kmax - kmin + 1 == h.n_freq;
  }
  std::vector<double> data, psd;
  if (ok) {
    const size_t nd = (size_t)2 * h.n_det * h.n_freq, np = (size_t)h.n_det * h.n_freq;
    data.resize(nd);
    psd.resize(np);
    ok = std::fread(data.data(), sizeof(double), nd, f) == nd && std::fread(psd.data(), sizeof(double), np, f) == np &&
         std::fgetc(f) == EOF;
  }
  std::fclose(f);
  if (!ok) return set_error(RB_EINVAL, "rb_event_load: %s is not a complete event file", path);
  rb_event_desc desc{};
  desc.n_det = h.n_det;
  desc.n_bins = h.n_bins;
  desc.T = h.T;
  desc.f_low = h.f_low;
  desc.f_high = h.f_high;
  desc.gmst = h.gmst;
  desc.data_on_device = 0;
  desc.bin_scheme = h.bin_scheme;
  desc.cuda_stream = stream;
  std::memcpy(desc.theta_ref, h.theta_ref, sizeof(desc.theta_ref));
  for (int d = 0; d < h.n_det; ++d) {
    rb_detector_desc& dd = desc.det[d];
    dd.lat = h.geom[d][0];
    dd.lon = h.geom[d][1];
    dd.elev_m = h.geom[d][2];
    dd.xarm_az = h.geom[d][3];
    dd.yarm_az = h.geom[d][4];
    dd.data = data.data() + (size_t)2 * d * h.n_freq;
    dd.psd = psd.data() + (size_t)d * h.n_freq;
  }
  return build_event(&desc, out, h.chunk_h0 == 1);
}

int rb_event_get_summary(rb_event_t ev, double* A0, double* A1, double* B0, double* B1, int64_t* edges) {
  RB_NVTX("rb_event_get_summary");
  if (!ev) return set_error(RB_EINVAL, "rb_event_get_summary: NULL event");
  const EventEntry& e = ev->e;
  const int D = e.n_det, B = e.n_bins;
  std::vector<double> s((size_t)6 * D * B);
  cudaError_t err = cudaMemcpy(s.data(), e.d_summ, sizeof(double) * s.size(), cudaMemcpyDeviceToHost);
  if (err != cudaSuccess) return cuda_fail(err, "copy summary");
  if (edges && (err = cudaMemcpy(edges, e.d_edges, sizeof(int64_t) * (B + 1), cudaMemcpyDeviceToHost)) != cudaSuccess)
    return cuda_fail(err, "copy edges");
  for (size_t i = 0; i < (size_t)D * B; ++i) {
    if (A0) { A0[2 * i] = s[6 * i]; A0[2 * i + 1] = s[6 * i + 1]; }
    if (A1) { A1[2 * i] = s[6 * i + 2]; A1[2 * i + 1] = s[6 * i + 3]; }
    if (B0) B0[i] = s[6 * i + 4];
    if (B1) B1[i] = s[6 * i + 5];
  }
  return RB_OK;
}

int rb_loglike_grad_batch(rb_event_t ev, const double* theta_dev, int64_t W, double* logl_dev, double* grad_dev,
                          int mode, void* stream) {
  RB_NVTX("rb_loglike_grad_batch");
  return rb::run_batch(event_entry(ev), theta_dev, W, logl_dev, grad_dev, mode & ~RB_SHARED, (cudaStream_t)stream, nullptr, nullptr,
                       !(mode & RB_SHARED));
}

namespace rb {
// The tangent and copy streams of the combined calls, created on an event's
// first combined call (most resident events never need them).
static cudaError_t ensure_stream(cudaStream_t& st, cudaEvent_t& ev) {
  cudaError_t err = cudaSuccess;
  if (!st && (err = cudaStreamCreateWithFlags(&st, cudaStreamNonBlocking)) != cudaSuccess) return err;
  if (!ev && (err = cudaEventCreateWithFlags(&ev, cudaEventDisableTiming)) != cudaSuccess) return err;
  return err;
}
}  // namespace rb

int rb_rebuild_loglike_grad(rb_event_t ev, const double* theta_dev, int64_t W, double* logl_dev, double* grad_dev,
                            int mode, void* stream) {
  RB_NVTX("rb_rebuild_loglike_grad");
  using namespace rb;
  if (!ev) return set_error(RB_EINVAL, "rb_rebuild_loglike_grad: NULL event");
  if (W < 0) return set_error(RB_EINVAL, "rb_rebuild_loglike_grad: W < 0");
  if (mode != RB_MIXED && mode != RB_FP64 && mode != RB_MIXED_F64PHASE)
    return set_error(RB_EINVAL, "rb_rebuild_loglike_grad: bad mode %d", mode);
  if (W > 0 && (!theta_dev || !logl_dev)) return set_error(RB_EINVAL, "rb_rebuild_loglike_grad: NULL theta or logl");
  return rebuild_and_batch(ev->e, theta_dev, W, logl_dev, grad_dev, mode, (cudaStream_t)stream, nullptr);
}

int rb_loglike_batch(rb_event_t ev, const double* theta_dev, int64_t W, double* logl_dev, int mode, void* stream) {
  RB_NVTX("rb_loglike_batch");
  return rb::run_batch(event_entry(ev), theta_dev, W, logl_dev, nullptr, mode & ~RB_SHARED, (cudaStream_t)stream, nullptr, nullptr,
                       !(mode & RB_SHARED));
}

namespace rb {
// Device address of a pinned, mapped host buffer that starts on an `align`
// boundary, or NULL (pageable memory, or unaligned).
static const double* mapped_host(const double* p, size_t align) {
  if (!p || reinterpret_cast<uintptr_t>(p) % align != 0) return nullptr;
  cudaPointerAttributes a{};
  if (cudaPointerGetAttributes(&a, p) != cudaSuccess) {
    cudaGetLastError();
    return nullptr;
  }
  if (a.type != cudaMemoryTypeHost || !a.devicePointer) return nullptr;
  if (reinterpret_cast<uintptr_t>(a.devicePointer) % align != 0) return nullptr;
  return static_cast<const double*>(a.devicePointer);
}

// Output buffers of the host-buffer calls: when log L (and the gradient, if
// asked for) are pinned, mapped host buffers, the likelihood kernel writes
// them directly over the host link and no copy back is needed.
struct HostOut {
  double* logl = nullptr;
  double* grad = nullptr;
  bool direct = false;
};

// The host-buffer batch's launches as a graph: captured (not run) for the
// walkers' and outputs' mapped addresses, W and mode on the event's capture
// stream, with a workspace of its own; replaced when the call changes.
// Returns false (nothing cached) if anything fails: the caller then launches
// the kernels directly.
static std::mutex g_hg_mu;
static bool host_batch_graph(EventEntry& e, const double* theta, int64_t W, double* logl, double* grad, int mode) {
  if (e.hg_exec && e.hg_theta == theta && e.hg_logl == logl && e.hg_grad == grad && e.hg_W == W && e.hg_mode == mode)
    return true;
  if (e.hg_exec) {
    cudaGraphExecDestroy(e.hg_exec);
    e.hg_exec = nullptr;
  }
  cudaError_t err = cudaSuccess;
  if (!e.hg_stream) err = cudaStreamCreateWithFlags(&e.hg_stream, cudaStreamNonBlocking);
  const size_t need = walker_ws_bytes(mode, grad != nullptr) * (size_t)W;
  if (err == cudaSuccess && e.hg_ws_bytes < need) {
    cudaFree(e.hg_ws);
    e.hg_ws = nullptr;
    e.hg_ws_bytes = 0;
    if ((err = cudaMalloc(&e.hg_ws, need)) == cudaSuccess) e.hg_ws_bytes = need;
  }
  if (err != cudaSuccess) {
    cudaGetLastError();
    return false;
  }
  cudaGraph_t g = nullptr;
  if (cudaStreamBeginCapture(e.hg_stream, cudaStreamCaptureModeThreadLocal) != cudaSuccess) {
    cudaGetLastError();
    return false;
  }
  const uint64_t n0 = t_launches;
  const int rc = run_batch(&e, theta, W, logl, grad, mode, e.hg_stream, e.hg_ws);
  e.hg_launches = t_launches - n0;
  count_launches((uint64_t)0 - e.hg_launches);  // the capture launched nothing
  err = cudaStreamEndCapture(e.hg_stream, &g);
  cudaGraphExec_t exec = nullptr;
  if (rc == RB_OK && err == cudaSuccess && g) err = cudaGraphInstantiate(&exec, g, 0);
  if (g) cudaGraphDestroy(g);
  if (rc != RB_OK || err != cudaSuccess || !exec) {
    cudaGetLastError();
    return false;
  }
  e.hg_exec = exec;
  e.hg_theta = theta;
  e.hg_logl = logl;
  e.hg_grad = grad;
  e.hg_W = W;
  e.hg_mode = mode;
  return false;  // captured for the next call; this one launches directly
}
static HostOut mapped_outputs(double* logl_host, double* grad_host) {
  HostOut o;
  o.logl = const_cast<double*>(mapped_host(logl_host, 8));
  o.grad = grad_host ? const_cast<double*>(mapped_host(grad_host, 8)) : nullptr;
  o.direct = o.logl && (!grad_host || o.grad);
  return o;
}
}  // namespace rb

int rb_loglike_grad_host(rb_event_t ev, const double* theta_host, int64_t W, double* logl_host, double* grad_host,
                         int mode, void* stream) {
  RB_NVTX("rb_loglike_grad_host");
  if (!ev) return set_error(RB_EINVAL, "rb_loglike_grad_host: NULL event");
  if (W < 0) return set_error(RB_EINVAL, "rb_loglike_grad_host: W < 0");
  if (W == 0) return RB_OK;
  if (!theta_host || !logl_host) return set_error(RB_EINVAL, "rb_loglike_grad_host: NULL buffer");
  cudaStream_t s = (cudaStream_t)stream;
  double *d_theta = nullptr, *d_logl = nullptr, *d_grad = nullptr;
  const rb::HostOut out = rb::mapped_outputs(logl_host, grad_host);
  // pinned (mapped) walkers are read by the set-up kernel over the host link;
  // others are copied in first
  const double* theta_in = rb::mapped_host(theta_host, 8);
  int rc = RB_OK;
  cudaError_t err;
  // everything pinned (a sampler's steady state): the launches replayed from
  // a graph captured for these buffers at the previous such call
  if (theta_in && out.direct && !rb::trace_events_set()) {
    bool replay;
    uint64_t launches;
    {
      std::lock_guard<std::mutex> lk(rb::g_hg_mu);
      replay = rb::host_batch_graph(ev->e, theta_in, W, out.logl, out.grad, mode);
      launches = ev->e.hg_launches;
      if (replay && (err = cudaGraphLaunch(ev->e.hg_exec, s)) != cudaSuccess) return cuda_fail(err, "graph launch");
    }
    if (replay) {
      rb::count_launches(launches);
      err = cudaStreamSynchronize(s);
      return err == cudaSuccess ? RB_OK : cuda_fail(err, "synchronise");
    }
  }
  do {
    if (!theta_in) {
      if ((err = ws_alloc(reinterpret_cast<void**>(&d_theta), sizeof(double) * kNPar * W, s)) != cudaSuccess) { rc = cuda_fail(err, "workspace allocation (theta)"); break; }
      if ((err = cudaMemcpyAsync(d_theta, theta_host, sizeof(double) * kNPar * W, cudaMemcpyHostToDevice, s)) != cudaSuccess) { rc = cuda_fail(err, "copy theta"); break; }
      theta_in = d_theta;
    }
    if (!out.direct) {
      if ((err = ws_alloc(reinterpret_cast<void**>(&d_logl), sizeof(double) * W, s)) != cudaSuccess) { rc = cuda_fail(err, "workspace allocation (logl)"); break; }
      if (grad_host && (err = ws_alloc(reinterpret_cast<void**>(&d_grad), sizeof(double) * kNPar * W, s)) != cudaSuccess) { rc = cuda_fail(err, "workspace allocation (grad)"); break; }
    }
    rc = rb::run_batch(&ev->e, theta_in, W, out.direct ? out.logl : d_logl, out.direct ? out.grad : d_grad, mode, s, nullptr);
    if (rc != RB_OK || out.direct) break;
    if ((err = cudaMemcpyAsync(logl_host, d_logl, sizeof(double) * W, cudaMemcpyDeviceToHost, s)) != cudaSuccess) { rc = cuda_fail(err, "copy logl"); break; }
    if (grad_host && (err = cudaMemcpyAsync(grad_host, d_grad, sizeof(double) * kNPar * W, cudaMemcpyDeviceToHost, s)) != cudaSuccess) { rc = cuda_fail(err, "copy grad"); break; }
  } while (false);
  if (d_theta) cudaFreeAsync(d_theta, s);
  if (d_logl) cudaFreeAsync(d_logl, s);
  if (d_grad) cudaFreeAsync(d_grad, s);
  err = cudaStreamSynchronize(s);
  if (rc == RB_OK && err != cudaSuccess) rc = cuda_fail(err, "synchronise");
  return rc;
}

namespace rb {
// The rebuild + batch of host buffers that are all pinned (mapped device
// addresses: strain, PSD, walkers, outputs), enqueued on s: the host-link read
// on the copy stream, the rebuild and batch (rebuild_and_batch, its
// data-independent kernels beside the read), the copy stream joined.
static int enqueue_host_step(EventEntry& e, const DataPtrs& src, const double* theta, int64_t W, double* logl,
                             double* grad, int mode, cudaStream_t s) {
  cudaError_t err;
  if ((err = cudaEventRecord(e.ev_fork, s)) != cudaSuccess || (err = cudaStreamWaitEvent(e.copy, e.ev_fork, 0)) != cudaSuccess)
    return cuda_fail(err, "copy fork");
  if ((err = launch_pull32(src, e.N, e.n_det, e.d_data, e.d_psd, e.d_w32, e.d_is32, e.d_wexp, sm_count(), e.copy)) != cudaSuccess) {
    e.w32_resident = false;
    cudaStreamWaitEvent(s, e.ev_fork, 0);
    return cuda_fail(err, "host-link read");
  }
  count_launches(1);
  e.w32_resident = true;  // once ev_data completes
  if ((err = cudaEventRecord(e.ev_data, e.copy)) != cudaSuccess) return cuda_fail(err, "copy strain");
  const int rc = rebuild_and_batch(e, theta, W, logl, grad, mode, s, e.ev_data);
  // the copy stream is joined into s (also when the rebuild failed early)
  cudaStreamWaitEvent(s, e.ev_data, 0);
  return rc;
}

// enqueue_host_step captured as a graph for these buffers, W and mode (not
// run); false if nothing is cached for them (the caller enqueues directly).
static bool host_step_graph(EventEntry& e, const DataPtrs& src, const double* theta, int64_t W, double* logl,
                            double* grad, int mode) {
  bool same = e.hs_exec && e.hs_theta == theta && e.hs_logl == logl && e.hs_grad == grad && e.hs_W == W &&
              e.hs_mode == mode;
  for (int d = 0; d < e.n_det && same; ++d) same = e.hs_data[d] == src.data[d] && e.hs_psd[d] == src.psd[d];
  if (same) return true;
  if (e.hs_exec) {
    cudaGraphExecDestroy(e.hs_exec);
    e.hs_exec = nullptr;
  }
  cudaError_t err = cudaSuccess;
  if (!e.hg_stream) err = cudaStreamCreateWithFlags(&e.hg_stream, cudaStreamNonBlocking);
  if (err != cudaSuccess || cudaStreamBeginCapture(e.hg_stream, cudaStreamCaptureModeThreadLocal) != cudaSuccess) {
    cudaGetLastError();
    return false;
  }
  const uint64_t n0 = t_launches;
  const int rc = enqueue_host_step(e, src, theta, W, logl, grad, mode, e.hg_stream);
  const uint64_t n = t_launches - n0;
  count_launches((uint64_t)0 - n);  // the capture launched nothing
  cudaGraph_t g = nullptr;
  err = cudaStreamEndCapture(e.hg_stream, &g);
  cudaGraphExec_t exec = nullptr;
  if (rc == RB_OK && err == cudaSuccess && g) err = cudaGraphInstantiate(&exec, g, 0);
  if (g) cudaGraphDestroy(g);
  if (rc != RB_OK || err != cudaSuccess || !exec) {
    cudaGetLastError();
    return false;
  }
  e.hs_exec = exec;
  for (int d = 0; d < e.n_det; ++d) {
    e.hs_data[d] = src.data[d];
    e.hs_psd[d] = src.psd[d];
  }
  e.hs_theta = theta;
  e.hs_logl = logl;
  e.hs_grad = grad;
  e.hs_W = W;
  e.hs_mode = mode;
  e.hs_launches = n;
  return false;
}
}  // namespace rb

int rb_rebuild_loglike_grad_host(rb_event_t ev, const double* const* data_host, const double* const* psd_host,
                                 const double* theta_host, int64_t W, double* logl_host, double* grad_host, int mode,
                                 void* stream) {
  RB_NVTX("rb_rebuild_loglike_grad_host");
  using namespace rb;
  if (!ev) return set_error(RB_EINVAL, "rb_rebuild_loglike_grad_host: NULL event");
  if (W < 0) return set_error(RB_EINVAL, "rb_rebuild_loglike_grad_host: W < 0");
  if (mode != RB_MIXED && mode != RB_FP64 && mode != RB_MIXED_F64PHASE)
    return set_error(RB_EINVAL, "rb_rebuild_loglike_grad_host: bad mode %d", mode);
  if (!data_host || !psd_host) return set_error(RB_EINVAL, "rb_rebuild_loglike_grad_host: NULL data or psd");
  EventEntry& e = ev->e;
  for (int d = 0; d < e.n_det; ++d)
    if (!data_host[d] || !psd_host[d]) return set_error(RB_EINVAL, "rb_rebuild_loglike_grad_host: detector %d has NULL data/psd", d);
  if (W > 0 && (!theta_host || !logl_host)) return set_error(RB_EINVAL, "rb_rebuild_loglike_grad_host: NULL buffer");
  cudaStream_t s = (cudaStream_t)stream;
  double *d_theta = nullptr, *d_logl = nullptr, *d_grad = nullptr;
  const HostOut out = W > 0 ? mapped_outputs(logl_host, grad_host) : HostOut{};
  int rc = RB_OK;
  cudaError_t err;
  // pinned (mapped) buffers are read by one kernel over the host link, which
  // writes the resident FP64 copies and the FP32 working copy together;
  // others are copied in by the copy engine (and converted by the rebuild)
  DataPtrs src{};
  bool mapped = true;
  for (int d = 0; d < e.n_det && mapped; ++d) {
    src.data[d] = mapped_host(data_host[d], 16);
    src.psd[d] = mapped_host(psd_host[d], 8);
    mapped = src.data[d] && src.psd[d];
  }
  if ((err = ensure_stream(e.copy, e.ev_data)) != cudaSuccess) return cuda_fail(err, "copy stream");
  // everything pinned (the steady state of a caller that streams data): the
  // call replayed from a graph captured for these buffers at the previous
  // such call, or enqueued directly
  const double* theta_in = W > 0 ? mapped_host(theta_host, 8) : nullptr;
  if (W > 0 && mapped && theta_in && out.direct && !trace_events_set()) {
    bool replay;
    uint64_t launches;
    {
      std::lock_guard<std::mutex> lk(g_hg_mu);
      replay = host_step_graph(e, src, theta_in, W, out.logl, out.grad, mode);
      launches = e.hs_launches;
      if (replay && (err = cudaGraphLaunch(e.hs_exec, s)) != cudaSuccess) return cuda_fail(err, "graph launch");
    }
    if (replay) count_launches(launches);
    else rc = enqueue_host_step(e, src, theta_in, W, out.logl, out.grad, mode, s);
    err = cudaStreamSynchronize(s);
    if (rc == RB_OK && err != cudaSuccess) rc = cuda_fail(err, "synchronise");
    return rc;
  }
  do {
    // strain and PSD into the event's resident copy on the copy stream, in
    // parallel with the data-independent kernels of the rebuild and batch
    if ((err = cudaEventRecord(e.ev_fork, s)) != cudaSuccess || (err = cudaStreamWaitEvent(e.copy, e.ev_fork, 0)) != cudaSuccess) { rc = cuda_fail(err, "copy fork"); break; }
    if (mapped) {
      err = launch_pull32(src, e.N, e.n_det, e.d_data, e.d_psd, e.d_w32, e.d_is32, e.d_wexp, sm_count(), e.copy);
      if (err == cudaSuccess) {
        count_launches(1);
        e.w32_resident = true;  // once ev_data completes
      } else {
        e.w32_resident = false;
      }
    } else {
      e.w32_resident = false;
      for (int d = 0; d < e.n_det && err == cudaSuccess; ++d) {
        err = cudaMemcpyAsync(e.d_data + 2 * (size_t)d * e.N, data_host[d], sizeof(double) * 2 * e.N, cudaMemcpyHostToDevice, e.copy);
        if (err == cudaSuccess)
          err = cudaMemcpyAsync(e.d_psd + (size_t)d * e.N, psd_host[d], sizeof(double) * e.N, cudaMemcpyHostToDevice, e.copy);
      }
    }
    if (err != cudaSuccess || (err = cudaEventRecord(e.ev_data, e.copy)) != cudaSuccess) { rc = cuda_fail(err, "copy strain"); break; }
    if (W > 0) {
      if ((err = ws_alloc(reinterpret_cast<void**>(&d_theta), sizeof(double) * kNPar * W, s)) != cudaSuccess) { rc = cuda_fail(err, "workspace allocation (theta)"); break; }
      if (!out.direct) {
        if ((err = ws_alloc(reinterpret_cast<void**>(&d_logl), sizeof(double) * W, s)) != cudaSuccess) { rc = cuda_fail(err, "workspace allocation (logl)"); break; }
        if (grad_host && (err = ws_alloc(reinterpret_cast<void**>(&d_grad), sizeof(double) * kNPar * W, s)) != cudaSuccess) { rc = cuda_fail(err, "workspace allocation (grad)"); break; }
      }
      if ((err = cudaMemcpyAsync(d_theta, theta_host, sizeof(double) * kNPar * W, cudaMemcpyHostToDevice, s)) != cudaSuccess) { rc = cuda_fail(err, "copy theta"); break; }
    }
    rc = rebuild_and_batch(e, d_theta, W, out.direct ? out.logl : d_logl, out.direct ? out.grad : d_grad, mode, s,
                           e.ev_data);
    if (rc != RB_OK || W == 0 || out.direct) break;
    if ((err = cudaMemcpyAsync(logl_host, d_logl, sizeof(double) * W, cudaMemcpyDeviceToHost, s)) != cudaSuccess) { rc = cuda_fail(err, "copy logl"); break; }
    if (grad_host && (err = cudaMemcpyAsync(grad_host, d_grad, sizeof(double) * kNPar * W, cudaMemcpyDeviceToHost, s)) != cudaSuccess) { rc = cuda_fail(err, "copy grad"); break; }
  } while (false);
  // the copy stream is joined into `stream` (also when the rebuild failed early)
  cudaStreamWaitEvent(s, e.ev_data, 0);
  if (d_theta) cudaFreeAsync(d_theta, s);
  if (d_logl) cudaFreeAsync(d_logl, s);
  if (d_grad) cudaFreeAsync(d_grad, s);
  err = cudaStreamSynchronize(s);
  if (rc == RB_OK && err != cudaSuccess) rc = cuda_fail(err, "synchronise");
  return rc;
}

int rb_strain(const double* geom, double gmst, const double* theta_host, double T, int64_t kmin, int64_t n_freq,
              double* h_dev, void* stream) {
  RB_NVTX("rb_strain");
  if (!geom || !theta_host || !h_dev) return set_error(RB_EINVAL, "rb_strain: NULL argument");
  if (!(T > 0.0) || n_freq < 1 || kmin < 1) return set_error(RB_EINVAL, "rb_strain: invalid grid");
  cudaStream_t s = (cudaStream_t)stream;
  EventConst ec;
  std::memset(&ec, 0, sizeof(ec));
  ec.n_det = 1;
  ec.gmst = gmst;
  split_pair(gmst, ec.gmst2);
  ec.det[0] = make_geom(geom[0], geom[1], geom[2], geom[3], geom[4]);
  double* d_theta = nullptr;
  RefValues* d_src = nullptr;
  int rc = RB_OK;
  cudaError_t err;
  do {
    if ((err = ws_alloc(reinterpret_cast<void**>(&d_theta), sizeof(double) * kNPar, s)) != cudaSuccess) { rc = cuda_fail(err, "workspace allocation (theta)"); break; }
    if ((err = ws_alloc(reinterpret_cast<void**>(&d_src), sizeof(RefValues), s)) != cudaSuccess) { rc = cuda_fail(err, "workspace allocation (values)"); break; }
    if ((err = cudaMemcpyAsync(d_theta, theta_host, sizeof(double) * kNPar, cudaMemcpyHostToDevice, s)) != cudaSuccess) { rc = cuda_fail(err, "copy theta"); break; }
    if ((err = launch_ref_values(d_theta, ec, d_src, s)) != cudaSuccess) { rc = cuda_fail(err, "values kernel"); break; }
    if ((err = launch_strain(d_src, kmin, n_freq, T, h_dev, s)) != cudaSuccess) { rc = cuda_fail(err, "strain kernel"); break; }
    count_launches(2);
  } while (false);
  if (d_theta) cudaFreeAsync(d_theta, s);
  if (d_src) cudaFreeAsync(d_src, s);
  return rc;
}

}  // extern "C"

namespace rb {

int rebuild_event(EventEntry& e, const DataPtrs* in_opt, int mode, cudaStream_t s, const SideSetup* ss, bool chunk_h0) {
  cudaError_t err;
  DataPtrs in{};
  if (in_opt) {
    in = *in_opt;
  } else {
    for (int d = 0; d < e.n_det; ++d) {
      in.data[d] = e.d_data + 2 * (size_t)d * e.N;
      in.psd[d] = e.d_psd + (size_t)d * e.N;
    }
  }
  const bool fast = mode != RB_FP64 && e.kmin >= 1024 && e.N <= (int64_t(1) << 30);
  // FP64 sums with h0 generated: from FP64 Taylor chunks for a theta_ref given with the
  // call, where the grid admits them; otherwise (creation, or a rebuild behind a change
  // of theta_ref that kept h0 away) directly at every point, so that events keep the bits
  // they are created with.  Which of the two it was is saved with the event: loading
  // takes the same one.  (k_summary_chunk64 counts points from 0 Hz in 32 bits)
  const bool chunk64 = mode == RB_FP64 && chunk_h0 && !e.h0_valid && e.kmin >= 1024 && e.N <= (int64_t(1) << 30) &&
                       e.kmin < (int64_t(1) << 30) - kChunk;
  if (ss && !(fast && mode == RB_MIXED)) return set_error(RB_EINVAL, "overlapped set-up needs the mixed fast rebuild");
  // Both sets of reference values are rebuilt: the float-float set (mixed
  // path, fast summary) and the FP64 set (FP64 paths, FP64 summary).  The
  // one this summary does not read runs on a forked stream, joined below.
  if ((err = cudaEventRecord(e.ev_fork, s)) != cudaSuccess || (err = cudaStreamWaitEvent(e.side, e.ev_fork, 0)) != cudaSuccess)
    return cuda_fail(err, "rebuild fork");
  int launches = 3;  // the two reference-value kernels and the summary kernel
  cudaStream_t ref_stream = e.side;  // where the FP64 reference set runs (joined by ev_join)
  // the float-float reference values head the critical path of the fast
  // rebuild: enqueued first
  if (fast && (err = launch_ref_dd(e.d_theta_ref, e.ec, e.d_ref, e.d_sync, s)) != cudaSuccess)
    return cuda_fail(err, "reference values kernel");
  if (ss && ss->grad) {
    // the tangents depend on theta only: on their own stream from the start
    if ((err = cudaStreamWaitEvent(e.tanst, e.ev_fork, 0)) != cudaSuccess) return cuda_fail(err, "rebuild fork");
    if ((err = launch_tangents(ss->theta, ss->W, e.ec, ss->tan, e.tanst)) != cudaSuccess) return cuda_fail(err, "tangent kernel");
    if ((err = cudaEventRecord(e.ev_tan, e.tanst)) != cudaSuccess) return cuda_fail(err, "rebuild join");
    ++launches;
  }
  if (fast) {
    if (!ss && (err = launch_ref_values(e.d_theta_ref, e.ec, e.d_ref, e.side)) != cudaSuccess)
      return cuda_fail(err, "reference values kernel");
    if (ss) {
      // the walkers' set-up reads the float-float reference values and theta
      // only: on the forked stream, launched as soon as they exist so that its
      // blocks are resident before the summary sums fill the GPU
      if ((err = cudaEventRecord(e.ev_ref, s)) != cudaSuccess || (err = cudaStreamWaitEvent(e.side, e.ev_ref, 0)) != cudaSuccess)
        return cuda_fail(err, "rebuild fork");
      if ((err = launch_setup(RB_MIXED, ss->theta, ss->W, e.ec, e.d_ref, ss->ws, nullptr, false, e.side)) != cudaSuccess)
        return cuda_fail(err, "set-up kernel");
      if ((err = cudaEventRecord(e.ev_setup, e.side)) != cudaSuccess) return cuda_fail(err, "rebuild join");
      // the FP64 set (off the critical path) behind the tangents, which end
      // early: behind the set-up it ran into the start of the likelihood
      // kernel, whose blocks each need a whole SM, and held one back
      ref_stream = ss->grad ? e.tanst : e.side;
      if ((err = launch_ref_values(e.d_theta_ref, e.ec, e.d_ref, ref_stream)) != cudaSuccess)
        return cuda_fail(err, "reference values kernel");
      ++launches;
    }
  } else {
    if ((err = launch_ref_dd(e.d_theta_ref, e.ec, e.d_ref, nullptr, e.side)) != cudaSuccess) return cuda_fail(err, "reference values kernel");
    // the streamed FP64 build (stored h0) does not read the reference values:
    // they are then rebuilt on the forked stream too
    if ((err = launch_ref_values(e.d_theta_ref, e.ec, e.d_ref, e.h0_valid ? e.side : s)) != cudaSuccess)
      return cuda_fail(err, "reference values kernel");
  }
  if ((err = cudaEventRecord(e.ev_join, ref_stream)) != cudaSuccess) return cuda_fail(err, "rebuild join");
  if (fast) {
    // with the walkers' set-up on the forked stream (rebuild + batch), the
    // chunk records are a launch of their own that overlaps the set-up (and
    // any data copies still in flight: they read the reference values only);
    // otherwise the summary kernel forms them in-block
    if (ss) {
      if ((err = launch_chunk_coef(e.N, e.n_det, e.d_ref, e.d_chunkq, e.d_chunks, s)) != cudaSuccess)
        return cuda_fail(err, "chunk record kernel");
      ++launches;
    }
    // the FP32 working copy follows the data the sums are taken over: data
    // read in place are converted every time, the resident data only after
    // they change
    if (ss && ss->data_ready && (err = cudaStreamWaitEvent(s, ss->data_ready, 0)) != cudaSuccess)
      return cuda_fail(err, "rebuild: wait for the data copies");
    if (in_opt || !e.w32_resident) {
      if ((err = launch_data32(in, e.N, e.n_det, e.d_w32, e.d_is32, e.d_wexp, s)) != cudaSuccess)
        return cuda_fail(err, "data conversion kernel");
      e.w32_resident = !in_opt;
      ++launches;
    }
    e.w32_current = true;
    err = launch_summary_parts(e.d_w32, e.d_is32, e.d_wexp, e.N, e.T, e.n_det, e.n_bins, e.d_edges, e.d_ref,
                               e.d_chunkq, ss ? e.d_chunks : nullptr, e.out(), s);
  } else if (chunk64) {
    // h0 generated from Taylor chunks, and stored for the next builds
    err = launch_summary_chunk64(in, e.d_h0, e.d_chunks, e.kmin, e.N, e.T, e.n_det, e.n_bins, e.d_edges, e.d_ref, e.out(),
                                 e.n_parts, s);
    e.h0_valid = err == cudaSuccess;
    e.h0_chunks = true;
    ++launches;
    e.w32_current = !in_opt && e.w32_resident;
  } else if (e.h0_valid) {
    // FP64 sums from the fiducial waveform stored by the last build that generated it
    // for this theta_ref: strain, PSD and h0 streamed, no waveform arithmetic;
    // its fixed-point sum starts from zero (a fast build leaves it set)
    if ((err = cudaMemsetAsync(&e.d_sync->base_acc, 0, sizeof(unsigned long long), s)) != cudaSuccess ||
        (err = cudaMemsetAsync(&e.d_sync->overflow, 0, sizeof(unsigned), s)) != cudaSuccess)
      return cuda_fail(err, "zero counters");
    err = launch_summary_stored(in, e.d_h0, e.N, e.T, e.n_det, e.n_bins, e.d_edges, e.out(), e.n_parts, s);
    e.w32_current = !in_opt && e.w32_resident;
  } else {
    // FP64 waveform evaluated at every point, and stored for the next builds
    err = launch_summary(in, e.kmin, e.N, e.T, e.n_det, e.n_bins, e.d_edges, e.d_ref, e.out(), e.d_h0, s);
    e.h0_valid = err == cudaSuccess;
    e.h0_chunks = false;
    e.w32_current = !in_opt && e.w32_resident;
  }
  e.last_in_place = in_opt != nullptr;
  if (err != cudaSuccess) return cuda_fail(err, "summary kernel");
  // with the overlapped set-up the caller's likelihood kernel waits for the
  // set-up (and tangents) only; it joins the FP64 reference set after that
  // kernel (finish_rebuild_join)
  if ((err = cudaStreamWaitEvent(s, ss ? e.ev_setup : e.ev_join, 0)) != cudaSuccess) return cuda_fail(err, "rebuild join");
  if (ss && ss->grad && (err = cudaStreamWaitEvent(s, e.ev_tan, 0)) != cudaSuccess) return cuda_fail(err, "rebuild join");
  count_launches(launches);
  return RB_OK;
}

static std::atomic<void*> g_trace_before{nullptr}, g_trace_after{nullptr};
bool trace_events_set() { return g_trace_before.load() != nullptr || g_trace_after.load() != nullptr; }
void set_trace_events(void* before, void* after) {
  g_trace_before.store(before);
  g_trace_after.store(after);
}

size_t walker_ws_bytes(int mode, bool grad) {
  size_t b = (mode == RB_MIXED) ? sizeof(WalkerMixed) : sizeof(WalkerF64);
  if (grad) b += (mode == RB_FP64) ? sizeof(WalkerTan<double>) : sizeof(WalkerTan<float>);
  return b;
}

// Set-up kernel + likelihood kernel for one batch.  If `scratch` is NULL the
// per-walker workspace is taken from the stream-ordered pool of `s`.
int run_batch(const EventEntry* e, const double* theta, int64_t W, double* logl, double* grad, int mode,
              cudaStream_t s, void* scratch, const MalaArgs* mala, bool spread) {
  if (!e) return set_error(RB_EINVAL, "NULL event");
  if (W < 0) return set_error(RB_EINVAL, "W < 0");
  if (mode != RB_MIXED && mode != RB_FP64 && mode != RB_MIXED_F64PHASE) return set_error(RB_EINVAL, "bad mode %d", mode);
  if (W == 0) return RB_OK;
  if (!theta || (!logl && !mala)) return set_error(RB_EINVAL, "NULL theta or logl");
  const bool want_grad = grad != nullptr || mala != nullptr;
  // set-up and likelihood in one launch where the batch allows it (not with
  // trace events, which bracket the likelihood kernel alone, nor for launches
  // that share the GPU with others, nor into theta's own memory: some blocks of that
  // kernel write results before others have read their walkers)
  const size_t theta_bytes = sizeof(double) * kNPar * W;
  if (mode == RB_MIXED && spread && !mala && !trace_events_set() && !overlap(theta, theta_bytes, logl, sizeof(double) * W) &&
      !(grad && overlap(theta, theta_bytes, grad, theta_bytes))) {
    bool done = false;
    const cudaError_t ferr = launch_rb_fused(e->dev, e->ec, theta, W, logl, grad, s, sm_count(), nullptr, &done);
    if (ferr != cudaSuccess) return cuda_fail(ferr, "likelihood kernel");
    if (done) {
      count_launches(1);
      return RB_OK;
    }
  }
  const size_t ws_bytes = (mode == RB_MIXED) ? sizeof(WalkerMixed) * W : sizeof(WalkerF64) * W;
  const size_t tan_bytes = !want_grad ? 0 : (mode == RB_FP64 ? sizeof(WalkerTan<double>) : sizeof(WalkerTan<float>)) * W;
  void* buf = scratch;
  cudaError_t err;
  if (!buf) {
    err = ws_alloc(reinterpret_cast<void**>(&buf), ws_bytes + tan_bytes, s);
    if (err != cudaSuccess) return cuda_fail(err, "workspace allocation");
  }
  void* ws = buf;
  void* tan = want_grad ? static_cast<void*>(static_cast<char*>(buf) + ws_bytes) : nullptr;
  int rc = RB_OK;
  err = launch_setup(mode, theta, W, e->ec, e->d_ref, ws, tan, want_grad, s);
  if (err == cudaSuccess) err = launch_batch_main(e, ws, tan, W, logl, grad, mode, spread, s, mala);
  if (err != cudaSuccess) rc = cuda_fail(err, "likelihood kernels");
  else count_launches(2);
  if (!scratch) cudaFreeAsync(buf, s);
  return rc;
}

// Rebuild from the resident data + batch, the walkers' set-up overlapped with
// the summary sums when the mixed chunk-expanded rebuild applies.  If
// data_ready is not NULL the resident data are complete only after it (the
// data-independent kernels run meanwhile).

int rebuild_and_batch(EventEntry& e, const double* theta, int64_t W, double* logl, double* grad, int mode,
                      cudaStream_t s, cudaEvent_t data_ready) {
  cudaError_t err;
  const bool overlap = W > 0 && mode == RB_MIXED && e.kmin >= 1024 && e.N <= (int64_t(1) << 30);
  if (!overlap) {  // the two calls in sequence
    if (data_ready && (err = cudaStreamWaitEvent(s, data_ready, 0)) != cudaSuccess)
      return cuda_fail(err, "wait for the data copies");
    int rc = rebuild_event(e, nullptr, mode, s);
    if (rc != RB_OK || W == 0) return rc;
    return run_batch(&e, theta, W, logl, grad, mode, s, nullptr);
  }
  const bool want_grad = grad != nullptr;
  if (want_grad && (err = ensure_stream(e.tanst, e.ev_tan)) != cudaSuccess) return cuda_fail(err, "tangent stream");
  const size_t ws_bytes = sizeof(WalkerMixed) * W, tan_bytes = want_grad ? sizeof(WalkerTan<float>) * W : 0;
  const size_t need = ws_bytes + tan_bytes;
  // the event's persistent workspace, grown when the stream is not being
  // captured; otherwise (or if too many buffers were outgrown) a per-call one
  if (e.step_ws_bytes < need) {
    cudaStreamCaptureStatus cs = cudaStreamCaptureStatusNone;
    if ((err = cudaStreamIsCapturing(s, &cs)) != cudaSuccess) return cuda_fail(err, "capture query");
    if (cs == cudaStreamCaptureStatusNone && e.n_step_ws_old < 16) {
      void* nb = nullptr;
      if ((err = cudaMalloc(&nb, need)) != cudaSuccess) return cuda_fail(err, "workspace allocation");
      if (e.step_ws) e.step_ws_old[e.n_step_ws_old++] = e.step_ws;
      e.step_ws = nb;
      e.step_ws_bytes = need;
    }
  }
  const bool own = e.step_ws_bytes >= need;
  void* buf = own ? e.step_ws : nullptr;
  if (!own && (err = ws_alloc(reinterpret_cast<void**>(&buf), need, s)) != cudaSuccess)
    return cuda_fail(err, "workspace allocation");
  void* tan = want_grad ? static_cast<void*>(static_cast<char*>(buf) + ws_bytes) : nullptr;
  const SideSetup ss{theta, W, buf, tan, want_grad, data_ready};
  int rc = rebuild_event(e, nullptr, mode, s, &ss);
  if (rc == RB_OK) {
    if ((err = launch_batch_main(&e, buf, tan, W, logl, grad, mode, true, s, nullptr)) != cudaSuccess)
      rc = cuda_fail(err, "likelihood kernel");
    else
      count_launches(1);
    // the FP64 reference set (forked stream) is complete before anything
    // that follows this call on `s`
    if ((err = cudaStreamWaitEvent(s, e.ev_join, 0)) != cudaSuccess && rc == RB_OK) rc = cuda_fail(err, "rebuild join");
  }
  if (!own) cudaFreeAsync(buf, s);
  return rc;
}

cudaError_t launch_batch_main(const EventEntry* e, void* ws, void* tan, int64_t W, double* logl, double* grad, int mode,
                              bool spread, cudaStream_t s, const MalaArgs* mala) {
  const int n_sm = sm_count();
  cudaEvent_t tb = static_cast<cudaEvent_t>(g_trace_before.load());
  cudaEvent_t ta = static_cast<cudaEvent_t>(g_trace_after.load());
  cudaError_t err = tb ? cudaEventRecord(tb, s) : cudaSuccess;
  if (err == cudaSuccess) {
    if (mode == RB_FP64)
      err = launch_rb_f64(e->dev, ws, tan, W, logl, grad, s, n_sm, mala);
    else
      err = launch_rb_mixed(e->dev, ws, tan, W, logl, grad, mode == RB_MIXED_F64PHASE, spread, s, n_sm, mala);
  }
  if (err == cudaSuccess && ta) err = cudaEventRecord(ta, s);
  return err;
}

}  // namespace rb
