// kf_chain.cu -- fused multi-layer chain: each track runs propagate + update
// through L detector layers inside one kernel (paper section 2 and the
// per-track layer loop of Figs. 3-5: for each layer, propagateTo{R,Z} then
// KalmanUpdate).
//
// One thread owns one track for the whole chain: state, covariance and
// charge are loaded once, kept in registers across all layers, and written
// back once; only the per-layer hits stream in (the next layer's hit is
// loaded while the current layer computes).  Per track that is 109 B in,
// 36 B per layer and 108 B out, against 253 B per layer for L separate
// single-step launches that round-trip the state through HBM.  The layer
// kind is uniform across the grid, so the p2z / p2r branch never diverges.
#include <cuda_runtime.h>

#include <atomic>
#include <cstdint>
#include <mutex>

#include "kf_common.cuh"
#include "kf_device.cuh"
#include "kf_step.cuh"
#include "kf_chain.cuh"
#include "kf_chain_kernel.cuh"
#include "kf_fp64_group.cuh"

namespace kf {
namespace staged {
// SM count of a device (cached; kf_step_staged.cu)
int sm_count(int dev, int *out);
}  // namespace staged

namespace {

// Tracks whose marks a block of the second pass gathers.
constexpr int kChainSpan = 2048;

// KF_ADAPTIVE's second pass for one marked track: the whole chain again
// from its (untouched) inputs, in double (chain_track_fp64).
__device__ __forceinline__ void chain_redo_track(const ChainArgs &a, int64_t i) {
  const ChainLoc l6 = chain_locate<6>(i, a.n, a.soa, a.lw);
  const ChainLoc l21 = chain_locate<21>(i, a.n, a.soa, a.lw);
  const ChainLoc l3 = chain_locate<3>(i, a.n, a.soa, a.lw);
  float p[6], C[21];
  for (int c = 0; c < 6; ++c) p[c] = a.state[l6.base + c * l6.stride];
  for (int e = 0; e < 21; ++e) C[e] = a.cov[l21.base + e * l21.stride];
  const float qf = (float)a.charge[i];
  unsigned st = chain_track_fp64(p, C, qf, a.bz, a.L, a.kinds, a.pos, a.hits, a.hit_stride,
                                 a.hitcovs, a.hc_stride, l3, l6);
  st |= finite_status(p, C);
  for (int c = 0; c < 6; ++c) a.state[l6.base + c * l6.stride] = p[c];
  for (int e = 0; e < 21; ++e) a.cov[l21.base + e * l21.stride] = C[e];
  a.status[i] = (uint8_t)st;
}

// The same for 32 tracks by the block's four warps (kf_fp64_group.cuh).
__device__ __forceinline__ void chain_redo_group(const ChainArgs &a, const f64::Group &g,
                                                 int64_t i, bool store) {
  const ChainLoc l6 = chain_locate<6>(i, a.n, a.soa, a.lw);
  const ChainLoc l21 = chain_locate<21>(i, a.n, a.soa, a.lw);
  const ChainLoc l3 = chain_locate<3>(i, a.n, a.soa, a.lw);
  const unsigned st =
      f64::group_chain(g, {a.state, a.cov, a.state, a.cov, l6, l21}, (float)a.charge[i], a.bz, a.L,
                       a.kinds, a.pos, a.hits, a.hit_stride, a.hitcovs, a.hc_stride, l3, store);
  if (g.role == 0 && store && a.status) a.status[i] = (uint8_t)st;
}

// The second pass over one list of the whole batch's marked tracks, which the
// first pass appends to (an atomic per marked track; the order of the list
// varies from run to run, the result of each track does not).
constexpr int kRedoListBlocksPerSm = 4;
// Up to this many tracks per SM four warps share 32 tracks of a KF_FP64 chain,
// beyond it each thread runs a track (chain_kernel).  15 layers, us: one group
// per SM (up to 4,864 tracks) 91, two 122, three 167, four 214; one thread per
// track 163 up to 10,000 tracks, 175 up to 19,000.
constexpr int kGroupTracksPerSm = 96;
// The same line for the list, whose kernel has 128 registers where a thread's
// track wants 150, and whose blocks land where the first pass leaves room.
// Adaptive chain, four warps against one thread: 2.6 M tracks (17,000 listed)
// 809 and 916 us, 5 M (33,000) 1,555 and 1,610, 8 M (52,000, 345 per SM) 2,377
// and 2,434, 9.5 M (62,000, 410 per SM) 2,838 and 2,769, 13 M 3,829 and 3,693.
constexpr int kListGroupTracksPerSm = 384;

__global__ void __launch_bounds__(f64::kGroupThreads, kRedoListBlocksPerSm)
    chain_redo_list_kernel(const __grid_constant__ ChainArgs a) {
  __shared__ f64::Shared sh;
  // the marking pass's list, complete once that kernel is
  asm volatile("griddepcontrol.wait;" ::: "memory");
  const int64_t total = *a.redo_count;
  const uint32_t *list = a.redo_list;
  if (total > (int64_t)(gridDim.x / kRedoListBlocksPerSm) * kListGroupTracksPerSm) {
    for (int64_t q = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; q < total;
         q += (int64_t)gridDim.x * blockDim.x)
      chain_redo_track(a, list[q]);
    return;
  }
  const f64::Group g{sh, (int)threadIdx.x >> 5, (int)threadIdx.x & 31};
  for (int64_t base = (int64_t)blockIdx.x * 32; base < total; base += (int64_t)gridDim.x * 32)
    chain_redo_group(a, g, list[f64::group_place(base, total, g.lane)], base + g.lane < total);
}

// KF_ADAPTIVE's second pass without a list (no scratch memory could be had,
// or more than 2^32 - 1 tracks): each block gathers the marked tracks of its
// span (gather_marked) and reruns them.
__global__ void __launch_bounds__(f64::kGroupThreads, 4) chain_redo_kernel(const ChainArgs a) {
  __shared__ f64::Shared sh;
  __shared__ uint16_t list[kChainSpan];
  __shared__ int count;
  const int64_t span0 = (int64_t)blockIdx.x * kChainSpan;
  const int cnt = gather_marked<kChainSpan, f64::kGroupThreads>(a.status, span0, a.n, list, &count);
  if (cnt > f64::kGroupMax) {
    for (int q = threadIdx.x; q < cnt; q += blockDim.x) chain_redo_track(a, span0 + list[q]);
    return;
  }
  const f64::Group g{sh, (int)threadIdx.x >> 5, (int)threadIdx.x & 31};
  for (int base = 0; base < cnt; base += 32)
    chain_redo_group(a, g, span0 + list[f64::group_place(base, cnt, g.lane)],
                     base + g.lane < cnt);
}

// KF_FP64 for batches too small to give every scheduler a warp of tracks.
__global__ void __launch_bounds__(f64::kGroupThreads, kRedoListBlocksPerSm)
    chain_group_kernel(const ChainArgs a) {
  __shared__ f64::Shared sh;
  const f64::Group g{sh, (int)threadIdx.x >> 5, (int)threadIdx.x & 31};
  const int64_t base = (int64_t)blockIdx.x * 32;
  chain_redo_group(a, g, f64::group_place(base, a.n, g.lane), base + g.lane < a.n);
}

// A stream-ordered memory pool per device for the second pass's list,
// created on first use and kept (with its memory: release threshold at the
// maximum) for the life of the process.  It is not created while the
// stream is being captured into a graph (creating a pool is not a
// capturable call); allocating from an existing pool is, and gives the
// graph an allocation node.
constexpr int kMaxPoolDevices = 64;
std::mutex g_redo_pool_mu;
cudaMemPool_t g_redo_pool[kMaxPoolDevices] = {};

bool redo_pool(int dev, bool may_create, cudaMemPool_t *out) {
  if (dev < 0 || dev >= kMaxPoolDevices) return false;
  std::lock_guard<std::mutex> lock(g_redo_pool_mu);
  if (!g_redo_pool[dev]) {
    if (!may_create) return false;
    cudaMemPoolProps props = {};
    props.allocType = cudaMemAllocationTypePinned;
    props.location.type = cudaMemLocationTypeDevice;
    props.location.id = dev;
    cudaMemPool_t pool = nullptr;
    if (cudaMemPoolCreate(&pool, &props) != cudaSuccess) {
      (void)cudaGetLastError();
      return false;
    }
    uint64_t keep = UINT64_MAX;
    (void)cudaMemPoolSetAttribute(pool, cudaMemPoolAttrReleaseThreshold, &keep);
    g_redo_pool[dev] = pool;
  }
  *out = g_redo_pool[dev];
  return true;
}

std::atomic<int> g_chain_redo{KF_CHAIN_REDO_LIST};

// Give the first pass a list for the tracks it marks, its count zeroed on
// stream s: stream-ordered scratch, to be returned with cudaFreeAsync.  False
// (and no list) when the marks alone have to do.
bool start_redo_list(ChainArgs &a, int dev, cudaStream_t s) {
  cudaMemPool_t pool = nullptr;
  void *buf = nullptr;
  cudaStreamCaptureStatus capture = cudaStreamCaptureStatusNone;
  const bool capturing = cudaStreamIsCapturing(s, &capture) != cudaSuccess ||
                         capture != cudaStreamCaptureStatusNone;
  if (g_chain_redo.load(std::memory_order_relaxed) == KF_CHAIN_REDO_LIST &&
      a.n < (int64_t)UINT32_MAX && redo_pool(dev, !capturing, &pool) &&
      cudaMallocFromPoolAsync(&buf, 4 * (size_t)(a.n + 1), pool, s) == cudaSuccess) {
    if (cudaMemsetAsync(buf, 0, sizeof(uint32_t), s) == cudaSuccess) {
      a.redo_count = static_cast<uint32_t *>(buf);
      a.redo_list = a.redo_count + 1;
      return true;
    }
    (void)cudaFreeAsync(buf, s);
  }
  (void)cudaGetLastError();  // a refused allocation is not the caller's error
  return false;
}

// KF_ADAPTIVE: the marking pass, then the second pass over its list, or per
// span where there is none (the same results).
int launch_chain_adaptive(ChainArgs &a, unsigned blocks, int threads, int dev, int sms,
                          cudaStream_t s) {
  const bool list = start_redo_list(a, dev, s);
  int rc = launch_chain_mark(a, blocks, threads, s);
  if (rc == KF_OK) {
    if (list) {
      // a programmatic dependent: set up while the marking pass drains
      cudaLaunchConfig_t cfg = {};
      cfg.gridDim = dim3((unsigned)(kRedoListBlocksPerSm * sms));
      cfg.blockDim = dim3(f64::kGroupThreads);
      cfg.stream = s;
      cudaLaunchAttribute attr[1];
      attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
      attr[0].val.programmaticStreamSerializationAllowed = 1;
      cfg.attrs = attr;
      cfg.numAttrs = 1;
      rc = check_cuda(cudaLaunchKernelEx(&cfg, chain_redo_list_kernel, a), "chain redo pass launch");
    } else {
      chain_redo_kernel<<<(unsigned)((a.n + kChainSpan - 1) / kChainSpan), f64::kGroupThreads, 0,
                          s>>>(a);
      rc = check_cuda(cudaGetLastError(), "chain redo pass launch");
    }
  }
  if (!list) return rc;
  const cudaError_t freed = cudaFreeAsync(a.redo_count, s);  // returned on every path
  return rc != KF_OK ? rc : check_cuda(freed, "cudaFreeAsync");
}

}  // namespace

bool chain_shares_warps(int precision, int64_t n, int sms) {
  return precision == KF_FP64 && n <= (int64_t)sms * kGroupTracksPerSm;
}

}  // namespace kf

extern "C" int kf_set_chain_redo(int32_t mode) {
  kf::clear_error();
  if (mode != KF_CHAIN_REDO_LIST && mode != KF_CHAIN_REDO_SPAN)
    return kf::set_error(KF_ERR_ARG, "chain redo mode %d is neither KF_CHAIN_REDO_LIST nor "
                         "KF_CHAIN_REDO_SPAN", mode);
  kf::g_chain_redo.store(mode, std::memory_order_relaxed);
  return KF_OK;
}

extern "C" int kf_kalman_chain(const kf_params *params, kf_layout layout, float *state,
                               float *cov, const int8_t *charge, const float *hits,
                               const float *hit_covs, const kf_layer *layers, int32_t L,
                               uint8_t *status, void *stream) {
  using namespace kf;
  clear_error();
  if (!params) return set_error(KF_ERR_ARG, "params is NULL");
  if (params->flags != 0) return set_error(KF_ERR_ARG, "params->flags must be 0");
  if (params->precision < KF_FP32 || params->precision > KF_DF_UPDATE)
    return set_error(KF_ERR_ARG, "unknown precision %d", params->precision);
  LayoutDesc d;
  if (int rc = check_layout(layout, &d)) return rc;
  if (L < 0 || L > KF_MAX_LAYERS)
    return set_error(KF_ERR_ARG, "L = %d not in [0, %d]", L, KF_MAX_LAYERS);
  if (d.n == 0 || L == 0) return KF_OK;
  if (!layers) return set_error(KF_ERR_ARG, "layers is NULL");
  ChainArgs a{};
  for (int l = 0; l < L; ++l) {
    if (layers[l].kind != KF_P2Z && layers[l].kind != KF_P2R)
      return set_error(KF_ERR_ARG, "layers[%d].kind = %d is neither KF_P2Z nor KF_P2R", l,
                       layers[l].kind);
    a.kinds[l] = layers[l].kind;
    a.pos[l] = layers[l].pos;
  }
  if (!aligned16(state) || !aligned16(cov) || !aligned16(hits) || !aligned16(hit_covs))
    return set_error(KF_ERR_ARG, "float arrays must be 16-byte aligned");
  const int64_t f3 = layout_floats(d, 3), f6 = layout_floats(d, 6), f21 = layout_floats(d, 21);
  if (int rc = check_device_range(state, 4 * f6, "state")) return rc;
  if (int rc = check_device_range(cov, 4 * f21, "cov")) return rc;
  if (int rc = check_device_range(charge, d.n, "charge")) return rc;
  if (int rc = check_device_range(hits, 4 * f3 * L, "hits")) return rc;
  if (int rc = check_device_range(hit_covs, 4 * f6 * L, "hit_covs")) return rc;
  if (status)
    if (int rc = check_device_range(status, d.n, "status")) return rc;
  if (!status && params->precision == KF_ADAPTIVE)
    return set_error(KF_ERR_ARG, "KF_ADAPTIVE needs a status array (its redo pass reads it)");

  a.state = state;
  a.cov = cov;
  a.charge = charge;
  a.hits = hits;
  a.hitcovs = hit_covs;
  a.status = status;
  a.n = d.n;
  a.hit_stride = f3;
  a.hc_stride = f6;
  a.soa = d.soa;
  a.lw = d.lw;
  a.bz = params->bz;
  a.L = L;
  int dev = 0, sms = 0;
  if (int rc = check_cuda(cudaGetDevice(&dev), "cudaGetDevice")) return rc;
  if (int rc = staged::sm_count(dev, &sms)) return rc;
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  if (chain_shares_warps(params->precision, d.n, sms)) {
    chain_group_kernel<<<(unsigned)((d.n + 31) / 32), f64::kGroupThreads, 0, s>>>(a);
    return check_cuda(cudaGetLastError(), "chain launch");
  }
  // CTA size: 64 threads spread a small batch over the SMs and waste least in
  // the last wave (us with 64, 128, 256 threads: FP32 5,000 tracks 15.0, 15.0,
  // 17.1, 440,000: 107, 107, 111; FP64 update 60,000: 144, 160, 160; KF_FP64
  // 20,000: 250, 322, 320).  The double-float update leads with 256 once the
  // device is full (60,000: 45.7, 45.7, 43.6; 1.75 M: 899, 889, 834) and with
  // 128 before (5,000: 25.2, 25.2, 27.3).
  const int df_threads = d.n > (int64_t)128 * sms ? 256 : 128;
  LaunchConfig cfg{KF_STEP_DIRECT, params->precision == KF_DF_UPDATE ? df_threads : 64, 0};
  if (const LaunchConfig *o = thread_override()) {
    cfg = *o;
  } else {
    LaunchConfig t;
    if (tune_lookup(kOpChain, 0, params->precision, d.soa, d.lw, d.n, &t)) cfg = t;
  }
  const int threads = (cfg.threads == 128 || cfg.threads == 64) ? cfg.threads : 256;
  const int64_t blocks = (d.n + threads - 1) / threads;
  if (blocks > 0x7fffffffLL) return set_error(KF_ERR_ARG, "n too large for one launch");
  const unsigned g = (unsigned)blocks;
  int rc = KF_OK;
  switch (params->precision) {
    case KF_FP32: rc = launch_chain_fp32(a, g, threads, s); break;
    case KF_ADAPTIVE: return launch_chain_adaptive(a, g, threads, dev, sms, s);
    case KF_FP64_UPDATE: chain_kernel<kFP64Update, 0><<<g, threads, 0, s>>>(a); break;
    case KF_JOSEPH: rc = launch_chain_joseph(a, g, threads, s); break;
    case KF_FP64: chain_kernel<kFP64, 0><<<g, threads, 0, s>>>(a); break;
    default: rc = launch_chain_df(a, g, threads, s); break;
  }
  if (rc != KF_OK) return rc;
  return check_cuda(cudaGetLastError(), "chain launch");
}
