// Allocation-free direct sum (dwfmm_direct_sum_noalloc): y = K x over all N
// sites, no tree.
//
// Some callers cannot call cudaMalloc: host applications whose framework
// owns the device memory pool (a caching allocator that has reserved nearly
// all of it, so a fresh cudaMalloc fails or fragments the pool), and
// latency-sensitive loops that cannot afford the device synchronisation
// that cudaMalloc/cudaFree imply.
//
// One CTA sums for 32 targets, one per lane; its 8 warps take 32 sources each
// of every staged tile of 256, four at a time in packed pairs, and add up at
// the end.  32 targets per CTA rather than 256 spread N = 1021 over 32 SMs
// instead of 4 (43 -> 6 us of kernel time); the sums need no other launch,
// because the CTA writes y itself.
//
// Up to kRawMaxN sites (y apart from the sites and charges) every CTA converts the float64 sites as it stages them:
// one launch, no scratch.  Above, those conversions (n d per CTA on a unit of
// 2 a clock) would cost more than the launch they save, so a first kernel
// leaves scaled float32 coordinates and charges in a file-scope array.  That
// array is shared by every call on a device; each call rewrites what it reads,
// and calls whose work overlaps on the GPU race on it.
#include <atomic>
#include <cmath>
#include <cstdint>
#include <string>

#include "dwfmm_internal.cuh"
#include "sum_f32.cuh"

namespace dw {

namespace {

using namespace sk;

constexpr int kNaThreads = 256;
constexpr int kNaWarps = kNaThreads / 32;
constexpr int kNaTile = 256;                        // sources staged at a time, 32 per warp
constexpr int kNaFold = 4;                          // tiles summed before the compensated sums take them
constexpr int kNaMaxN = 8192;                       // largest N
constexpr int kNaMaxD = 16;                         // largest d (padded dimension <= 16)
constexpr int kRawMaxN = 1536;
constexpr size_t kNaFloats = static_cast<size_t>(kNaMaxN) * (kNaMaxD + 1 + kRC);

static __device__ __align__(256) float g_noalloc_scratch[kNaFloats];

struct NaArgs {
  const double* pts;
  int n, d;
  int64_t ldp;
  double scale;
  const double* x;
  double* y;
  int R;
  int64_t ldx, ldy;
  float* scratch;   // [D + 1 + RC][npad] coordinates, squared norms, charges; not used on the raw path
  int npad;         // n rounded up to kNaTile
  bool raw;         // one launch on the caller's buffers
};

double coordinate_scale(int kernel, double sigma) {
  if (kernel == DWFMM_K_GAUSS) return std::sqrt(1.4426950408889634 / (2.0 * sigma * sigma));
  if (kernel == DWFMM_K_EXP) return 1.4426950408889634 / sigma;
  return 1.7320508075688772 / sigma;
}

// Scaled coordinates, squared norm and charges of site j, `stride` floats
// apart (sites from n on repeat the first with zero charges).
template <int D, int RC>
__device__ __forceinline__ void na_load(const NaArgs& a, int j, float* dst, int stride) {
  const int64_t s = j < a.n ? j : 0;
  double n2 = 0.0;
#pragma unroll
  for (int k = 0; k < D; ++k) {
    const float f = k < a.d ? static_cast<float>(a.pts[s * a.ldp + k] * a.scale) : 0.0f;
    dst[k * stride] = f;
    n2 += static_cast<double>(f) * static_cast<double>(f);
  }
  dst[D * stride] = static_cast<float>(n2);
#pragma unroll
  for (int r = 0; r < RC; ++r)
    dst[(D + 1 + r) * stride] = (j < a.n && r < a.R) ? static_cast<float>(a.x[r * a.ldx + j]) : 0.0f;
}

template <int D, int RC>
__global__ void k_na_prepare(const NaArgs a) {
  const int j = static_cast<int>(blockIdx.x) * blockDim.x + threadIdx.x;
  if (j < a.npad) na_load<D, RC>(a, j, a.scratch + j, a.npad);
}

template <int D, int RC>
constexpr size_t na_smem() {
  return (static_cast<size_t>(D + 1 + RC) * kNaTile + 2 * static_cast<size_t>(RC) * kNaThreads) * sizeof(float);
}

template <int D, int RC, int KER, bool RAW>
__global__ void __launch_bounds__(kNaThreads, RC > 4 ? 2 : 3) k_na_sum(const NaArgs a) {
  constexpr int ROWS = D + 1 + RC;
  extern __shared__ __align__(16) float nsm[];
  float* tile = nsm;                          // [ROWS][kNaTile]
  float* ks = nsm + ROWS * kNaTile;           // [RC][kNaThreads] compensated sums
  float* kc = ks + RC * kNaThreads;           // [RC][kNaThreads]
  const int tid = static_cast<int>(threadIdx.x), warp = tid >> 5, lane = tid & 31;
  const int i = static_cast<int>(blockIdx.x) * 32 + lane;
  u64 x2[D], nt2;   // the target, (c x_k, c x_k), c = 2 for the Gaussian, and -(|x|^2, |x|^2)
  {
    float v[ROWS];
    if constexpr (RAW) {
      na_load<D, RC>(a, i, v, 1);
    } else {
      const int t = i < a.n ? i : 0;
#pragma unroll
      for (int k = 0; k <= D; ++k) v[k] = a.scratch[static_cast<int64_t>(k) * a.npad + t];
    }
#pragma unroll
    for (int k = 0; k < D; ++k) {
      const float f = KER == DWFMM_K_GAUSS ? 2.0f * v[k] : v[k];
      x2[k] = pk2(f, f);
    }
    nt2 = pk2(-v[D], -v[D]);
  }
#pragma unroll
  for (int r = 0; r < RC; ++r) ks[r * kNaThreads + tid] = kc[r * kNaThreads + tid] = 0.0f;
  u64 acc[RC];
#pragma unroll
  for (int r = 0; r < RC; ++r) acc[r] = 0ull;
  auto fold = [&]() {
#pragma unroll
    for (int r = 0; r < RC; ++r) {
      float f0, f1;
      up2(acc[r], f0, f1);
      acc[r] = 0ull;
      float* s = ks + r * kNaThreads + tid;
      float* c = kc + r * kNaThreads + tid;
      const float v = (f0 + f1) - *c, t = *s + v;
      *c = (t - *s) - v;
      *s = t;
    }
  };
  for (int t0 = 0, nt = 0; t0 < a.n; t0 += kNaTile) {
    __syncthreads();
    if constexpr (RAW) {
      na_load<D, RC>(a, t0 + tid, tile + tid, kNaTile);
    } else {
      for (int q = tid; q < ROWS * (kNaTile / 4); q += kNaThreads) {
        const int row = q / (kNaTile / 4), col = q % (kNaTile / 4);
        reinterpret_cast<float4*>(tile)[q] =
            reinterpret_cast<const float4*>(a.scratch + static_cast<int64_t>(row) * a.npad + t0)[col];
      }
    }
    __syncthreads();
    const int j1 = min(32, a.n - t0 - warp * 32);   // the tail's padding is whole groups of 4 with zero charges
    const float* w = tile + warp * 32;
    for (int j = 0; j < j1; j += 4) {
      u64 e0, e1;
      if (KER == DWFMM_K_GAUSS) {
        const ulonglong2 ns = *reinterpret_cast<const ulonglong2*>(w + D * kNaTile + j);
        e0 = fsub2(nt2, ns.x);
        e1 = fsub2(nt2, ns.y);
      } else {
        e0 = e1 = 0ull;
      }
#pragma unroll
      for (int k = 0; k < D; ++k) {
        const ulonglong2 sv = *reinterpret_cast<const ulonglong2*>(w + k * kNaTile + j);
        if (KER == DWFMM_K_GAUSS) {
          e0 = ffma2(x2[k], sv.x, e0);
          e1 = ffma2(x2[k], sv.y, e1);
        } else {
          const u64 d0 = fsub2(x2[k], sv.x), d1 = fsub2(x2[k], sv.y);
          e0 = ffma2(d0, d0, e0);
          e1 = ffma2(d1, d1, e1);
        }
      }
      float p0, p1, p2, p3;
      up2(e0, p0, p1);
      up2(e1, p2, p3);
      const u64 f0 = pk2(phi_scaled<KER>(p0), phi_scaled<KER>(p1)), f1 = pk2(phi_scaled<KER>(p2), phi_scaled<KER>(p3));
#pragma unroll
      for (int r = 0; r < RC; ++r) {
        const ulonglong2 q = *reinterpret_cast<const ulonglong2*>(w + (D + 1 + r) * kNaTile + j);
        acc[r] = ffma2(f0, q.x, acc[r]);
        acc[r] = ffma2(f1, q.y, acc[r]);
      }
    }
    if (++nt % kNaFold == 0) fold();
  }
  fold();
  __syncthreads();
  // the warps' sums of each target, in order
  for (int o = tid; o < 32 * RC; o += kNaThreads) {
    const int r = o >> 5, t = o & 31, at = r * kNaThreads + t;
    if (r >= a.R || static_cast<int>(blockIdx.x) * 32 + t >= a.n) continue;
    float s = ks[at], c = kc[at];
#pragma unroll
    for (int u = 1; u < kNaWarps; ++u) {
      const float v = ks[at + 32 * u] - (kc[at + 32 * u] + c), z = s + v;
      c = (z - s) - v;
      s = z;
    }
    a.y[r * a.ldy + static_cast<int64_t>(blockIdx.x) * 32 + t] = static_cast<double>(s) - static_cast<double>(c);
  }
}

template <int D, int RC, int KER>
void na_launch_k(const NaArgs& a, cudaStream_t s) {
  const int grid = ceil_div(a.n, 32);
  if (a.raw) {
    k_na_sum<D, RC, KER, true><<<grid, kNaThreads, na_smem<D, RC>(), s>>>(a);
    return;
  }
  k_na_prepare<D, RC><<<ceil_div(a.npad, 128), 128, 0, s>>>(a);
  k_na_sum<D, RC, KER, false><<<grid, kNaThreads, na_smem<D, RC>(), s>>>(a);
}

template <int D, int RC>
void na_launch(int kernel, const NaArgs& a, cudaStream_t s) {
  if (kernel == DWFMM_K_EXP) na_launch_k<D, RC, DWFMM_K_EXP>(a, s);
  else if (kernel == DWFMM_K_MATERN32) na_launch_k<D, RC, DWFMM_K_MATERN32>(a, s);
  else na_launch_k<D, RC, DWFMM_K_GAUSS>(a, s);
}

template <int D, int RC, int KER>
void na_attr_k() {
  const int b = static_cast<int>(na_smem<D, RC>());
  DW_CUDA(cudaFuncSetAttribute(k_na_sum<D, RC, KER, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, b));
  DW_CUDA(cudaFuncSetAttribute(k_na_sum<D, RC, KER, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, b));
}

template <int D, int RC>
void na_attr() {
  na_attr_k<D, RC, DWFMM_K_EXP>();
  na_attr_k<D, RC, DWFMM_K_MATERN32>();
  na_attr_k<D, RC, DWFMM_K_GAUSS>();
}

// f.template operator()<D, RC>() for the padded sizes.
#define DW_NA_RC(DV, CALL)                            \
  switch (RC) {                                       \
    case 1: CALL(DV, 1); break;                       \
    case 4: CALL(DV, 4); break;                       \
    case 8: CALL(DV, 8); break;                       \
    default: CALL(DV, 16); break;                     \
  }
#define DW_NA_D(CALL)                                 \
  switch (D) {                                        \
    case 4: DW_NA_RC(4, CALL) break;                  \
    case 8: DW_NA_RC(8, CALL) break;                  \
    case 10: DW_NA_RC(10, CALL) break;                \
    case 12: DW_NA_RC(12, CALL) break;                \
    default: DW_NA_RC(16, CALL) break;                \
  }

void na_dispatch(int D, int RC, int kernel, const NaArgs& a, cudaStream_t s) {
#define DW_NA_GO(DV, RV) na_launch<DV, RV>(kernel, a, s)
  DW_NA_D(DW_NA_GO)
#undef DW_NA_GO
}

void na_attrs() {
  // the shapes whose shared memory passes the default limit
  for (int D : {4, 8, 10, 12, 16}) {
    const int RC = 16;
#define DW_NA_AT(DV, RV) na_attr<DV, RV>()
    DW_NA_D(DW_NA_AT)
#undef DW_NA_AT
  }
}
static_assert(na_smem<16, 8>() <= 48 * 1024, "the shapes below 16 right-hand sides fit the default limit");

// Device address of the scratch array.  Outside stream capture it is looked
// up on every call (cudaGetSymbolAddress allocates nothing), so a context
// that was reset still gets the right address; the last address seen per
// device serves calls made during capture, where the first call on a device
// must not load the module or set kernel attributes.
constexpr int kNaMaxDevices = 64;
std::atomic<float*> g_na_ptr[kNaMaxDevices];

float* na_scratch_for_current_device(int dev, cudaStream_t s) {
  if (dev < 0 || dev >= kNaMaxDevices) fail(DWFMM_ERR_INVALID_ARG, "device index out of range");
  cudaStreamCaptureStatus cap = cudaStreamCaptureStatusNone;
  DW_CUDA(cudaStreamIsCapturing(s, &cap));
  float* p = g_na_ptr[dev].load();
  if (cap != cudaStreamCaptureStatusNone) {
    if (!p)
      fail(DWFMM_ERR_STATE,
           "direct_sum_noalloc: the first call on a device sets it up and must come before any stream capture");
    return p;
  }
  if (!p) na_attrs();
  void* q = nullptr;
  DW_CUDA(cudaGetSymbolAddress(&q, g_noalloc_scratch));
  g_na_ptr[dev].store(static_cast<float*>(q));
  return static_cast<float*>(q);
}

// Buffers the kernels read or write directly: device (or managed) memory of
// the current device.  A host pointer would fault on the GPU.
void na_check_device_buffer(const void* p, int dev, const char* name) {
  cudaPointerAttributes a;
  const cudaError_t e = cudaPointerGetAttributes(&a, p);
  if (e != cudaSuccess) (void)cudaGetLastError();
  const bool ok = e == cudaSuccess &&
                  ((a.type == cudaMemoryTypeDevice && a.device == dev) || a.type == cudaMemoryTypeManaged);
  if (!ok)
    fail(DWFMM_ERR_INVALID_ARG, std::string("direct_sum_noalloc: ") + name +
                                    " must be device memory of the current device");
}

}  // namespace

dwfmm_status direct_sum_noalloc(int kernel, double sigma, const double* pts, int64_t n, int d, int64_t ldp,
                                const double* x, double* y, int R, int64_t ldx, int64_t ldy,
                                cudaStream_t s) {
  if (kernel < 0 || kernel > 2 || !(sigma > 0.0) || n < 0 || n > kNaMaxN || d < 1 || d > kNaMaxD ||
      R < 1 || R > kRC)
    fail(DWFMM_ERR_INVALID_ARG, "direct_sum_noalloc: needs N <= 8192, 1 <= d <= 16, 1 <= nrhs <= 16");
  if (n == 0) return DWFMM_OK;
  if (!pts || !x || !y || ldp < d || ldx < n || ldy < n)
    fail(DWFMM_ERR_INVALID_ARG, "direct_sum_noalloc: NULL buffer or leading dimension too small");
  int dev = 0;
  DW_CUDA(cudaGetDevice(&dev));
  na_check_device_buffer(pts, dev, "pts");
  na_check_device_buffer(x, dev, "x");
  na_check_device_buffer(y, dev, "y");
  NaArgs a{};
  a.pts = pts;
  a.n = static_cast<int>(n);
  a.d = d;
  a.ldp = ldp;
  a.scale = coordinate_scale(kernel, sigma);
  a.x = x;
  a.y = y;
  a.R = R;
  a.ldx = ldx;
  a.ldy = ldy;
  a.scratch = na_scratch_for_current_device(dev, s);
  a.npad = round_up(a.n, kNaTile);
  // y over the sites or the charges: they are read in full before y is written
  auto apart = [](const double* p, int64_t np, const double* q, int64_t nq) { return p + np <= q || q + nq <= p; };
  const int64_t ny = (R - 1) * ldy + n;
  a.raw = n <= kRawMaxN && apart(y, ny, x, (R - 1) * ldx + n) && apart(y, ny, pts, (n - 1) * ldp + d);
  na_dispatch(sum_padded_dim(d), sum_padded_rc(R), kernel, a, s);
  DW_CUDA(cudaGetLastError());
  return DWFMM_OK;
}

}  // namespace dw
