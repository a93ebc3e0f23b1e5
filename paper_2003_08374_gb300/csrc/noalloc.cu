// noalloc.cu -- mdbs_field_stats_static: the field-statistics reduction
// (liquid volume, alpha min / max, non-finite sentinel) for callers that
// cannot allocate device memory.  Its scratch (per-block partial results)
// lives in a file-scope __device__ array instead of a cudaMalloc'ed arena.
#include <math.h>
#include <stdint.h>

#include <mutex>

#include "../../include/mdbs.h"

namespace {

constexpr int kThreads = 512;
constexpr int kMaxDevices = 64;
constexpr int kUnroll = 4;      // pairs of cells of each field that a thread has in flight
constexpr int kBlocksMost = 304;  // two blocks an SM (152): all resident, 196 KB of loads in flight an SM
static_assert(kBlocksMost <= MDBS_STATIC_STATS_MAX_BLOCKS && kBlocksMost <= kThreads, "scratch and the final fold");

// 4 channels (volume, min, max, non-finite count) x MDBS_STATIC_STATS_MAX_BLOCKS partials.
// Every device that loads the library holds this array until the process exits.
static __device__ __align__(256) double g_stats_scratch[4 * MDBS_STATIC_STATS_MAX_BLOCKS];

std::mutex g_setup_mutex;
double* g_scratch_ptr[kMaxDevices] = {};  // device address of g_stats_scratch, per device

// Order-preserving integer keys: the signed order of key(a) is the IEEE order of a, so the
// minimum and maximum are integer operations (GB300 runs FP64 compares on its narrow FP64
// pipe).  A NaN is left out, as fmin and
// fmax leave it out.
__device__ __forceinline__ long long key_of(double a) {
  const long long b = __double_as_longlong(a);
  return b ^ ((b >> 63) & 0x7fffffffffffffffll);
}
__device__ __forceinline__ double of_key(long long k) {
  return __longlong_as_double(k ^ ((k >> 63) & 0x7fffffffffffffffll));
}
// exponent field all ones: infinite or NaN; and the mantissa not zero: NaN
constexpr long long kExp = 0x7ff0000000000000ll;
__device__ __forceinline__ bool not_finite(double a) { return (__double_as_longlong(a) & kExp) == kExp; }

struct Acc {
  double mass[2];  // sums of porosity * alpha (two chains)
  long long lo, hi;
  unsigned bad;
  __device__ __forceinline__ void add(double phi, double a, double p, int chain) {
    mass[chain] = fma(phi, a, mass[chain]);
    const long long b = __double_as_longlong(a), k = key_of(a);
    const bool nan = (b & 0x7fffffffffffffffll) > kExp;
    lo = !nan && k < lo ? k : lo;
    hi = !nan && k > hi ? k : hi;
    bad += not_finite(a) || not_finite(p);
  }
};

// block fold of the four channels; the sums in a fixed order; result in thread 0
__device__ __forceinline__ void fold(double& mass, long long& lo, long long& hi, double& bad) {
  __shared__ double s_m[kThreads / 32], s_b[kThreads / 32];
  __shared__ long long s_l[kThreads / 32], s_h[kThreads / 32];
  auto warp = [&](int from) {
    for (int o = from; o > 0; o >>= 1) {
      mass += __shfl_down_sync(0xffffffffu, mass, o);
      bad += __shfl_down_sync(0xffffffffu, bad, o);
      const long long l = __shfl_down_sync(0xffffffffu, lo, o), h = __shfl_down_sync(0xffffffffu, hi, o);
      lo = l < lo ? l : lo;
      hi = h > hi ? h : hi;
    }
  };
  warp(16);
  const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
  if (lane == 0) {
    s_m[w] = mass;
    s_b[w] = bad;
    s_l[w] = lo;
    s_h[w] = hi;
  }
  __syncthreads();
  if (w == 0) {
    const int q = lane % (kThreads / 32);  // the upper lanes repeat the lower ones and are not folded in
    mass = s_m[q];
    bad = s_b[q];
    lo = s_l[q];
    hi = s_h[q];
    warp(kThreads / 64);
  }
}

// Stage 1: each block writes its partials into the static scratch.  Bound by its three
// reads of 8 bytes a cell: 16-byte loads (VEC: the fields are 16-byte aligned), kUnroll
// of each field in flight a thread.  256^3 cells, both kernels: 406 us before (one 8-byte
// load of each field in flight, FP64 minima, a serial second stage), 80 us now (5.0 TB/s;
// with evict-first loads 107, with 64 warps an SM and one pair each in flight 117).
template <bool VEC>
__global__ void __launch_bounds__(kThreads, 2)
    k_stats_partials(long long cells, const double* __restrict__ phi, const double* __restrict__ alpha,
                     const double* __restrict__ p, double* __restrict__ scratch, int nb) {
  asm volatile("griddepcontrol.launch_dependents;\n" ::: "memory");
  Acc acc{{0.0, 0.0}, key_of(INFINITY), key_of(-INFINITY), 0u};
  const long long stride = (long long)gridDim.x * kThreads, t = blockIdx.x * (long long)kThreads + threadIdx.x;
  long long done = 0;
  if (VEC) {
    const double2* __restrict__ phi2 = reinterpret_cast<const double2*>(phi);
    const double2* __restrict__ alpha2 = reinterpret_cast<const double2*>(alpha);
    const double2* __restrict__ p2 = reinterpret_cast<const double2*>(p);
    const long long pairs = cells / 2;
    long long c = t;
    for (; c + (kUnroll - 1) * stride < pairs; c += kUnroll * stride) {
      double2 f[kUnroll], a[kUnroll], q[kUnroll];
#pragma unroll
      for (int u = 0; u < kUnroll; u++) {
        f[u] = phi2[c + u * stride];
        a[u] = alpha2[c + u * stride];
        q[u] = p2[c + u * stride];
      }
#pragma unroll
      for (int u = 0; u < kUnroll; u++) {
        acc.add(f[u].x, a[u].x, q[u].x, 0);
        acc.add(f[u].y, a[u].y, q[u].y, 1);
      }
    }
    for (; c < pairs; c += stride) {
      const double2 f = phi2[c], a = alpha2[c], q = p2[c];
      acc.add(f.x, a.x, q.x, 0);
      acc.add(f.y, a.y, q.y, 1);
    }
    done = 2 * pairs;
  }
  for (long long c = done + t; c < cells; c += stride) acc.add(phi[c], alpha[c], p[c], 0);
  double mass = acc.mass[0] + acc.mass[1], bad = (double)acc.bad;
  long long lo = acc.lo, hi = acc.hi;
  fold(mass, lo, hi, bad);
  if (threadIdx.x == 0) {
    scratch[blockIdx.x] = mass;
    scratch[nb + blockIdx.x] = of_key(lo);
    scratch[2 * nb + blockIdx.x] = of_key(hi);
    scratch[3 * nb + blockIdx.x] = bad;
  }
}

// stage 2: one block folds the partials in a fixed order into the caller's output
__global__ void __launch_bounds__(kThreads)
    k_stats_final(const double* __restrict__ scratch, int nb, double volume, double* __restrict__ out) {
  asm volatile("griddepcontrol.wait;\n" ::: "memory");
  const int b = threadIdx.x;
  double mass = 0.0, bad = 0.0;
  long long lo = key_of(INFINITY), hi = key_of(-INFINITY);
  if (b < nb) {
    mass = __ldcg(scratch + b);
    lo = key_of(__ldcg(scratch + nb + b));
    hi = key_of(__ldcg(scratch + 2 * nb + b));
    bad = __ldcg(scratch + 3 * nb + b);
  }
  fold(mass, lo, hi, bad);
  if (b != 0) return;
  out[0] = mass * volume;
  out[1] = of_key(lo);
  out[2] = of_key(hi);
  out[3] = bad;
}

// Device address of the static scratch on the current device, looked up once per
// device (cudaGetSymbolAddress) with that device current.
cudaError_t scratch_for_current_device(double** out) {
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  if (dev < 0 || dev >= kMaxDevices) return cudaErrorInvalidDevice;
  std::lock_guard<std::mutex> lock(g_setup_mutex);
  if (!g_scratch_ptr[dev]) {
    void* ptr = nullptr;
    e = cudaGetSymbolAddress(&ptr, g_stats_scratch);
    if (e != cudaSuccess) return e;
    g_scratch_ptr[dev] = (double*)ptr;
  }
  *out = g_scratch_ptr[dev];
  return cudaSuccess;
}

}  // namespace

extern "C" int mdbs_field_stats_static(int64_t cells, double cell_volume, const double* porosity,
                                       const double* alpha, const double* p, double* out, void* stream) {
  if (cells < 1 || cells > MDBS_STATIC_STATS_MAX_CELLS) return MDBS_ERR_ARG;
  if (!porosity || !alpha || !p || !out || !(cell_volume > 0.0)) return MDBS_ERR_ARG;
  double* scratch = nullptr;
  if (scratch_for_current_device(&scratch) != cudaSuccess) return MDBS_ERR_CUDA;
  const long long blocks = (cells + 2 * kThreads - 1) / (2 * kThreads);
  const int nb = (int)(blocks < kBlocksMost ? blocks : kBlocksMost);
  cudaStream_t s = (cudaStream_t)stream;
  // An error already pending on this thread belongs to the caller's earlier work: report
  // it as MDBS_ERR_CUDA without launching and leave it pending (cudaPeekAtLastError does
  // not clear it).  Otherwise any error after the launches is theirs and is cleared.
  if (cudaPeekAtLastError() != cudaSuccess) return MDBS_ERR_CUDA;
  const bool vec = (((uintptr_t)porosity | (uintptr_t)alpha | (uintptr_t)p) & 15) == 0;
  if (vec)
    k_stats_partials<true><<<nb, kThreads, 0, s>>>(cells, porosity, alpha, p, scratch, nb);
  else
    k_stats_partials<false><<<nb, kThreads, 0, s>>>(cells, porosity, alpha, p, scratch, nb);
  // the second kernel's launch overlaps the first; it waits for the first's results
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(1);
  cfg.blockDim = dim3(kThreads);
  cfg.stream = s;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  cudaLaunchKernelEx(&cfg, k_stats_final, (const double*)scratch, nb, cell_volume, out);
  return cudaGetLastError() == cudaSuccess ? MDBS_OK : MDBS_ERR_CUDA;
}
