// rewl_thermo.cu -- canonical thermodynamics from a density of states: for
// every temperature T (k_B = 1, beta = 1/T), with the Boltzmann weights
// w(E) = g(E) exp(-beta E) taken in log space,
//   ln Z = ln sum_E w(E)              (shifted by the largest term)
//   U    = <E>,  C = beta^2 <(E - U)^2>   (two passes: mean, then centred moment)
//   F    = -T ln Z,  S = (U - F) / T.
// One CTA per temperature (and table); block reductions over the energy bins.
// rewl_thermo_jackknife adds the resampling errors over independent runs
// (join paragraph: statistical errors by resampling): the same quantities of
// the mean ln g and of every leave-one-out mean, combined into jackknife errors.
#include <cuda_runtime.h>

#include <cmath>
#include <cstdint>
#include <mutex>

#include "rewl.h"
#include "rewl_ctx.h"

namespace {

// Sum over the CTA, the same for all threads.  The warps' sums are added up by the first warp alone: done by every
// thread, these few additions were half of the FP64 pipe's work.
__device__ __forceinline__ double block_sum(double v, double* sh) {
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, nw = (blockDim.x + 31) >> 5;
  for (int o = 16; o; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  if (nw == 1) return v;
  __syncthreads();  // the last sum has been read
  if (lane == 0) sh[wid] = v;
  __syncthreads();
  if (wid == 0) {
    double r = lane < nw ? sh[lane] : 0.0;
    for (int o = 4; o; o >>= 1) r += __shfl_xor_sync(0xffffffffu, r, o);  // at most eight warps
    __syncwarp();
    if (lane == 0) sh[0] = r;
  }
  __syncthreads();
  return sh[0];
}
__device__ __forceinline__ long long block_max(long long v, long long* sh) {
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, nw = (blockDim.x + 31) >> 5;
  for (int o = 16; o; o >>= 1) v = max(v, __shfl_xor_sync(0xffffffffu, v, o));
  if (lane == 0) sh[wid] = v;
  __syncthreads();
  for (int i = 0; i < nw; ++i) v = max(v, sh[i]);
  return v;
}

// 2^(j/64), rounded.
__device__ const double kExp2[64] = {
    0x1.0000000000000p+0, 0x1.02c9a3e778061p+0, 0x1.059b0d3158574p+0, 0x1.0874518759bc8p+0,
    0x1.0b5586cf9890fp+0, 0x1.0e3ec32d3d1a2p+0, 0x1.11301d0125b51p+0, 0x1.1429aaea92de0p+0,
    0x1.172b83c7d517bp+0, 0x1.1a35beb6fcb75p+0, 0x1.1d4873168b9aap+0, 0x1.2063b88628cd6p+0,
    0x1.2387a6e756238p+0, 0x1.26b4565e27cddp+0, 0x1.29e9df51fdee1p+0, 0x1.2d285a6e4030bp+0,
    0x1.306fe0a31b715p+0, 0x1.33c08b26416ffp+0, 0x1.371a7373aa9cbp+0, 0x1.3a7db34e59ff7p+0,
    0x1.3dea64c123422p+0, 0x1.4160a21f72e2ap+0, 0x1.44e086061892dp+0, 0x1.486a2b5c13cd0p+0,
    0x1.4bfdad5362a27p+0, 0x1.4f9b2769d2ca7p+0, 0x1.5342b569d4f82p+0, 0x1.56f4736b527dap+0,
    0x1.5ab07dd485429p+0, 0x1.5e76f15ad2148p+0, 0x1.6247eb03a5585p+0, 0x1.6623882552225p+0,
    0x1.6a09e667f3bcdp+0, 0x1.6dfb23c651a2fp+0, 0x1.71f75e8ec5f74p+0, 0x1.75feb564267c9p+0,
    0x1.7a11473eb0187p+0, 0x1.7e2f336cf4e62p+0, 0x1.82589994cce13p+0, 0x1.868d99b4492edp+0,
    0x1.8ace5422aa0dbp+0, 0x1.8f1ae99157736p+0, 0x1.93737b0cdc5e5p+0, 0x1.97d829fde4e50p+0,
    0x1.9c49182a3f090p+0, 0x1.a0c667b5de565p+0, 0x1.a5503b23e255dp+0, 0x1.a9e6b5579fdbfp+0,
    0x1.ae89f995ad3adp+0, 0x1.b33a2b84f15fbp+0, 0x1.b7f76f2fb5e47p+0, 0x1.bcc1e904bc1d2p+0,
    0x1.c199bdd85529cp+0, 0x1.c67f12e57d14bp+0, 0x1.cb720dcef9069p+0, 0x1.d072d4a07897cp+0,
    0x1.d5818dcfba487p+0, 0x1.da9e603db3285p+0, 0x1.dfc97337b9b5fp+0, 0x1.e502ee78b3ff6p+0,
    0x1.ea4afa2a490dap+0, 0x1.efa1bee615a27p+0, 0x1.f50765b6e4540p+0, 0x1.fa7c1819e90d8p+0,
};

// exp(x) for -746 < x <= 0 by a table of 2^(j/64) and a polynomial on the rest (P. T. P. Tang, Table-driven
// implementation of the exponential function, ACM TOMS 15, 144 (1989)): x = n ln2/64 + r, |r| <= ln2/128, and
// e^r - 1 to r^5 (the next term is below 3.5e-17).  Ten FP64 operations: the FP64 pipe (2.2 lane operations a
// cycle and SM) is what bounds these sums.  tab: kExp2 in shared memory.
__device__ __forceinline__ double exp_of_nonpositive(double x, const double* tab) {
  constexpr double kMagic = 6755399441055744.0;  // 1.5 * 2^52: the sum's low word is the rounded integer
  const double t = fma(x, 0x1.71547652b82fep+6, kMagic);
  const int n = __double2loint(t);
  const double f = t - kMagic;
  const double r = fma(f, -0x1.abc9e3b39803fp-62, fma(f, -0x1.62e42fefa39efp-7, x));
  double q = fma(r, 1.0 / 120.0, 1.0 / 24.0);
  q = fma(r, q, 1.0 / 6.0);
  q = fma(r, q, 0.5);
  const double s = tab[n & 63];
  const double v = fma(s, fma(r * r, q, r), s);
  const int k = n >> 6;  // -1077 .. 0
  if (k >= -1021) return __hiloint2double(__double2hiint(v) + (k << 20), __double2loint(v));
  return __hiloint2double(__double2hiint(v) + ((k + 128) << 20), __double2loint(v)) * 0x1p-128;  // into the denormals
}

// One CTA per (temperature, table): table blockIdx.y of n_bins values, output
// [table][temperature][5].  Each weight is computed once and kept in shared memory for the
// centred moment (s_w holds n_bins of them, or none and they are computed again); a term of
// exp(-746) or less, which is 0 in FP64, is not computed at all; the largest term is found
// on the integer pipe.  rewl_thermo_jackknife of 8 runs of 1025 levels at 300 temperatures
// (2700 CTAs) before -> after: 583 -> 348 us a call, with CUDA's exp 451; 197 since the call no longer allocates.
constexpr uint32_t kZeroHi = 0x40875000u;  // upper word of 746
__device__ __forceinline__ long long order_key(double v) {  // orders as the numbers do (no NaN)
  const long long i = __double_as_longlong(v);
  return i ^ (long long)((unsigned long long)(i >> 63) >> 1);
}
__global__ void __launch_bounds__(256) k_thermo(const double* __restrict__ lng_tables, int n_bins, int e_min,
                                                int e_step, const double* __restrict__ T,
                                                double* __restrict__ out_tables, int keep) {
  extern __shared__ double s_w[];
  __shared__ double sh[8], tab[64];
  __shared__ long long sh_max[8];
  const double* lng = lng_tables + (size_t)blockIdx.y * n_bins;
  double* out = out_tables + (size_t)blockIdx.y * gridDim.x * 5;
  const double t = T[blockIdx.x];
  const double beta = 1.0 / t;
  for (int j = threadIdx.x; j < 64; j += blockDim.x) tab[j] = kExp2[j];  // block_max synchronises before its use
  // E of the thread's bins: integers well below 2^53, so the steps are exact
  const double e_first = (double)(e_min + (int)threadIdx.x * e_step), e_stride = (double)blockDim.x * (double)e_step;
  long long top = order_key(-INFINITY);
  double e = e_first;
  for (int b = threadIdx.x; b < n_bins; b += blockDim.x, e += e_stride) {
    const double l = lng[b];
    const double a = isfinite(l) ? l - beta * e : -INFINITY;
    if (keep) s_w[b] = a;  // its own thread reads it back
    top = max(top, order_key(a));
  }
  top = block_max(top, sh_max);
  const double mx = __longlong_as_double(top ^ (long long)((unsigned long long)(top >> 63) >> 1));
  double z = 0.0, ze = 0.0;
  e = e_first;
  for (int b = threadIdx.x; b < n_bins; b += blockDim.x, e += e_stride) {
    const double a = keep ? s_w[b] : isfinite(lng[b]) ? lng[b] - beta * e : -INFINITY;
    const double x = a - mx;
    double wgt = 0.0;
    if ((uint32_t)(__double2hiint(x) & 0x7fffffff) < kZeroHi) {  // |x| < 746
      wgt = exp_of_nonpositive(x, tab);
      z += wgt;
      ze += wgt * e;
    }
    if (keep) s_w[b] = wgt;
  }
  z = block_sum(z, sh);
  ze = block_sum(ze, sh);
  const double U = ze / z;
  double zc = 0.0;
  e = e_first;
  for (int b = threadIdx.x; b < n_bins; b += blockDim.x, e += e_stride) {
    double wgt = 0.0;
    if (keep) {
      wgt = s_w[b];
    } else {
      const double x = (isfinite(lng[b]) ? lng[b] - beta * e : -INFINITY) - mx;
      if ((uint32_t)(__double2hiint(x) & 0x7fffffff) < kZeroHi) wgt = exp_of_nonpositive(x, tab);
    }
    if (__double_as_longlong(wgt) != 0) {
      const double d = e - U;
      zc += wgt * d * d;
    }
  }
  zc = block_sum(zc, sh);
  if (threadIdx.x == 0) {
    const double lnZ = mx + log(z);
    const double F = -t * lnZ;
    double* o = out + 5 * (size_t)blockIdx.x;
    o[0] = lnZ;
    o[1] = U;
    o[2] = beta * beta * (zc / z);
    o[3] = F;
    o[4] = (U - F) / t;
  }
}

constexpr int kKeepBins = 4096;  // weights kept up to here: 32 KB of shared memory, seven CTAs an SM
// Threads a CTA: few temperatures and tables are latency-bound, eight warps each; many fill the SMs, and then fewer
// warps share out a table, with fewer additions across warps (that call, while it allocated, with 256 threads 388 us,
// 128 353, 64 348).
constexpr int kFewCtas = 304;  // two an SM
void launch_thermo(const double* tables, int n_tables, int n_bins, int e_min, int e_step, const double* T, int n_T,
                   double* out) {
  const int keep = n_bins <= kKeepBins;
  const int threads = (int64_t)n_T * n_tables <= kFewCtas || n_bins > 8192 ? 256 : n_bins > 2048 ? 128 : 64;
  k_thermo<<<dim3(n_T, (unsigned)n_tables), threads, keep ? sizeof(double) * n_bins : 0>>>(tables, n_bins, e_min, e_step,
                                                                                          T, out, keep);
}

// Jackknife tables: [0] the mean ln g over the R runs, [1 + i] the mean
// without run i; a bin counts only where every run is finite (else -inf).
// Sums in run order.  One thread per bin.
__global__ void k_jack_tables(const double* __restrict__ runs, int R, int n_bins, double* __restrict__ tables) {
  const int b = blockIdx.x * blockDim.x + threadIdx.x;
  if (b >= n_bins) return;
  bool fin = true;
  for (int i = 0; i < R; ++i) fin = fin && isfinite(runs[(size_t)i * n_bins + b]);
  if (!fin) {
    for (int i = 0; i <= R; ++i) tables[(size_t)i * n_bins + b] = -INFINITY;
    return;
  }
  double total = runs[b];
  for (int i = 1; i < R; ++i) total = __dadd_rn(total, runs[(size_t)i * n_bins + b]);
  tables[b] = __ddiv_rn(total, (double)R);
  for (int i = 0; i < R; ++i)
    tables[(size_t)(1 + i) * n_bins + b] = __ddiv_rn(__dsub_rn(total, runs[(size_t)i * n_bins + b]), (double)(R - 1));
}

// est = quantity of the mean table; err = sqrt((R-1)/R * sum_i (Q_(i) - Qbar)^2)
// over the leave-one-out tables.  One thread per (temperature, quantity).
__global__ void k_jack_combine(const double* __restrict__ q, int R, int n_T, double* __restrict__ est,
                               double* __restrict__ err) {
  const int j = blockIdx.x * blockDim.x + threadIdx.x;
  if (j >= n_T * 5) return;
  const size_t stride = (size_t)n_T * 5;
  double m = q[stride + j];
  for (int i = 1; i < R; ++i) m = __dadd_rn(m, q[(size_t)(1 + i) * stride + j]);
  m = __ddiv_rn(m, (double)R);
  double ss = 0.0;
  for (int i = 0; i < R; ++i) {
    const double d = __dsub_rn(q[(size_t)(1 + i) * stride + j], m);
    ss = __dadd_rn(ss, __dmul_rn(d, d));
  }
  est[j] = q[j];
  err[j] = sqrt(__dmul_rn(__ddiv_rn((double)(R - 1), (double)R), ss));
}

// A call's device memory, one block: a fixed array of the library while it fits (32 runs of 1025 levels at 300
// temperatures do), held by one call at a time, else an allocation.  Allocating and releasing the only block of a
// process maps and unmaps a page of device memory: 59 us of the 107 us that the smallest call took.  The array's
// address is looked up in every call and belongs to the current device.
constexpr size_t kScratchDoubles = 1u << 17;
static __device__ double g_thermo_scratch[kScratchDoubles];
std::mutex g_scratch_mutex;
struct DeviceBlock {
  double* d = nullptr;
  bool own = false;
  std::unique_lock<std::mutex> lock;
  explicit DeviceBlock(size_t n) {
    if (n <= kScratchDoubles) {
      lock = std::unique_lock<std::mutex>(g_scratch_mutex);
      void* p = nullptr;
      if (cudaGetSymbolAddress(&p, g_thermo_scratch) == cudaSuccess) {
        d = static_cast<double*>(p);
        return;
      }
      lock.unlock();
    }
    own = cudaMalloc(&d, sizeof(double) * n) == cudaSuccess;
    if (!own) d = nullptr;
  }
  ~DeviceBlock() {
    if (own) cudaFree(d);
  }
  DeviceBlock(const DeviceBlock&) = delete;
  DeviceBlock& operator=(const DeviceBlock&) = delete;
};
bool to_device(double* d, const double* h, size_t n) {
  return cudaMemcpy(d, h, sizeof(double) * n, cudaMemcpyHostToDevice) == cudaSuccess;
}
bool from_device(double* h, const double* d, size_t n) {
  return cudaMemcpy(h, d, sizeof(double) * n, cudaMemcpyDeviceToHost) == cudaSuccess;
}
rewl_status failed(rewl_status st, const char* msg) {
  rewl_set_last_error(msg);
  return st;
}

rewl_status check_temperatures(const double* temperatures, int32_t n_T) {
  for (int i = 0; i < n_T; ++i)
    if (!(temperatures[i] > 0.0) || !std::isfinite(temperatures[i])) {
      rewl_set_last_error("temperatures must be positive and finite");
      return REWL_EINVAL;
    }
  return REWL_OK;
}

}  // namespace

extern "C" rewl_status rewl_thermo_jackknife(const double* lng_runs, int32_t n_runs, int32_t n_bins, int32_t e_min,
                                             int32_t e_step, const double* temperatures, int32_t n_T, double* est,
                                             double* err) {
  if (!lng_runs || !temperatures || !est || !err || n_runs < 2 || n_bins < 1 || n_T < 1 || e_step < 1 ||
      (int64_t)n_T * 5 * (n_runs + 1) > (1ll << 31)) {
    rewl_set_last_error("rewl_thermo_jackknife: invalid argument");
    return REWL_EINVAL;
  }
  if (check_temperatures(temperatures, n_T) != REWL_OK) return REWL_EINVAL;
  bool any = false;
  for (int b = 0; b < n_bins && !any; ++b) {
    bool all = true;
    for (int i = 0; i < n_runs && all; ++i) all = std::isfinite(lng_runs[(size_t)i * n_bins + b]) != 0;
    any = all;
  }
  if (!any) {
    rewl_set_last_error("rewl_thermo_jackknife: no bin is finite in every run");
    return REWL_EINVAL;
  }
  const size_t nt = (size_t)n_runs + 1, n_in = (size_t)n_runs * n_bins, n_out = (size_t)n_T * 5;
  DeviceBlock mem((size_t)n_T + n_in + nt * n_bins + nt * n_out + 2 * n_out);
  if (!mem.d) return failed(REWL_ENOMEM, "rewl_thermo_jackknife: device allocation failed");
  double *d_T = mem.d, *d_runs = d_T + n_T, *d_tab = d_runs + n_in, *d_q = d_tab + nt * n_bins;
  double *d_est = d_q + nt * n_out, *d_err = d_est + n_out;
  if (!to_device(d_T, temperatures, n_T) || !to_device(d_runs, lng_runs, n_in))
    return failed(REWL_ECUDA, "rewl_thermo_jackknife: copy failed");
  k_jack_tables<<<(n_bins + 255) / 256, 256>>>(d_runs, n_runs, n_bins, d_tab);
  launch_thermo(d_tab, (int)nt, n_bins, e_min, e_step, d_T, n_T, d_q);
  k_jack_combine<<<(n_T * 5 + 127) / 128, 128>>>(d_q, n_runs, n_T, d_est, d_err);
  if (cudaGetLastError() != cudaSuccess || !from_device(est, d_est, n_out) || !from_device(err, d_err, n_out))
    return failed(REWL_ECUDA, "rewl_thermo_jackknife: kernel failed");
  return REWL_OK;
}

extern "C" rewl_status rewl_thermo(const double* lng, int32_t n_bins, int32_t e_min, int32_t e_step,
                                   const double* temperatures, int32_t n_T, double* out) {
  if (!lng || !temperatures || !out || n_bins < 1 || n_T < 1 || e_step < 1) {
    rewl_set_last_error("rewl_thermo: invalid argument");
    return REWL_EINVAL;
  }
  if (check_temperatures(temperatures, n_T) != REWL_OK) return REWL_EINVAL;
  bool any = false;
  for (int b = 0; b < n_bins; ++b) any |= std::isfinite(lng[b]) != 0;
  if (!any) {
    rewl_set_last_error("rewl_thermo: no finite ln g");
    return REWL_EINVAL;
  }
  DeviceBlock mem((size_t)n_T + n_bins + 5 * (size_t)n_T);
  if (!mem.d) return failed(REWL_ENOMEM, "rewl_thermo: device allocation failed");
  double *d_T = mem.d, *d_lng = d_T + n_T, *d_out = d_lng + n_bins;
  if (!to_device(d_T, temperatures, n_T) || !to_device(d_lng, lng, n_bins))
    return failed(REWL_ECUDA, "rewl_thermo: copy failed");
  launch_thermo(d_lng, 1, n_bins, e_min, e_step, d_T, n_T, d_out);
  if (cudaGetLastError() != cudaSuccess || !from_device(out, d_out, 5 * (size_t)n_T))
    return failed(REWL_ECUDA, "rewl_thermo: kernel failed");
  return REWL_OK;
}
