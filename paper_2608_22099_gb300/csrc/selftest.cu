// selftest.cu -- self-test hooks (declared in include/bandlu_selftest.h): the
// integer-pipe reciprocal used on the pivot chain and the known-divisor division
// of the back substitution, callable on the host and on the device so tests can
// compare them bit for bit with IEEE division (and the quotient with its zero test
// on the host), the choice of the factorisation kernel, and the solve's CTA sweeps with
// a value that never arrives.
#include "bandlu_selftest.h"
#include "common.cuh"
#include "rcp.cuh"
#include "trwin.cuh"

namespace {
// x / d as the sweeps form it, a zero dividend divided like any other.
__host__ __device__ double quotient(double x, double d) {
  bool unsure;
  const double q = bandlu::div_quick(x, bandlu::div_known_prep(d), &unsure);
  return unsure ? x / d : q;
}
// The sweeps' quotient with its zero test.
double quotient_nz(double x, double d) {
  bool unsure, nonzero;
  const double q = bandlu::div_quick(x, bandlu::div_known_prep(d), &unsure);
  return unsure ? bandlu::div_unsure(x, d, true, &nonzero) : q;
}
// A straight-line reciprocal and whether it leaves this operand to the division.
__host__ __device__ double reciprocal(int which, double x, int *special) {
  bool s;
  const double y = which == 0 ? bandlu::rcp_rn_quick(x, &s) : bandlu::rcp_rn_fast(x, &s);
  *special = s ? 1 : 0;
  return y;
}
__global__ void k_rcp_raw(int which, const double *__restrict__ x, double *__restrict__ y, int *__restrict__ special,
                          long long n) {
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x)
    y[i] = reciprocal(which, x[i], special + i);
}
__global__ void k_rcp(const double *__restrict__ x, double *__restrict__ y, long long n) {
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x)
    y[i] = bandlu::rcp_rn(x[i]);
}
__global__ void k_div(const double *__restrict__ x, double *__restrict__ y, long long n) {
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x)
    y[i] = 1.0 / x[i];
}
__global__ void k_divk(const double *__restrict__ x, const double *__restrict__ d, double *__restrict__ q,
                       long long n, int use_division) {
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x) {
    if (use_division) {
      q[i] = x[i] / d[i];
    } else {
      q[i] = quotient(x[i], d[i]);
    }
  }
}

// The sweeps' hand-over with the value (or the copied column) of one step lost.
struct LossyRing : bandlu::trwin::Ring {
  int lost;
  __device__ __forceinline__ void put(int k, double v, bool c) { bandlu::trwin::Ring::put(k, v, c && k != lost); }
};
struct LossyStage : bandlu::trwin::Stage {
  int lost;
  __device__ __forceinline__ void copy(int k, const double *from, unsigned bytes, unsigned bar) const {
    if (k != lost) bandlu::trwin::Stage::copy(k, from, bytes, bar);
  }
};

__global__ void __launch_bounds__(256) k_sweep_lost(int what, int lost, int n, int kl, int ku, const double *AB,
                                                    int ldab, const int *ipiv, double *b, int *d_info) {
  extern __shared__ __align__(16) double columns[];
  __shared__ LossyRing ring;
  __shared__ bandlu::trwin::BlockShared bs;
  __shared__ unsigned long long full[2];
  const int kv = kl + ku;
  if (threadIdx.x == 0) ring.lost = what == 0 ? -1 : lost;
  if (what == 2) {
    bandlu::trwin::ring_sweep_div<8, false>(b, n, kv, bandlu::trwin::GbUpper{AB, ldab, kv, n}, ring, d_info);
  } else {
    const LossyStage st{{columns, bandlu::trwin::stage_pitch(kl), full}, what == 0 ? lost : -1};
    bandlu::trwin::block_sweep_piv<true>(b, n, kl, bandlu::trwin::GbLower{AB, ldab, kv}, ipiv, ring, st, bs, d_info);
  }
}
}  // namespace

extern "C" {

int bandlu_selftest_sweep_lost(int what, int lost, int n, int kl, int ku, const double *AB, int ldab, const int *ipiv,
                               double *b, int *d_info, cudaStream_t stream) {
  if (what < 0 || what > 2) return -1;
  if (n < 1 || kl < 33 || kl > 128 || ku < 0 || kl + ku > 160 || ldab < 2 * kl + ku + 1) return -3;
  const int threads = what == 2 ? bandlu::trwin::ring_threads_div(kl + ku) : bandlu::trwin::block_threads(kl);
  const size_t smem = 64 * (size_t)bandlu::trwin::stage_pitch(kl) * sizeof(double);
  if (!bandlu::allow_dynamic_smem(reinterpret_cast<const void *>(k_sweep_lost), (int)smem)) return BANDLU_ERR_CUDA;
  k_sweep_lost<<<1, threads, smem, stream>>>(what, lost, n, kl, ku, AB, ldab, ipiv, b, d_info);
  BANDLU_CHECK_LAUNCH();
  return BANDLU_OK;
}

void bandlu_selftest_div_host(const double *x, const double *d, double *q, int64_t n) {
  for (int64_t i = 0; i < n; ++i) {
    q[i] = quotient(x[i], d[i]);
  }
}

void bandlu_selftest_div_nz_host(const double *x, const double *d, double *q, int64_t n) {
  for (int64_t i = 0; i < n; ++i) {
    q[i] = quotient_nz(x[i], d[i]);
  }
}

int bandlu_selftest_div_device(const double *x, const double *d, double *q, int64_t n, int use_division,
                               cudaStream_t stream) {
  if (n < 0) return -4;
  if (n == 0) return BANDLU_OK;
  if (x == nullptr) return -1;
  if (d == nullptr) return -2;
  if (q == nullptr) return -3;
  long long blocks = (n + 255) / 256;
  if (blocks > 152ll * 64) blocks = 152ll * 64;
  k_divk<<<(unsigned)blocks, 256, 0, stream>>>(x, d, q, n, use_division);
  BANDLU_CHECK_LAUNCH();
  return BANDLU_OK;
}

int bandlu_selftest_gbtrf_path(int64_t n, int kl, int ku, int64_t ldab) {
  return bandlu::gbtrf_path(n, kl, ku, ldab);
}

void bandlu_selftest_rcp_host(const double *x, double *y, int64_t n) {
  for (int64_t i = 0; i < n; ++i) y[i] = bandlu::rcp_rn(x[i]);
}

void bandlu_selftest_rcp_raw_host(int which, const double *x, double *y, int *special, int64_t n) {
  for (int64_t i = 0; i < n; ++i) y[i] = reciprocal(which, x[i], special + i);
}

int bandlu_selftest_rcp_raw_device(int which, const double *x, double *y, int *special, int64_t n,
                                   cudaStream_t stream) {
  if (which < 0 || which > 1) return -1;
  if (n < 0) return -5;
  if (n == 0) return BANDLU_OK;
  if (x == nullptr) return -2;
  if (y == nullptr) return -3;
  if (special == nullptr) return -4;
  long long blocks = (n + 255) / 256;
  if (blocks > 152ll * 64) blocks = 152ll * 64;
  k_rcp_raw<<<(unsigned)blocks, 256, 0, stream>>>(which, x, y, special, n);
  BANDLU_CHECK_LAUNCH();
  return BANDLU_OK;
}

int bandlu_selftest_rcp_device(const double *x, double *y, int64_t n, int use_division, cudaStream_t stream) {
  if (n < 0) return -3;
  if (n == 0) return BANDLU_OK;
  if (x == nullptr) return -1;
  if (y == nullptr) return -2;
  long long blocks = (n + 255) / 256;
  if (blocks > 152ll * 64) blocks = 152ll * 64;
  if (use_division)
    k_div<<<(unsigned)blocks, 256, 0, stream>>>(x, y, n);
  else
    k_rcp<<<(unsigned)blocks, 256, 0, stream>>>(x, y, n);
  BANDLU_CHECK_LAUNCH();
  return BANDLU_OK;
}

}  // extern "C"
