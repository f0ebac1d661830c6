// batched.cu -- the strategy of Sec. II-A over a batch of independent matrices,
// with no host round trip: every matrix gets its own identification, decision,
// conversion and factorisation.
//
//  * k_batch_scan_convert: one block per matrix.  Warps stride over rows and
//    lanes over 16-byte vectors of a row (consecutive addresses); the block
//    folds the largest i-j / j-i over nonzeros, applies the dispatch predicate
//    and, for a banded matrix, writes its band storage (reading the band back
//    from the matrix it has just scanned, which is still in L2).
//  * k_batch_factor: one warp per matrix, or per pair of matrices where both
//    windows fit 16 lanes, in place on their band storage, in the xGBTRF order of
//    operations.  Bands whose active window fits a register a lane, or, in batches
//    of few warps, up to nine (takes_window), are factored with the window in registers
//    (window_gbtrf): no shared memory, one argmax, a few shuffles, and a DMUL and a
//    DFMA per plane and column; the others column by column through memory
//    (warp_gbtrf).  One matrix's chain of columns bounds it: 500 matrices of n = 201,
//    kl = ku = 5 take 130 us (three planes; column by column they took 619), 4096 of n =
//    256, kl = ku = 2 take 136 us (201 with the windows kept in order).
//  The band storage written by the first kernel (58.7 MB for 4096 matrices of
//  n = 256, kl = ku = 2) stays in L2 for the second.  (A single kernel with
//  scanner and factor warps side by side was slower: the factor warps' loads
//  queue behind the scanners' HBM stream.)
#include <climits>

#include "common.cuh"
#include "rcp.cuh"
#include "regwin.cuh"

namespace bandlu {
namespace {

constexpr int kFlatLoads = 4;  // 16-byte loads a thread keeps in flight

__global__ void __launch_bounds__(256) k_batch_scan_convert(const double *__restrict__ A, long long n, long long lda,
                                                            long long strideA, long long batch, double *__restrict__ AB,
                                                            long long ldab, long long strideAB, int *__restrict__ d_kl,
                                                            int *__restrict__ d_ku, int *__restrict__ d_info,
                                                            int *__restrict__ d_status, int vec, int flat) {
  __shared__ int s_l[8], s_u[8];
  __shared__ int s_kl, s_ku, s_banded;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, nw = blockDim.x >> 5;
  for (long long b = blockIdx.x; b < batch; b += gridDim.x) {
    const double *Ab = A + b * strideA;
    int lmax = 0, umax = 0;
    if (flat) {
      // the matrix as one run of elements, padding and all, in 16-byte vectors from the first aligned
      // one on; an element's row and column matter only where it is nonzero
      const unsigned ld = (unsigned)lda, total = (unsigned)((n - 1) * lda + n);
      const unsigned head = (unsigned)(reinterpret_cast<uintptr_t>(Ab) >> 3) & 1u;
      const unsigned V = (total - head) / 2;  // (total >= 1)
      const ulonglong2 *run = reinterpret_cast<const ulonglong2 *>(Ab + head);
      auto see = [&](unsigned e) {
        const int i = (int)(e / ld), j = (int)(e - (unsigned)i * ld);
        if (j < (int)n) {
          lmax = max(lmax, i - j);
          umax = max(umax, j - i);
        }
      };
      for (unsigned f0 = threadIdx.x; f0 < V; f0 += kFlatLoads * 256) {
        ulonglong2 x[kFlatLoads];
#pragma unroll
        for (int u = 0; u < kFlatLoads; ++u) {
          const unsigned f = f0 + 256u * u;
          x[u] = f < V ? __ldcs(run + f) : make_ulonglong2(0ull, 0ull);
        }
#pragma unroll
        for (int u = 0; u < kFlatLoads; ++u) {
          if (((x[u].x << 1) | (x[u].y << 1)) != 0ull) {
            const unsigned e = head + 2u * (f0 + 256u * u);
            if (nz_bits(x[u].x)) see(e);
            if (nz_bits(x[u].y)) see(e + 1u);
          }
        }
      }
      const unsigned long long *el = reinterpret_cast<const unsigned long long *>(Ab);
      if (threadIdx.x == 0 && head != 0u && nz_bits(__ldcs(el))) see(0u);
      if (threadIdx.x == 32 && ((total - head) & 1u) != 0u && nz_bits(__ldcs(el + (total - 1u)))) see(total - 1u);
    } else if (vec) {
      const long long nv = (n + 1) / 2;
      for (long long i = warp; i < n; i += nw) {
        const ulonglong2 *row = reinterpret_cast<const ulonglong2 *>(Ab + i * lda);
        for (long long v0 = lane; v0 < nv; v0 += 32 * 4) {
          ulonglong2 x[4];
#pragma unroll
          for (int u = 0; u < 4; ++u) {
            const long long v = v0 + 32 * u;
            x[u] = v < nv ? __ldcs(row + v) : make_ulonglong2(0ull, 0ull);
          }
#pragma unroll
          for (int u = 0; u < 4; ++u) {
            if (((x[u].x << 1) | (x[u].y << 1)) != 0ull) {
              const long long j0 = 2 * (v0 + 32 * u);
              if (nz_bits(x[u].x)) {
                lmax = max(lmax, (int)(i - j0));
                umax = max(umax, (int)(j0 - i));
              }
              if (nz_bits(x[u].y) && j0 + 1 < n) {
                lmax = max(lmax, (int)(i - j0 - 1));
                umax = max(umax, (int)(j0 + 1 - i));
              }
            }
          }
        }
      }
    } else {
      for (long long i = warp; i < n; i += nw) {
        const unsigned long long *row = reinterpret_cast<const unsigned long long *>(Ab + i * lda);
        for (long long j = lane; j < n; j += 32) {
          if (nz_bits(__ldcs(row + j))) {
            lmax = max(lmax, (int)(i - j));
            umax = max(umax, (int)(j - i));
          }
        }
      }
    }
    lmax = __reduce_max_sync(FULL, lmax);
    umax = __reduce_max_sync(FULL, umax);
    if (lane == 0) {
      s_l[warp] = lmax;
      s_u[warp] = umax;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
      int kl = 0, ku = 0;
      for (int w = 0; w < nw; ++w) {
        kl = max(kl, s_l[w]);
        ku = max(ku, s_u[w]);
      }
      const bool banded = predicate_banded(n, kl, ku, ldab);
      s_kl = kl;
      s_ku = ku;
      s_banded = banded ? 1 : 0;
      d_kl[b] = kl;
      d_ku[b] = ku;
      d_info[b] = 0;
      d_status[b] = banded ? BANDLU_OK : BANDLU_NOT_BANDED;
    }
    __syncthreads();
    if (s_banded) {
      const long long kl = s_kl, ku = s_ku, kv = kl + ku;
      double *ABb = AB + b * strideAB;
      const long long total = n * ldab;
      if (total <= INT_MAX - 256) {  // one 32-bit division an entry (a 64-bit one is five times as long)
        const unsigned ld = (unsigned)ldab;
        for (unsigned e = threadIdx.x; e < (unsigned)total; e += blockDim.x) {
          const int j = (int)(e / ld), r = (int)(e - (unsigned)j * ld), i = j - (int)kv + r;
          double v = 0.0;
          if (r >= kl && r <= kv + kl && i >= 0 && i < n) v = Ab[i * lda + j];
          ABb[e] = v;
        }
      } else {
        for (long long e = threadIdx.x; e < total; e += blockDim.x) {
          const long long j = e / ldab;
          const long long r = e - j * ldab;
          const long long i = j - kv + r;
          double v = 0.0;
          if (r >= kl && r <= kv + kl && i >= 0 && i < n) v = Ab[i * lda + j];
          ABb[e] = v;
        }
      }
    }
    __syncthreads();
  }
}

// Unblocked banded elimination by one warp on band storage `ab` (shared or
// global memory), in the xGBTRF order of operations.  32-bit indices (n < 2^31).
// Candidates of a pivot column sit one per lane; the first-max argmax is the
// exact integer reduction over |x|'s bit pattern.  Returns info.
__device__ int warp_gbtrf(double *ab, int ldab, int n, int kl, int ku, int *ipiv) {
  const int lane = threadIdx.x & 31;
  const int kv = kl + ku;
  if (kl > 0) {
    for (long long e = lane; e < (long long)n * kl; e += 32) {
      const long long c = e / kl, r = e - c * kl;
      ab[r + c * ldab] = 0.0;
    }
  }
  __syncwarp();
  int ju = 0;
  int info = 0;
  for (int j = 0; j < n; ++j) {
    const int km = min(kl, n - 1 - j);
    double *col = ab + (long long)j * ldab;
    int p;
    if (km < 32) {
      const double x = lane <= km ? col[kv + lane] : 0.0;
      bool allz;
      p = warp_argmax_first_z(lane <= km ? pivot_abs_key(x, lane == 0) : 0ull, &allz);
    } else {
      KeyIdx best{0ull, LLONG_MAX};
      for (int t = lane; t <= km; t += 32) best = better(best, KeyIdx{pivot_abs_key(col[kv + t], t == 0), t});
      p = (int)warp_reduce_keyidx(best).idx;
    }
    const double pv = col[kv + p];
    if (lane == 0) ipiv[j] = j + p + 1;
    if (nz(pv)) {
      ju = max(ju, min(j + ku + p, n - 1));
      if (p != 0) {
        for (int c = j + lane; c <= ju; c += 32) {
          double *x = ab + (kv + j - c) + (long long)c * ldab;
          double *y = ab + (kv + j + p - c) + (long long)c * ldab;
          const double t0 = *x;
          *x = *y;
          *y = t0;
        }
      }
      if (km > 0) {
        const double r = rcp_rn(pv);  // IEEE 1/pv on the integer pipes
        __syncwarp();
        for (int t = 1 + lane; t <= km; t += 32) col[kv + t] *= r;
        __syncwarp();
        const int ncol = ju - j;
        for (int e = lane; e < ncol * km; e += 32) {
          const int cc = e / km, t = 1 + (e - cc * km);
          const int c = j + 1 + cc;
          double *colc = ab + (long long)c * ldab;
          const double u = colc[kv + j - c];
          if (nz(u)) colc[kv + j + t - c] = fma(-col[kv + t], u, colc[kv + j + t - c]);
        }
      }
    } else if (info == 0) {
      info = j + 1;
    }
    __syncwarp();
  }
  return info;
}

// One matrix by one warp with its window in NR registers a lane.
template <int NR>
__device__ __forceinline__ int one_window(double *ab, unsigned ldab, int n, int kl, int ku, int *ipiv) {
  double *const abp[1] = {ab};
  int *const pvp[1] = {ipiv};
  const int klt[1] = {kl}, kut[1] = {ku};
  int inf[1];
  regwin::window_gbtrf<1, NR, unsigned>(abp, ldab, n, klt, kut, pvp, inf);
  return inf[0];
}

// Whether a band of np planes goes to a register window, in a batch of `load` warps to each of
// the chip's sub-partitions (at most kPlanesLoad, all resident with the 128 registers of nine
// planes).  A window's instructions grow with its planes, those of a column through memory
// with its kl*kv updates, and more warps hide its latencies.  us a call with windows of up to
// nine planes / column by column (n = 128: 600 and 1200 matrices; n = 64: 1800 and 2400):
//   kl, ku        600          1200         1800         2400
//   4, 4          105 / 161    137 / 185     88 / 110    108 / 117     3 planes
//   6, 6          142 / 206    186 / 233    128 / 133    161 / 143     4
//   7, 7          143 / 244    191 / 275    130 / 151    163 / 161     4
//   4, 27         149 / 374    215 / 410    133 / 202    175 / 211     5
//   10, 5         218 / 284    285 / 315    201 / 169    261 / 182     6
//   5, 20         219 / 320    295 / 363    205 / 186    264 / 200     6
//   8, 8          219 / 225    289 / 259    206 / 144    263 / 157     9
//   8, 23         225 / 525    317 / 572    210 / 277    270 / 297     9
// Beyond kPlanesLoad column by column is faster for any of them (4096 of n = 64: kl = ku = 4 182
// with planes, 147 without, 8, 23 475, 352; 20000: 764, 639 and 2044, 1582), in the kernel of one
// plane, whose 72 registers keep seven warps a sub-partition resident.
// Instantiated are 3, 5 and 9 planes; a count between runs the next one's window.  That costs it up to
// 22% of a call (600 of n = 128 with a window of its own / the next one's: kl = ku = 4, two planes, 84 / 105
// us, 6, 6, four, 129 / 141, 5, 20, six, 171 / 219, 7, 24, eight, 207 / 224), and a window each would more
// than double the time to compile this kernel (11 to 24 s).
constexpr int kPlanesLoad = 4;
__device__ __forceinline__ bool takes_window(int np, int load, int kl, int ku) {
  if (np <= 3) return true;
  if (np > 9) return false;
  const int work = kl * (kl + ku);
  if (np <= 5) return load <= 3 || work >= 100;
  return load <= 2 || work >= 200;
}

// Warp b of the first half of the grid takes matrices 2b and 2b+1 together, in
// 16-lane windows, when both bands fit one; otherwise it takes matrix 2b and its
// counterpart in the second half (which leaves at once in the first case) takes
// matrix 2b+1: in a register window, of one plane or (kPlanes) of up to nine, or
// column by column.
template <bool kPlanes>
__global__ void __launch_bounds__(128) k_batch_factor(long long n, long long batch, double *__restrict__ AB,
                                                      long long ldab, long long strideAB, int *__restrict__ ipiv,
                                                      long long strideP, const int *__restrict__ d_kl,
                                                      const int *__restrict__ d_ku, int *__restrict__ d_info,
                                                      const int *__restrict__ d_status, int win_ok, int load) {
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, wpb = blockDim.x >> 5;
  const long long half = gridDim.x >> 1;
  const bool second = blockIdx.x >= half;
  const long long b0 = 2 * ((blockIdx.x - (second ? half : 0)) * wpb + warp);
  if (b0 >= batch) return;  // whole warp leaves together
  bool ok[2];
  int kl[2], ku[2];
  for (int t = 0; t < 2; ++t) {
    const long long b = b0 + t;
    ok[t] = b < batch && d_status[b] == BANDLU_OK;
    kl[t] = ok[t] ? d_kl[b] : 0;
    ku[t] = ok[t] ? d_ku[b] : 0;
  }
  auto planes = [&](int t, int width) { return win_ok ? regwin::planes_of(kl[t], kl[t] + ku[t], width) : INT_MAX; };
  if (ok[0] && ok[1] && planes(0, 16) == 1 && planes(1, 16) == 1) {
    if (second) return;
    double *const abp[2] = {AB + b0 * strideAB, AB + (b0 + 1) * strideAB};
    int *const pvp[2] = {ipiv + b0 * strideP, ipiv + (b0 + 1) * strideP};
    int info[2];
    regwin::window_gbtrf<2, 1, unsigned>(abp, (unsigned)ldab, (int)n, kl, ku, pvp, info);
    if (lane == 0) {
      d_info[b0] = info[0];
      d_info[b0 + 1] = info[1];
    }
    return;
  }
  const int t = second ? 1 : 0;
  if (!ok[t]) return;
  const long long b = b0 + t;
  double *ABb = AB + b * strideAB;
  int *pv = ipiv + b * strideP;
  const int np = planes(t, 32);
  int info;
  if (np == 1) {
    info = one_window<1>(ABb, (unsigned)ldab, (int)n, kl[t], ku[t], pv);
  } else if (kPlanes && takes_window(np, load, kl[t], ku[t])) {
    if (np <= 3) info = one_window<3>(ABb, (unsigned)ldab, (int)n, kl[t], ku[t], pv);
    else if (np <= 5) info = one_window<5>(ABb, (unsigned)ldab, (int)n, kl[t], ku[t], pv);
    else info = one_window<9>(ABb, (unsigned)ldab, (int)n, kl[t], ku[t], pv);
  } else {
    info = warp_gbtrf(ABb, (int)ldab, (int)n, kl[t], ku[t], pv);
  }
  if (lane == 0) d_info[b] = info;
}

}  // namespace

int launch_batched(const double *A, int64_t n, int64_t lda, int64_t strideA, int64_t batch, double *AB, int64_t ldab,
                   int64_t strideAB, int *ipiv, int64_t strideP, int *d_kl, int *d_ku, int *d_info, int *d_status,
                   cudaStream_t s) {
  if (batch == 0) return BANDLU_OK;
  const int vec = ((reinterpret_cast<uintptr_t>(A) & 15u) == 0) && (lda % 2 == 0) && (strideA % 2 == 0);
  // Rows with little padding are read as one run of vectors, whatever their alignment, unless
  // each row is a whole number of a warp's four loads.  (Row by row the last loads of a row are
  // part empty, and rows of odd length or on odd addresses went element by element.  500 of
  // n = 201, lda = 203: 37 us against 50; 2000 of n = 40, lda = 41: 14 against 23; 4096 of n = 256
  // by rows 337, as one run 342.)
  const int flat = n >= 1 && !(vec && ((n + 1) / 2) % 128 == 0) && lda - n <= 2 + n / 32 &&
                   n * lda < (1ll << 31) - 4096;
  long long grid1 = batch;
  const long long cap = (long long)device_sms() * 64;
  if (grid1 > cap) grid1 = cap;
  k_batch_scan_convert<<<(unsigned)grid1, 256, 0, s>>>(A, n, lda, strideA, batch, AB, ldab, strideAB, d_kl, d_ku,
                                                       d_info, d_status, vec, flat);
  BANDLU_CHECK_LAUNCH();
  if (n == 0) return BANDLU_OK;
  const int wpb = 4;
  const long long grid2 = 2 * (((batch + 1) / 2 + wpb - 1) / wpb);  // two warps per pair of matrices
  const int win_ok = ldab <= (INT_MAX - 1) / (n + 1);  // 32-bit offsets in window_gbtrf: (n + 1) * ldab < INT_MAX
  // warps to a sub-partition (every band that storage of up to seven rows admits goes in pairs)
  const long long subs = 4ll * device_sms(), load = ((ldab <= 7 ? (batch + 1) / 2 : batch) + subs - 1) / subs;
  if (load <= kPlanesLoad)
    k_batch_factor<true><<<(unsigned)grid2, 32 * wpb, 0, s>>>(n, batch, AB, ldab, strideAB, ipiv, strideP, d_kl, d_ku,
                                                              d_info, d_status, win_ok, (int)load);
  else
    k_batch_factor<false><<<(unsigned)grid2, 32 * wpb, 0, s>>>(n, batch, AB, ldab, strideAB, ipiv, strideP, d_kl,
                                                               d_ku, d_info, d_status, win_ok, 0);
  BANDLU_CHECK_LAUNCH();
  return BANDLU_OK;
}

}  // namespace bandlu
