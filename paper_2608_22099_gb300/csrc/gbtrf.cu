// gbtrf.cu -- banded LU with partial pivoting (Sec. II-A step 3; f(N) ~ O(N*P*Q), Eq. S-N-N3).
//
// Two single-matrix kernels here, after the narrowest bands (a one-warp
// register window, k_gbtrf_regwin) and before the wide ones (the multi-CTA
// kernel of gbtrf_wide.cu, when it can be launched):
//
//  * k_gbtrf_window (kl <= 27, the narrow bands the method targets).  One CTA.
//    The active part of the band at step j is the dense (kl+1) x (kv+1) block
//    of the rows at positions j..j+kl and columns j..j+kv.  Nothing in it
//    moves: a row keeps its slot from the step it enters to the step it is
//    chosen as a pivot, a column keeps its slot (column mod C, C = kv+1), and
//    the slots of the retired pivot row and of column j are given to the
//    entering row j+1+kl and the entering column j+C.
//      Warp 0 (the panel) runs the pivot chain: lane = row slot, columns j, j+1
//    and j+2 in registers.  It finds the pivot (one reduction, beside every
//    candidate's reciprocal), forms the multipliers, publishes them, applies step
//    j to column j+1, which is the next pivot column, and, off the chain, to
//    column j+2, which it takes from the updaters with steps 0..j-1 applied.
//      12 updater warps own the other elements in registers, one (row slot,
//    column slot) a lane and plane, row slots fastest; each step they apply the
//    rank-1 update to columns j+3..j+kv and write their elements through to the
//    next step's copy of the window in shared memory, from which the next pivot
//    row and the panel's next column are read.
//      Three I/O warps move data: two the finished U row, the pivot and the
//    multipliers to AB, one the rows that enter the window from AB into a ring kEnt
//    steps deep (cp.async).  They share no SMSP with the panel (up to four planes): there
//    their instructions took the panel's issue slots.
//      Four named barriers hand over (Pub and Col below).
//    What bounds it: the panel warp's instruction stream and chain, 290 ns a column (argmax |
//    reciprocal -> shuffle -> DMUL -> DFMA), and beside it the updaters' FP64 instructions
//    on the SM's one unit (18.4 clk each; kl = ku = 27 issues 51 a column: 450 ns).  Loops
//    are unrolled by the publication's depth, so that barrier numbers and buffer offsets are
//    constants, and warps skip planes that hold none of their elements.  Measured at n =
//    4096, ns a column, against the first kernel of this layout / its predecessor (logical
//    rows, an exact two-word argmax, a helper warp on column j+2): kl = ku = 5: 289 / 349 /
//    394; 16: 316 / 384 / 411; kl = 8, ku = 64: 359 / 426 / 494; kl = ku = 27: 560 / 738 /
//    1029; kl = 27, ku = 74: 933 / 984 / 1337.
//
//  * k_gbtrf_generic (any kl, ku).  One CTA works directly on AB in global
//    memory (the active window stays L2-resident), one column at a time.
//
// Both follow the xGBTRF order of operations exactly (first-max pivot,
// interchange, reciprocal then multiply, fma(-l, u, a) updates applied in
// column order, zero-u skip), so they reproduce the unblocked elimination
// bit for bit.  Entries of U beyond the running column reach ju are structural
// zeros in both interchanged rows, so interchanging and (skipped) updating the
// whole window is the same as LAPACK's restriction to columns j..ju.
#include <climits>
#include <type_traits>

#include "common.cuh"
#include "rcp.cuh"
#include "regwin.cuh"
#include "sync.cuh"

namespace bandlu {
namespace {

constexpr int kWinMaxKl = 27;
constexpr int kWinMaxTrail = 2816;  // elements a step updates beyond column j+2 (so L*C <= 2900 <= 8 * kNUT)
constexpr int kNU = 12;            // updater warps: warps 1..15 but 4, 8, 12 (none on the panel's SMSP)
constexpr int kNUT = 32 * kNU;     // updater threads
// Warps of a window kernel with K planes: warp 0 panel, 12 updaters, 3 I/O warps.  The I/O warps
// stay off the panel's SMSP too (warps 17..19; 4, 8, 12 and 16 leave at once) where registers
// allow 20 warps.
constexpr int kWinWarps = 20;
constexpr int win_warps(int K) { return K <= 4 ? kWinWarps : 16; }
constexpr int kEnt = 16;           // entering rows in shared memory (a power of two)
constexpr int kAhead = 12;         // steps an entering row is asked for before its step
constexpr int kPub = 4;            // published steps kept

// What a step publishes beside its multipliers.
struct __align__(16) StepMeta {
  int wl;     // row slot of the pivot row
  int zp;     // exact zero pivot
  int p;      // pivot offset
  int pad;
  double u1;  // U(j, j+1)
  double pad2;
};

// Named barriers of the window kernel (0 is __syncthreads), two of each kind for
// even and odd steps:
//   Pub(j) = kBarPub0 + (j & 1): the panel arrives once step j is published; the
//            updaters and the I/O warps sync on it, so it also orders all their
//            step j-1 work before any step j.
//   Col(j) = kBarCol0 + (j & 1): the updaters arrive once they hold step j; the panel
//            syncs on it in step j+1, before it reads column j+3.
// Every participating warp executes its barrier operations unconditionally, once per
// step.  No barrier has two open phases: the panel arrives at Pub(j) after its sync on
// Col(j-2), which the updaters reach only after Pub(j-2) has completed; the updaters
// arrive at Col(j) after Pub(j), which needs the panel's arrival after its sync on
// Col(j-2).
// Buffers: step j's publication (slot j % kPub) is overwritten by step j+4, published
// after Col(j+2), so after Pub(j+2), which every reader joined after its step j+1.  The
// window copy of step j (j & 1) is overwritten in step j+1 by updaters that have passed
// Pub(j+1): the panel arrives there after its reads of step j, the others sync there
// after theirs.  Entering rows: the row of step j+kAhead is asked for after Pub(j) and
// takes the slot of step j-4's, which the panel read before it arrived at Pub(j-4) and
// the updaters read before Pub(j-3).  Rows of steps up to s+3 have landed before the
// row-in warp joins Pub(s); the panel reads that of step j after Col(j-2), so after
// Pub(j-2), the updaters after Pub(j).
constexpr int kBarPub0 = 1, kBarCol0 = 3;
constexpr int kPubCount = 32 * (1 + kNU + 3);
constexpr int kColCount = 32 * (1 + kNU);

#ifdef BANDLU_BOUNDED_SYNC
// Checked build (development and tests only): the same protocol on mbarriers
// with bounded waits.  A protocol slip (a missing participant, a miscounted
// barrier) ends the kernel with info = -BANDLU_ERR_TIMEOUT instead of a hang.
struct BarState {
  unsigned long long mb[5];
  int abort_flag;
};
__device__ __forceinline__ void bar_init(BarState &st) {
  mbar_init(&st.mb[kBarPub0], kPubCount / 32);
  mbar_init(&st.mb[kBarPub0 + 1], kPubCount / 32);
  mbar_init(&st.mb[kBarCol0], kColCount / 32);
  mbar_init(&st.mb[kBarCol0 + 1], kColCount / 32);
  st.abort_flag = 0;
}
__device__ __forceinline__ void bar_arrive_x(BarState &st, int id) {
  __syncwarp();
  if ((threadIdx.x & 31) == 0) mbar_arrive(&st.mb[id]);
}
// phase: how many times this warp has synced on barrier `id` so far
__device__ __forceinline__ bool bar_sync_x(BarState &st, int id, unsigned phase) {
  bar_arrive_x(st, id);
  return mbar_wait_warp(&st.mb[id], phase & 1u, &st.abort_flag);
}
#define BAR_SYNC(id, count, phase) bar_sync_x(sh.bars, (id), (unsigned)(phase))
#define BAR_ARRIVE(id, count) bar_arrive_x(sh.bars, (id))
#define BAR_FAILED() (sh.bars.abort_flag != 0)
#else
__device__ __forceinline__ bool bar_sync(int id, int count) {
  asm volatile("bar.sync %0, %1;" ::"r"(id), "r"(count) : "memory");
  return true;
}
__device__ __forceinline__ void bar_arrive(int id, int count) {
  asm volatile("bar.arrive %0, %1;" ::"r"(id), "r"(count) : "memory");
}
#define BAR_SYNC(id, count, phase) bar_sync((id), (count))
#define BAR_ARRIVE(id, count) bar_arrive((id), (count))
#define BAR_FAILED() false
#endif

struct WinShared {
  StepMeta meta[kPub];
  double l[kPub][32];  // by row slot: the multiplier, the pivot itself for the pivot row
  int t[kPub][32];     // by row slot: the row's position after the interchange, less j
#ifdef BANDLU_BOUNDED_SYNC
  BarState bars;
#endif
};

// Asynchronous global -> shared copies (the entering rows).
__device__ __forceinline__ void cp_async8(double *dst, const double *src) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"((unsigned)__cvta_generic_to_shared(dst)), "l"(src)
               : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_async_wait() {
  asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory");
}

// The window factorisation (win_warps(K) warps or more), for k_gbtrf_window and the device-side
// dispatch.  W: window_smem(kl, ku) bytes of dynamic shared memory: two copies of
// the window, element (row slot r, column slot c) at c*L + r, and the ring of
// entering rows.  K: planes an updater thread holds, L*C <= K * kNUT.
template <int K>
__device__ __forceinline__ void window_factor(int n, int kl, int ku, double *__restrict__ AB, long long ldab,
                                              int *__restrict__ ipiv, int *__restrict__ d_info, double *W,
                                              WinShared &sh) {
  const int kv = kl + ku, L = kl + 1, C = kv + 1, LC = L * C;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  // the U rows, pivots and multipliers; the U rows' other columns; the entering rows
  constexpr int kRowOutWarp = K <= 4 ? 17 : 4, kRowOut2Warp = K <= 4 ? 18 : 12, kRowInWarp = K <= 4 ? 19 : 8;
  double *const ent = W + 2 * LC;  // row i's entry of the column in slot c: ent[(i - L) % kEnt * C + c]

#ifdef BANDLU_BOUNDED_SYNC
  if (threadIdx.x == 0) bar_init(sh.bars);
#endif
  // Fill-row entries of the top-left corner (element row < 0) are cleared, as
  // the elimination clears every fill row before it starts.
  for (int e = threadIdx.x; e < kl * kv; e += blockDim.x) {
    const int r = e / kv, c = e - r * kv;
    if (c < kv - r && c < n) AB[r + (long long)c * ldab] = 0.0;
  }
  // Rows 0..kl go to slots 0..kl, columns 0..kv to slots 0..kv.
  for (int e = threadIdx.x; e < LC; e += blockDim.x) {
    const int c = e / L, i = e - c * L;
    W[e] = (i < n && c < n && c <= i + ku) ? AB[(kv + i - c) + (long long)c * ldab] : 0.0;
  }
  // Row i = s+1+kl enters at step s; in slot c it has the column of s+1..s+1+kv that is c mod C.
  int first = 1 % C;  // slot of column s+1 for the next row asked for
  auto ask_row = [&](int s) {  // by one warp, s = 0, 1, ..: row of step s into the ring
    double *dst = ent + (s & (kEnt - 1)) * C;
    const double *src = AB + (kv + kl) + (long long)(s + 1) * ldab;  // its column s+1
    const int last = s + 1 + kl < n ? n - 2 - s : -1;                // columns past s+1 inside the matrix
    for (int c = lane; c < C; c += 32) {
      int d = c - first;
      if (d < 0) d += C;  // column s+1+d
      if (d <= last)
        cp_async8(dst + c, src + d * (ldab - 1));
      else
        dst[c] = 0.0;
    }
    first = first + 1 == C ? 0 : first + 1;
  };
  if (warp == kRowInWarp) {
    for (int s = 0; s < kAhead; ++s) ask_row(s);
    cp_async_commit();
    cp_async_wait<0>();
  }
  __syncthreads();

  int info = 0;
  if (warp == 0) {
    // ---------------- panel warp: the pivot chain ----------------
    // One pass of the loop runs from step j's multipliers to step j+1's pivot, so that the
    // work on column j+2 and the publication fill the latencies of the next pivot search.
    const int rs = min(lane, L - 1);  // a slot to read for the lanes that hold none
    int pos = lane < L ? lane : INT_MAX;
    double cur = W[rs], v1 = W[L + rs];  // columns j, j+1
    int q1 = 1, q2 = 2;                  // column slots of columns j+1, j+2 (C >= 3: factor_path)
    // the step's pivot: its slot, its offset, an exact zero; the multipliers; U(j, j+1)
    int wl = 0, p = 0;
    bool zp = false;
    double rc = 0.0, l = 0.0, u1 = 0.0;
    unsigned hk = 0, mh = 0;
    bool unsure = false;
    // The largest modulus by its high word, of which the low five bits make room for the
    // lane: one reduction gives the winner, provided it is alone with its upper 27 bits,
    // nonzero and no infinity or NaN (checked beside the chain; else decided in full).
    auto search = [&]() {
      hk = pos < n ? ((unsigned)__double2hiint(cur) & 0x7fffffe0u) | lane : 0u;
      mh = __reduce_max_sync(FULL, hk);
      rc = rcp_rn_quick(cur, &unsure);  // every candidate's, beside the reduction
      wl = mh & 31;
    };
    auto settle = [&](int j) {
      // the multipliers first: the checks run in the product's latency
      l = cur * __shfl_sync(FULL, rc, wl);
      u1 = __shfl_sync(FULL, v1, wl);
      p = __shfl_sync(FULL, pos, wl) - j;
      zp = false;
      const unsigned same = __ballot_sync(FULL, hk >= (mh & ~31u) && hk >= 32u);
      const unsigned odd = __ballot_sync(FULL, unsure) >> wl;
      if ((same & (same - 1u)) != 0u || (odd & 1u) != 0u || mh - 32u >= 0x7ff00000u - 32u) {  // uniform, rare
        // exact keys, then the lowest position
        const unsigned long long key = pos < n ? pivot_abs_key(cur, pos == j) : 0ull;
        const unsigned m1 = __reduce_max_sync(FULL, (unsigned)(key >> 32));
        const unsigned m2 = __reduce_max_sync(FULL, (unsigned)(key >> 32) == m1 ? (unsigned)key : 0u);
        const bool top = pos < n && key == (((unsigned long long)m1 << 32) | m2);
        const int mp = __reduce_min_sync(FULL, top ? pos : INT_MAX);
        wl = __ffs(__ballot_sync(FULL, top && pos == mp)) - 1;
        zp = (m1 | m2) == 0u;
        u1 = __shfl_sync(FULL, v1, wl);
        p = mp - j;
        const double pv = __shfl_sync(FULL, cur, wl);
        if (!zp) l = cur * rcp_division(pv);
        if (zp && info == 0) info = j + 1;
      }
    };
    search();
    settle(0);
    bool ok = true;
    for (int j0 = 0; ok && j0 < n; j0 += kPub) {
#pragma unroll
      for (int b = 0; b < kPub; ++b) {
        const int j = j0 + b;
        if (j >= n) break;
        const double *en = ent + (j & (kEnt - 1)) * C;
        const bool piv = lane == wl;
        const int np = pos == j ? j + p : pos;
        sh.t[b][lane] = np - j;
        if (piv) {
          *reinterpret_cast<int4 *>(&sh.meta[b]) = make_int4(wl, zp ? 1 : 0, p, 0);
          sh.meta[b].u1 = u1;
        }
        const double e1 = en[q1], e2 = en[q2];  // the entering row's columns j+1, j+2
        const double t1 = fma(-l, u1, v1);
        sh.l[b][lane] = (piv || zp) ? cur : l;
        __syncwarp();
        BAR_ARRIVE(kBarPub0 + (b & 1), kPubCount);
        // step j on column j+2 (steps 0..j-1 applied by the updaters), in column j+1's latency and
        // the next search's
        if (j >= 1) ok = BAR_SYNC(kBarCol0 + ((b + 1) & 1), kColCount, (j - 1) >> 1);
        if (!ok) break;
        const double v2 = W[(b & 1) * LC + q2 * L + rs];
        const double u2 = __shfl_sync(FULL, v2, wl);
        const double t2 = fma(-l, u2, v2);
        const bool act2 = nz(u2) && !zp;
        cur = piv ? e1 : ((nz(u1) && !zp) ? t1 : v1);
        pos = piv ? j + 1 + kl : np;
        search();
        v1 = piv ? e2 : (act2 ? t2 : v2);
        q1 = q2;
        q2 = q2 + 1 == C ? 0 : q2 + 1;
        if (j + 1 < n) settle(j + 1);
      }
    }
    if (ok) BAR_SYNC(kBarCol0 + ((n - 1) & 1), kColCount, (n - 1) >> 1);  // the updaters' arrival of the last step
  } else if (warp == kRowOutWarp || warp == kRowOut2Warp) {
    // ---------------- U row, pivot and multipliers of step j to AB ----------------
    int jc = 0;
    bool ok = true;
    for (int j0 = 0; ok && j0 < n; j0 += kPub) {
#pragma unroll
      for (int b = 0; b < kPub; ++b) {
        const int j = j0 + b;
        if (j >= n) break;
        ok = BAR_SYNC(kBarPub0 + (b & 1), kPubCount, j >> 1);
        if (!ok) break;
        const int wl = sh.meta[b].wl;
        const double *Wj = W + (b & 1) * LC + wl;
        double *ABj = AB + (long long)j * ldab;
        if (warp == kRowOutWarp) {
          const double l = sh.l[b][lane];
          const int t = sh.t[b][lane];
          if (lane == 0) ipiv[j] = j + sh.meta[b].p + 1;
          if (lane < L && lane != wl && t < n - j) ABj[kv + t] = l;
        }
        for (int c = lane + (warp == kRowOutWarp ? 0 : 32); c < C; c += 64) {
          int d = c - jc;  // column j+d
          if (d < 0) d += C;
          const double u = d >= 2 ? Wj[c * L] : (d == 1 ? sh.meta[b].u1 : sh.l[b][wl]);
          if (d < n - j) ABj[(kv - d) + (long long)d * ldab] = u;
        }
        jc = jc + 1 == C ? 0 : jc + 1;
      }
    }
  } else if (warp == kRowInWarp) {
    // ---------------- entering rows ----------------
    // Before this warp joins step s's kBarPub, every row but those asked for in the
    // last kAhead - 4 steps has landed: the rows of steps up to s+3.
    bool ok = true;
    for (int j0 = 0; ok && j0 < n; j0 += 2) {
#pragma unroll
      for (int b = 0; b < 2; ++b) {
        const int j = j0 + b;
        if (j >= n) break;
        cp_async_wait<kAhead - 4>();
        ok = BAR_SYNC(kBarPub0 + b, kPubCount, j >> 1);
        if (!ok) break;
        ask_row(j + kAhead);
        cp_async_commit();
      }
    }
    cp_async_wait<0>();
  } else if ((warp & 3) != 0 && warp < 16) {
    // ---------------- updater warps: columns j+3 .. j+kv ----------------
    const int tu = (warp - 1 - (warp >> 2)) * 32 + lane;  // warps 1,2,3,5,6,7,9,.. -> 0..kNU-1
    int rs[K], cL[K], cs[K], coff[K];  // row slot, c*L, column slot (-1: no element), columns after j
    double w[K];
#pragma unroll
    for (int k = 0; k < K; ++k) {
      const int e = tu + kNUT * k;
      const bool has = e < LC;
      const int c = has ? e / L : 0;
      rs[k] = has ? e - c * L : 0;
      cs[k] = has ? c : -1;
      cL[k] = c * L;
      coff[k] = c;
      w[k] = W[cL[k] + rs[k]];
    }
    // P: planes this warp holds elements of (uniform; the last planes may be short of warps, and
    // a multiply-add without an element would still take its turn on the FP64 unit)
    auto steps = [&](auto planes) {
      constexpr int P = decltype(planes)::value;
      bool ok = true;
      for (int j0 = 0; ok && j0 < n; j0 += kPub) {
#pragma unroll
        for (int b = 0; b < kPub; ++b) {
          const int j = j0 + b;
          if (j >= n) break;
          ok = BAR_SYNC(kBarPub0 + (b & 1), kPubCount, j >> 1);
          if (!ok) break;
          if constexpr (P > 0) {
            const double *Wj = W + (b & 1) * LC;
            double *Wn = W + ((b & 1) ^ 1) * LC;
            const double *en = ent + (j & (kEnt - 1)) * C;
            const int2 m = *reinterpret_cast<const int2 *>(&sh.meta[b]);
            const int wl = m.x;
            const bool zp = m.y != 0;
            double l[P], u[P], t[P];
#pragma unroll
            for (int k = 0; k < P; ++k) l[k] = sh.l[b][rs[k]];
#pragma unroll
            for (int k = 0; k < P; ++k) u[k] = Wj[cL[k] + wl];
#pragma unroll
            for (int k = 0; k < P; ++k) t[k] = fma(-l[k], u[k], w[k]);
#pragma unroll
            for (int k = 0; k < P; ++k) {
              const bool piv = rs[k] == wl;
              // a slot that changes hands (the pivot row's, column j's), or no update
              double keep = coff[k] == 0 ? 0.0 : w[k];
              if (piv) keep = en[max(cs[k], 0)];
              const bool up = coff[k] >= 3 && !piv && !zp && nz(u[k]);
              w[k] = up ? t[k] : keep;
              if (cs[k] >= 0) Wn[cL[k] + rs[k]] = w[k];
              coff[k] = coff[k] == 0 ? kv : coff[k] - 1;
            }
            __syncwarp();
          }
          BAR_ARRIVE(kBarCol0 + (b & 1), kColCount);
        }
      }
    };
    const int planes = (LC - (tu - lane) + kNUT - 1) / kNUT;
    if (planes >= K) steps(std::integral_constant<int, K>());
    else if (planes == K - 1) steps(std::integral_constant<int, K - 1>());
    else steps(std::integral_constant<int, (K > 2 ? K - 2 : 0)>());
  }
  __syncthreads();
  if (threadIdx.x == 0) *d_info = BAR_FAILED() ? -BANDLU_ERR_TIMEOUT : info;
}

template <int K>
__global__ void __launch_bounds__(win_warps(K) * 32, 1) k_gbtrf_window(int n, int kl, int ku, double *__restrict__ AB,
                                                                  long long ldab, int *__restrict__ ipiv,
                                                                  int *__restrict__ d_info) {
  extern __shared__ double W[];
  __shared__ WinShared sh;
  window_factor<K>(n, kl, ku, AB, ldab, ipiv, d_info, W, sh);
}

// Column-by-column elimination by the whole block (any block size) on AB in
// global memory, for k_gbtrf_generic and the device-side dispatch.
__device__ __forceinline__ void generic_factor(long long n, int kl, int ku, double *__restrict__ AB, long long ldab,
                                               int *__restrict__ ipiv, int *__restrict__ d_info) {
  __shared__ KeyIdx s_red[32];
  __shared__ int s_p;
  __shared__ double s_r;
  const long long kv = (long long)kl + ku;
  const int tid = threadIdx.x, B = blockDim.x, lane = tid & 31, warp = tid >> 5, nw = B >> 5;
  if (kl > 0) {
    for (long long e = tid; e < n * kl; e += B) {
      const long long c = e / kl, r = e - c * kl;
      AB[r + c * ldab] = 0.0;
    }
  }
  __syncthreads();
  long long ju = 0;
  int info = 0;
  for (long long j = 0; j < n; ++j) {
    const long long km = min((long long)kl, n - 1 - j);
    double *colj = AB + j * ldab;
    KeyIdx best{0ull, LLONG_MAX};
    for (long long t = tid; t <= km; t += B) best = better(best, KeyIdx{pivot_abs_key(colj[kv + t], t == 0), t});
    best = warp_reduce_keyidx(best);
    if (lane == 0) s_red[warp] = best;
    __syncthreads();
    if (warp == 0) {
      KeyIdx v = lane < nw ? s_red[lane] : KeyIdx{0ull, LLONG_MAX};
      v = warp_reduce_keyidx(v);
      if (lane == 0) s_p = (int)v.idx;
    }
    __syncthreads();
    const long long p = s_p;
    const double piv = colj[kv + p];
    if (tid == 0) ipiv[j] = (int)(j + p + 1);
    if (nz(piv)) {
      ju = max(ju, min(j + ku + p, n - 1));
      if (p != 0) {
        for (long long c = j + tid; c <= ju; c += B) {
          double *x = AB + (kv + j - c) + c * ldab;
          double *y = AB + (kv + j + p - c) + c * ldab;
          const double t0 = *x;
          *x = *y;
          *y = t0;
        }
        __syncthreads();
      }
      if (km > 0) {
        if (tid == 0) s_r = 1.0 / colj[kv];
        __syncthreads();
        const double r = s_r;
        for (long long t = 1 + tid; t <= km; t += B) colj[kv + t] *= r;
        __syncthreads();
        const long long tot = (ju - j) * km;
        for (long long e = tid; e < tot; e += B) {
          const long long cc = e / km, t = 1 + (e - cc * km);
          const long long c = j + 1 + cc;
          double *colc = AB + c * ldab;
          const double u = colc[kv + j - c];
          if (nz(u)) colc[kv + j + t - c] = fma(-colj[kv + t], u, colc[kv + j + t - c]);
        }
        __syncthreads();
      }
    } else if (info == 0) {
      info = (int)(j + 1);
    }
  }
  if (tid == 0) *d_info = info;
}

__global__ void __launch_bounds__(1024) k_gbtrf_generic(long long n, int kl, int ku, double *__restrict__ AB,
                                                         long long ldab, int *__restrict__ ipiv,
                                                         int *__restrict__ d_info) {
  generic_factor(n, kl, ku, AB, ldab, ipiv, d_info);
}

// The narrowest bands, (kl+1)*(kl+ku+1) <= 32: one warp with the active window
// in registers (regwin.cuh).  Fill-row entries above the matrix are cleared
// first, as the elimination clears every fill row; the window writes the rest.
// Called by one whole warp.
template <class Off>
__device__ __forceinline__ void regwin_factor(int n, int kl, int ku, double *__restrict__ AB, Off ldab,
                                              int *__restrict__ ipiv, int *__restrict__ d_info) {
  const int kv = kl + ku, lane = threadIdx.x & 31;
  if (kl > 0) {
    for (int e = lane; e < kl * min(n, kv); e += 32) {
      const int jj = e / kl, rr = e - jj * kl;
      if (rr < kv - jj) AB[rr + jj * ldab] = 0.0;
    }
  }
  __syncwarp();
  double *const abp[1] = {AB};
  int *const pvp[1] = {ipiv};
  const int klv[1] = {kl}, kuv[1] = {ku};
  int info[1];
  regwin::window_gbtrf<1, 1, Off>(abp, ldab, n, klv, kuv, pvp, info);
  if (lane == 0) *d_info = info[0];
}

template <class Off>
__global__ void __launch_bounds__(32) k_gbtrf_regwin(int n, int kl, int ku, double *__restrict__ AB, Off ldab,
                                                     int *__restrict__ ipiv, int *__restrict__ d_info) {
  regwin_factor<Off>(n, kl, ku, AB, ldab, ipiv, d_info);
}

// The register window's 32-bit offsets reach every entry.
__host__ __device__ inline bool offsets_fit(long long n, long long ldab) {
  return ldab <= (INT_MAX - 1) / (n + 1);  // (n + 1) * ldab < INT_MAX
}

// The path choice of launch_gbtrf (without the multi-CTA kernel), shared by the
// host launcher and the device-side dispatch: 0 register window, 1 shared-memory
// window (*K: its template parameter, *smem: its bytes), 2 generic.  Every band with
// L*C <= 32 takes path 0, whatever its storage, so path 1 has C >= 6 (C >= L); its
// panel warp requires 3 (columns j+1 and j+2 beside column j, in slots of their own).
// The windows count rows a few steps past the last one in 32 bits.
__host__ __device__ inline int factor_path(long long n, int kl, int ku, long long ldab, int *K, size_t *smem) {
  const long long kv = (long long)kl + ku;
  const long long L = kl + 1LL, C = kv + 1;
  if (n > INT_MAX - 64) return 2;
  if (L * C <= 32) return 0;
  if (kl <= kWinMaxKl && kl + kv + 1 <= 256 && L * (kv - 2) <= kWinMaxTrail) {
    const int k = (int)((L * C + kNUT - 1) / kNUT);
    *smem = (size_t)((2 * L + kEnt) * C) * sizeof(double);
    *K = k <= 4 ? k : (k <= 6 ? 6 : 8);  // (K - 2 planes at least are full)
    return 1;
  }
  return 2;
}

__device__ __forceinline__ void window_factor_k(int K, int n, int kl, int ku, double *AB, long long ldab, int *ipiv,
                                                int *d_info, double *W, WinShared &sh) {
  if (K == 1) window_factor<1>(n, kl, ku, AB, ldab, ipiv, d_info, W, sh);
  else if (K == 2) window_factor<2>(n, kl, ku, AB, ldab, ipiv, d_info, W, sh);
  else if (K == 3) window_factor<3>(n, kl, ku, AB, ldab, ipiv, d_info, W, sh);
  else if (K == 4) window_factor<4>(n, kl, ku, AB, ldab, ipiv, d_info, W, sh);
  else if (K == 6) window_factor<6>(n, kl, ku, AB, ldab, ipiv, d_info, W, sh);
  else window_factor<8>(n, kl, ku, AB, ldab, ipiv, d_info, W, sh);
}

// Device-side dispatch: the factorisation of dispatch_lu_async, with (kl, ku)
// and the dispatch decision read from device memory.  kWinWarps warps and
// smem_bytes of dynamic shared memory, enough for every shared-memory window
// that fits the band storage (2*kl+ku+1 <= ldab); the block takes the path
// launch_gbtrf would take.  A band beyond the windows is left to the multi-CTA
// kernel enqueued behind this one where that kernel takes it (up to wide_rows_cap
// panel rows); else the block runs the generic elimination itself.
// All windows share the 96 registers of 640 threads, and the widest spill (120 bytes):
// n = 4096, us dispatch_lu / dispatch_lu_async: kl = ku = 16 1509 / 1406, 27 2509 / 2408, kl = 27, ku =
// 74 4042 / 4091, kl = 20, ku = 100 3668 / 3723 (dispatch_lu's host round trip and scratch take about 90).
__global__ void __launch_bounds__(kWinWarps * 32, 1) k_gbtrf_on_device(int n, double *__restrict__ AB, long long ldab,
                                                                     int *__restrict__ ipiv,
                                                                     const int *__restrict__ d_kl,
                                                                     const int *__restrict__ d_ku,
                                                                     const int *__restrict__ d_status,
                                                                     int *__restrict__ d_info, size_t smem_bytes,
                                                                     int wide_rows_cap, int *__restrict__ wide_flag) {
  extern __shared__ double W[];
  __shared__ WinShared sh;
  if (*d_status != BANDLU_OK) return;  // declined: nothing is written
  const int kl = *d_kl, ku = *d_ku;
  int K = 1;
  size_t smem = 0;
  int path = factor_path(n, kl, ku, ldab, &K, &smem);
  if (path == 1 && smem > smem_bytes) path = 2;
  if (path == 2 && wide_flag != nullptr && wide_pair_takes(n, kl, ku, wide_rows_cap)) {
    // the cluster-pair kernel enqueued after this one factors the band
    if (threadIdx.x == 0) *wide_flag = 1;
    return;
  }
  if (path == 0) {
    if (threadIdx.x < 32) {
      if (offsets_fit(n, ldab)) regwin_factor<unsigned>(n, kl, ku, AB, (unsigned)ldab, ipiv, d_info);
      else regwin_factor<long long>(n, kl, ku, AB, ldab, ipiv, d_info);
    }
  } else if (path == 1) {
    window_factor_k(K, n, kl, ku, AB, ldab, ipiv, d_info, W, sh);
  } else {
    generic_factor(n, kl, ku, AB, ldab, ipiv, d_info);
  }
}

template <int K>
int launch_window(long long n, int kl, int ku, double *AB, long long ldab, int *ipiv, int *d_info, size_t smem,
                  cudaStream_t s) {
  if (!allow_dynamic_smem(reinterpret_cast<const void *>(k_gbtrf_window<K>), 200 * 1024)) return BANDLU_ERR_CUDA;
  k_gbtrf_window<K><<<1, win_warps(K) * 32, smem, s>>>((int)n, kl, ku, AB, ldab, ipiv, d_info);
  BANDLU_CHECK_LAUNCH();
  return BANDLU_OK;
}

}  // namespace

int gbtrf_path(int64_t n, int kl, int ku, int64_t ldab) {
  int K = 0;
  size_t smem = 0;
  return factor_path(n, kl, ku, ldab, &K, &smem);
}

int launch_gbtrf(int64_t n, int kl, int ku, double *AB, int64_t ldab, int *ipiv, int *d_info, cudaStream_t s,
                 bool allow_alloc) {
  if (n == 0) {
    if (cudaMemsetAsync(d_info, 0, sizeof(int), s) != cudaSuccess) return BANDLU_ERR_CUDA;
    return BANDLU_OK;
  }
  int K = 1;
  size_t smem = 0;
  const int path = factor_path(n, kl, ku, ldab, &K, &smem);
  if (path == 0) {
    if (offsets_fit(n, ldab)) k_gbtrf_regwin<unsigned><<<1, 32, 0, s>>>((int)n, kl, ku, AB, (unsigned)ldab, ipiv, d_info);
    else k_gbtrf_regwin<long long><<<1, 32, 0, s>>>((int)n, kl, ku, AB, ldab, ipiv, d_info);
    BANDLU_CHECK_LAUNCH();
    return BANDLU_OK;
  }
  if (path == 1) {
    if (K == 1) return launch_window<1>(n, kl, ku, AB, ldab, ipiv, d_info, smem, s);
    if (K == 2) return launch_window<2>(n, kl, ku, AB, ldab, ipiv, d_info, smem, s);
    if (K == 3) return launch_window<3>(n, kl, ku, AB, ldab, ipiv, d_info, smem, s);
    if (K == 4) return launch_window<4>(n, kl, ku, AB, ldab, ipiv, d_info, smem, s);
    if (K == 6) return launch_window<6>(n, kl, ku, AB, ldab, ipiv, d_info, smem, s);
    return launch_window<8>(n, kl, ku, AB, ldab, ipiv, d_info, smem, s);
  }
  if (allow_alloc) {
    bool used = false;
    const int rc = launch_gbtrf_wide(n, kl, ku, AB, ldab, ipiv, d_info, s, &used);
    if (rc != BANDLU_OK || used) return rc;
  }
  k_gbtrf_generic<<<1, 1024, 0, s>>>(n, kl, ku, AB, ldab, ipiv, d_info);
  BANDLU_CHECK_LAUNCH();
  return BANDLU_OK;
}

}  // namespace bandlu

namespace bandlu {

int launch_gbtrf_on_device(int64_t n, double *AB, int64_t ldab, int *ipiv, const int *d_kl, const int *d_ku,
                           const int *d_status, int *d_info, cudaStream_t s) {
  if (n == 0) return BANDLU_OK;
  // every shared-memory window that fits the band storage: C = kl+ku+1 <= min(ldab, 256)
  // columns and L*C <= (kWinMaxKl+1)*C elements, at most kWinMaxTrail + 3*(kWinMaxKl+1)
  const long long cs = ldab < 256 ? ldab : 256;
  const long long most = kWinMaxTrail + 3 * (kWinMaxKl + 1);
  const long long lc = (kWinMaxKl + 1) * cs < most ? (kWinMaxKl + 1) * cs : most;
  const size_t smem = (size_t)(2 * lc + kEnt * cs) * sizeof(double);
  if (!allow_dynamic_smem(reinterpret_cast<const void *>(k_gbtrf_on_device), 200 * 1024)) return BANDLU_ERR_CUDA;
  // a band storage that admits kl >= kWinMaxKl + 1 may hold a band no window takes:
  // the multi-CTA kernel is enqueued too and runs only if the decision on the device is its
  WideDeferred wd;
  if (ldab >= 2 * (kWinMaxKl + 1) + 1) {
    const int rc = prepare_gbtrf_wide_deferred(n, ldab, s, &wd);
    if (rc != BANDLU_OK) return rc;
  }
  k_gbtrf_on_device<<<1, kWinWarps * 32, smem, s>>>((int)n, AB, ldab, ipiv, d_kl, d_ku, d_status, d_info, smem,
                                                 wd.rows_cap, wd.flags != nullptr ? wd.flags + 1 : nullptr);
  if (cudaPeekAtLastError() != cudaSuccess) {
    if (wd.flags != nullptr) cudaFreeAsync(wd.flags, s);
    return BANDLU_ERR_CUDA;
  }
  if (wd.rows_cap > 0) return launch_gbtrf_wide_deferred(wd, n, AB, ldab, ipiv, d_kl, d_ku, d_info, s);
  return BANDLU_OK;
}

}  // namespace bandlu
