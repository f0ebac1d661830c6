// regwin.cuh -- banded LU with the active window (kl+1) x (kl+ku+1) in the
// registers of one warp (Sec. II-A step 3; f(N) ~ O(N*P*Q), Eq. S-N-N3).  Used
// by the single-matrix gbtrf for the narrowest bands and by the batched
// factorisation.
#pragma once

#include <climits>

#include "common.cuh"
#include "rcp.cuh"

namespace bandlu {
namespace regwin {

constexpr int kWinPrefetch = 8;  // entering rows a window keeps in flight

// Rows per register plane and planes of a window of kl+1 rows, kv+1 columns in a
// segment of W lanes.
__host__ __device__ __forceinline__ int planes_of(int kl, int kv, int W) {
  const int C = kv + 1;
  if (C > W) return INT_MAX;
  const int rr = W / C;
  return (kl + rr) / rr;  // ceil((kl+1) / rr)
}

// Banded elimination with the active window in registers, in place on band
// storage (ldab x n).  It reads only the band's own entries and writes U's rows
// and the multipliers; fill-row entries above the matrix, which no step
// writes, are the caller's (the elimination clears them).  The warp is cut into S
// segments of W = 32/S lanes; segment s factors its own matrix (ab[s], kl[s],
// ku[s], ipiv[s]), all of the same order n.  Every warp instruction thus serves S
// matrices.  NR registers a lane (NR = 1 when S > 1): planes_of(kl, kv, W) <= NR.
//
// At step j a segment's window holds the physical rows at positions j..j+kl and
// columns j..j+kv (kv = kl+ku).  Nothing moves between lanes: a row keeps its slot
// from the step it enters to the step it is chosen as a pivot (pos: its current
// position; an interchange changes pos), a column keeps its slot (column mod C,
// C = kv+1), and the slots of the retired pivot row and of column j are given to
// the entering row j+1+kl and the entering column j+C.  Row slot s sits in plane
// s / RR on segment lanes (s % RR)*C .. +C-1.  (The former layout kept rows and
// columns in order: two 64-bit shuffles for the interchange and one for the move
// down the diagonal, at 16 clk a 32-bit shuffle, sat on every step's chain.)
// Step j: first-max argmax over column j, beside it each candidate's reciprocal and
// the copy of column j to every lane of its row; then one shuffle of the winner's
// reciprocal, the multiplier (formed by every lane of the row), the rank-1 update
// with the zero-u skip.  The pivot row (U row j) and column j's multipliers are
// written to their places in AB.  The entering column holds structural zeros except
// in the entering row, which is the untouched original row, read kWinPrefetch steps
// ahead (every lane holds its column's entry, so any slot can take it).  Every AB
// entry a step writes belongs to a row that entered the window earlier, so reading
// and writing in place do not collide.  Same operations in the same order as the
// unblocked elimination: the factors are bit-identical to it.
// Off: the type of offsets into AB; unsigned requires (n+1) * ldab < 2^31, long long takes any
// storage.  A lane's offsets run on past column n, by up to C + kWinPrefetch columns, to places
// that nothing reads: a 32-bit type must wrap there, not overflow.
template <int S, int NR, class Off>
__device__ __forceinline__ void window_gbtrf(double *const (&abs)[S], Off ldab, int n, const int (&kls)[S],
                                             const int (&kus)[S], int *const (&ipivs)[S], int (&infos)[S]) {
  static_assert(S == 1 || NR == 1, "several segments or several planes");
  static_assert(sizeof(Off) == 8 || Off(-1) > Off(0), "32-bit offsets wrap");
  constexpr int W = 32 / S;
  const int lane = threadIdx.x & 31;
  const int seg = lane / W, sl = lane - seg * W, base = seg * W;
  int kl = kls[0], ku = kus[0];
  double *ab = abs[0];
  int *ipiv = ipivs[0];
#pragma unroll
  for (int t = 1; t < S; ++t)
    if (seg == t) {
      kl = kls[t];
      ku = kus[t];
      ab = abs[t];
      ipiv = ipivs[t];
    }
  const int kv = kl + ku, C = kv + 1, L = kl + 1;
  const int RR = W / C;  // row slots of a plane
  const bool inw = sl < RR * C;
  const int r = inw ? sl / C : 0, c = inw ? sl - r * C : 0;
  const int rb = base + r * C;  // first lane of this row
  double w[NR];
  int pos[NR];  // position of the row in plane k's slot here (n or more: none)
#pragma unroll
  for (int k = 0; k < NR; ++k) {
    const int s = k * RR + r;
    pos[k] = (inw && s < L) ? s : INT_MAX;
    w[k] = 0.0;
    if (pos[k] < n && c < n && c - s <= ku) w[k] = __ldcg(ab + (kv + s - c) + c * ldab);
  }
  // this lane's column in the window: coff columns after j, at ab + cb
  int coff = c;
  Off cb = c * ldab;
  int jc = 0;  // column slot of column j
  // q[s] holds the entry of the entering row of the next step j with j % kWinPrefetch == s
  // (row j+1+kl) in this lane's column of that window (columns j+1..j+1+kv); it is refilled
  // kWinPrefetch steps ahead.  The step loop is unrolled by kWinPrefetch so that every slot is
  // one register (rotating the slots would wait on each load a step after issuing it).
  int qoff = c == 0 ? kv : c - 1, qcol = c == 0 ? C : c;  // for the next refill: offset in its window, column
  Off qat = (kv + kl - qoff) + qcol * ldab;
  double q[kWinPrefetch];
  auto refill = [&](int row) {
    double v = 0.0;
    if (inw && row < n && qcol < n) v = __ldcg(ab + qat);
    const bool wrap = qoff == 0;
    qat += wrap ? C * ldab - kv : 1;
    qcol += wrap ? C : 0;
    qoff = wrap ? kv : qoff - 1;
    return v;
  };
#pragma unroll
  for (int k = 0; k < kWinPrefetch; ++k) q[k] = refill(kl + 1 + k);
  int info = 0;
  auto step = [&](int j, double &qs) {
    const bool head = inw && coff == 0;  // this lane's column is column j
    const int hl = inw ? rb + jc : lane;
    // every lane's copy of its row's entry of column j
    double a[NR];
#pragma unroll
    for (int k = 0; k < NR; ++k) a[k] = __shfl_sync(FULL, w[k], hl);
    // The largest modulus of the segment by its high word, of which the low five bits make
    // room for the lane: one reduction gives the winner, provided it is alone with its upper
    // 27 bits, nonzero and no infinity or NaN (checked beside the chain; else decided in full).
    unsigned hk[NR], hmax = 0;
#pragma unroll
    for (int k = 0; k < NR; ++k) {
      hk[k] = (head && pos[k] < n) ? ((unsigned)__double2hiint(w[k]) & 0x7fffffe0u) : 0u;
      hmax = max(hmax, hk[k]);
    }
    double cand = w[0];
    int mykp = 0, cnt = 0;
    if (NR > 1) {
#pragma unroll
      for (int k = 1; k < NR; ++k) {
        cand = hk[k] == hmax ? w[k] : cand;
        mykp = hk[k] == hmax ? k : mykp;
      }
#pragma unroll
      for (int k = 0; k < NR; ++k) cnt += hk[k] == hmax ? 1 : 0;
    }
    unsigned mh = 0, bad = 0;
#pragma unroll
    for (int t = 0; t < S; ++t) {
      const unsigned v = __reduce_max_sync(FULL, S == 1 || seg == t ? (hmax | lane) : 0u);
      if (S == 1 || seg == t) mh = v;
      bad |= (v - 32u >= 0x7ff00000u - 32u) ? 1u : 0u;
    }
    bool unsure;
    const double myr = rcp_rn_quick(cand, &unsure);
    int wl = mh & 31;  // the pivot row's lane of column j
    int kp = NR > 1 ? __shfl_sync(FULL, mykp, wl) : 0;
    bool zp = false;  // exact zero pivot (then the row at position j)
    double rc = __shfl_sync(FULL, myr, wl);
    double wsel = w[0];
    int psel = pos[0];
    auto pick = [&]() {  // the pivot row's plane
      wsel = w[0];
      psel = pos[0];
#pragma unroll
      for (int k = 1; k < NR; ++k) {
        wsel = kp == k ? w[k] : wsel;
        psel = kp == k ? pos[k] : psel;
      }
    };
    pick();
    double u = __shfl_sync(FULL, wsel, wl - jc + c);  // the pivot row's entry in this lane's column
    int p = __shfl_sync(FULL, psel, wl) - j;
    // not alone (a second candidate with the same upper bits), or the reciprocal is unsure
    const unsigned same = __ballot_sync(FULL, (hmax | lane) - (mh & ~31u) < 32u && hmax != 0u);
    const unsigned odd = __ballot_sync(FULL, (lane == wl && unsure) || (NR > 1 && hmax != 0u && cnt > 1));
    bool rare = (bad | odd) != 0u;
#pragma unroll
    for (int t = 0; t < S; ++t) {
      const unsigned v = S == 1 ? same : same & (((1u << (W & 31)) - 1u) << (t * W));
      rare = rare || (v & (v - 1u)) != 0u;
    }
    if (rare) {  // uniform: exact keys, then the lowest position
      unsigned long long key[NR];
      unsigned m1 = 0, m2 = 0, x1 = 0, x2 = 0;
#pragma unroll
      for (int k = 0; k < NR; ++k) {
        key[k] = (head && pos[k] < n) ? pivot_abs_key(w[k], pos[k] == j) : 0ull;
        x1 = max(x1, (unsigned)(key[k] >> 32));
      }
#pragma unroll
      for (int t = 0; t < S; ++t) {
        const unsigned v = __reduce_max_sync(FULL, S == 1 || seg == t ? x1 : 0u);
        if (S == 1 || seg == t) m1 = v;
      }
#pragma unroll
      for (int k = 0; k < NR; ++k)
        if ((unsigned)(key[k] >> 32) == m1) x2 = max(x2, (unsigned)key[k]);
#pragma unroll
      for (int t = 0; t < S; ++t) {
        const unsigned v = __reduce_max_sync(FULL, S == 1 || seg == t ? x2 : 0u);
        if (S == 1 || seg == t) m2 = v;
      }
      int lpos = INT_MAX, mpos = 0;
#pragma unroll
      for (int k = 0; k < NR; ++k)
        if (head && pos[k] < n && key[k] == (((unsigned long long)m1 << 32) | m2) && pos[k] < lpos) {
          lpos = pos[k];
          mykp = k;
        }
#pragma unroll
      for (int t = 0; t < S; ++t) {
        const int v = __reduce_min_sync(FULL, S == 1 || seg == t ? lpos : INT_MAX);
        if (S == 1 || seg == t) mpos = v;
      }
      unsigned win = __ballot_sync(FULL, lpos == mpos && lpos != INT_MAX);
      if (S > 1) win &= ((1u << (W & 31)) - 1u) << base;
      zp = (m1 | m2) == 0u;
      wl = __ffs(win) - 1;
      kp = NR > 1 ? __shfl_sync(FULL, mykp, wl) : 0;
      pick();
      u = __shfl_sync(FULL, wsel, wl - jc + c);
      p = __shfl_sync(FULL, psel, wl) - j;
      const double pv = __shfl_sync(FULL, wsel, wl);
      if (!zp) rc = rcp_division(pv);
      if (zp && info == 0) info = j + 1;
    }
    const bool prow = inw && rb + jc == wl;
    const bool act = nz(u) && !zp;
#pragma unroll
    for (int k = 0; k < NR; ++k) {
      const bool piv = prow && (NR == 1 || k == kp);
      const int np = pos[k] == j ? j + p : pos[k];
      // U(j, j+coff) -> AB(kv-coff, j+coff); l_{pos, j} -> AB(kv+pos-j, j)
      const Off at = cb + kv + (piv ? -coff : np - j);
      const bool put = piv ? j + coff < n : (head && np < n);
      const double keep = piv ? qs : (head ? 0.0 : w[k]);  // a slot that changes hands, or no update
      const double l = a[k] * rc;                          // multiplier l_{pos, j}
      const double t = fma(-l, u, w[k]);
      if (put) ab[at] = (piv || zp) ? w[k] : l;
      w[k] = (act && !piv && !head) ? t : keep;
      pos[k] = piv ? j + 1 + kl : np;
    }
    if (sl == 0) ipiv[j] = j + p + 1;
    cb += coff == 0 ? C * ldab : 0;
    coff = coff == 0 ? kv : coff - 1;
    jc = jc + 1 == C ? 0 : jc + 1;
    qs = refill(j + 1 + kl + kWinPrefetch);
  };
  int j0 = 0;
  for (; j0 + kWinPrefetch <= n; j0 += kWinPrefetch) {
#pragma unroll
    for (int s = 0; s < kWinPrefetch; ++s) step(j0 + s, q[s]);
  }
#pragma unroll
  for (int s = 0; s < kWinPrefetch - 1; ++s)
    if (j0 + s < n) step(j0 + s, q[s]);
#pragma unroll
  for (int t = 0; t < S; ++t) infos[t] = __shfl_sync(FULL, info, t * W);
}

}  // namespace regwin
}  // namespace bandlu
