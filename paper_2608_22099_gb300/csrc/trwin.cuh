// trwin.cuh -- one sweep of a banded triangular solve by one warp, with the
// active part of the right-hand side in registers.  Both halves of the band
// solve after gbtrf (xGBTRS) and the banded triangular solves of the dispatch
// (xTBSV, no transpose) are such sweeps.
//
// A sweep visits positions k = 0..n-1 (row k going forward, row n-1-k going
// backward).  Step k, with x the value at position k:
//   sweep_piv: x and the value at position k + p_k are interchanged first;
//   if x != 0 (the reference-BLAS zero test):
//     sweep_div: x = x / c(k, 0)          (IEEE quotient: div_quick)
//     position k + t takes fma(-c(k, t), x, .) for t = 1..min(kw, n-1-k);
//   x is final and is stored.
// c(k, t) is the coefficient at the source functor's address at(k, t) (t = 0:
// the divisor).
//
// What bounds a sweep: the chain of its steps -- a multiply-add (64 clk on GB300),
// the broadcast of x (a 64-bit shuffle), and going backward the quotient -- and, as
// in every one-warp kernel here, the number of instructions beside it.  So a step
// moves no data between lanes but that broadcast: the window of W = 32*RW positions
// ROTATES.  Without interchanges position m lives on lane m % 32, register
// (m / 32) % RW; a finished position's slot takes the position W further on.  The
// owner of position k divides (every lane runs div_quick on what it holds, with the
// divisor of its own position of the block of 32) and the quotient is broadcast.
// With interchanges an element keeps its slot and its position is tracked instead
// (pos): a finished element's slot takes the position W further on.  The tracking
// needs the interchanges only, so it runs kPf steps ahead, with the coefficient
// loads, and the chain has no interchange at all.
// Each lane loads the coefficients of what it holds kPf steps ahead into registers
// (the step loop is unrolled by kPf, one register per slot), as predicated loads
// that nothing consumes before their step.  (Measured on GB300: a per-warp
// shared-memory ring filled by cp.async, waited on one commit group per step,
// made every step slower than these register loads do.)
// Measured (n = 4096, ns a row): triangular solve, k = 16 137 (315 with the quotient from
// a two-term reciprocal on the FP64 pipe and the divisor broadcast); both sweeps after
// gbtrf, kl = ku = 16 271 (602, with the interchanges as moves of data inside each step).
#pragma once

#include "common.cuh"
#include "rcp.cuh"
#include "sync.cuh"

namespace bandlu {
namespace trwin {

// Coefficients of the sweeps.  k is the step; t >= 0 the offset from the
// eliminated position.
// at(k, t): the coefficient's address.  prefetch(k, kw, n, lane): called once
// per step k by every lane, asks L2 for data the sweep reads kPrefetchSteps
// steps later (a no-op for the band storage, which the factorisation has just
// left in L2).
constexpr int kPrefetchSteps = 48;

// prefetch_cta(k, kw, n, lane): the same from one warp of a CTA-wide sweep: the band of a wide
// factorisation does not stay in L2.
__device__ __forceinline__ void prefetch_l2_line(const double *p) {
  asm volatile("prefetch.global.L2 [%0];" ::"l"(p));
}
__device__ __forceinline__ void prefetch_l2_run(const double *p, int len, int lane) {
  for (int i = lane * 16; i < len; i += 32 * 16) prefetch_l2_line(p + i);
}

struct GbLower {  // forward half of xGBTRS: multipliers l_{k+t,k} = AB(kv+t, k)
  const double *AB;
  int ldab, kv;
  __device__ __forceinline__ const double *at(int k, int t) const { return AB + (kv + t) + (long long)k * ldab; }
  __device__ __forceinline__ void prefetch(int, int, int, int) const {}
};
struct GbUpper {  // backward half of xGBTRS: j = n-1-k, U(j-t, j) = AB(kv-t, j)
  const double *AB;
  int ldab, kv, n;
  __device__ __forceinline__ const double *at(int k, int t) const {
    return AB + (kv - t) + (long long)(n - 1 - k) * ldab;
  }
  __device__ __forceinline__ void prefetch(int, int, int, int) const {}
  __device__ __forceinline__ void prefetch_cta(int k, int kw, int, int lane) const {
    const int m = k + kPrefetchSteps, mk = min(kw, n - 1 - m);
    if (m < n) prefetch_l2_run(at(m, mk), mk + 1, lane);
  }
};
// In the dense matrix the coefficients of one step lie in different rows (one
// 32-byte sector each), but row m's band segment -- used over kw consecutive
// steps -- is contiguous: lane L prefetches the L-th 128-byte line of the
// segment of the row whose first use is kPrefetchSteps steps ahead.
struct DenseLower {  // lower triangular, row-major dense: L(k+t, k) = A[(k+t)*lda + k]
  const double *A;
  long long lda;
  __device__ __forceinline__ const double *at(int k, int t) const { return A + (long long)(k + t) * lda + k; }
  // row m = k + kw + kPrefetchSteps is first read at step m - kw; its segment is
  // A[m*lda + m-kw .. m-1]
  __device__ __forceinline__ void prefetch(int k, int kw, int n, int lane) const {
    const int m = k + kw + kPrefetchSteps;
    if (m < n && lane * 16 < kw) prefetch_l2_line(A + (long long)m * lda + (m - kw) + lane * 16);
  }
  __device__ __forceinline__ void prefetch_cta(int k, int kw, int n_, int lane) const {
    const int m = k + kw + kPrefetchSteps;
    if (m < n_) prefetch_l2_run(A + (long long)m * lda + (m - kw), kw, lane);
  }
};
struct DenseUpper {  // upper triangular, row-major dense: j = n-1-k, U(j-t, j) = A[(j-t)*lda + j]
  const double *A;
  long long lda;
  int n;
  __device__ __forceinline__ const double *at(int k, int t) const {
    const int j = n - 1 - k;
    return A + (long long)(j - t) * lda + j;
  }
  // row m = j - kw - kPrefetchSteps is first read at column m + kw; its segment
  // is A[m*lda + m+1 .. m+kw]
  __device__ __forceinline__ void prefetch(int k, int kw, int, int lane) const {
    const int m = n - 1 - k - kw - kPrefetchSteps;
    if (m >= 0 && lane * 16 < kw) prefetch_l2_line(A + (long long)m * lda + (m + 1) + lane * 16);
  }
  __device__ __forceinline__ void prefetch_cta(int k, int kw, int, int lane) const {
    const int m = n - 1 - k - kw - kPrefetchSteps;
    if (m >= 0) prefetch_l2_run(A + (long long)m * lda + (m + 1), kw, lane);
  }
};

// *p where c holds, else 0.0, as one predicated load: a load followed by a
// select would make the select (and so the step that issues the read-ahead)
// wait for the data.  ld_coef reads through the read-only path (coefficients);
// ld_rhs through the ordinary one (the right-hand side, which the sweep writes).
__device__ __forceinline__ double ld_coef(const double *p, bool c) {
  double v;
  asm("{\n\t.reg .pred q;\n\tsetp.ne.u32 q, %2, 0;\n\tmov.b64 %0, 0;\n\t@q ld.global.nc.f64 %0, [%1];\n\t}"
      : "=d"(v)
      : "l"(p), "r"((unsigned)c));
  return v;
}
__device__ __forceinline__ double ld_rhs(const double *p, bool c) {
  double v;
  // (never an entry the sweep has written: positions are read once, before their step)
  asm("{\n\t.reg .pred q;\n\tsetp.ne.u32 q, %2, 0;\n\tmov.b64 %0, 0;\n\t@q ld.global.f64 %0, [%1];\n\t}"
      : "=d"(v)
      : "l"(p), "r"((unsigned)c));
  return v;
}

// *p = v where c holds: predicated, no branch.
__device__ __forceinline__ void st_rhs(double *p, double v, bool c) {
  asm volatile("{\n\t.reg .pred q;\n\tsetp.ne.u32 q, %2, 0;\n\t@q st.global.f64 [%0], %1;\n\t}" ::"l"(p), "d"(v),
               "r"((unsigned)c));
}

// Sweeps with a division and no interchanges.  b: the right-hand side (n doubles,
// overwritten with the result); kw: the band width of the update, W >= kw + 1.
template <int RW, int kPf, bool kFwd, class Src>
__device__ __forceinline__ void sweep_div(double *b, int n, int kw, const Src &src) {
  constexpr int W = 32 * RW;
  static_assert(32 % kPf == 0, "blocks of 32 steps");
  const int lane = threadIdx.x & 31;
  auto row = [&](int m) { return kFwd ? m : n - 1 - m; };
  double w[RW];
#pragma unroll
  for (int r = 0; r < RW; ++r) {
    const int m = lane + 32 * r;
    w[r] = ld_rhs(b + row(m), m < n);
  }
  // coefficients of step k0+s for the positions this lane holds
  double cf[kPf][RW];
  auto fill = [&](int s, int k) {
    const unsigned mk = (unsigned)max(min(kw, n - 1 - k), 0);
#pragma unroll
    for (int r = 0; r < RW; ++r) {
      const int t = (lane + 32 * r - k) & (W - 1);
      cf[s][r] = ld_coef(src.at(k, t), (unsigned)(t - 1) < mk);
    }
    src.prefetch(k, kw, n, lane);
  };
#pragma unroll
  for (int s = 0; s < kPf; ++s) fill(s, s);
  // Per block of 32 steps, lane L: the divisor of position 32*B + L (the next block's is read a
  // block ahead), the position W further on, which takes its slot, and the block's results.
  double nd = __ldg(src.at(min(lane, n - 1), 0));
  double nx = ld_rhs(b + row(W + lane), W + lane < n);
  int rr = 0;  // register of the block's positions
  for (int kb = 0; kb < n; kb += 32) {
    const double bd = nd, in = nx;
    const Divisor dv = div_known_prep(bd);
    nd = __ldg(src.at(min(kb + 32 + lane, n - 1), 0));
    nx = ld_rhs(b + row(kb + 32 + W + lane), kb + 32 + W + lane < n);
    double out = 0.0;
    for (int k0 = kb; k0 < kb + 32; k0 += kPf) {
      if (k0 >= n) break;  // uniform
#pragma unroll
      for (int s = 0; s < kPf; ++s) {
        const int k = k0 + s;  // past the end (k >= n): no coefficient, and nothing is stored
        const unsigned mk = (unsigned)max(min(kw, n - 1 - k), 0);
        const int o = k & 31;
        double mine = w[0];
#pragma unroll
        for (int r = 1; r < RW; ++r) mine = rr == r ? w[r] : mine;
        bool unsure;
        const double q = div_quick(mine, dv, &unsure);
        double x = __shfl_sync(FULL, q, o);
        bool go = true;
        if ((__ballot_sync(FULL, unsure) >> o) & 1u) {  // uniform, rare
          const double xo = __shfl_sync(FULL, mine, o), d = __shfl_sync(FULL, bd, o);
          x = div_unsure(xo, d, k < n, &go);
        }
#pragma unroll
        for (int r = 0; r < RW; ++r) {
          const int t = (lane + 32 * r - k) & (W - 1);
          if (go && (unsigned)(t - 1) < mk) w[r] = fma(-cf[s][r], x, w[r]);
        }
        // position k leaves, position k+W enters
        out = lane == o ? x : out;
#pragma unroll
        for (int r = 0; r < RW; ++r) w[r] = (lane == o && rr == r) ? in : w[r];
        fill(s, k + kPf);
      }
    }
    if (kb + lane < n) b[row(kb + lane)] = out;
    rr = rr + 1 == RW ? 0 : rr + 1;
  }
}

// The forward half of xGBTRS: interchanges (ipiv, 1-based; entries outside the
// window's reach k..k+min(kw, n-1-k) are ignored) and no division; W >= kw + 1.
template <int RW, int kPf, class Src>
__device__ __forceinline__ void sweep_piv(double *b, int n, int kw, const Src &src, const int *ipiv) {
  constexpr int W = 32 * RW;
  const int lane = threadIdx.x & 31;
  double w[RW];
  int pos[RW];  // position of the element in this slot, after the interchanges of the steps asked for
#pragma unroll
  for (int r = 0; r < RW; ++r) {
    pos[r] = lane + 32 * r;
    w[r] = ld_rhs(b + pos[r], pos[r] < n);
  }
  // step k0+s: the coefficients, which registers take the update (bit r of up), the slot of the
  // element at position k (lane, register) and the value that takes it over (its owner only)
  double cf[kPf][RW], en[kPf];
  unsigned up[kPf];
  int sl[kPf], sr[kPf], pv[kPf];
  auto ask = [&](int k) { return __ldg(ipiv + min(k, n - 1)); };
  auto fill = [&](int s, int k, int piv) {  // piv: ipiv of step k
    const int mk = max(min(kw, n - 1 - k), 0);
    int to = piv - 1;
    if ((unsigned)(to - k) > (unsigned)mk) to = k;  // past the end, or outside the reach: ignored
    unsigned who = 0;
    int reg = 0;
#pragma unroll
    for (int r = 0; r < RW; ++r) {
      const unsigned v = __ballot_sync(FULL, pos[r] == to);
      reg = v != 0u ? r : reg;
      who |= v;
    }
    sl[s] = __ffs(who) - 1;  // every position k..k+W-1 is held by one slot
    sr[s] = reg;
    up[s] = 0u;
    en[s] = ld_rhs(b + k + W, lane == sl[s] && k + W < n);
#pragma unroll
    for (int r = 0; r < RW; ++r) {
      const bool leaves = lane == sl[s] && reg == r;
      pos[r] = pos[r] == k ? to : pos[r];
      const int t = pos[r] - k;
      const bool in = !leaves && (unsigned)(t - 1) < (unsigned)mk;
      cf[s][r] = ld_coef(src.at(k, t), in);
      up[s] |= in ? 1u << r : 0u;
      pos[r] = leaves ? k + W : pos[r];
    }
  };
#pragma unroll
  for (int s = 0; s < kPf; ++s) pv[s] = ask(s);
#pragma unroll
  for (int s = 0; s < kPf; ++s) {
    fill(s, s, pv[s]);
    pv[s] = ask(s + kPf);
  }
  for (int k0 = 0; k0 < n; k0 += kPf) {
#pragma unroll
    for (int s = 0; s < kPf; ++s) {
      const int k = k0 + s;
      if (k >= n) break;
      double mine = w[0];
#pragma unroll
      for (int r = 1; r < RW; ++r) mine = sr[s] == r ? w[r] : mine;
      const double x = __shfl_sync(FULL, mine, sl[s]);
      const bool go = nz(x);
#pragma unroll
      for (int r = 0; r < RW; ++r)
      {  // (the test is a select after the multiply-add, off the chain)
        const double u = fma(-cf[s][r], x, w[r]);
        w[r] = (go && ((up[s] >> r) & 1u)) ? u : w[r];
      }
      // x is final; position k+W takes its slot
      st_rhs(b + k, x, lane == sl[s]);
#pragma unroll
      for (int r = 0; r < RW; ++r) w[r] = (lane == sl[s] && sr[s] == r) ? en[s] : w[r];
      const int piv = pv[s];
      pv[s] = ask(k + 2 * kPf);
      fill(s, k + kPf, piv);
    }
  }
}

// ---------------------------------------------------------------------------
// The same sweeps by a CTA of NW = blockDim.x / 32 warps, for windows where one
// warp's multiply-adds (64 clk each, one at a time) would outlast the chain: every
// thread holds one position, W = 32*NW.
// The values x are handed on through a ring in shared memory, two blocks of 32 steps
// deep, without a barrier per step: a slot holds kEmpty until its x is written, and a
// reader polls it (one 8-byte word is value and flag at once, so no fence is needed).
// A value that happens to have kEmpty's high word, a NaN no operation here produces, is
// handed on as the canonical NaN.  A barrier every 32 steps lets the slots of the block
// before be emptied again: step k of block B reads slot k % 64, which is emptied during
// block B+1 (every reader has passed the barrier after block B) and written again in
// block B+2 (after the barrier that follows the emptying).
// Measured (n = 4096, ns a row): triangular solve, k = 300 210 (1061 with one warp and 16
// registers a lane), k = 100 178 (542; 218 when a follower polled every step by itself);
// both sweeps after gbtrf, kl = ku = 100 338 (645 with a CTA-wide window and a barrier per
// step), 256 433 (1035), 400 521 (1080).
// A poll gives up after kWaitLimitCycles, says so in *d_info and raises giveup, on which
// every wait of the CTA returns at once; what it waited for is then NaN, and so is all that
// the sweep forms from it.  In a correct run none does.
constexpr unsigned long long kEmpty = 0xfff8badc0ffee123ull;
constexpr int kRing = 64;
// An empty slot, told by its high word alone.
__device__ __forceinline__ bool slot_empty(unsigned long long v) {
  return (unsigned)(v >> 32) == (unsigned)(kEmpty >> 32);
}

struct Ring {
  alignas(16) unsigned long long x[kRing];
  int *status;  // *d_info, or null
  int giveup;

  __device__ __forceinline__ void init(int *d_info) {  // by the whole CTA, a barrier after it
    for (int i = threadIdx.x; i < kRing; i += blockDim.x) x[i] = kEmpty;
    if (threadIdx.x == 0) {
      status = d_info;
      giveup = 0;
    }
  }
  __device__ __forceinline__ bool gave_up() const { return *reinterpret_cast<const volatile int *>(&giveup) != 0; }
  // The lane where c holds writes v (predicated: a divergent branch would cost each step more than
  // the store).
  __device__ __forceinline__ void put(int k, double v, bool c) {
    unsigned long long u = (unsigned long long)__double_as_longlong(v);
    u = slot_empty(u) ? 0x7fffffffffffffffull : u;
    asm volatile("{\n\t.reg .pred q;\n\tsetp.ne.u32 q, %2, 0;\n\t@q st.volatile.shared.u64 [%0], %1;\n\t}" ::"r"(
                     smem_addr(&x[k & (kRing - 1)])),
                 "l"(u), "r"((unsigned)c)
                 : "memory");
  }
  __device__ __forceinline__ double peek(int k) {
    unsigned long long v;
    asm volatile("ld.volatile.shared.u64 %0, [%1];" : "=l"(v) : "r"(smem_addr(&x[k & (kRing - 1)])) : "memory");
    return __longlong_as_double((long long)v);
  }
  // Polls until get() returns true; false when that does not come about.
  template <class Get>
  __device__ __forceinline__ bool poll(Get get) {
    bool ok = get();
    if (!ok) {
      const long long t0 = clock64();
      for (unsigned it = 0; !(ok = get()); ++it) {
        if ((it & 1023u) == 0 && (gave_up() || clock64() - t0 > kWaitLimitCycles)) {
          *reinterpret_cast<volatile int *>(&giveup) = 1;
          if (status != nullptr) *status = -BANDLU_ERR_TIMEOUT;
          break;
        }
      }
    }
    __syncwarp();
    return ok;
  }
  // x of steps k..k+3, k a multiple of 4, polled by a whole warp (an empty slot's NaN when the
  // poll gave up).
  __device__ __forceinline__ void get4(int k, double (&out)[4]) {
    unsigned long long v[4];
    const unsigned a = smem_addr(&x[k & (kRing - 1)]);
    auto get = [&] {
      asm volatile("ld.volatile.shared.v2.u64 {%0, %1}, [%2];" : "=l"(v[0]), "=l"(v[1]) : "r"(a) : "memory");
      asm volatile("ld.volatile.shared.v2.u64 {%0, %1}, [%2];" : "=l"(v[2]), "=l"(v[3]) : "r"(a + 16u) : "memory");
      return !(slot_empty(v[0]) || slot_empty(v[1]) || slot_empty(v[2]) || slot_empty(v[3]));
    };
    poll(get);
#pragma unroll
    for (int s = 0; s < 4; ++s) out[s] = __longlong_as_double((long long)v[s]);
  }
  __device__ __forceinline__ void empty(int B) {  // by one warp: the slots of block B
    asm volatile("st.volatile.shared.u64 [%0], %1;" ::"r"(
                     smem_addr(&x[(32 * B + (threadIdx.x & 31)) & (kRing - 1)])),
                 "l"(kEmpty)
                 : "memory");
  }
};

// Threads of a CTA-wide sweep with update width kw <= kRingMax.
constexpr int kRingMax = 992;  // 1024 threads hold kw + 32 positions
constexpr int ring_threads_div(int kw) { return kw < 1 ? 64 : (kw + 63) / 32 * 32; }

// sweep_div by a CTA, W >= kw + 32.  Warp w holds chunk c = w (positions 32c..32c+31),
// then c + NW, ...: the chunk of block B is led by its warp, in which the chain of the
// block stays (quotient, shuffle, multiply-add, as in sweep_div); the other warps follow
// from the ring, as far behind as they like within the block.
template <int kPf, bool kFwd, class Src, class Ring>
__device__ __forceinline__ void ring_sweep_div(double *b, int n, int kw, const Src &src, Ring &ring, int *d_info) {
  static_assert(32 % kPf == 0 && kPf % 4 == 0, "blocks of 32 steps, polled by fours");
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
  auto row = [&](int m) { return kFwd ? m : n - 1 - m; };
  ring.init(d_info);
  int c = warp;   // this warp's chunk
  int cf_c = c;   // the chunk of the next coefficients asked for
  auto pos = [&](int chunk) { return 32 * chunk + lane; };
  double w = ld_rhs(b + row(pos(c)), pos(c) < n);
  double nx = ld_rhs(b + row(pos(c + nw)), pos(c + nw) < n);  // the chunk it takes next
  double bd = __ldg(src.at(min(pos(c), n - 1), 0));           // the divisors of its chunk
  Divisor dv = div_known_prep(bd);
  double cf[kPf];
  auto fill = [&](int s, int k) {
    if ((k & 31) == 0 && cf_c < (k >> 5)) cf_c += nw;  // uniform: block k / 32 begins, this warp led the one before
    const unsigned mk = (unsigned)max(min(kw, n - 1 - k), 0);
    const int t = pos(cf_c) - k;
    cf[s] = ld_coef(src.at(k, t), (unsigned)(t - 1) < mk);
  };
#pragma unroll
  for (int s = 0; s < kPf; ++s) fill(s, s);
  __syncthreads();
  for (int kb = 0, B = 0; kb < n; kb += 32, ++B) {
    if (warp == nw - 1 && B >= 1) ring.empty(B - 1);
    if (c == B) {
      double out = 0.0;
      for (int k0 = kb; k0 < kb + 32; k0 += kPf) {
        if (k0 >= n) break;  // uniform
#pragma unroll
        for (int s = 0; s < kPf; ++s) {
          const int k = k0 + s, o = k & 31;  // past the end (k >= n): no coefficient, and nothing is stored
          bool unsure;
          const double q = div_quick(w, dv, &unsure);
          double x = __shfl_sync(FULL, q, o);
          bool go = true;
          if ((__ballot_sync(FULL, unsure) >> o) & 1u) {  // uniform, rare
            const double xo = __shfl_sync(FULL, w, o), d = __shfl_sync(FULL, bd, o);
            x = div_unsure(xo, d, k < n, &go);
          }
          const int t = lane - o;
          const double u = fma(-cf[s], x, w);
          ring.put(k, x, lane == o);
          out = lane == o ? x : out;
          w = (go && t >= 1 && t <= min(kw, n - 1 - k)) ? u : w;
          fill(s, k + kPf);
        }
      }
      if (pos(c) < n) b[row(pos(c))] = out;
      c += nw;
      w = nx;
      bd = __ldg(src.at(min(pos(c), n - 1), 0));
      nx = ld_rhs(b + row(pos(c + nw)), pos(c + nw) < n);
    } else {
      if (c == B + 1) dv = div_known_prep(bd);
      for (int k0 = kb; k0 < kb + 32; k0 += kPf) {
        if (k0 >= n) break;
#pragma unroll
        for (int s4 = 0; s4 < kPf; s4 += 4) {
          const int k4 = k0 + s4;
          // some position within reach of one of the four steps (none is past the end)
          if (32 * c - k4 - 3 <= kw && 32 * c < n) {  // uniform
            double x[4];
            ring.get4(k4, x);
#pragma unroll
            for (int s = 0; s < 4; ++s) {
              const int k = k4 + s, t = pos(c) - k;
              const double u = fma(-cf[s4 + s], x[s], w);
              w = (nz(x[s]) && t <= min(kw, n - 1 - k)) ? u : w;
            }
          }
#pragma unroll
          for (int s = 0; s < 4; ++s) {
            fill(s4 + s, k4 + s + kPf);
            if (c == B + nw - 1) src.prefetch_cta(k4 + s, kw, n, lane);  // the warp with the least in reach
          }
        }
      }
    }
    __syncthreads();
  }
}

// ---------------------------------------------------------------------------
// Multipliers of the band storage staged in shared memory, a block of 32 columns at a time in
// two buffers: one bulk copy a column, issued by one warp a block ahead.  A copy starts at a
// 16-byte boundary, so a column whose first multiplier is not on one carries the entry before
// it, the diagonal, and one more at the end if need be (inside AB: a column with multipliers
// is not the last one).
struct Stage {
  double *buf;               // 64 columns of `pitch` doubles
  int pitch;                 // even
  unsigned long long *full;  // [2]: block B's columns have landed, phase B / 2
  __device__ __forceinline__ double *col(int k) const { return buf + (k & 63) * pitch; }
  // column k's copy, on the barrier of its block
  __device__ __forceinline__ void copy(int k, const double *from, unsigned bytes, unsigned bar) const {
    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
                     smem_addr(col(k))),
                 "l"(from), "r"(bytes), "r"(bar)
                 : "memory");
  }
};
constexpr int stage_pitch(int entries) { return (entries + 3) & ~1; }

// The first entry of a copied column sits at col(k)[stage_off(first)], first its global address.
__device__ __forceinline__ int stage_off(const double *first) {
  return (int)((reinterpret_cast<unsigned long long>(first) >> 3) & 1ull);
}
// By one warp: `len` entries from `first` (this lane's column; len 0 or less: none) for block B.
template <class Stage>
__device__ __forceinline__ void stage_block(const Stage &st, int B, int k, const double *first, int len) {
  const int lane = threadIdx.x & 31;
  const int off = stage_off(first);
  const unsigned bytes = len > 0 ? (unsigned)((off + len + 1) & ~1) * 8u : 0u;
  const unsigned total = __reduce_add_sync(FULL, bytes);
  const unsigned bar = smem_addr(st.full + (B & 1));
  asm volatile("fence.proxy.async.shared::cta;" ::: "memory");  // (its buffer has been read through ordinary loads)
  if (lane == 0)
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(total) : "memory");
  __syncwarp();
  if (bytes != 0u) st.copy(k, first - off, bytes, bar);
}
// Block B's columns have landed; false: they never did.
__device__ __forceinline__ bool stage_wait(const Stage &st, int B, Ring &ring) {
  return ring.poll([&] { return mbar_try_wait(st.full + (B & 1), (unsigned)(B >> 1) & 1u); });
}

// sweep_piv by a CTA, the chain of a block of 32 steps in one warp: the interchanges of a block
// are known before it starts, so which elements it eliminates is too.  (With the elements in
// fixed threads, whichever held the next one publishing it, every warp was on the chain:
// kl = 100 260 ns a row, now 140.)  Warp 0 (the leader) gathers those 32, lane s the one eliminated in the block's step s,
// and runs the block's triangle with a shuffle and a multiply-add a step; the follower warps
// hold the elements that survive the block, thread t the one that ends it at position
// kb + 32 + t, and take the block's values from the ring four steps at a time, as far behind as
// they like; the last warp (the keeper) prepares the next block.  Elements pass from block to
// block through shared memory by their positions (val, two copies: a block reads one and
// writes the other); within a block everyone tracks its element's position.
// (Where kw > 960 the keeper follows too, after its preparations.)
constexpr int kStageWidth = 397;     // 2 * 32 columns of kStageWidth + 2 entries: 199 KB
constexpr int kValRing = 1024 + 64;  // >= kRingMax + 64 positions
constexpr int block_threads(int kw) { return kw > 960 ? 1024 : 32 * ((kw + 31) / 32 + 2); }

struct BlockShared {
  double val[2][kValRing];        // position p's element at the start of block B: val[B & 1][p % kValRing]
  int from[2][kRingMax + 32];     // element that block B leaves at offset o (o < 32: eliminates in step o): its offset at the start
  alignas(16) int swap_to[128];   // slot k % 128: the position that k is interchanged with in step k
};

// kStaged: the multipliers through shared memory (kw <= kStageWidth, where the buffers fit), else
// from memory a group of four steps ahead.
template <bool kStaged, class Ring, class Stage>
__device__ __forceinline__ void block_sweep_piv(double *b, int n, int kw, const GbLower &src, const int *ipiv,
                                                Ring &ring, const Stage &st, BlockShared &bs, int *d_info) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
  const bool keeper = warp == nw - 1;
  auto ask_swap = [&](int B) { return __ldg(ipiv + min(32 * B + lane, n - 1)); };
  auto put_swaps = [&](int B, int piv) {
    const int k = 32 * B + lane, mk = max(min(kw, n - 1 - k), 0);
    bs.swap_to[k & 127] = (unsigned)(piv - 1 - k) > (unsigned)mk ? k : piv - 1;  // outside the reach: ignored
  };
  auto stage = [&](int B) {
    const int k = 32 * B + lane;
    stage_block(st, B, k, src.at(k, 1), min(kw, n - 1 - k));
  };
  // positions 32B+kw .. 32B+kw+31 are new in block B
  auto ask_new = [&](int B) { return ld_rhs(b + 32 * B + kw + lane, 32 * B + kw + lane < n); };
  auto put_new = [&](int B, double v) { bs.val[B & 1][(32 * B + kw + lane) % kValRing] = v; };
  auto put_from = [&](int B) {  // by the keeper, block B's interchanges in shared memory
    volatile int *f = bs.from[B & 1];
    for (int o = lane; o < kw + 32; o += 32) f[o] = o;
    __syncwarp();
    if (lane == 0) {
      for (int s = 0; s < 32; ++s) {
        const int o = bs.swap_to[(32 * B + s) & 127] - 32 * B, x = f[s], y = f[o];
        f[s] = y;
        f[o] = x;
      }
    }
    __syncwarp();
  };
  ring.init(d_info);
  if (kStaged && threadIdx.x == 0) {
    mbar_init(st.full, 1);
    mbar_init(st.full + 1, 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  for (int p = threadIdx.x; p < kw + 32; p += blockDim.x) bs.val[0][p] = ld_rhs(b + p, p < n);
  __syncthreads();
  int piv = 0;
  double in = 0.0;
  if (keeper) {
    if (kStaged) {
      stage(0);
      if (32 < n) stage(1);
    }
    put_swaps(0, ask_swap(0));
    put_swaps(1, ask_swap(1));
    __syncwarp();
    put_from(0);
    piv = ask_swap(2);
    in = ask_new(1);
  }
  __syncthreads();
  for (int kb = 0, B = 0; kb < n; kb += 32, ++B) {
    if (keeper) {
      if (B >= 1) {
        b[kb - 32 + lane] = ring.peek(kb - 32 + lane);
        ring.empty(B - 1);
        // (no arrival on a barrier whose phase has never completed: that is a fault)
        if (kStaged && kb + 32 < n && !__any_sync(FULL, ring.gave_up())) stage(B + 1);
      }
      put_new(B + 1, in);
      in = ask_new(B + 2);
      put_swaps(B + 2, piv);
      piv = ask_swap(B + 3);
      put_from(B + 1);
      for (int s = 0; s < 32 && !kStaged; ++s)  // the block after next from HBM to L2: a wide band does not stay there
        if (kb + 64 + s < n) prefetch_l2_run(src.at(kb + 64 + s, 1), min(kw, n - 1 - (kb + 64 + s)), lane);
    }
    if (!keeper || 32 * (warp - 1) < kw) {  // uniform in a warp
      const int at = warp == 0 ? lane : threadIdx.x;  // offset that this thread's element has at the block's end (or lane)
      const bool has = warp == 0 || at - 32 < kw;
      const int o0 = has ? bs.from[B & 1][at] : 0;
      int pos = kb + o0;
      double w = has ? bs.val[B & 1][pos % kValRing] : 0.0;
      if (kStaged && !stage_wait(st, B, ring)) w = __longlong_as_double(0x7fffffffffffffffll);  // all of the block
      double cf[4];
      unsigned in4 = 0;
      const int a0 = stage_off(src.at(0, 1));
      auto fill = [&](int k0) {  // four steps' coefficients
        const int4 t4 = *reinterpret_cast<const int4 *>(&bs.swap_to[k0 & 127]);
        const int tos[4] = {t4.x, t4.y, t4.z, t4.w};
        in4 = 0;
#pragma unroll
        for (int s = 0; s < 4; ++s) {
          const int k = k0 + s, to = tos[s];
          const bool out = pos == to;  // eliminated (the leader's): never in reach again
          pos = pos == k ? to : pos;
          pos = out ? -1 : pos;
          const bool use = pos > k && pos <= min(k + kw, n - 1);
          if (kStaged) {
            // l_{pos, k} sits at col(k)[off + pos - k - 1], off = stage_off(src.at(k, 1))
            const int at0 = (k & 63) * st.pitch + ((a0 + (k & src.ldab)) & 1) - k - 1;
            cf[s] = use ? st.buf[at0 + pos] : 0.0;
          } else {
            cf[s] = ld_coef(src.at(k, pos - k), use);
          }
          in4 |= use ? 1u << s : 0u;
        }
      };
      if (!has) pos = -1;
      fill(kb);
      for (int k0 = kb; k0 < kb + 32 && k0 < n; k0 += 4) {
        double c4[4];
        const unsigned m4 = in4;
#pragma unroll
        for (int s = 0; s < 4; ++s) c4[s] = cf[s];
        if (k0 + 4 < kb + 32) fill(k0 + 4);
        if (warp == 0) {
#pragma unroll
          for (int s = 0; s < 4; ++s) {
            const int o = (k0 + s) & 31;
            const double x = __shfl_sync(FULL, w, o);
            const double u = fma(-c4[s], x, w);
            ring.put(k0 + s, w, lane == o);
            w = (((m4 >> s) & 1u) && nz(x)) ? u : w;
          }
        } else if (__any_sync(FULL, m4 != 0u)) {
          double x[4];
          ring.get4(k0, x);  // (the leader writes all four, past the last position too)
#pragma unroll
          for (int s = 0; s < 4; ++s) {
            const double u = fma(-c4[s], x[s], w);
            w = (((m4 >> s) & 1u) && nz(x[s])) ? u : w;
          }
        }
      }
      if (warp != 0 && has) bs.val[(B + 1) & 1][(kb + at) % kValRing] = w;
    }
    __syncthreads();
  }
  const int last = (n - 1) / 32 * 32 + threadIdx.x;
  if (threadIdx.x < 32 && last < n) b[last] = ring.peek(last);
}

}  // namespace trwin
}  // namespace bandlu
