// The resident kernel: one cooperative launch refactors and solves one
// system; its CTAs stay on the SMs from the value permutation to the true
// residual.  The phases of the factorisation and of the sweeps, the products
// and the updates are stages separated by grid barriers with bounded waits.
//
// Why: a launch per stage pays a launch boundary, the chain of dependent loads
// that finds a warp's work (entry, descriptor, row pointers, columns) and, at
// a dot product, the chain of fences and atomics that finds the last CTA.
// Here a warp's first unit of the next stage is found, and its constant data
// loaded, before the barrier's wait.
//
// What bounds it for small systems is latency: a grid barrier takes 2,500
// cycles on 152 SMs (1,500 up to 8 CTAs), a dependent FP64 FMA 65, a quotient
// or a square root 650, a load from L2 300 and more, and code that is not in
// the instruction caches is fetched from L2 too.  The last is why every stage
// exists once, with run-time flags for the two halves of an iteration and for
// the two sweeps, and why loops over blocks are not unrolled: with an
// instance per flag the kernel's text was 415 KB and a 500-row iteration took
// 50 us, most of it instruction fetches.
//
// The arithmetic is that of the launch-per-phase kernels, expression by
// expression, and every sum has their order (unit sums of a warp, tiles of
// eight units, groups of 32 tiles, see red_end), so the results are bitwise
// those of the other launch forms, alone and in a batch.
#pragma once

#include <type_traits>

#include "factor.cuh"
#include "kernels.cuh"
#include "sweeps.cuh"

namespace opm {

enum ResidentWork { kResFactor = 1, kResSolve = 2, kResApply = 4 };

// Device words of one runner, zero between launches: the CTA that leaves
// last clears them.
struct ResidentCtl {
  uint32_t arrive, pad0[31];  // barrier arrivals, counted up over the launch
  uint32_t exits, pad1[31];   // CTAs that have left
  uint32_t abort, pad2[31];   // a bounded wait expired
};

// The warps' unit sums of one kind of dot product: up to three planes of
// units, grouped by 256.
struct DotUnits {
  double *sums;
  int32_t ngrp, nunits;
};

struct Resident {
  Batch B;
  Sys sys;                // the system's descriptor (B.sys is not read)
  ResidentCtl *ctl;
  int32_t *err;           // factorisation error: status, 0x7fffffff - smallest row (both 0: none)
  const int32_t *prod;    // every slice for the products, the heaviest first
  DotUnits ds, du;        // slice units (whole 256-row tiles), update units (whole 1024-row tiles)
  double *gpart;          // group sums, three values per group
  Result *res;            // the outcome, in page-locked host memory
  int32_t nupd, work;
};

// The Krylov scalars, kept by every CTA in shared memory.
struct Scal {
  double n0, tol, rho, alpha, omega, beta, relres;
  double tot[3], part[3];  // a complete sum and the slow parts of its decision
  int32_t status, k, iters, maxit, half, pad;
};

// Between two looks at the clock a wait counts at most this long: a context
// that was switched out (a time slice, a debugger) has not waited.
constexpr uint64_t kPollGapNs = 1000000;

constexpr int kTrios = 5;       // trios of a CTA of the trio form
constexpr int kTrioThreads = 32 * (3 * kTrios + 1);  // and one warp more: the boss's
constexpr int kResidentThreads = 1024;               // the wide form

struct ResShared {
  Sys sys;  // k_resident_apply's
  Scal sc;
  int dead, last;
  int32_t phase0;                           // entries of the first forward phase
  int4 first[kResidentThreads / 32];        // the warps' first entry of it
  double ex[kTrios][2][4][3][32];  // a trio's exchange: two units in turn, up to four rows per lane
};

// The steps of a solve: each ends with a dot product and what it decides.
enum ResStep { kStepSetup, kStepP, kStepS, kStepUpdate, kStepFinish };

// The slow operations of a decision, one per warp.
__device__ __forceinline__ int dot_parts(int step) { return step == kStepS ? 2 : step == kStepUpdate ? 3 : 1; }

__device__ __forceinline__ double dot_part(int step, const Scal &c, int part) {
  const bool root = (step == kStepS || step == kStepUpdate) ? part == 1 : step != kStepP;
  if (root) {
    const double r = sqrt(c.tot[step == kStepS ? 2 : 0]);
    return step == kStepFinish ? r / c.n0 : r;
  }
  const double num = step == kStepP ? c.rho : step == kStepS ? c.tot[0] : part == 0 ? c.tot[1] : c.alpha;
  const double den = step == kStepP ? c.tot[0] : step == kStepS ? c.tot[1] : part == 0 ? c.rho : c.omega;
  return num / den;
}

// The decision (setup_scalars, and the ends of k_spmv_v, k_spmv_t, k_update,
// k_finish) from the sums in c.tot and the parts in c.part.
__device__ __forceinline__ void dot_decide(int step, Scal &c) {
  const double *tot = c.tot, *part = c.part;
  if (step == kStepSetup) {
    c.n0 = part[0];
    c.tol *= part[0];  // holds rtol until here
    c.k = 1;
    c.rho = tot[0];
    c.alpha = 1.0;
    c.omega = 1.0;
    c.beta = tot[0];
    if (c.status != kRunning) return;  // the factorisation failed
    if (!isfinite(c.n0)) c.status = OPM_ERR_NONFINITE;
    else if (c.n0 == 0.0) c.status = OPM_OK;
    else if (c.maxit < 1) c.status = OPM_NOT_CONVERGED;
  } else if (step == kStepP) {
    if (tot[0] == 0.0) {
      c.status = OPM_ERR_BREAKDOWN;
      c.iters = c.k;
    } else {
      c.alpha = part[0];
    }
  } else if (step == kStepS) {
    if (part[1] <= c.tol) {
      c.half = 1;
    } else if (tot[1] == 0.0) {
      c.status = OPM_ERR_BREAKDOWN;
      c.iters = c.k;
    } else {
      c.omega = part[0];
      if (c.omega == 0.0) {
        c.status = OPM_ERR_BREAKDOWN;
        c.iters = c.k;
      }
    }
  } else if (step == kStepUpdate) {
    c.iters = c.k;
    if (c.half || part[1] <= c.tol) {
      c.status = OPM_OK;
    } else if (c.k >= c.maxit) {
      c.status = OPM_NOT_CONVERGED;
    } else if (tot[1] == 0.0) {
      c.status = OPM_ERR_BREAKDOWN;
      c.iters = c.k + 1;
    } else {
      c.rho = tot[1];
      c.beta = part[0] * part[2];
      c.k += 1;
    }
  } else {
    const bool ok = c.status == OPM_OK || c.status == OPM_NOT_CONVERGED;
    c.relres = !ok ? nan("") : (c.n0 > 0.0 ? part[0] : 0.0);
  }
}

__device__ __forceinline__ void red_release(uint32_t *p) {
  asm volatile("red.release.gpu.global.add.u32 [%0], 1;" ::"l"(p) : "memory");
}

// One thread's view of the launch.
struct ResCtx {
  const Resident &R;
  ResShared &sm;
  const Sys &S;      // the system's descriptor
  int lane, wp, nw;  // lane, warp of the CTA, warps per CTA
  int g, W;          // first unit of a stage of this warp (trio), the units' stride
  int r, trio;       // component and trio of the warp (trios only)
  int flip;          // exchange buffer of the trio's next unit
  uint32_t target;   // arrivals that complete the current barrier
  bool dead;         // a bounded wait expired: every CTA leaves
  bool boss;         // the thread that arrives and polls: one of the last warp

  // The trio's three warps meet.
  __device__ __forceinline__ void trio_sync() const {
    asm volatile("bar.sync %0, 96;" ::"r"(trio + 1) : "memory");
  }
  // All warps of the grid, consecutive ones on different SMs.
  __device__ __forceinline__ int warp_id() const { return wp * gridDim.x + blockIdx.x; }
  __device__ __forceinline__ int warps() const { return nw * gridDim.x; }

  // Ends a stage: this CTA's writes are released to the grid.
  __device__ __forceinline__ void arrive() {
    __syncthreads();
    target += gridDim.x;
    if (boss && gridDim.x > 1 && (int)blockIdx.x != R.B.skip_cta) red_release(&R.ctl->arrive);
  }
  // Waits until every CTA has ended the last stage.  Every warp calls it
  // once per stage.  The CTA numbered skip_cta (a test hook) has not arrived
  // and leaves at once, so the others' waits run out.
  __device__ __forceinline__ void wait() {
    if (gridDim.x == 1) return;  // arrive()'s CTA barrier was enough
    if (boss) {
      bool d = dead || (int)blockIdx.x == R.B.skip_cta;
      if (!d) {
        uint64_t last = gtimer(), waited = 0;
        for (uint32_t it = 1; (int32_t)(ld_acquire(&R.ctl->arrive) - target) < 0; ++it) {
          if ((it & 63u) == 0u) {
            const uint64_t now = gtimer(), gap = now - last;
            last = now;
            waited += gap < kPollGapNs ? gap : kPollGapNs;
            if (ld_acquire(&R.ctl->abort) != 0u) d = true;
            else if (waited > R.B.spin_limit_ns) {
              atomicExch(&R.ctl->abort, 1u);
              d = true;
            }
            if (d) break;
          }
        }
      }
      sm.dead = d;
    }
    __syncthreads();
    dead = sm.dead != 0;
  }
  // Whether the iteration goes on.
  __device__ __forceinline__ bool runs() const { return sm.sc.status == kRunning; }
};

using First = std::true_type;
using Rest = std::false_type;

// A stage: units e0 + g, e0 + g + W, ... below e1.  The first goes to
// body(e, First{}), which calls wait() once, at the place that suits it; the
// others to body(e, Rest{}).
template <typename Body>
__device__ __forceinline__ void stage(ResCtx &c, int e0, int e1, Body body) {
  int e = e0 + c.g;
  if (e < e1) body(e, First{});
  else c.wait();
#pragma unroll 1
  for (e += c.W; e < e1 && !c.dead; e += c.W) body(e, Rest{});
  c.arrive();
}

// Writes a warp's sums of unit u.
__device__ __forceinline__ void store_unit(const DotUnits &D, int u, const double (&v)[3]) {
  const double s = warp_sum_split<3>(v);
  const int q = warp_sum_of<3>(threadIdx.x & 31);
  if (q >= 0) D.sums[(size_t)q * D.nunits + u] = s;
}

// Completes a step's dot product after the wait: group sums (red_end's order:
// the butterflies over a tile's eight units and over 32 tiles), then the sum
// and what it decides, by every CTA for itself, a value and a slow operation
// per warp.  A single group (a system of up to 8,192 rows) is summed by every
// CTA; more are spread over the grid, with one more barrier: read by every
// CTA, the unit sums of a 249,053-row system took 35 us per three-value dot,
// the barrier 1.3.
__device__ __forceinline__ void finish_dot(ResCtx &c, int step) {
  const DotUnits &D = (step == kStepSetup || step == kStepUpdate) ? c.R.du : c.R.ds;
  const bool local = D.ngrp == 1, every = step == kStepSetup || step == kStepFinish;
  const int nv = step == kStepS ? 3 : step == kStepUpdate ? 2 : 1;
  double *gp = c.R.gpart;
  Scal &sc = c.sm.sc;
#pragma unroll 1
  for (int q = local ? c.wp : c.warp_id(); q < D.ngrp * nv; q += local ? c.nw : c.warps()) {
    const int grp = q / nv, v = q - grp * nv;
    const int u0 = 256 * grp + 8 * c.lane;
    double t[1] = {0.0};
    if (u0 < D.nunits) {
      const double *p = D.sums + (size_t)v * D.nunits + u0;
      double a[8];
#pragma unroll
      for (int w = 0; w < 8; ++w) a[w] = __ldcg(p + w);
      t[0] = ((a[0] + a[4]) + (a[2] + a[6])) + ((a[1] + a[5]) + (a[3] + a[7]));
    }
    warp_sum<1>(t);
    if (c.lane == 0) {
      if (local) sc.tot[v] = t[0];
      else gp[(size_t)grp * 3 + v] = t[0];
    }
  }
  if (!local) {
    c.arrive();
    c.wait();
#pragma unroll 1
    for (int v = c.wp; v < nv; v += c.nw) {
      double t[1] = {0.0};
#pragma unroll 1
      for (int q = c.lane; q < D.ngrp; q += 32) t[0] += __ldcg(gp + (size_t)q * 3 + v);
      warp_sum<1>(t);
      if (c.lane == 0) sc.tot[v] = t[0];
    }
  }
  __syncthreads();
  const int parts = dot_parts(step);
  if (c.wp < parts && c.lane == 0) sc.part[c.wp] = dot_part(step, sc, c.wp);
  __syncthreads();
  if (threadIdx.x == 0 && (every || sc.status == kRunning)) dot_decide(step, sc);
  __syncthreads();
}

// ------------------------------------------------ units of one warp
//
// The wide form: a lane per row, as in the launch-per-phase kernels.  The
// caller has waited.

// The earlier phases' results for a sweep: y (forward) or z (backward); with
// FP32 factors from f, y or the floats of z (Sys::zf).  A conversion from
// FP64 costs the FP64 pipe what an FMA does: three per gathered block and
// warp of a trio took a refactorisation and solve of 21,793 rows from 157.8
// to 168.3 us.  (The launches per phase keep the conversions: there the
// floats' stores cost as much, 3270 against 3247 us at 949,871 rows.)
template <typename TF>
__device__ __forceinline__ Vec3<TF> sweep_gather(const void *y, const double *z, const float *f, bool fwd, int j) {
  if constexpr (sizeof(TF) == 4) {
    return load3cg(f + 3ll * j);
  } else {
    const Vec3<double> v = load3cg((fwd ? static_cast<const double *>(y) : z) + 3ll * j);
    return {(TF)v.c0, (TF)v.c1, (TF)v.c2};
  }
}

// One slice of a sweep over the phase's rows [E.z, E.w): fwd_rows (fwd; the
// right-hand side p in the first half of an iteration, s in the second, the
// caller's vector in a standalone application) or bwd_rows.  A standalone
// application reads and writes the caller's order in place.
template <typename TF, int MODE>
__device__ __forceinline__ void sweep_unit(ResCtx &c, int4 E, bool fwd, bool second) {
  const Sys &S = c.S;
  const int lane = c.lane, sl = E.y, s0 = sl * 32, i = s0 + lane;
  constexpr bool kPlain = MODE == kModePlain;
  TF *y = static_cast<TF *>(S.y);
  double *z = kPlain ? S.t : second ? S.sh : S.ph;
  const uint2 M = __ldg(S.sl_mask + sl);
  const bool eager = (M.x >> lane) & 1u;
  const bool act = i >= E.z && i < E.w && (fwd || !eager);
  const int32_t *rp = fwd ? S.l_rp : S.u_rp, *col = fwd ? S.l_col : S.u_col;
  const TF *lu = static_cast<const TF *>(S.lu);
  const TF *vals = lu + (fwd ? 0 : S.u_off);
  const float *zf = sizeof(TF) == 4 ? (fwd ? static_cast<const float *>(S.y) : S.zf) : nullptr;
  const int len = (i < S.n) ? __ldg(rp + i + 1) - __ldg(rp + i) : 0;
  int base = __ldg(rp + s0);
  const int maxlen = __reduce_max_sync(0xffffffffu, len);
  Vec3<TF> a{TF(0), TF(0), TF(0)};
  const int64_t o = kPlain && act ? 3ll * __ldg(S.perm + i) : 0;
  if (act && fwd && kPlain) {
    const Vec3<double> h = load3cg(S.b_in + o);
    a = {(TF)h.c0, (TF)h.c1, (TF)h.c2};
  } else if (act && fwd) {
    Vec3<double> h = load3cg(S.r + 3ll * i);
    const Vec3<double> vo = load3cg(S.v + 3ll * i);
    const Scal &sc = c.sm.sc;
    if (second) {
      const double c1 = sc.alpha;
      h.c0 = fma(-c1, vo.c0, h.c0);
      h.c1 = fma(-c1, vo.c1, h.c1);
      h.c2 = fma(-c1, vo.c2, h.c2);
    } else {
      const Vec3<double> po = load3cg(S.p + 3ll * i);
      const double c1 = sc.beta, c2 = sc.omega;
      h.c0 = fma(c1, fma(-c2, vo.c0, po.c0), h.c0);
      h.c1 = fma(c1, fma(-c2, vo.c1, po.c1), h.c1);
      h.c2 = fma(c1, fma(-c2, vo.c2, po.c2), h.c2);
    }
    double *ho = (second ? S.s : S.p) + 3ll * i;
    ho[0] = h.c0; ho[1] = h.c1; ho[2] = h.c2;
    a = {(TF)h.c0, (TF)h.c1, (TF)h.c2};
  } else if (act) {
    a = load3cg(static_cast<const TF *>(y) + 3ll * i);
  }
  const unsigned lt = lanemask_lt();
#pragma unroll 1
  for (int k = 0; k < maxlen; k += 2) {  // two slabs per step for memory-level parallelism
    const unsigned m0 = __ballot_sync(0xffffffffu, len > k), m1 = __ballot_sync(0xffffffffu, len > k + 1);
    const int b0 = base, b1 = base + __popc(m0), q0 = __popc(m0 & lt), q1 = __popc(m1 & lt);
    base = b1 + __popc(m1);
    const bool u0 = act && len > k, u1 = act && len > k + 1;
    int j0 = 0, j1 = 0;
    if (u0) j0 = __ldcs(col + b0 + q0);
    if (u1) j1 = __ldcs(col + b1 + q1);
    if (u0) {
      const Vec3<TF> v = sweep_gather<TF>(S.y, z, zf, fwd, j0);
      blk_sub<TF>(vals + 9ll * b0 + q0, __popc(m0), v.c0, v.c1, v.c2, a.c0, a.c1, a.c2);
    }
    if (u1) {
      const Vec3<TF> v = sweep_gather<TF>(S.y, z, zf, fwd, j1);
      blk_sub<TF>(vals + 9ll * b1 + q1, __popc(m1), v.c0, v.c1, v.c2, a.c0, a.c1, a.c2);
    }
  }
  if (!act) return;
  if (!kPlain && !fwd && sizeof(TF) == sizeof(double) && S.uz && ((__ldg(S.sp_mask + sl).y >> lane) & 1u)) {
    const Vec3<TF> yr = load3cg(static_cast<const TF *>(y) + 3ll * i);
    double *w = S.uz + 3ll * i;
    w[0] = (double)(yr.c0 - a.c0);
    w[1] = (double)(yr.c1 - a.c1);
    w[2] = (double)(yr.c2 - a.c2);
  }
  if (!fwd || eager) {
    TF d[9];
    load_dinv<TF>(lu + S.d_off + (int64_t)kSliceVals * sl + lane, d);
    const Vec3<TF> v = store_dinv_product<TF>(z + 3ll * i, d, a.c0, a.c1, a.c2);
    if constexpr (sizeof(TF) == 4) {
      float *f = S.zf + 3ll * i;
      f[0] = v.c0; f[1] = v.c1; f[2] = v.c2;
    }
    if (kPlain) store_dinv_product<TF>(S.x_out + o, d, a.c0, a.c1, a.c2);
  }
  if (fwd && ((M.y >> lane) & 1u)) {
    TF *yi = y + 3ll * i;
    yi[0] = a.c0; yi[1] = a.c1; yi[2] = a.c2;
  }
}

// The wells' term of perforated row i, component r: k_wells' expressions on
// t2, the row's perforations in order.
__device__ __forceinline__ double wells_term(const Sys &S, int i, int r) {
  double s = 0.0;
#pragma unroll 1
  for (int q = __ldg(S.w_rptr + i); q < __ldg(S.w_rptr + i + 1); ++q) {
    const int p = __ldg(S.w_rperf + q);
    const double *t2 = S.w_t2 + 4ll * __ldg(S.w_of + p);
    const double *Cp = S.w_C + 12ll * p + r;
    s += fma(__ldg(Cp), __ldcg(t2),
             fma(__ldg(Cp + 3), __ldcg(t2 + 1), fma(__ldg(Cp + 6), __ldcg(t2 + 2), __ldg(Cp + 9) * __ldcg(t2 + 3))));
  }
  return s;
}

// Which vectors a product's step reads and writes.
struct ProductIo {
  const double *x, *xin;  // the operator's input; what the application that gave it started from
  double *out;
  const double *dot;      // (r^, v) or (t, s)
  __device__ __forceinline__ ProductIo(const Sys &S, int step)
      : x(step == kStepFinish ? S.x : step == kStepS ? S.sh : S.ph), xin(step == kStepS ? S.s : S.p),
        out(step == kStepS ? S.t : S.v), dot(step == kStepS ? S.s : S.rh) {}
};

// A product's slice: v = A p^ and (r^, v); t = A s^, (t,s), (t,t), (s,s); or
// the true residual and x back in the caller's order (zeros on failure).
// row_operator_applied with reuse, row_operator without.
__device__ __forceinline__ void product_unit(ResCtx &c, int sl, int step, bool reuse) {
  const Sys &S = c.S;
  const bool fin = step == kStepFinish;
  const int status = c.sm.sc.status;
  const bool ok = !fin || status == OPM_OK || status == OPM_NOT_CONVERGED;
  const ProductIo io(S, step);
  reuse = reuse && !fin;
  const int lane = c.lane, n = S.n, s0 = sl * 32, i = s0 + lane;
  const bool in = i < n;
  const int len = in ? __ldg(S.a_rp + i + 1) - __ldg(S.a_rp + i) : 0;
  const uint2 M = reuse ? __ldg(S.sp_mask + sl) : make_uint2(0u, 0u);
  const int lead = reuse ? (in ? __ldg(S.sp_len + i) : 0) : len;
  int base = __ldg(S.a_rp + s0);
  const int maxlead = __reduce_max_sync(0xffffffffu, lead);
  const unsigned lt = lanemask_lt();
  Vec3<double> y{0.0, 0.0, 0.0};
  if (in) {
    if (S.nwells > 0 && ((__ldg(S.w_mask + sl) >> lane) & 1u))
      y = {-wells_term(S, i, 0), -wells_term(S, i, 1), -wells_term(S, i, 2)};
    const double *e = ((M.x >> lane) & 1u) ? io.xin + 3ll * i : ((M.y >> lane) & 1u) ? S.uz + 3ll * i : nullptr;
    if (e) {
      const Vec3<double> v = load3cg(e);
      y.c0 += v.c0;
      y.c1 += v.c1;
      y.c2 += v.c2;
    }
  }
#pragma unroll 1
  for (int k = 0; k < maxlead; ++k) {
    const unsigned m = __ballot_sync(0xffffffffu, len > k);
    if (lead > k) {
      const int cnt = __popc(m), q = __popc(m & lt);
      const Vec3<double> x = load3cg(io.x + 3ll * __ldcs(S.a_col + base + q));
      const double *av = S.a_val + 9ll * base + q;
      double b[9];
#pragma unroll
      for (int e = 0; e < 9; ++e) b[e] = __ldcs(av + e * cnt);
      y.c0 = fma(b[0], x.c0, fma(b[1], x.c1, fma(b[2], x.c2, y.c0)));
      y.c1 = fma(b[3], x.c0, fma(b[4], x.c1, fma(b[5], x.c2, y.c1)));
      y.c2 = fma(b[6], x.c0, fma(b[7], x.c1, fma(b[8], x.c2, y.c2)));
    }
    base += __popc(m);
  }
  double acc[3] = {0.0, 0.0, 0.0};
  if (in && fin) {
    const int o = __ldg(S.perm + i);
    if (ok) {
      const Vec3<double> b = load3cg(S.b_in + 3ll * o);
      const double d0 = b.c0 - y.c0, d1 = b.c1 - y.c1, d2 = b.c2 - y.c2;
      acc[0] = fma(d0, d0, fma(d1, d1, fma(d2, d2, acc[0])));
    }
    const Vec3<double> x = load3cg(S.x + 3ll * i);
    double *xo = S.x_out + 3ll * o;
    xo[0] = ok ? x.c0 : 0.0;
    xo[1] = ok ? x.c1 : 0.0;
    xo[2] = ok ? x.c2 : 0.0;
  } else if (in) {
    double *out = io.out + 3ll * i;
    out[0] = y.c0; out[1] = y.c1; out[2] = y.c2;
    const Vec3<double> q = load3cg(io.dot + 3ll * i);
    acc[0] = fma(q.c0, y.c0, fma(q.c1, y.c1, fma(q.c2, y.c2, acc[0])));
    if (step == kStepS) {
      acc[1] = fma(y.c0, y.c0, fma(y.c1, y.c1, fma(y.c2, y.c2, acc[1])));
      acc[2] = fma(q.c0, q.c0, fma(q.c1, q.c1, fma(q.c2, q.c2, acc[2])));
    }
  }
  store_unit(c.R.ds, sl, acc);
}

// inv(D) B x of every well, one warp per well (k_wells).
__device__ __forceinline__ void wells_stage(ResCtx &c, int step) {
  c.wait();
  const Sys &S = c.S;
  if (!c.dead) {
    const double *x = step == kStepFinish ? S.x : step == kStepS ? S.sh : S.ph;
#pragma unroll 1
    for (int w = c.warp_id(); w < S.nwells; w += c.warps()) {
      double t1[4] = {0.0, 0.0, 0.0, 0.0};
      const int p1 = __ldg(S.w_ptr + w + 1);
#pragma unroll 1
      for (int p = __ldg(S.w_ptr + w) + c.lane; p < p1; p += 32) {
        const Vec3<double> v = load3cg(x + 3ll * __ldg(S.w_cell + p));
        const double *Bp = S.w_B + 12ll * p;
#pragma unroll
        for (int r = 0; r < 4; ++r)
          t1[r] = fma(__ldg(Bp + 3 * r), v.c0, fma(__ldg(Bp + 3 * r + 1), v.c1, fma(__ldg(Bp + 3 * r + 2), v.c2, t1[r])));
      }
      warp_sum<4>(t1);
      if (c.lane < 4) {
        const double *Dw = S.w_Dinv + 16ll * w + 4 * c.lane;
        S.w_t2[4ll * w + c.lane] =
            fma(__ldg(Dw), t1[0], fma(__ldg(Dw + 1), t1[1], fma(__ldg(Dw + 2), t1[2], __ldg(Dw + 3) * t1[3])));
      }
    }
  }
  c.arrive();
}

// Setup unit u (k_setup's rows of one warp: r = r^ = P b, x = p = v = 0 and
// the unit's part of ||b||^2) or update unit u (k_update's rows).
__device__ __forceinline__ void vector_unit(ResCtx &c, int u, bool setup) {
  const Sys &S = c.S;
  const double alpha = c.sm.sc.alpha, omega = c.sm.sc.omega;
  const bool half = c.sm.sc.half;
  double acc[3] = {0.0, 0.0, 0.0};
#pragma unroll 1
  for (int p = 0, i = (u >> 3) * kTileRows + (u & 7) * 32 + c.lane; p < 4; ++p, i += 256) {
    if (i >= S.n) break;
    const size_t e = 3ll * i;
    if (setup) {
      const Vec3<double> b = load3cg(S.b_in + 3ll * __ldg(S.perm + i));
      S.r[e] = b.c0; S.r[e + 1] = b.c1; S.r[e + 2] = b.c2;
      S.rh[e] = b.c0; S.rh[e + 1] = b.c1; S.rh[e + 2] = b.c2;
#pragma unroll
      for (int q = 0; q < 3; ++q) {
        S.x[e + q] = 0.0;
        S.p[e + q] = 0.0;
        S.v[e + q] = 0.0;
      }
      acc[0] = fma(b.c0, b.c0, fma(b.c1, b.c1, fma(b.c2, b.c2, acc[0])));
      continue;
    }
    Vec3<double> x = load3cg(S.x + e);
    const Vec3<double> ph = load3cg(S.ph + e);
    if (!half) {
      const Vec3<double> sh = load3cg(S.sh + e), t = load3cg(S.t + e), s = load3cg(S.s + e), q = load3cg(S.rh + e);
      x.c0 = fma(omega, sh.c0, x.c0);
      x.c1 = fma(omega, sh.c1, x.c1);
      x.c2 = fma(omega, sh.c2, x.c2);
      const double r0 = fma(-omega, t.c0, s.c0), r1 = fma(-omega, t.c1, s.c1), r2 = fma(-omega, t.c2, s.c2);
      S.r[e] = r0; S.r[e + 1] = r1; S.r[e + 2] = r2;
      acc[0] = fma(r2, r2, fma(r1, r1, fma(r0, r0, acc[0])));
      acc[1] = fma(q.c2, r2, fma(q.c1, r1, fma(q.c0, r0, acc[1])));
    }
    S.x[e] = fma(alpha, ph.c0, x.c0);
    S.x[e + 1] = fma(alpha, ph.c1, x.c1);
    S.x[e + 2] = fma(alpha, ph.c2, x.c2);
  }
  if (setup || !half) store_unit(c.R.du, u, acc);
}

// ------------------------------------------------ units of three warps
//
// The trio form, for systems whose phases leave the chip short of work: the
// three warps of a trio compute the three components of a slice's rows.  An
// FP64 instruction of a warp takes 64 cycles of its scheduler's quarter of the
// SM, so a slice of six-block rows costs one warp 70 x 64 cycles and a trio a
// third of that, on three schedulers; and with a third of a row's blocks to
// hold, the first kPre blocks are loaded before the wait without spills.  A
// component's chain of operations is that of the one-warp form.

// The blocks and their columns are loaded with the default cache policy, not as
// streams: a system of these sizes stays in L2 from one product to the next.
// Evict-first loads took (us, refactor + solve) 252.4 against 249.7 at 44,431
// rows, 449.4 against 433.0 at 60,793, 32.8 against 31.4 for an application
// alone at 44,431.
constexpr int kPre = 6;  // blocks loaded ahead: the couplings of a cell on a grid

// The first kPre blocks of the lane's row, row r of each: columns and values.
// Blocks that the row has not are zero: left undefined, the arrays would count
// as carried around the solve's loop and be spilled (3.4 KB per thread).
template <typename T>
__device__ __forceinline__ int preload_row(const int32_t *col, const T *vals, int len, int lead, int base, int r,
                                           int (&jp)[kPre], T (&bp)[kPre][3]) {
  const unsigned lt = lanemask_lt();
#pragma unroll
  for (int k = 0; k < kPre; ++k) {
    const unsigned m = __ballot_sync(0xffffffffu, len > k);
    jp[k] = 0;
    bp[k][0] = bp[k][1] = bp[k][2] = T(0);
    if (lead > k) {
      const int q = __popc(m & lt), cnt = __popc(m);
      const T *v = vals + 9ll * base + q + 3 * r * cnt;
      jp[k] = __ldca(col + base + q);
      bp[k][0] = __ldca(v);
      bp[k][1] = __ldca(v + cnt);
      bp[k][2] = __ldca(v + 2 * cnt);
    }
    base += __popc(m);
  }
  return base;
}

// sweep_unit by a trio; FIRST: wait() is called here.
template <typename TF, int MODE, bool FIRST>
__device__ __forceinline__ void sweep_trio(ResCtx &c, int4 E, bool fwd, bool second) {
  const Sys &S = c.S;
  const int lane = c.lane, r = c.r, sl = E.y, s0 = sl * 32, i = s0 + lane;
  constexpr bool kPlain = MODE == kModePlain;
  TF *y = static_cast<TF *>(S.y);
  double *z = kPlain ? S.t : second ? S.sh : S.ph;
  const uint2 M = __ldg(S.sl_mask + sl);
  const bool eager = (M.x >> lane) & 1u;
  const bool act = i >= E.z && i < E.w && (fwd || !eager);
  const int32_t *rp = fwd ? S.l_rp : S.u_rp, *col = fwd ? S.l_col : S.u_col;
  const TF *lu = static_cast<const TF *>(S.lu);
  const TF *vals = lu + (fwd ? 0 : S.u_off);
  const float *zf = sizeof(TF) == 4 ? (fwd ? static_cast<const float *>(S.y) : S.zf) : nullptr;
  const int len = (i < S.n) ? __ldg(rp + i + 1) - __ldg(rp + i) : 0;
  const int lead = act ? len : 0;
  int base = __ldg(rp + s0);
  const int maxlen = __reduce_max_sync(0xffffffffu, len);
  const bool use_d = act && (!fwd || eager);
  int jp[kPre];
  TF bp[kPre][3], d[3] = {TF(0), TF(0), TF(0)};
  base = preload_row<TF>(col, vals, len, lead, base, r, jp, bp);
  if (use_d) {
    const TF *D = lu + S.d_off + (int64_t)kSliceVals * sl + lane + 96 * r;
    d[0] = __ldca(D);
    d[1] = __ldca(D + 32);
    d[2] = __ldca(D + 64);
  }
  if (FIRST) c.wait();
  double h = 0.0, vo = 0.0, po = 0.0;
  TF a = TF(0);
  const int64_t e = 3ll * i + r, o = kPlain && act ? 3ll * __ldg(S.perm + i) + r : 0;
  if (act) {
    if (fwd && kPlain) {
      h = __ldcg(S.b_in + o);
    } else if (fwd) {
      h = __ldcg(S.r + e);
      vo = __ldcg(S.v + e);
      if (!second) po = __ldcg(S.p + e);
    } else {
      a = __ldcg(y + e);
    }
  }
  Vec3<TF> vv[kPre];
#pragma unroll
  for (int k = 0; k < kPre; ++k) {
    vv[k] = {TF(0), TF(0), TF(0)};
    if (lead > k) vv[k] = sweep_gather<TF>(S.y, z, zf, fwd, jp[k]);
  }
  const TF y0 = a;  // the backward sweep's y_i
  if (act && fwd && kPlain) {
    a = (TF)h;
  } else if (act && fwd) {
    const Scal &sc = c.sm.sc;
    h = second ? fma(-sc.alpha, vo, h) : fma(sc.beta, fma(-sc.omega, vo, po), h);
    (second ? S.s : S.p)[e] = h;
    a = (TF)h;
  }
#pragma unroll
  for (int k = 0; k < kPre; ++k)
    if (lead > k) a = fma(-bp[k][0], vv[k].c0, fma(-bp[k][1], vv[k].c1, fma(-bp[k][2], vv[k].c2, a)));
  const unsigned lt = lanemask_lt();
#pragma unroll 1
  for (int k = kPre; k < maxlen; ++k) {
    const unsigned m = __ballot_sync(0xffffffffu, len > k);
    if (lead > k) {
      const int cnt = __popc(m), q = __popc(m & lt);
      const Vec3<TF> v = sweep_gather<TF>(S.y, z, zf, fwd, __ldca(col + base + q));
      const TF *b = vals + 9ll * base + q + 3 * r * cnt;
      const TF b0 = __ldca(b), b1 = __ldca(b + cnt), b2 = __ldca(b + 2 * cnt);
      a = fma(-b0, v.c0, fma(-b1, v.c1, fma(-b2, v.c2, a)));
    }
    base += __popc(m);
  }
  double(*ex)[32] = c.sm.ex[c.trio][c.flip][0];
  c.flip ^= 1;
  ex[r][lane] = (double)a;
  c.trio_sync();
  const TF a0 = (TF)ex[0][lane], a1 = (TF)ex[1][lane], a2 = (TF)ex[2][lane];
  if (!act) return;
  if (!kPlain && !fwd && sizeof(TF) == sizeof(double) && S.uz && ((__ldg(S.sp_mask + sl).y >> lane) & 1u))
    S.uz[e] = (double)(y0 - a);
  if (use_d) {
    const TF f = fma(d[0], a0, fma(d[1], a1, d[2] * a2));
    const double v = (double)f;
    z[e] = v;
    if constexpr (sizeof(TF) == 4) S.zf[e] = f;
    if (kPlain) S.x_out[o] = v;
  }
  if (fwd && ((M.y >> lane) & 1u)) y[e] = a;
}

// product_unit by a trio; FIRST: wait() is called here.
template <bool FIRST>
__device__ __forceinline__ void product_trio(ResCtx &c, int sl, int step, bool reuse) {
  const Sys &S = c.S;
  const bool fin = step == kStepFinish;
  const int status = c.sm.sc.status;
  const bool ok = !fin || status == OPM_OK || status == OPM_NOT_CONVERGED;
  const ProductIo io(S, step);
  reuse = reuse && !fin;
  const int lane = c.lane, r = c.r, n = S.n, s0 = sl * 32, i = s0 + lane;
  const bool in = i < n;
  const int len = in ? __ldg(S.a_rp + i + 1) - __ldg(S.a_rp + i) : 0;
  const uint2 M = reuse ? __ldg(S.sp_mask + sl) : make_uint2(0u, 0u);
  const int lead = reuse ? (in ? __ldg(S.sp_len + i) : 0) : len;
  int base = __ldg(S.a_rp + s0);
  const int maxlead = __reduce_max_sync(0xffffffffu, lead);
  int jp[kPre];
  double bp[kPre][3];
  base = preload_row<double>(S.a_col, S.a_val, len, lead, base, r, jp, bp);
  if (FIRST) c.wait();
  const int64_t e = 3ll * i + r;
  double y = 0.0;
  if (in) {
    if (S.nwells > 0 && ((__ldg(S.w_mask + sl) >> lane) & 1u)) y = -wells_term(S, i, r);
    if ((M.x >> lane) & 1u) y += __ldcg(io.xin + e);
    else if ((M.y >> lane) & 1u) y += __ldcg(S.uz + e);
  }
  Vec3<double> xv[kPre], q{0.0, 0.0, 0.0};
#pragma unroll
  for (int k = 0; k < kPre; ++k) {
    xv[k] = {0.0, 0.0, 0.0};
    if (lead > k) xv[k] = load3cg(io.x + 3ll * jp[k]);
  }
  const int o = (in && fin) ? __ldg(S.perm + i) : i;
  if (in) q = load3cg((fin ? S.b_in : io.dot) + 3ll * o);
#pragma unroll
  for (int k = 0; k < kPre; ++k)
    if (lead > k) y = fma(bp[k][0], xv[k].c0, fma(bp[k][1], xv[k].c1, fma(bp[k][2], xv[k].c2, y)));
  const unsigned lt = lanemask_lt();
#pragma unroll 1
  for (int k = kPre; k < maxlead; ++k) {
    const unsigned m = __ballot_sync(0xffffffffu, len > k);
    if (lead > k) {
      const int cnt = __popc(m), p = __popc(m & lt);
      const Vec3<double> x = load3cg(io.x + 3ll * __ldca(S.a_col + base + p));
      const double *b = S.a_val + 9ll * base + p + 3 * r * cnt;
      const double b0 = __ldca(b), b1 = __ldca(b + cnt), b2 = __ldca(b + 2 * cnt);
      y = fma(b0, x.c0, fma(b1, x.c1, fma(b2, x.c2, y)));
    }
    base += __popc(m);
  }
  if (in && !fin) io.out[e] = y;
  double(*ex)[32] = c.sm.ex[c.trio][c.flip][0];
  c.flip ^= 1;
  ex[r][lane] = y;
  c.trio_sync();
  // past the trio's reads of b: x may be written in its place
  if (in && fin) S.x_out[3ll * o + r] = ok ? __ldcg(S.x + e) : 0.0;
  // the dot products, one per warp: (q, y), (y, y), (q, q)
  if (r > 0 && step != kStepS) return;
  double v[1] = {0.0};
  if (in && ok) {
    const double y0 = ex[0][lane], y1 = ex[1][lane], y2 = ex[2][lane];
    Vec3<double> f = q, g{y0, y1, y2};
    if (fin) f = g = {q.c0 - y0, q.c1 - y1, q.c2 - y2};
    if (r == 1) f = g;
    if (r == 2) g = q;
    v[0] = fma(f.c0, g.c0, fma(f.c1, g.c1, fma(f.c2, g.c2, v[0])));
  }
  warp_sum<1>(v);
  if (lane == 0) c.R.ds.sums[(size_t)r * c.R.ds.nunits + sl] = v[0];
}

// vector_unit by a trio.
__device__ __forceinline__ void vector_trio(ResCtx &c, int u, bool setup) {
  const Sys &S = c.S;
  const double alpha = c.sm.sc.alpha, omega = c.sm.sc.omega;
  const bool half = c.sm.sc.half;
  const int lane = c.lane, r = c.r, i0 = (u >> 3) * kTileRows + (u & 7) * 32 + lane;
  double(*ex)[3][32] = c.sm.ex[c.trio][c.flip];
  c.flip ^= 1;
  double x[4], ph[4], sh[4], t[4], s[4];
#pragma unroll
  for (int p = 0; p < 4; ++p) {
    const int i = i0 + 256 * p;
    const int64_t e = 3ll * i + r;
    x[p] = ph[p] = sh[p] = t[p] = s[p] = 0.0;
    if (i < S.n) {
      if (setup) {
        s[p] = __ldcg(S.b_in + 3ll * __ldg(S.perm + i) + r);
      } else {
        x[p] = __ldcg(S.x + e);
        ph[p] = __ldcg(S.ph + e);
        if (!half) {
          sh[p] = __ldcg(S.sh + e);
          t[p] = __ldcg(S.t + e);
          s[p] = __ldcg(S.s + e);
        }
      }
    }
  }
#pragma unroll
  for (int p = 0; p < 4; ++p) {
    const int i = i0 + 256 * p;
    const int64_t e = 3ll * i + r;
    double rr = s[p];
    if (i < S.n) {
      if (setup) {
        S.r[e] = rr;
        S.rh[e] = rr;
        S.x[e] = 0.0;
        S.p[e] = 0.0;
        S.v[e] = 0.0;
      } else if (half) {
        S.x[e] = fma(alpha, ph[p], x[p]);
      } else {
        S.x[e] = fma(alpha, ph[p], fma(omega, sh[p], x[p]));
        rr = fma(-omega, t[p], s[p]);
        S.r[e] = rr;
      }
    }
    ex[p][r][lane] = rr;
  }
  c.trio_sync();
  if (!setup && half) return;
  // ||b||^2, or ||r||^2 and (r^, r): one per warp
  if (r > (setup ? 0 : 1)) return;
  double acc[1] = {0.0};
#pragma unroll
  for (int p = 0; p < 4; ++p) {
    const int i = i0 + 256 * p;
    if (i >= S.n) break;
    const double r0 = ex[p][0][lane], r1 = ex[p][1][lane], r2 = ex[p][2][lane];
    if (setup) {
      acc[0] = fma(r0, r0, fma(r1, r1, fma(r2, r2, acc[0])));
    } else {
      const Vec3<double> q = r == 0 ? Vec3<double>{r0, r1, r2} : load3cg(S.rh + 3ll * i);
      acc[0] = fma(q.c2, r2, fma(q.c1, r1, fma(q.c0, r0, acc[0])));
    }
  }
  warp_sum<1>(acc);
  if (lane == 0) c.R.du.sums[(size_t)r * c.R.du.nunits + u] = acc[0];
}

// copy_row_to_factors by a trio: row r of every block of slice sl.
template <typename TF>
__device__ __forceinline__ void copy_trio(const ResCtx &c, const Sys &S, int sl) {
  const int lane = c.lane, r = c.r, s0 = sl * 32, i = s0 + lane;
  TF *lu = static_cast<TF *>(S.lu);
  const unsigned lt = lanemask_lt();
  const int len = (i < S.n) ? __ldg(S.a_rp + i + 1) - __ldg(S.a_rp + i) : 0;
  int base = __ldg(S.a_rp + s0);
  const int maxlen = __reduce_max_sync(0xffffffffu, len);
#pragma unroll 4
  for (int k = 0; k < maxlen; ++k) {
    const unsigned m = __ballot_sync(0xffffffffu, len > k);
    if (len > k) {
      const int cnt = __popc(m), w = base + __popc(m & lt);
      const int64_t dst = __ldg(S.a_dst + w);
      double *av = S.a_val + 9ll * base + __popc(m & lt) + 3 * r * cnt;
      double e[3];
      if (S.vals_in) {
        const double *src = S.vals_in + 9ll * __ldg(S.a_src + w) + 3 * r;
#pragma unroll
        for (int q = 0; q < 3; ++q) e[q] = __ldg(src + q);
#pragma unroll
        for (int q = 0; q < 3; ++q) av[q * cnt] = e[q];
      } else {
#pragma unroll
        for (int q = 0; q < 3; ++q) e[q] = av[q * cnt];
      }
      if (dst >= 0) {
        TF *t = lu + (dst >> 6) + 3 * r * (int)(dst & 63);
#pragma unroll
        for (int q = 0; q < 3; ++q) t[q * (int)(dst & 63)] = (TF)e[q];
      }
    }
    base += __popc(m);
  }
}

// eliminate_row and invert_diagonal by a trio: row r of the slice's blocks,
// whose updates need no other row of them until the inversion.
template <typename TF, typename Note>
__device__ __forceinline__ void eliminate_trio(ResCtx &c, const Sys &S, int4 E, const Note &note) {
  const int lane = c.lane, r = c.r, sl = E.y, s0 = sl * 32, i = s0 + lane;
  const bool act = i >= E.z && i < E.w;
  TF *lu = static_cast<TF *>(S.lu);
  const unsigned lt = lanemask_lt();
  const int lrow = (i < S.n) ? __ldg(S.l_rp + i) : 0;
  const int len = (i < S.n) ? __ldg(S.l_rp + i + 1) - lrow : 0;
  int base = __ldg(S.l_rp + s0);
  const int maxlen = __reduce_max_sync(0xffffffffu, act ? len : 0);
#pragma unroll 1
  for (int k = 0; k < maxlen; ++k) {
    const unsigned m = __ballot_sync(0xffffffffu, len > k);
    if (act && len > k) {
      const int cnt = __popc(m), q = __popc(m & lt);
      const int kc = __ldg(S.l_col + base + q);
      TF *Lp = lu + 9ll * base + q + 3 * r * cnt;
      const TF *Dk = lu + S.d_off + (int64_t)kSliceVals * (kc >> 5) + (kc & 31);
      TF a[3], d[9], l[3];
#pragma unroll
      for (int e = 0; e < 3; ++e) a[e] = Lp[e * cnt];
#pragma unroll
      for (int e = 0; e < 9; ++e) d[e] = __ldcg(Dk + 32 * e);
#pragma unroll
      for (int e = 0; e < 3; ++e) l[e] = fma(a[0], d[e], fma(a[1], d[3 + e], a[2] * d[6 + e]));
#pragma unroll
      for (int e = 0; e < 3; ++e) Lp[e * cnt] = l[e];
      const int u1 = __ldg(S.upd_ptr + lrow + k + 1);
#pragma unroll 1
      for (int u = __ldg(S.upd_ptr + lrow + k); u < u1; ++u) {
        const int64_t ds = __ldg(S.upd_dst + u), ss = __ldg(S.upd_src + u);
        const int dstr = (int)(ds & 63), sstr = (int)(ss & 63);
        TF *Ap = lu + (ds >> 6) + 3 * r * dstr;
        const TF *Up = lu + (ss >> 6);
        TF uu[9];
#pragma unroll
        for (int e = 0; e < 9; ++e) uu[e] = __ldcg(Up + e * sstr);
#pragma unroll
        for (int e = 0; e < 3; ++e) {
          TF *ap = Ap + e * dstr;
          *ap = fma(-l[0], uu[e], fma(-l[1], uu[3 + e], fma(-l[2], uu[6 + e], *ap)));
        }
      }
    }
    base += __popc(m);
  }
  // the eliminated diagonal block, then its inverse
  TF *Dp = lu + S.d_off + (int64_t)kSliceVals * sl + lane;
  double(*ex)[3][32] = c.sm.ex[c.trio][c.flip];
  c.flip ^= 1;
#pragma unroll
  for (int e = 0; e < 3; ++e) ex[r][e][lane] = act ? (double)Dp[32 * (3 * r + e)] : 0.0;
  c.trio_sync();
  TF a[9], o[9];
#pragma unroll
  for (int e = 0; e < 9; ++e) a[e] = (TF)ex[e / 3][e % 3][lane];
  if (!act) return;
  if (!inv3<TF>(a, o) && r == 0) note(i);
#pragma unroll
  for (int e = 0; e < 3; ++e) Dp[32 * (3 * r + e)] = r == 0 ? o[e] : r == 1 ? o[3 + e] : o[6 + e];
}

// ------------------------------------------------ the kernel

// A singular pivot of the lane's row.
__device__ __forceinline__ void note_singular(int32_t *err, int i) {
  atomicCAS(err, 0, (int32_t)OPM_ERR_ZERO_PIVOT);
  atomicMax(err + 1, 0x7fffffff - i);
}

// ILU0, phase by phase.  Trios copy the rows of all phases first, so that a
// phase only eliminates; the wide form is that of the large phases' launches
// (factor_rows).
template <typename TF, bool TRIO>
__device__ __forceinline__ void resident_factor(ResCtx &c) {
  const Batch &B = c.R.B;
  if (TRIO) {
#pragma unroll 1
    for (int sl = c.g; sl < B.nall; sl += c.W) copy_trio<TF>(c, c.S, sl);
    c.arrive();
  }
#pragma unroll 1
  for (int p = 0; p < B.nphases && !c.dead; ++p) {
    if (TRIO || p > 0) c.wait();
    const int e1 = __ldg(B.fwd_ptr + p + 1);
#pragma unroll 1
    for (int e = __ldg(B.fwd_ptr + p) + c.g; e < e1 && !c.dead; e += c.W) {
      const int4 E = __ldg(B.ent + e);
      const Sys &S = c.S;
      const auto note = [&](int i) { note_singular(c.R.err, i); };
      if constexpr (TRIO) eliminate_trio<TF>(c, S, E, note);
      else factor_rows<TF, true, false, sizeof(TF) == 4>(S, E.y, E.z, E.w, note);
    }
    c.arrive();
  }
  c.wait();
  if (threadIdx.x == 0 && __ldcg(c.R.err) != 0) c.sm.sc.status = OPM_ERR_ZERO_PIVOT;
  __syncthreads();
}

// One preconditioner application.  The first forward phase follows the
// caller's wait; the last phase ends with an arrival.
template <typename TF, int MODE, bool TRIO>
__device__ __forceinline__ void resident_apply(ResCtx &c, bool second) {
  const Batch &B = c.R.B;
  // The first phase's rows have no L blocks, so there is nothing to load ahead
  // of the wait but the warp's entry, which is kept: finding it again took two
  // loads from L2, one after the other.
#pragma unroll 1
  for (int e = c.g, e1 = c.sm.phase0; e < e1; e += c.W) {
    const int4 E = e == c.g ? c.sm.first[c.wp] : __ldg(B.ent + e);
    if constexpr (TRIO) sweep_trio<TF, MODE, false>(c, E, true, second);
    else sweep_unit<TF, MODE>(c, E, true, second);
  }
  c.arrive();
  // forward phases 1 .. np - 1, then backward phases np - 1 .. 0
  const int np = B.nphases;
#pragma unroll 1
  for (int q = 1; q < 2 * np && !c.dead; ++q) {
    const bool fwd = q < np;
    const int32_t *ptr = fwd ? B.fwd_ptr + q : B.bwd_ptr + (2 * np - 1 - q);
    const int e0 = __ldg(ptr), e1 = __ldg(ptr + 1);
    if (!fwd && e0 == e1) continue;
    stage(c, e0, e1, [&](int e, auto first) {
      constexpr bool F = decltype(first)::value;
      const int4 E = __ldg(B.ent + e);
      if (F && !TRIO) c.wait();
      if constexpr (TRIO) sweep_trio<TF, MODE, F>(c, E, fwd, second);
      else sweep_unit<TF, MODE>(c, E, fwd, second);
    });
  }
}

// The start of a launch: the scalars into shared memory, and the warp's place
// among the units.  COPY: the descriptor too.  A solve reads it where it is, in
// the launch's parameters (FP64, 44,431 rows: 307 us against 316 from shared
// memory; 116 phases 2306 against 2467); an application alone would wait for
// its fields one after the other (45 us against 42).
template <bool TRIO, bool COPY>
__device__ __forceinline__ ResCtx resident_enter(const Resident &R, ResShared &sm) {
  const Batch &B = R.B;
  const int wp = threadIdx.x >> 5, nt = blockDim.x;
  ResCtx c{R, sm, COPY ? sm.sys : R.sys, (int)(threadIdx.x & 31), wp, nt / 32, 0, 0, 0, 0, 0, 0u, false,
           (int)threadIdx.x == nt - 32};
  if (TRIO) {
    c.r = wp % 3;
    c.trio = wp / 3;
    c.g = c.trio < kTrios ? c.trio * gridDim.x + blockIdx.x : 0x40000000;  // the last warp takes no units
    c.W = kTrios * gridDim.x;
  } else {
    c.g = c.warp_id();  // consecutive units go to different SMs
    c.W = c.warps();
  }
  const int phase0 = __ldg(B.fwd_ptr + 1);
  if (threadIdx.x == 0) sm.phase0 = phase0;
  if (c.lane == 0 && c.g < phase0) sm.first[wp] = __ldg(B.ent + c.g);
  if (COPY) {
    const int2 *src = reinterpret_cast<const int2 *>(&R.sys);
    int2 *dst = reinterpret_cast<int2 *>(&sm.sys);
    static_assert(sizeof(Sys) % sizeof(int2) == 0, "the descriptor is copied in 8-byte pieces");
    for (int q = threadIdx.x; q < (int)(sizeof(Sys) / sizeof(int2)); q += nt) dst[q] = src[q];
  }
  if (threadIdx.x == 0) {
    Scal z{};
    z.tol = R.sys.rtol;
    z.maxit = R.sys.maxit;
    // an earlier factorisation's failure makes the solve fail
    const int32_t ferr = R.work == kResSolve ? R.sys.st->ferror : 0;
    z.status = ferr != 0 ? ferr : kRunning;
    sm.sc = z;
  }
  __syncthreads();
  return c;
}

// The end: the last CTA to leave writes the outcome and clears the device
// words.  After an expired wait no stage has written x: it zeroes it, as the
// finish stage does for every other failure.
__device__ __forceinline__ void resident_leave(ResCtx &c) {
  const Resident &R = c.R;
  ResShared &sm = c.sm;
  const bool factor = R.work & kResFactor, solve = R.work & kResSolve;
  __syncthreads();
  if (threadIdx.x == 0) {
    __threadfence();
    sm.last = atomicAdd(&R.ctl->exits, 1u) == gridDim.x - 1;
    __threadfence();
  }
  __syncthreads();
  if (!sm.last) return;
  const bool aborted = ld_acquire(&R.ctl->abort) != 0u;
  const Sys &S = R.sys;
  if (aborted && solve)
    for (int64_t e = threadIdx.x; e < 3ll * S.n; e += blockDim.x) S.x_out[e] = 0.0;
  if (threadIdx.x == 0) {
    const int32_t ferr = __ldcg(R.err);
    DevState *st = S.st;
    Result r{};
    r.status = aborted ? (int32_t)OPM_ERR_TIMEOUT : solve ? sm.sc.status : ferr;  // 0 after an application
    r.iters = sm.sc.iters;
    r.relres = aborted ? nan("") : sm.sc.relres;
    r.err_row = ferr != 0 ? 0x7fffffff - __ldcg(R.err + 1) : 0x7fffffff;
    if (factor) {
      st->ferror = aborted ? (int32_t)OPM_ERR_TIMEOUT : ferr;
      st->err_row = r.err_row;
    }
    if (factor || solve) {
      st->error = aborted ? (int32_t)OPM_ERR_TIMEOUT : 0;
      st->status = r.status;
    }
    *R.res = r;
    R.err[0] = 0;
    R.err[1] = 0;
    R.ctl->arrive = 0;
    R.ctl->exits = 0;
    R.ctl->abort = 0;
  }
}

// A standalone application z = inv(LU) r (opm_ilu_apply).
template <typename TF, bool TRIO, int NT>
__global__ void __launch_bounds__(NT, 1) k_resident_apply(const __grid_constant__ Resident R) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  ResCtx c = resident_enter<TRIO, true>(R, *reinterpret_cast<ResShared *>(smem_raw));
  resident_apply<TF, kModePlain, TRIO>(c, false);
  resident_leave(c);
}

// Factorisation and solve.  TF: factor precision; TRIO: three warps per slice
// (with one warp more for the barrier) or one; NT: threads per CTA, one CTA
// per SM.
template <typename TF, bool TRIO, int NT>
__global__ void __launch_bounds__(NT, 1) k_resident(const __grid_constant__ Resident R) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  ResShared &sm = *reinterpret_cast<ResShared *>(smem_raw);
  const Batch &B = R.B;
  static_assert(!TRIO || NT == kTrioThreads, "the trios and one warp more");
  ResCtx c = resident_enter<TRIO, false>(R, sm);
  const bool factor = R.work & kResFactor, solve = R.work & kResSolve;
  const bool wells = R.sys.nwells > 0, reuse = R.sys.uz != nullptr;
  auto vector_stage = [&](bool setup) {
#pragma unroll 1
    for (int u = c.g; u < R.nupd; u += c.W) {
      if constexpr (TRIO) vector_trio(c, u, setup);
      else vector_unit(c, u, setup);
    }
  };

  // the setup needs only b: it runs ahead of the factorisation's phases
  if (solve) vector_stage(true);
  if (factor) {
    resident_factor<TF, TRIO>(c);
  } else {
    c.arrive();
    c.wait();
  }

  int step = kStepSetup;
#pragma unroll 1
  while (solve && !c.dead) {
    // after a wait
    if (step == kStepUpdate) {
      vector_stage(false);
      c.arrive();
    } else if (step != kStepSetup) {
      const bool second = step == kStepS;
      if (step != kStepFinish) {
        resident_apply<TF, kModeP, TRIO>(c, second);
      } else {
        c.arrive();
      }
      if (wells && !c.dead) wells_stage(c, step);
      stage(c, 0, B.nall, [&](int u, auto first) {
        constexpr bool F = decltype(first)::value;
        const int sl = __ldg(R.prod + u);
        if (F && !TRIO) c.wait();
        if constexpr (TRIO) product_trio<F>(c, sl, step, reuse);
        else product_unit(c, sl, step, reuse);
      });
    }
    if (step != kStepSetup) c.wait();
    if (c.dead) break;
    finish_dot(c, step);
    if (step == kStepFinish) break;
    step = !c.runs() ? kStepFinish : step == kStepP ? kStepS : step == kStepS ? kStepUpdate : kStepP;
  }

  resident_leave(c);
}

}  // namespace opm
