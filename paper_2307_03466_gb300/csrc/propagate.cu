// Bound propagation on the GPU (Section 2.3's activity-based tightening), in rounds:
// every active row computes, from the domains at the start of the round, the
// tightened bounds it implies for its columns (the arithmetic of one visit of the
// sequential propagation, in CSR order, one thread per row); then every column takes
// the largest proposed lower and the smallest proposed upper bound over its rows
// (read through the stored transpose; no atomics on the domains).  A row whose
// activity bounds already exclude [lo, hi], or that would empty a domain, is ignored
// from then on; a column whose merged proposals cross keeps its domain and counts a
// conflict.  The rows of the columns that changed are the next round's active rows.
// On integer data without ignored rows or conflicts this is the fixpoint of the
// sequential queue (the greatest fixpoint of a monotone tightening), bit for bit.
#include <cuda_runtime.h>

#include <cmath>
#include <cstdint>

#include "internal.h"

namespace scylla {

namespace {

constexpr int kPropThreads = 256;

int prop_grid(long long items) {
  long long g = (items + kPropThreads - 1) / kPropThreads;
  const long long cap = 8LL * device_sm_count();
  if (g > cap) g = cap;
  if (g < 1) g = 1;
  return int(g);
}

// position in A of every entry of the transpose: entry q of column j lies in row
// i = rows[q], whose column indices are ascending, so a binary search finds j
__global__ void k_prop_perm(int n, const int* __restrict__ t_rowptr, const int* __restrict__ t_rows,
                            const int* __restrict__ a_rowptr, const int* __restrict__ a_cols, int* __restrict__ perm) {
  for (int j = blockIdx.x * blockDim.x + threadIdx.x; j < n; j += gridDim.x * blockDim.x) {
    for (int q = t_rowptr[j]; q < t_rowptr[j + 1]; ++q) {
      const int i = t_rows[q];
      int lo = a_rowptr[i], hi = a_rowptr[i + 1] - 1;
      while (lo < hi) {
        const int mid = (lo + hi) >> 1;
        if (a_cols[mid] < j) lo = mid + 1;
        else hi = mid;
      }
      perm[q] = lo;
    }
  }
}

// The start of a call: the caller's domains side by side, and whether an integer column's
// is fractional (then no row is screened: the rounding alone changes such a bound); no
// column has a proposal, no row is ignored, every row is active.
__global__ void k_prop_in(PropDev P, unsigned char* __restrict__ active) {
  bool frac = false;
  const int t0 = blockIdx.x * blockDim.x + threadIdx.x, stride = gridDim.x * blockDim.x;
  for (int j = t0; j < P.n; j += stride) {
    const double l = P.dl[j], u = P.du[j];
    P.dom[j] = make_double2(l, u);
    P.flag[j] = 0;
    frac = frac || (P.is_int[j] && (l != floor(l) || u != floor(u)));
  }
  for (int i = t0; i < P.m; i += stride) {
    P.state[i] = 0;
    active[i] = 1;
  }
  if (frac) P.ctl->fractional = 1;
}
__global__ void k_prop_out(PropDev P) {
  for (int j = blockIdx.x * blockDim.x + threadIdx.x; j < P.n; j += gridDim.x * blockDim.x) {
    const double2 d = P.dom[j];
    P.dl[j] = d.x;
    P.du[j] = d.y;
  }
}

__device__ __forceinline__ bool prop_inf(double v) {
  return (__double_as_longlong(v) & 0x7fffffffffffffffLL) == 0x7ff0000000000000LL;
}

// Whether a round has anything to do: the first of a call, or its predecessor marked a row.
__device__ __forceinline__ bool prop_on(const PropCtl* c, int slot) { return slot == 0 || c->round[slot - 1].marked != 0u; }

// One round, first half: the activity bounds of every active row (one thread per row, in
// CSR order).  A row whose sides' slacks both exceed its largest single-column span
// |a_j| (u_j - l_j) by a relative margin of 1e-6 cannot change a domain: its visit ends
// here, without the divisions of the candidates (95% of the visits of the packing/covering
// workload; the whole propagation was bound by them).  The others go on a list for the
// second half.  state[i]: 0 no proposals this round, 1 proposals in plb/pub at the row's
// CSR positions (-inf / +inf where a bound is not tightened), 2 ignored for good.
__global__ void __launch_bounds__(kPropThreads)
    k_prop_rows(PropDev P, int slot, const unsigned char* __restrict__ active, unsigned char* __restrict__ active_next) {
  PropCtl* ctl = P.ctl;
  if (!prop_on(ctl, slot)) return;
  if (blockIdx.x == 0 && threadIdx.x == 0) ++ctl->rounds;
  const double inf = __longlong_as_double(0x7ff0000000000000LL);
  const bool screen = ctl->fractional == 0;
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < P.m; i += gridDim.x * blockDim.x) {
    active_next[i] = 0;
    const unsigned char st = P.state[i];
    if (st == 2) continue;
    if (st != 0) P.state[i] = 0;
    if (!active[i]) continue;
    const double lo_i = P.lo[i], hi_i = P.hi[i];
    if (lo_i == -inf && hi_i == inf) continue;
    const int p0 = P.rowptr[i], p1 = P.rowptr[i + 1];
    double minf = 0.0, maxf = 0.0, span = 0.0;
    int nmin = 0, nmax = 0;
    bool zero = false;
    for (int p = p0; p < p1; ++p) {
      const double a = P.vals[p];
      const double2 d = P.dom[P.cols[p]];
      const bool pos = __double_as_longlong(a) > 0;
      const double bmin = pos ? d.x : d.y, bmax = pos ? d.y : d.x;
      if (prop_inf(bmin)) ++nmin;
      else minf = __dadd_rn(minf, __dmul_rn(a, bmin));
      if (prop_inf(bmax)) ++nmax;
      else maxf = __dadd_rn(maxf, __dmul_rn(a, bmax));
      span = fmax(span, fabs(a) * (d.y - d.x));
      zero = zero || a == 0.0;
    }
    if ((nmin == 0 && hi_i != inf && minf > __dadd_rn(hi_i, 1e-9)) ||
        (nmax == 0 && lo_i != -inf && maxf < __dsub_rn(lo_i, 1e-9))) {
      P.state[i] = 2;
      continue;
    }
    constexpr double kMarg = 1e-6;
    const bool hi_side = hi_i != inf && (nmin == 1 || (nmin == 0 && !((hi_i - minf) > span * (1.0 + kMarg) +
                                                       kMarg * (1.0 + fabs(hi_i) + fabs(minf)))));
    const bool lo_side = lo_i != -inf && (nmax == 1 || (nmax == 0 && !((maxf - lo_i) > span * (1.0 + kMarg) +
                                                        kMarg * (1.0 + fabs(lo_i) + fabs(maxf)))));
    if (screen && !zero && !hi_side && !lo_side) continue;
    P.act[i] = make_double2(minf, maxf);
    P.ninf[i] = make_int2(nmin, nmax);
    P.list[atomicAdd(&ctl->round[slot].listed, 1u)] = i;
  }
}

// Second half: the candidates of the listed rows, a warp per row, a lane per entry.  The
// columns that get a proposal are flagged for the merge.
__global__ void __launch_bounds__(kPropThreads) k_prop_visit(PropDev P, int slot) {
  PropCtl* ctl = P.ctl;
  if (!prop_on(ctl, slot)) return;
  const double inf = __longlong_as_double(0x7ff0000000000000LL);
  const int lane = threadIdx.x & 31, count = int(ctl->round[slot].listed);
  for (int v = (blockIdx.x * blockDim.x + threadIdx.x) >> 5; v < count; v += (gridDim.x * blockDim.x) >> 5) {
    const int i = P.list[v];
    const double lo_i = P.lo[i], hi_i = P.hi[i];
    const double2 act = P.act[i];
    const int2 ni = P.ninf[i];
    const double minf = act.x, maxf = act.y;
    const int nmin = ni.x, nmax = ni.y, p1 = P.rowptr[i + 1];
    bool ignore = false;
    for (int p = P.rowptr[i] + lane; p < p1; p += 32) {
      const int j = P.cols[p];
      const double a = P.vals[p];
      const double2 d = P.dom[j];
      const double old_lb = d.x, old_ub = d.y;
      const double bmin = a > 0.0 ? old_lb : old_ub;
      const double bmax = a > 0.0 ? old_ub : old_lb;
      double rmin, rmax;
      if (isinf(bmin)) rmin = nmin == 1 ? minf : -inf;
      else rmin = nmin == 0 ? __dsub_rn(minf, __dmul_rn(a, bmin)) : -inf;
      if (isinf(bmax)) rmax = nmax == 1 ? maxf : inf;
      else rmax = nmax == 0 ? __dsub_rn(maxf, __dmul_rn(a, bmax)) : inf;
      double cand_lb = -inf, cand_ub = inf;
      if (hi_i != inf && rmin != -inf) {
        const double t = __ddiv_rn(__dsub_rn(hi_i, rmin), a);
        if (a > 0.0) cand_ub = t;
        else cand_lb = t;
      }
      if (lo_i != -inf && rmax != inf) {
        const double t = __ddiv_rn(__dsub_rn(lo_i, rmax), a);
        if (a > 0.0) cand_lb = t;
        else cand_ub = t;
      }
      double new_lb = old_lb, new_ub = old_ub;
      if (P.is_int[j]) {
        if (cand_ub != inf) {
          const double v2 = floor(__dadd_rn(cand_ub, 1e-6));
          if (v2 < old_ub) new_ub = v2;
        }
        if (cand_lb != -inf) {
          const double v2 = ceil(__dsub_rn(cand_lb, 1e-6));
          if (v2 > old_lb) new_lb = v2;
        }
      } else {
        if (cand_ub != inf &&
            (old_ub == inf || cand_ub < __dsub_rn(old_ub, __dmul_rn(1e-3, fmax(1.0, fabs(old_ub))))))
          new_ub = cand_ub;
        if (cand_lb != -inf &&
            (old_lb == -inf || cand_lb > __dadd_rn(old_lb, __dmul_rn(1e-3, fmax(1.0, fabs(old_lb))))))
          new_lb = cand_lb;
      }
      const bool moved = new_lb != old_lb || new_ub != old_ub;
      if (moved && new_lb > __dadd_rn(new_ub, 1e-9)) ignore = true;
      P.plb[p] = new_lb != old_lb ? new_lb : -inf;
      P.pub[p] = new_ub != old_ub ? new_ub : inf;
      if (moved) P.flag[j] = 1;
    }
    ignore = __any_sync(0xffffffffu, ignore);
    if (lane == 0) P.state[i] = ignore ? 2 : 1;
  }
}

// The merge of one round: each flagged column over its rows' proposals; changed columns
// mark their rows active for the next round.
__global__ void __launch_bounds__(kPropThreads)
    k_prop_cols(PropDev P, int slot, unsigned char* __restrict__ active_next) {
  PropCtl* ctl = P.ctl;
  if (!prop_on(ctl, slot)) return;
  for (int j = blockIdx.x * blockDim.x + threadIdx.x; j < P.n; j += gridDim.x * blockDim.x) {
    if (!P.flag[j]) continue;
    P.flag[j] = 0;
    const int q0 = P.t_rowptr[j], q1 = P.t_rowptr[j + 1];
    const double2 d = P.dom[j];
    double nl = d.x, nu = d.y;
    for (int q = q0; q < q1; ++q) {
      const int i = P.t_rows[q];
      if (i >= P.m || P.state[i] != 1) continue;
      const int p = P.perm[q];
      nl = fmax(nl, P.plb[p]);
      nu = fmin(nu, P.pub[p]);
    }
    if (nl == d.x && nu == d.y) continue;
    if (nl > __dadd_rn(nu, 1e-9)) {
      atomicAdd(&ctl->conflicts, 1ULL);
      continue;
    }
    P.dom[j] = make_double2(nl, nu);
    bool marked = false;
    for (int q = q0; q < q1; ++q) {
      const int i = P.t_rows[q];
      if (i >= P.m || P.state[i] == 2) continue;
      active_next[i] = 1;
      marked = true;
    }
    if (marked) ctl->round[slot].marked = 1u;
  }
}

}  // namespace

cudaError_t propagate_perm(int n, const int* t_rowptr, const int* t_rows, const int* a_rowptr, const int* a_cols,
                           int* perm, cudaStream_t st) {
  if (n > 0) k_prop_perm<<<prop_grid(n), kPropThreads, 0, st>>>(n, t_rowptr, t_rows, a_rowptr, a_cols, perm);
  return cudaGetLastError();
}

cudaError_t propagate_start(const PropDev& P, unsigned char* active, cudaStream_t st) {
  const cudaError_t e = cudaMemsetAsync(P.ctl, 0, sizeof(PropCtl), st);
  if (e != cudaSuccess) return e;
  k_prop_in<<<prop_grid(P.m > P.n ? P.m : P.n), kPropThreads, 0, st>>>(P, active);
  return cudaGetLastError();
}

cudaError_t propagate_round(const PropDev& P, int slot, const unsigned char* active, unsigned char* active_next,
                            cudaStream_t st) {
  if (P.m > 0) {
    k_prop_rows<<<prop_grid(P.m), kPropThreads, 0, st>>>(P, slot, active, active_next);
    k_prop_visit<<<prop_grid(32LL * P.m), kPropThreads, 0, st>>>(P, slot);
  }
  if (P.n > 0) k_prop_cols<<<prop_grid(P.n), kPropThreads, 0, st>>>(P, slot, active_next);
  return cudaGetLastError();
}

cudaError_t propagate_end(const PropDev& P, cudaStream_t st) {
  if (P.n > 0) k_prop_out<<<prop_grid(P.n), kPropThreads, 0, st>>>(P);
  return cudaGetLastError();
}

}  // namespace scylla
