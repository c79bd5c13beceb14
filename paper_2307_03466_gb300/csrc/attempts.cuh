// The resident form of the per-attempt kernels: all the attempts between two checks in
// one launch, for LPs whose matrix fits in the shared memory of the blocks.
//
// As separate launches an attempt of such an LP is mostly latency: two launches, each
// with its ramp, its tail and the last block's reduction and decision, and in each a
// chain of dependent loads (tile bounds, row ranges, indices, gathered entries).  Here
// the blocks stay resident.  Every warp keeps its tiles' indices and values of A and of
// the transpose in shared memory and the vectors of the rows and columns that its lanes
// own (x, y, A x, A^T y, the averages, costs and bounds) in registers, so an attempt
// loads nothing but the gathered entries.  A barrier separates the phases.  After the
// dual's barrier the last three warps of every block reduce the partial sums in one fixed order
// and a thread takes the step-size decision on the block's own copy of the control
// block, while the other warps already form the row sums A^T y' that the next primal
// step needs when the attempt is accepted (a rejected attempt keeps the old ones).
//
// Two scopes, by size (resident_plan):
//   cluster  1 to 16 blocks; the gathered vectors and the partial sums are replicated in
//            every block's shared memory through distributed shared memory, and the
//            barrier is the hardware cluster barrier;
//   grid     one block per SM (a cooperative launch); the gathered vectors are in global
//            memory (L2), and the barrier is a counter there, every wait on it bounded.
//
// The results are those of the launched form bit for bit.  The launched form deals tile
// t to warp (t div G) mod 8 of block t mod G (G its grid) and sums the block's eight
// warps, then the blocks, in a fixed order.  Here one warp stands for warp s div G of
// block s mod G and takes that warp's tiles s, s + 8 G, ... in the same order; the eight
// of a block are summed in order, and the block sums are reduced in the launched form's
// order.
#pragma once

constexpr int kResTile = kTileNnz;  // entries of a tile's slot in shared memory
constexpr int kResMaxVb = 8;        // virtual blocks per block in the grid scope

// most threads of a block: as many warps per SM as the launched form keeps resident
// (FP32: four blocks of 256 threads at 64 registers; FP64: two at 128)
template <typename T>
struct ResidentThreads {
  static constexpr int value = sizeof(T) == 4 ? 1024 : 512;
};

// most tiles of a side in the cluster scope: FP32 what 8 blocks of 32 warps hold beside three
// control warps each; FP64 where the grid's SMs are worth more than its barrier (resident_plan)
template <typename T>
struct ResidentTiles {
  static constexpr int value = sizeof(T) == 4 ? 8 * (ResidentThreads<T>::value / 32 - 3) : 64;
};

struct ResidentArgs {
  int slots_t, slots_a;  // tile slots per block in shared memory, of the transpose and of A
};

// Weak load through L1 of a vector that other blocks wrote earlier in this launch: the
// barrier's acquire drops this SM's L1 lines.  Not ld.global.nc, which a compiler may
// choose for a const restrict pointer.
__device__ __forceinline__ float ld_ca(const float* p) {
  float v;
  asm volatile("ld.global.ca.f32 %0, [%1];" : "=f"(v) : "l"(p) : "memory");
  return v;
}
__device__ __forceinline__ double ld_ca(const double* p) {
  double v;
  asm volatile("ld.global.ca.f64 %0, [%1];" : "=d"(v) : "l"(p) : "memory");
  return v;
}
// store to the same shared-memory place of block `rank` of the cluster
__device__ __forceinline__ void st_cluster(float* p, unsigned rank, float v) {
  unsigned a;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(a) : "r"(smem_addr(p)), "r"(rank));
  asm volatile("st.shared::cluster.f32 [%0], %1;" ::"r"(a), "f"(v) : "memory");
}
__device__ __forceinline__ void st_cluster(double* p, unsigned rank, double v) {
  unsigned a;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(a) : "r"(smem_addr(p)), "r"(rank));
  asm volatile("st.shared::cluster.f64 [%0], %1;" ::"r"(a), "d"(v) : "memory");
}

// Barrier over the blocks of the launch.  The grid's is a monotonic arrival counter
// (zeroed before the launch) that one thread per block adds to and polls; false when the
// wait ran out here or in another block, and then all blocks leave.
struct ResidentBar {
  unsigned int count;
  int err;
};
template <int SCOPE>
__device__ __forceinline__ bool resident_barrier(ResidentBar* b, unsigned int& target, unsigned long long limit_ns) {
  if constexpr (SCOPE == kScopeCluster) {
    if (gridDim.x == 1) {
      __syncthreads();
    } else {
      asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
      asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
    }
    return true;
  } else {
    __shared__ int ok;
    target += gridDim.x;
    __syncthreads();
    if (threadIdx.x == 0) {
      int good = 1;
      asm volatile("red.release.gpu.global.add.u32 [%0], 1;" ::"l"(&b->count) : "memory");
      unsigned int v;
      const unsigned long long t0 = clock_ns();
      int spins = 0;
      while (true) {
        asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(&b->count) : "memory");
        if (int(v - target) >= 0) break;
        int e = 0;
        if ((++spins & 15) == 0)
          asm volatile("ld.relaxed.gpu.global.s32 %0, [%1];" : "=r"(e) : "l"(&b->err) : "memory");
        if (e != 0 || clock_ns() - t0 > limit_ns) {
          atomicExch(&b->err, 1);
          good = 0;
          break;
        }
      }
      ok = good;
    }
    __syncthreads();
    return ok != 0;
  }
}

// One side (A or its transpose) of the LP.
template <typename T>
struct ResSide {
  const int2* tiles;
  const int* rowptr;
  const int* cols;
  const T* vals;
  int ntiles;
  int G;        // the launched form's grid
  bool spread;  // at most G tiles: tile s is the only one of its virtual block
};

// What a warp keeps of one of its tiles.
struct ResTile {
  int t;          // the tile, -1 for none
  int row;        // the row this lane owns, -1 for none
  int q0, q1;     // that lane's share of the tile's entries: q0, q0 + L, ... < q1
  int len, lsh;   // entries of the tile (kResTile + 1: a long row, read from global memory); log2 L
  int slot;       // its slot in shared memory
};

// First tile of this warp (its virtual warp's s), -1 for none.
template <typename T>
__device__ __forceinline__ int res_first(const ResSide<T>& S, int w, int nw) {
  const int c = blockIdx.x, P = gridDim.x;
  if (S.spread) {
    const int s = c + P * w;
    return s < S.ntiles ? s : -1;
  }
  const int nb = nw >> 3, b = c + P * (w % nb), s = b + (w / nb) * S.G;
  return b < S.G && s < S.ntiles ? s : -1;
}

// the warp's tile number i (s, s + 8 G, ...): its row map, and its entries into its slot
template <typename T, int TPW>
__device__ __forceinline__ void res_load(const ResSide<T>& S, int i, ResTile& R, int* idx, T* val) {
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, nw = blockDim.x >> 5;
  R.t = R.row = -1;
  R.q0 = R.q1 = R.len = R.lsh = R.slot = 0;
  const int s = res_first(S, w, nw);
  const int t = s < 0 ? -1 : s + i * 8 * S.G;
  if (t < 0 || t >= S.ntiles) return;
  R.t = t;
  // slots: the warps' first tiles, then the second ones in warp order
  R.slot = w;
  if (TPW > 1 && i > 0) {
    int k = nw;
    for (int v = 0; v < w; ++v) {
      const int sv = res_first(S, v, nw);
      k += sv >= 0 && sv + 8 * S.G < S.ntiles ? 1 : 0;
    }
    R.slot = k;
  }
  const int2 ta = __ldg(S.tiles + t), tb = __ldg(S.tiles + t + 1);
  const int nr = tb.x - ta.x, n = tb.y - ta.y;
  R.lsh = row_lanes_log2(nr);
  const int rl = lane >> R.lsh, sub = lane & ((1 << R.lsh) - 1);
  if (rl < nr) {
    R.q0 = __ldg(S.rowptr + ta.x + rl) - ta.y + sub;
    R.q1 = __ldg(S.rowptr + ta.x + rl + 1) - ta.y;
    if (sub == 0) R.row = ta.x + rl;
  }
  if (n > kResTile) {
    R.len = kResTile + 1;
    return;
  }
  R.len = n;
  int* ip = idx + R.slot * kResTile;
  T* vp = val + R.slot * kResTile;
  for (int q = lane; q < n; q += 32) {
    ip[q] = __ldg(S.cols + ta.y + q);
    vp[q] = __ldg(S.vals + ta.y + q);
  }
}

// the row sums of a tile whose products are in sm
template <typename T>
__device__ __forceinline__ T res_sums(const ResTile& R, const T* sm) {
  __syncwarp();
  T s = T(0);
  const int L = 1 << R.lsh;
  int q = R.q0;
  for (; q + 3 * L < R.q1; q += 4 * L) {
    const T a = sm[skew(q)], b = sm[skew(q + L)], c = sm[skew(q + 2 * L)], e = sm[skew(q + 3 * L)];
    s += a;
    s += b;
    s += c;
    s += e;
  }
  for (; q < R.q1; q += L) s += sm[skew(q)];
  for (int o = L >> 1; o > 0; o >>= 1) s += __shfl_down_sync(0xffffffffu, s, o);
  __syncwarp();
  return s;
}

// Row sum of the lane's row (on the lane that owns it) with the vector x: products
// rounded, then summed as spmv_tiles does.  VS: x is in shared memory.
template <typename T, bool VS>
__device__ __forceinline__ T res_rowsum(const ResSide<T>& S, const ResTile& R, const int* idx, const T* val,
                                        const T* x, T* sm) {
  const int lane = threadIdx.x & 31;
  if (R.len > kResTile) {
    const int2 ta = __ldg(S.tiles + R.t), tb = __ldg(S.tiles + R.t + 1);
    T s[1];
    auto gat = [&](int i, T(&g)[1]) { g[0] = VS ? x[i] : ld_ca(x + i); };
    long_row_sum<1, false>(ta.y, tb.y, S.cols, S.vals, gat, s);
    return s[0];
  }
  const int* ip = idx + R.slot * kResTile + lane;
  const T* vp = val + R.slot * kResTile + lane;
  int c[kResTile / 32];
  T g[kResTile / 32];
#pragma unroll
  for (int j = 0; j < kResTile / 32; ++j) c[j] = lane + 32 * j < R.len ? ip[32 * j] : -1;
#pragma unroll
  for (int j = 0; j < kResTile / 32; ++j) {
    g[j] = T(0);
    if (c[j] >= 0) g[j] = VS ? x[c[j]] : ld_ca(x + c[j]);
  }
#pragma unroll
  for (int j = 0; j < kResTile / 32; ++j)
    if (c[j] >= 0) sm[lane + 33 * j] = vp[32 * j] * g[j];
  return res_sums(R, sm);
}

// Sum of count partials (stride apart) by one warp in the order of reduce_step: thread i
// of 224 takes i, i + 224, ..., the 224 are summed by 32 lanes in turns, then the lanes.
template <bool kShared, typename A>
__device__ __forceinline__ A res_reduce(const A* p, int count, int stride) {
  constexpr int nt = kThreads - 32;
  const int lane = threadIdx.x & 31;
  A v = A(0);
  if (count <= 3 * nt) {
    A a[nt / 32][3];
#pragma unroll
    for (int j = 0; j < nt / 32; ++j)
#pragma unroll
      for (int r = 0; r < 3; ++r) {
        const int b = lane + 32 * j + nt * r;
        a[j][r] = b < count ? (kShared ? p[stride * b] : ldcg_t(p + stride * b)) : A(0);
      }
#pragma unroll
    for (int j = 0; j < nt / 32; ++j) {
      // count <= 224 in the cluster scope's common case: one term
      A t = a[j][0];
      if (count > nt) t += a[j][1];
      if (count > 2 * nt) t += a[j][2];
      v += t;
    }
  } else {
    for (int j = 0; j < nt / 32; ++j) {
      A t = A(0);
      for (int b = lane + 32 * j; b < count; b += nt) t += kShared ? p[stride * b] : ldcg_t(p + stride * b);
      v += t;
    }
  }
  return warp_sum(v);
}

// The attempts up to the next check.  TPW: most tiles of a side per warp.
template <typename T, int SCOPE, int TPW>
__global__ void __launch_bounds__(ResidentThreads<T>::value, 1)
    k_attempts(DevLP<T> d, ResidentArgs ra, ResidentBar* bar, unsigned long long limit_ns) {
  constexpr bool VS = SCOPE == kScopeCluster;
  extern __shared__ __align__(16) char rsm[];
  __shared__ Control sc;
  __shared__ StepPre spre;
  __shared__ T red[kNP + kND];
  __shared__ T shw[2][kResMaxVb][8];
  constexpr int kP = VS ? ResidentTiles<T>::value : 1;
  __shared__ T bpart[4 * kP];  // cluster scope: primal sums (two buffers), dual sums (pairs)
  if (d.ctl->done || d.ctl->k >= d.ctl->iter_limit) return;
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, nw = blockDim.x >> 5, P = gridDim.x;
  const ResSide<T> St{d.t_tiles, d.t_rowptr, d.t_cols, d.t_vals, d.t_ntiles, d.grid_p, d.t_ntiles <= d.grid_p};
  const ResSide<T> Sa{d.a_tiles, d.a_rowptr, d.a_cols, d.a_vals, d.a_ntiles, d.grid_d, d.a_ntiles <= d.grid_d};
  // shared memory: tile values, product buffers, the gathered vectors, tile indices
  T* val_t = reinterpret_cast<T*>(rsm);
  T* val_a = val_t + ra.slots_t * kResTile;
  T* sm = val_a + ra.slots_a * kResTile + w * kSmemPerWarp;
  T* xs = val_a + ra.slots_a * kResTile + nw * kSmemPerWarp;
  T* ys = xs + (VS ? d.n : 0);
  int* idx_t = reinterpret_cast<int*>(ys + (VS ? d.m : 0));
  int* idx_a = idx_t + ra.slots_t * kResTile;
  static_assert(sizeof(Control) % 4 == 0, "word copy");
  for (int i = threadIdx.x; i < int(sizeof(Control) / 4); i += blockDim.x)
    reinterpret_cast<int*>(&sc)[i] = reinterpret_cast<const int*>(d.ctl)[i];
  if (VS)
    for (int i = threadIdx.x; i < 4 * kP; i += blockDim.x) bpart[i] = T(0);
  ResTile Rt[TPW], Ra[TPW];
#pragma unroll
  for (int i = 0; i < TPW; ++i) {
    res_load<T, TPW>(St, i, Rt[i], idx_t, val_t);
    res_load<T, TPW>(Sa, i, Ra[i], idx_a, val_a);
  }
  __syncthreads();
  // the lanes' own entries
  T xc[TPW], xa[TPW], xn[TPW], aty[TPW], cj[TPW], lj[TPW], uj[TPW], sp[TPW];
  T yc[TPW], ya[TPW], yn[TPW], ax[TPW], axn[TPW], lo[TPW], hi[TPW];
#pragma unroll
  for (int i = 0; i < TPW; ++i) {
    xc[i] = xa[i] = xn[i] = aty[i] = cj[i] = lj[i] = uj[i] = sp[i] = T(0);
    yc[i] = ya[i] = yn[i] = ax[i] = axn[i] = lo[i] = hi[i] = T(0);
    const int j = Rt[i].row, r = Ra[i].row;
    if (j >= 0) {
      xc[i] = d.X[sc.ix_cur][j];
      xa[i] = d.X[sc.ix_avg][j];
      aty[i] = d.ATY[sc.ia_cur][j];
      cj[i] = d.c[j];
      lj[i] = d.l[j];
      uj[i] = d.u[j];
    }
    if (r >= 0) {
      yc[i] = d.Y[sc.ix_cur][r];
      ya[i] = d.Y[sc.ix_avg][r];
      ax[i] = d.AX[sc.ix_cur][r];
      lo[i] = d.lo[r];
      hi[i] = d.hi[r];
    }
  }
  unsigned int target = 0;
  bool ok = true;
  // every block runs before another writes its shared memory
  if (VS) resident_barrier<SCOPE>(bar, target, limit_ns);
  if (!sc.aty_valid) {  // after a check A^T y is always at hand; otherwise form it
    if (VS) {
      const T* y = d.Y[sc.ix_cur];
      for (int i = threadIdx.x; i < d.m; i += blockDim.x) ys[i] = y[i];
      __syncthreads();
    }
#pragma unroll
    for (int i = 0; i < TPW; ++i)
      if (Rt[i].t >= 0) sp[i] = res_rowsum<T, VS>(St, Rt[i], idx_t, val_t, VS ? ys : d.Y[sc.ix_cur], sm);
    if (VS) __syncthreads();
  }
  // a block sum to every block: the tile's own (spread), or the eight warps' of a
  // virtual block in order
  auto publish = [&](const ResSide<T>& S, const ResTile& R0, T* part, auto& a, auto nv) {
    constexpr int NV = decltype(nv)::value;
    const int nb = nw >> 3;
#pragma unroll
    for (int k = 0; k < NV; ++k) {
      a[k] = warp_sum(a[k]);
      if (VS) {
        if (R0.t >= 0 && lane < P) {
          if (P == 1) part[NV * R0.t + k] = a[k];
          else st_cluster(part + NV * R0.t + k, unsigned(lane), a[k]);
        }
      } else if (S.spread) {
        if (R0.t >= 0 && lane == 0) part[NV * R0.t + k] = a[k];
      } else if (lane == 0) {
        shw[k][w % nb][w / nb] = a[k];
      }
    }
    if (VS || S.spread) return;
    __syncthreads();
    if (int(threadIdx.x) < NV * nb) {
      const int k = threadIdx.x % NV, v = threadIdx.x / NV, b = int(blockIdx.x) + P * v;
      if (b < S.G) {
        T t = T(0);
#pragma unroll
        for (int q = 0; q < 8; ++q) t += shw[k][v][q];
        part[NV * b + k] = t;
      }
    }
  };
  for (int a = 0; a < d.n_check; ++a) {
    if (sc.done || sc.k >= sc.iter_limit) break;
    const SlotView<T> v = make_view<T>(&sc);
    const bool more = a + 1 < d.n_check && sc.k + 1 < sc.iter_limit;
    T* part_p = VS ? bpart + (a & 1) * kP : acc_part<T>(d.part_p) + (a & 1) * d.grid_p;
    T* part_d = VS ? bpart + 2 * kP : acc_part<T>(d.part_d);
    // the control warps are the last three: the deal of the tiles leaves them without
    // one before any other
    const int cw = w - (nw - 3);
    if (cw == 0 && lane == 0) spre = step_pre<T>(&sc, d.step_fac, d.n_check);
    {
      T acc[1] = {T(0)};
#pragma unroll
      for (int i = 0; i < TPW; ++i) {
        const int j = Rt[i].row;
        if (j < 0) continue;
        // a retry keeps A^T y
        if (!v.aty_valid) aty[i] = sp[i];
        if (v.do_avg) xa[i] = blend(xa[i], xc[i], v.w1, v.w);
        if (v.copy_lr) d.XLR[j] = xc[i];
        T z = xc[i] + v.tau * (aty[i] - cj[i]);
        if (d.q) z = z / (T(1) + v.tau * d.q[j]);
        xn[i] = clampv<T>(z, lj[i], uj[i]);
        const T dx = xn[i] - xc[i];
        acc[0] += dx * dx;
        if (!VS) d.X[v.nxt][j] = xn[i];
        else if (P == 1) xs[j] = xn[i];
        else
          for (int r = 0; r < P; ++r) st_cluster(xs + j, unsigned(r), xn[i]);
      }
      publish(St, Rt[0], part_p, acc, std::integral_constant<int, 1>());
    }
    ok = resident_barrier<SCOPE>(bar, target, limit_ns);
    if (!ok) break;
    {
      T acc[2] = {T(0), T(0)};
#pragma unroll
      for (int i = 0; i < TPW; ++i) {
        if (Ra[i].t < 0) continue;
        const T s = res_rowsum<T, VS>(Sa, Ra[i], idx_a, val_a, VS ? xs : d.X[v.nxt], sm);
        const int r = Ra[i].row;
        if (r < 0) continue;
        if (v.do_avg) ya[i] = blend(ya[i], yc[i], v.w1, v.w);
        if (v.copy_lr) d.YLR[r] = yc[i];
        const T axt = T(2) * s - ax[i];
        yn[i] = dual_prox<T>(yc[i], v.sigma, axt, lo[i], hi[i]);
        axn[i] = s;
        const T dy = yn[i] - yc[i];
        acc[0] += dy * dy;
        acc[1] += dy * (s - ax[i]);
        if (!VS) d.Y[v.nxt][r] = yn[i];
        else if (P == 1) ys[r] = yn[i];
        else
          for (int q = 0; q < P; ++q) st_cluster(ys + r, unsigned(q), yn[i]);
      }
      publish(Sa, Ra[0], part_d, acc, std::integral_constant<int, 2>());
    }
    ok = resident_barrier<SCOPE>(bar, target, limit_ns);
    if (!ok) break;
    // the decision (the control warps), and meanwhile the next primal step's row sums
    if (cw >= 0) {
      const T s = cw == 0 ? res_reduce<VS>(part_p, d.grid_p, 1) : res_reduce<VS>(part_d + (cw - 1), d.grid_d, 2);
      if (lane == 0) red[cw] = s;
      asm volatile("bar.sync 1, 96;" ::: "memory");
      if (cw == 0 && lane == 0)
        step_control<T>(&sc, spre, red[0], red[1], red[2], blockIdx.x == 0 ? d.trace_steps : nullptr, d.trace_cap);
      __syncwarp();
    }
    if (more) {
#pragma unroll
      for (int i = 0; i < TPW; ++i)
        if (Rt[i].t >= 0) sp[i] = res_rowsum<T, VS>(St, Rt[i], idx_t, val_t, VS ? ys : d.Y[v.nxt], sm);
    }
    __syncthreads();
    if (!sc.aty_valid) {  // accepted
#pragma unroll
      for (int i = 0; i < TPW; ++i) {
        xc[i] = xn[i];
        yc[i] = yn[i];
        ax[i] = axn[i];
      }
    }
  }
  // the lanes' entries back to the pools (the check that follows reads the current and
  // the averaged point and refreshes the products)
#pragma unroll
  for (int i = 0; i < TPW; ++i) {
    const int j = Rt[i].row, r = Ra[i].row;
    if (j >= 0) {
      d.X[sc.ix_cur][j] = xc[i];
      d.X[sc.ix_avg][j] = xa[i];
      d.ATY[sc.ia_cur][j] = aty[i];
    }
    if (r >= 0) {
      d.Y[sc.ix_cur][r] = yc[i];
      d.Y[sc.ix_avg][r] = ya[i];
      d.AX[sc.ix_cur][r] = ax[i];
    }
  }
  if (blockIdx.x == 0) {
    __syncthreads();
    if (!ok && threadIdx.x == 0) {
      sc.done = 1;
      sc.status = SCYLLA_DEVICE_TIMEOUT;
    }
    __syncthreads();
    for (int i = threadIdx.x; i < int(sizeof(Control) / 4); i += blockDim.x)
      reinterpret_cast<int*>(d.ctl)[i] = reinterpret_cast<const int*>(&sc)[i];
  }
}

// ------------------------------------------------------------- plan and launch ---
template <typename T>
static const void* resident_kernel(const ResidentPlan& p) {
  if (p.scope == kScopeCluster) return (const void*)k_attempts<T, kScopeCluster, 1>;
  if constexpr (sizeof(T) == 8)
    if (p.tpw == 2) return (const void*)k_attempts<T, kScopeGrid, 2>;
  return (const void*)k_attempts<T, kScopeGrid, 1>;
}

template <typename T>
static size_t resident_smem(const DevLP<T>& d, const ResidentPlan& p) {
  const size_t slots = size_t(p.slots_t) + size_t(p.slots_a);
  return slots * kResTile * (sizeof(T) + sizeof(int)) + size_t(p.threads / 32) * kSmemPerWarp * sizeof(T) +
         (p.scope == kScopeCluster ? (size_t(d.n) + size_t(d.m)) * sizeof(T) : 0);
}

static void resident_config(const ResidentPlan& p, cudaLaunchConfig_t& cfg, cudaLaunchAttribute (&attr)[1]) {
  cfg.gridDim = dim3(unsigned(p.blocks));
  cfg.blockDim = dim3(unsigned(p.threads));
  cfg.dynamicSmemBytes = p.smem;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  if (p.scope == kScopeGrid) {
    attr[0].id = cudaLaunchAttributeCooperative;
    attr[0].val.cooperative = 1;
  } else {
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = unsigned(p.blocks);
    attr[0].val.clusterDim.y = attr[0].val.clusterDim.z = 1;
  }
}

// whether the plan's launch can run on this device; sets the kernel's limits
template <typename T>
static bool resident_fits(const DevLP<T>& d, ResidentPlan& p) {
  p.smem = resident_smem(d, p);
  const void* k = resident_kernel<T>(p);
  int dev = 0, most = 0;
  cudaFuncAttributes fa{};
  cudaError_t e = cudaGetDevice(&dev);
  if (e == cudaSuccess) e = cudaDeviceGetAttribute(&most, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
  if (e == cudaSuccess) e = cudaFuncGetAttributes(&fa, k);
  if (e != cudaSuccess || p.smem + fa.sharedSizeBytes > size_t(most)) {
    cudaGetLastError();
    return false;
  }
  // the limit is per kernel, not per handle: the largest any handle may ask for
  e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, int(size_t(most) - fa.sharedSizeBytes));
  int n = 0;
  if (p.scope == kScopeCluster) {
    if (e == cudaSuccess) e = cudaFuncSetAttribute(k, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
    cudaLaunchConfig_t cfg = {};
    cudaLaunchAttribute attr[1];
    resident_config(p, cfg, attr);
    if (e == cudaSuccess) e = cudaOccupancyMaxActiveClusters(&n, k, &cfg);
  } else if (e == cudaSuccess) {
    e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, k, p.threads, p.smem);
  }
  if (e != cudaSuccess) cudaGetLastError();
  return e == cudaSuccess && n >= 1;
}

template <typename T>
bool resident_plan(const DevLP<T>& d, ResidentPlan* out) {
  const int sms = device_sm_count(), warps = ResidentThreads<T>::value / 32;
  const bool spread = d.t_ntiles <= d.grid_p && d.a_ntiles <= d.grid_d;
  const int most = d.t_ntiles > d.a_ntiles ? d.t_ntiles : d.a_ntiles;
  ResidentPlan p{};
  // A cluster as long as it beats the grid.  Its barrier is cheaper (0.34 us against
  // 1.3), but it has fewer SMs, and every new entry of x and y is stored to each of its
  // blocks.  Measured per 64 attempts, cluster of 8 / 16 / grid: FP32, 125 tiles 397 / 398
  // / 522 us, 330 tiles - / 610 / 562; FP64 (bound by the SMs' FP64 pipes), 44 tiles 659 /
  // 596 / 760, 125 tiles - / 834 / 774.
  // Few tiles take fewer blocks; with their check, 1 / 4 / 8 / 16 blocks: FP64, 2 tiles 397 /
  // 418 / 419 / 432 us, 8 tiles 557 / 425 / 427 / 439, 9 tiles 603 / 434 / 430 / 440, 24 tiles
  // - / 526 / 451 / 460; FP32, 2 tiles 187 / 236 / 239 / 246, 8 tiles 201 / 239 / 240 / 248, 24
  // tiles 286 / 249 / 246 / 262 (one block is the faster one there up to some 16 tiles).
  const int top = sizeof(T) == 4 ? 8 : 16;
  if (spread && most <= ResidentTiles<T>::value) {
    for (int P = most > 8 ? top : most > 2 ? 4 : 1; P >= 1; P /= 2) {
      const int per = (most + P - 1) / P;
      if (per + 3 > warps) break;
      p = ResidentPlan{};
      p.scope = kScopeCluster;
      p.blocks = P;
      p.threads = 32 * (per + 3);
      p.tpw = 1;
      p.slots_t = p.slots_a = per;
      if (resident_fits(d, p)) {
        *out = p;
        return true;
      }
    }
  }
  // one block per SM; every block's virtual warps fit its warps, one tile each (FP64:
  // up to two)
  p = ResidentPlan{};
  p.scope = kScopeGrid;
  p.blocks = sms;
  p.threads = ResidentThreads<T>::value;
  p.tpw = 1;
  auto slots = [&](int ntiles, int G) {
    if (ntiles <= G) return ntiles <= sms * warps ? (ntiles + sms - 1) / sms : -1;
    const int nb = warps / 8;
    if ((G + sms - 1) / sms > nb || nb > kResMaxVb) return -1;
    if (ntiles > 8 * G * (sizeof(T) == 8 ? 2 : 1)) return -1;
    if (ntiles <= 8 * G) return warps;
    p.tpw = 2;
    // second tiles s + 8 G of the block with most of them
    int top = 0;
    for (int c = 0; c < sms; ++c) {
      int k = 0;
      for (int v = 0; v < nb; ++v)
        for (int q = 0; q < 8; ++q) {
          const int b = c + sms * v, s = b + q * G;
          k += b < G && s + 8 * G < ntiles ? 1 : 0;
        }
      top = k > top ? k : top;
    }
    return warps + top;
  };
  p.slots_t = slots(d.t_ntiles, d.grid_p);
  p.slots_a = slots(d.a_ntiles, d.grid_d);
  if (p.slots_t < 0 || p.slots_a < 0) return false;
  if (!resident_fits(d, p)) return false;
  *out = p;
  return true;
}

template <typename T>
cudaError_t launch_attempts(const DevLP<T>& d, const ResidentPlan& p, void* bar, cudaStream_t st) {
  if (p.scope == kScopeGrid) {
    const cudaError_t e = cudaMemsetAsync(bar, 0, sizeof(ResidentBar), st);
    if (e != cudaSuccess) return e;
  }
  cudaLaunchConfig_t cfg = {};
  cudaLaunchAttribute attr[1];
  resident_config(p, cfg, attr);
  cfg.stream = st;
  DevLP<T> arg = d;
  ResidentArgs ra{p.slots_t, p.slots_a};
  ResidentBar* b = static_cast<ResidentBar*>(bar);
  unsigned long long limit = d.wait_ns;
  void* args[] = {&arg, &ra, &b, &limit};
  return cudaLaunchKernelExC(&cfg, resident_kernel<T>(p), args);
}
