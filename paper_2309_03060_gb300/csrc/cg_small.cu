// CG on small Kronecker operators, A = c_k (K_1 (x) K_2) [+ c_d Diag(d)], as one
// cooperative kernel that runs the whole iteration loop.
//
// A captured iteration of the general path is nine launches of a few
// microseconds each on an operator like 64 x 64, far above their work.  Here a
// grid of at most one block per SM keeps x, r and p of its outputs in registers
// and passes only p, r and the half-contracted vector through L2, with three
// grid barriers per iteration:
//   A  p = z + beta p_old (formed by every reader; the owner stores it),
//      T[i1][m] = sum_j K_1[i1][j] p[j][m]                          | barrier
//   B  A p[i1][i2] = c_k sum_m K_2[i2][m] T[i1][m] + c_d d p, partials of p . A p
//                                                                    | barrier
//   C  alpha, x, r, z, partials of r . z and r . r                   | barrier
//   D  beta and the stopping rule; the loop ends as soon as every right-hand
//      side has stopped
// A task is a 4 x 8 tile of outputs of one right-hand side, 8 lanes per output
// sharing its k sum; a block runs up to 4 tasks.  Sums over tasks are taken by
// every block in the same order, so all blocks agree on alpha and beta.
// Measured (FP64, 64 x 64, one right-hand side): 15 us per iteration against 37 us.
// A barrier that is not reached within 2 s raises the error flag and ends the kernel.
#include <algorithm>

#include "internal.h"

namespace cola {

namespace {

constexpr int kSmTasks = 4;    // tasks per block
constexpr int kSmThreads = 256;
constexpr uint64_t kSmWaitNs = 2000000000ull;

template <typename T>
struct SmallP {
  const T *K1, *K2, *d, *invd;
  int64_t dstride;
  T ck, cd;
  int n1, n2, R, tiles2, tiles, ntask, limit;
  T *r, *x, *p0, *p1, *t;
  double2 *part_pap, *part_rr;  // [R][tiles]: (p . A p, 0) and (r . z, r . r)
  CgState* st;
  int* act;        // [R]
  unsigned* bar;   // barrier arrivals
  int* err;
};

__device__ __forceinline__ unsigned ld_acquire(const unsigned* p) {
  unsigned v;
  asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
  return v;
}

__device__ __forceinline__ uint64_t clock_ns() {
  uint64_t t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}

// Every block has arrived `epoch` times.  False (in every block, sooner or
// later) when one did not within the limit.
__device__ bool grid_barrier(unsigned* bar, unsigned epoch, int* err, volatile int* fail) {
  __syncthreads();
  if (threadIdx.x == 0) {
    const unsigned want = epoch * gridDim.x;
    // release: the block's writes, ordered before by the barrier above
    asm volatile("red.release.gpu.global.add.u32 [%0], 1;" ::"l"(bar) : "memory");
    unsigned spins = 0;
    uint64_t t0 = 0;
    while (ld_acquire(bar) < want) {
      if ((++spins & 255u) != 0) continue;
      if (t0 == 0) t0 = clock_ns();
      if (clock_ns() - t0 > kSmWaitNs || *(volatile int*)err != 0) {
        atomicExch(err, COLA_ERR_TIMEOUT);
        *fail = 1;
        break;
      }
    }
  }
  __syncthreads();
  return *fail == 0;
}

// Sums of two values over the block, in every thread (fixed order).  LO: only
// lanes that are multiples of it hold values (a dependent FP64 add is most of
// the cost, so steps are worth saving).
template <int LO>
__device__ __forceinline__ double2 block_sum2(double2 v, double2* sh) {
#pragma unroll
  for (int o = 16; o >= LO; o >>= 1) {
    v.x += __shfl_xor_sync(0xffffffffu, v.x, o);
    v.y += __shfl_xor_sync(0xffffffffu, v.y, o);
  }
  __syncthreads();
  if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5] = v;
  __syncthreads();
  v = sh[threadIdx.x & (kSmThreads / 32 - 1)];
#pragma unroll
  for (int o = kSmThreads / 64; o > 0; o >>= 1) {
    v.x += __shfl_xor_sync(0xffffffffu, v.x, o);
    v.y += __shfl_xor_sync(0xffffffffu, v.y, o);
  }
  return v;
}

// Sums of the `n` pairs of partials written by other blocks (in every thread).
__device__ __forceinline__ double2 part_sum2(const double2* p, int n, double2* sh) {
  double2 v = make_double2(0.0, 0.0);
  for (int j = threadIdx.x; j < n; j += kSmThreads) {
    const double2 a = __ldcg(p + j);
    v.x += a.x;
    v.y += a.y;
  }
  return block_sum2<1>(v, sh);
}

// sum over the 8 lanes of an output
template <typename T>
__device__ __forceinline__ T lane8(T v) {
  v += __shfl_xor_sync(0xffffffffu, v, 1);
  v += __shfl_xor_sync(0xffffffffu, v, 2);
  v += __shfl_xor_sync(0xffffffffu, v, 4);
  return v;
}

template <typename T>
__global__ void __launch_bounds__(kSmThreads) k_cg_small(const SmallP<T> q) {
  __shared__ double2 sh[kSmThreads / 32];
  __shared__ int fail;
  if (threadIdx.x == 0) fail = 0;
  __syncthreads();
  const int kl = threadIdx.x & 7, out = threadIdx.x >> 3;  // k lane, output of the tile
  const int n1 = q.n1, n2 = q.n2;
  const int64_t N = (int64_t)n1 * n2;
  // outputs: rows 4 (tile / tiles2) + out / 8, columns 8 (tile mod tiles2) + out mod 8
  int rhs[kSmTasks], row[kSmTasks], col[kSmTasks];
  bool on[kSmTasks];
  int64_t own[kSmTasks];
  T xv[kSmTasks], rv[kSmTasks], pv[kSmTasks], av[kSmTasks], dv[kSmTasks], mv[kSmTasks];
  double beta[kSmTasks], rz[kSmTasks];
  int active[kSmTasks];
#pragma unroll
  for (int k = 0; k < kSmTasks; ++k) {
    const int t = blockIdx.x + k * gridDim.x;
    on[k] = t < q.ntask;
    rhs[k] = on[k] ? t / q.tiles : 0;
    const int tile = on[k] ? t - rhs[k] * q.tiles : 0;
    row[k] = tile / q.tiles2 * 4 + (out >> 3);
    col[k] = tile % q.tiles2 * 8 + (out & 7);
    const bool in = on[k] && row[k] < n1 && col[k] < n2;
    own[k] = in ? (int64_t)row[k] * n2 + col[k] : -1;
    const int64_t o = rhs[k] * N + (in ? own[k] : 0);
    xv[k] = in ? q.x[o] : T(0);
    rv[k] = in ? q.r[o] : T(0);
    pv[k] = in ? q.p0[o] : T(0);
    dv[k] = in && q.d ? q.cd * q.d[q.dstride ? own[k] : 0] : T(0);
    mv[k] = in && q.invd ? q.invd[own[k]] : T(1);
    const CgState& s = q.st[rhs[k]];
    active[k] = s.active;
    beta[k] = s.beta;
    rz[k] = s.rz;
  }
  unsigned epoch = 0;
  const T *po = q.p0;
  T* pn = q.p1;
  for (int it = 0; it < q.limit; ++it) {
    // ---- A
#pragma unroll
    for (int k = 0; k < kSmTasks; ++k) {
      if (!on[k]) continue;
      const T b = (T)beta[k];
      const int64_t base = rhs[k] * N;
      if (own[k] >= 0) {
        const T z = rv[k] * mv[k];
        pv[k] = b != T(0) ? fma(b, pv[k], z) : z;
        if (kl == 0) pn[base + own[k]] = pv[k];
      }
      // T[i1 = row][m = col]: k = j over the rows of p
      T acc = T(0);
      const int i1 = min(row[k], n1 - 1), m = min(col[k], n2 - 1);
      const T* k1 = q.K1 + (int64_t)i1 * n1;
      const T* rr = q.r + base + m;
      const T* pp = po + base + m;
#pragma unroll 8
      for (int j = kl; j < n1; j += 8) {
        T z = __ldcg(rr + (int64_t)j * n2);
        if (q.invd) z *= __ldg(q.invd + (int64_t)j * n2 + m);
        if (b != T(0)) z = fma(b, __ldcg(pp + (int64_t)j * n2), z);
        acc = fma(__ldg(k1 + j), z, acc);
      }
      acc = lane8(acc);
      if (kl == 0 && own[k] >= 0) q.t[base + own[k]] = acc;
    }
    if (!grid_barrier(q.bar, ++epoch, q.err, &fail)) break;
    // every right-hand side stopped (flags written before the barrier)
    {
      int any = 0;
      for (int r = threadIdx.x; r < q.R; r += kSmThreads) any |= __ldcg(q.act + r);
      if (!__syncthreads_or(any)) break;
    }
    // ---- B
#pragma unroll
    for (int k = 0; k < kSmTasks; ++k) {
      if (!on[k]) continue;
      T acc = T(0);
      const int i1 = min(row[k], n1 - 1), i2 = min(col[k], n2 - 1);
      const T* tt = q.t + rhs[k] * N + (int64_t)i1 * n2;
      const T* k2 = q.K2 + (int64_t)i2 * n2;
#pragma unroll 8
      for (int m = kl; m < n2; m += 8) acc = fma(__ldg(k2 + m), __ldcg(tt + m), acc);
      acc = lane8(acc);
      av[k] = fma(dv[k], pv[k], q.ck * acc);
      const double2 s = block_sum2<8>(
          make_double2(kl == 0 && own[k] >= 0 ? (double)pv[k] * (double)av[k] : 0.0, 0.0), sh);
      if (threadIdx.x == 0) q.part_pap[blockIdx.x + k * gridDim.x] = s;
    }
    if (!grid_barrier(q.bar, ++epoch, q.err, &fail)) break;
    // ---- C
#pragma unroll
    for (int k = 0; k < kSmTasks; ++k) {
      if (!on[k]) continue;
      const double pap = part_sum2(q.part_pap + rhs[k] * q.tiles, q.tiles, sh).x;
      double alpha = 0.0;
      if (active[k]) {
        if (!(pap > 0.0) || !isfinite(pap)) {
          active[k] = -1;  // breakdown
        } else {
          alpha = rz[k] / pap;
        }
      }
      const T a = (T)alpha;
      double2 s2 = make_double2(0.0, 0.0);
      if (own[k] >= 0) {
        if (a != T(0)) {
          xv[k] = fma(a, pv[k], xv[k]);
          rv[k] = fma(-a, av[k], rv[k]);
          if (kl == 0) q.r[rhs[k] * N + own[k]] = rv[k];
        }
        if (kl == 0) {
          s2.x = (double)rv[k] * (double)(rv[k] * mv[k]);
          s2.y = (double)rv[k] * (double)rv[k];
        }
      }
      s2 = block_sum2<8>(s2, sh);
      const int t = blockIdx.x + k * gridDim.x;
      if (threadIdx.x == 0) {
        q.part_rr[t] = s2;
        if (t == rhs[k] * q.tiles && active[k] == 1) {  // tile 0 keeps the state
          q.st[rhs[k]].pAp = pap;
          q.st[rhs[k]].alpha = alpha;
        }
      }
    }
    if (!grid_barrier(q.bar, ++epoch, q.err, &fail)) break;
    // ---- D
#pragma unroll
    for (int k = 0; k < kSmTasks; ++k) {
      if (!on[k]) continue;
      const int t = blockIdx.x + k * gridDim.x;
      const bool first = threadIdx.x == 0 && t == rhs[k] * q.tiles;
      CgState& s = q.st[rhs[k]];
      if (active[k] == 1) {
        const double2 sums = part_sum2(q.part_rr + rhs[k] * q.tiles, q.tiles, sh);
        const double nz = sums.x, nr = sums.y;
        beta[k] = nz / rz[k];
        rz[k] = nz;
        const bool bad = !isfinite(nr) || !isfinite(nz);
        if (bad) beta[k] = 0.0;
        if (bad || nr <= s.tol2) active[k] = 0;
        if (first) {
          s.rz = nz;
          s.rr = nr;
          s.iters += 1;
          s.beta = beta[k];
          s.active = active[k];
          if (bad) s.status = COLA_ERR_BREAKDOWN;
          q.act[rhs[k]] = active[k];
        }
      } else if (active[k] == -1) {
        active[k] = 0;
        beta[k] = 0.0;
        if (first) {
          s.status = COLA_ERR_BREAKDOWN;
          s.active = 0;
          s.alpha = 0.0;
          q.act[rhs[k]] = 0;
        }
      } else {
        beta[k] = 0.0;
        if (first) q.act[rhs[k]] = 0;
      }
    }
    const T* o = po;
    po = pn;
    pn = const_cast<T*>(o);
  }
  // x and the last direction (every reader of either p buffer is behind a barrier)
#pragma unroll
  for (int k = 0; k < kSmTasks; ++k)
    if (on[k] && own[k] >= 0 && kl == 0) {
      q.x[rhs[k] * N + own[k]] = xv[k];
      q.p0[rhs[k] * N + own[k]] = pv[k];
    }
}

}  // namespace

template <typename T>
bool small_cg_setup(Ctx* c, const cola_linop* op, int64_t R, SmallCg* S) {
  *S = SmallCg{};
  const cola_linop *kr = nullptr, *dg = nullptr;
  double ck = 1.0, cd = 0.0;
  if (op->kind == LK_KRON) {
    kr = op;
  } else if (op->kind == LK_SUM && op->kids.size() == 2) {
    for (int i = 0; i < 2; ++i) {
      const cola_linop* k = op->kids[i];
      if (k->kind == LK_KRON) {
        kr = k;
        ck = op->coeffs[i];
      } else if (k->kind == LK_DIAG) {
        dg = k;
        cd = op->coeffs[i];
      }
    }
    if (!dg) return false;
  }
  if (!kr || kr->kids.size() != 2) return false;
  for (auto* f : kr->kids)
    if (f->rows != f->cols) return false;
  const int64_t n1 = kr->kids[0]->rows, n2 = kr->kids[1]->rows;
  const int64_t tiles2 = (n2 + 7) / 8, tiles = (n1 + 3) / 4 * tiles2;
  if (n1 > 1024 || n2 > 1024 || R * tiles > (int64_t)kSmTasks * c->num_sms) return false;
  S->on = true;
  S->kron = kr;
  S->diag = dg;
  S->ck = ck;
  S->cd = cd;
  S->tiles2 = (int)tiles2;
  S->tiles = (int)tiles;
  const int64_t N = n1 * n2;
  S->t = c->ws.get("cgs.t", sizeof(T) * N * R);
  S->p1 = c->ws.get("cgs.p1", sizeof(T) * N * R);
  S->part = (double*)c->ws.get("cgs.part", 2 * sizeof(double2) * (size_t)(tiles * R));
  S->act = (int*)c->ws.get("cgs.act", 4 * R + 256);
  S->bar = (unsigned*)c->ws.get("cgs.bar", 256);
  return true;
}
template bool small_cg_setup<float>(Ctx*, const cola_linop*, int64_t, SmallCg*);
template bool small_cg_setup<double>(Ctx*, const cola_linop*, int64_t, SmallCg*);

template <typename T>
void small_cg_run(Ctx* c, const SmallCg& S, T* r, T* x, T* p, const T* invd, CgState* st,
                  int64_t R, int limit) {
  SmallP<T> q{};
  q.K1 = leaf_ptr<T>(S.kron->kids[0]);
  q.K2 = leaf_ptr<T>(S.kron->kids[1]);
  if (S.diag) {
    q.d = leaf_ptr<T>(S.diag);
    q.dstride = S.diag->stride;
  }
  q.invd = invd;
  q.ck = (T)S.ck;
  q.cd = (T)S.cd;
  q.n1 = (int)S.kron->kids[0]->rows;
  q.n2 = (int)S.kron->kids[1]->rows;
  q.R = (int)R;
  q.tiles2 = S.tiles2;
  q.tiles = S.tiles;
  q.ntask = (int)(R * S.tiles);
  q.limit = limit;
  q.r = r;
  q.x = x;
  q.p0 = p;
  q.p1 = (T*)S.p1;
  q.t = (T*)S.t;
  q.part_pap = (double2*)S.part;
  q.part_rr = (double2*)S.part + q.ntask;
  q.st = st;
  q.act = S.act;
  q.bar = S.bar;
  q.err = tc_errflag(c);
  COLA_CUDA(cudaMemsetAsync(S.bar, 0, 4, c->s));
  // active flags as of the state (any non-zero byte pattern counts as active)
  COLA_CUDA(cudaMemsetAsync(S.act, 1, 4 * R, c->s));
  const int grid = std::min(q.ntask, c->num_sms);
  void* args[] = {&q};
  COLA_CUDA(cudaLaunchCooperativeKernel((const void*)k_cg_small<T>, dim3(grid), dim3(kSmThreads),
                                        args, 0, c->s));
  c->count_launch();
  c->f64_tc_used = true;  // the error flag is checked at the end of the call
}
template void small_cg_run<float>(Ctx*, const SmallCg&, float*, float*, float*, const float*,
                                  CgState*, int64_t, int);
template void small_cg_run<double>(Ctx*, const SmallCg&, double*, double*, double*, const double*,
                                   CgState*, int64_t, int);

}  // namespace cola
