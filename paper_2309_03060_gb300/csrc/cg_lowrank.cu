// FP32 CG iteration for A = c_s (T_1 (+) T_2) + c_d Diag(d) + c_u U U^T with
// tridiagonal T_k (a 2-D stencil), optionally Jacobi preconditioned, in two
// large kernels and two small ones.
//
// The generic iteration reads U twice (U^T p, then U W), and p, A p, r, z several
// times in separate passes.  Here U is read once per iteration:
//   * p . A p = p . (S p) + c_u ||U^T p||^2 with S the stencil and the diagonal,
//     so alpha is known before U W is formed;
//   * U^T p_new = U^T z + beta U^T p_old, so the pass over U that forms
//     A p = S p + c_u U (U^T p), updates x and r and forms z = M^-1 r also
//     accumulates U^T z for the next direction.
// The recurrence for U^T p (kept in FP64) is as exact as the one for p itself,
// and a solve that meets its tolerance is checked on the true residual formed
// by the ordinary MVM.  Bytes per iteration and vector entry: r, p read, p, q
// written (k_lr_pq); q, p, r, x read, r, x written (k_lr_update); U once per 8
// right-hand sides.  Measured on the 2^20-point, rank 32, 8-right-hand-side
// solve: 127 us per iteration against 164 us (k_lr_update 78, k_lr_pq 35; 326 and 170 MB).
#include <algorithm>

#include "internal.h"

namespace cola {

namespace {

constexpr int kLrRank = 32;     // largest rank of this path
constexpr int kLrRows = 128;    // rows per stage of the pass over U
constexpr int kLrPad = 36;      // floats per staged row of U (16-byte chunks, no conflicts)
constexpr int kLrStages = 3;
// floats per stage: 128 rows of U, then q, p, r, x of 8 right-hand sides
constexpr int kLrStage = kLrRows * kLrPad + 4 * 8 * kLrRows;
constexpr size_t kLrSmem = sizeof(float) * (kLrStages * kLrStage + kLrRank * 8);

__device__ __forceinline__ float4 ld4f(const float* p) {
  return *reinterpret_cast<const float4*>(p);
}

// Sum over the block, valid in thread 0 (fixed order).
__device__ __forceinline__ double block_sum_d(double v, double* sh) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  __syncthreads();
  if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5] = v;
  __syncthreads();
  double t = 0.0;
  if (threadIdx.x == 0)
    for (int w = 0; w < (int)(blockDim.x >> 5); ++w) t += sh[w];
  return t;
}

// p_new = M^-1 r + beta p_old, q = (c_s stencil + c_d Diag(d)) p_new and the
// partials of p_new . q.  A thread walks strips of S rows of one column quad,
// forming each row of p once (plus one halo row at each end) from r, 1/diag
// and p_old; left and right neighbours come from the adjacent lanes.
// grid.y = right-hand side.
__global__ void __launch_bounds__(256, 2)
    k_lr_pq(int n1, int n2, int S, const float* __restrict__ bands, const float* __restrict__ r,
            const float* __restrict__ invd, const float* __restrict__ p_old,
            float* __restrict__ p_new, float* __restrict__ q, const float* __restrict__ dg,
            int64_t dstride, float cs, float cd, const CgState* st, double* part) {
  __shared__ double sh[8];
  const int q4 = n2 / 4, ns = (n1 + S - 1) / S;
  const int64_t N = (int64_t)n1 * n2;
  const int v = blockIdx.y, lane = threadIdx.x & 31;
  const float beta = (float)st[v].beta;
  const float* rv = r + v * N;
  const float* po = p_old + v * N;
  float* pn = p_new + v * N;
  float* qv = q + v * N;
  const float *lo0 = bands, *di0 = bands + n1, *up0 = bands + 2 * n1;
  const float *lo1 = bands + 3 * n1, *di1 = lo1 + n2, *up1 = lo1 + 2 * n2;
  // one row of a quad as loaded (r, 1/diag, p_old, and the scalar neighbours of
  // the lanes at a warp's ends): loaded one row ahead of its use
  struct Raw {
    float4 r, m, b;
    float lr, lm, lb, rr, rm, rb;
  };
  auto load = [&](int64_t o, bool l_ld, bool r_ld, Raw& w) {
    w.r = ld4f(rv + o);
    if (invd) w.m = ld4f(invd + o);
    if (beta != 0.0f) w.b = ld4f(po + o);
    if (l_ld) {
      w.lr = rv[o - 1];
      w.lm = invd ? invd[o - 1] : 1.0f;
      w.lb = beta != 0.0f ? po[o - 1] : 0.0f;
    }
    if (r_ld) {
      w.rr = rv[o + 4];
      w.rm = invd ? invd[o + 4] : 1.0f;
      w.rb = beta != 0.0f ? po[o + 4] : 0.0f;
    }
  };
  auto p4 = [&](const Raw& w, float (&out)[4]) {
    float4 z = w.r;
    if (invd) z = make_float4(z.x * w.m.x, z.y * w.m.y, z.z * w.m.z, z.w * w.m.w);
    if (beta != 0.0f) {
      z.x = fmaf(beta, w.b.x, z.x);
      z.y = fmaf(beta, w.b.y, z.y);
      z.z = fmaf(beta, w.b.z, z.z);
      z.w = fmaf(beta, w.b.w, z.w);
    }
    out[0] = z.x;
    out[1] = z.y;
    out[2] = z.z;
    out[3] = z.w;
  };
  auto p1 = [&](float r1, float m1, float b1) {
    const float z = invd ? r1 * m1 : r1;
    return beta != 0.0f ? fmaf(beta, b1, z) : z;
  };
  const int items = ns * q4;
  float dot = 0.0f;
  for (int t0 = blockIdx.x * 256 + (threadIdx.x & ~31); t0 < items; t0 += gridDim.x * 256) {
    const int t = t0 + lane;
    const bool on = t < items;
    const int tt = on ? t : items - 1;
    const int cq = tt % q4, i1a = tt / q4 * S, i2 = cq * 4;
    const int i1b = min(i1a + S, n1);
    // neighbours from the adjacent lanes where those hold the same rows
    const bool l_sh = lane > 0 && cq > 0;
    const bool r_sh = lane < 31 && cq < q4 - 1 && t + 1 < items;
    const bool l_ld = !l_sh && cq > 0, r_ld = !r_sh && cq < q4 - 1;
    float b_lo[4], b_di[4], b_up[4];
#pragma unroll
    for (int e = 0; e < 4; ++e) {
      b_lo[e] = lo1[i2 + e];
      b_di[e] = di1[i2 + e];
      b_up[e] = up1[i2 + e];
    }
    float xu[4] = {0.f, 0.f, 0.f, 0.f}, xc[4], xd[4] = {0.f, 0.f, 0.f, 0.f};
    Raw w;
    {
      Raw h;
      const bool up = i1a > 0;
      load((int64_t)(up ? i1a - 1 : i1a) * n2 + i2, false, false, h);
      load((int64_t)i1a * n2 + i2, l_ld, r_ld, w);
      if (up) p4(h, xu);
    }
    p4(w, xc);
    float el = l_ld ? p1(w.lr, w.lm, w.lb) : 0.0f, er = r_ld ? p1(w.rr, w.rm, w.rb) : 0.0f;
    if (i1a + 1 < n1) load((int64_t)(i1a + 1) * n2 + i2, l_ld, r_ld, w);
    // every lane takes S steps (the exchanges need the whole warp)
    for (int k = 0; k < S; ++k) {
      const int i1 = i1a + k;
      const bool act = i1 < i1b;
      const int64_t o = (int64_t)(act ? i1 : i1a) * n2 + i2;
      float nl = 0.0f, nr = 0.0f;  // the next row's end neighbours
      if (act && i1 + 1 < n1) {
        p4(w, xd);
        if (l_ld) nl = p1(w.lr, w.lm, w.lb);
        if (r_ld) nr = p1(w.rr, w.rm, w.rb);
        if (k + 1 < S && i1 + 2 < n1) load(o + 2 * n2, l_ld, r_ld, w);
      }
      float xl = __shfl_up_sync(0xffffffffu, xc[3], 1);
      float xr = __shfl_down_sync(0xffffffffu, xc[0], 1);
      if (!act) continue;
      if (!l_sh) xl = el;
      if (!r_sh) xr = er;
      const float a0 = di0[i1], l0 = lo0[i1], u0 = up0[i1];
      float out[4];
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        const int j = i2 + e;
        float s = a0 * xc[e];
        if (i1 > 0) s = fmaf(l0, xu[e], s);
        if (i1 < n1 - 1) s = fmaf(u0, xd[e], s);
        s = fmaf(b_di[e], xc[e], s);
        if (j > 0) s = fmaf(b_lo[e], e > 0 ? xc[e - 1] : xl, s);
        if (j < n2 - 1) s = fmaf(b_up[e], e < 3 ? xc[e + 1] : xr, s);
        out[e] = s * cs;
      }
      if (dg) {
        const float d0 = dstride ? 0.0f : dg[0];
        const float4 d = dstride ? ld4f(dg + o) : make_float4(d0, d0, d0, d0);
        out[0] = fmaf(cd * d.x, xc[0], out[0]);
        out[1] = fmaf(cd * d.y, xc[1], out[1]);
        out[2] = fmaf(cd * d.z, xc[2], out[2]);
        out[3] = fmaf(cd * d.w, xc[3], out[3]);
      }
      if (on) {
        *reinterpret_cast<float4*>(pn + o) = make_float4(xc[0], xc[1], xc[2], xc[3]);
        *reinterpret_cast<float4*>(qv + o) = make_float4(out[0], out[1], out[2], out[3]);
#pragma unroll
        for (int e = 0; e < 4; ++e) dot = fmaf(xc[e], out[e], dot);
      }
      el = nl;
      er = nr;
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        xu[e] = xc[e];
        xc[e] = xd[e];
      }
    }
  }
  const double s = block_sum_d((double)dot, sh);
  if (threadIdx.x == 0) part[(int64_t)v * gridDim.x + blockIdx.x] = s;
}

// One block per right-hand side: W = U^T p_new = U^T z + beta U^T p_old,
// p . A p = the partials + c_u ||W||^2, alpha (as k_cg_alpha).
__global__ void k_lr_alpha(CgState* st, const double* part, int nparts, int rank, int64_t R,
                           const double* Wz, double* W, double cu) {
  __shared__ double sh[8];
  const int64_t r = blockIdx.x;
  CgState& s = st[r];
  double v = 0.0;
  for (int j = threadIdx.x; j < nparts; j += blockDim.x) v += part[r * nparts + j];
  if (threadIdx.x < rank) {
    const int64_t o = threadIdx.x * R + r;
    double w = Wz[o];
    const double be = (double)(float)s.beta;  // as k_lr_pq applied it
    if (be != 0.0) w = fma(be, W[o], w);
    W[o] = w;
    v = fma(cu * w, w, v);
  }
  v = block_sum_d(v, sh);
  if (threadIdx.x != 0) return;
  if (!s.active || s.paused) {
    s.alpha = 0.0;
    return;
  }
  s.pAp = v;
  if (!(v > 0.0) || !isfinite(v)) {
    s.status = COLA_ERR_BREAKDOWN;
    s.active = 0;
    s.alpha = 0.0;
    return;
  }
  s.alpha = s.rz / v;
}

__device__ __forceinline__ void cp16(float* dst, const float* src, bool ok) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(
                   (unsigned)__cvta_generic_to_shared(dst)),
               "l"(src), "r"(ok ? 16 : 0)
               : "memory");
}

// The pass over U: A p = q + c_u U W, x += alpha p, r -= alpha A p, z = M^-1 r, the
// partials of r . z, r . r and U^T z.  A block owns the contiguous rows
// [rb0, rb0 + rpb) for the 8 right-hand sides of grid.y; U and the vectors
// arrive in stages of 128 rows by cp.async, two stages ahead.  Thread (row,
// half) forms 4 right-hand sides of one row and leaves z where q was; then
// lane (c, g) of warp w multiplies columns
// 4 c .. + 3 of rows 16 w + 4 g .. + 3 with the 8 z's, as k_lr_vtx_cp.
__global__ void __launch_bounds__(256, 2)
    k_lr_update(const float* U, int rank, int64_t n, int64_t R, int64_t rpb, const double* W,
                const float* q, const float* p, float* r, float* x, const float* invd, float cu,
                const CgState* st, double* part_rz, double* part_rr, double* part_w) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  float* us = reinterpret_cast<float*>(smem_raw);
  float* ws = us + kLrStages * kLrStage;  // [32][8]
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int64_t r0 = (int64_t)blockIdx.y * 8;
  const int64_t rb0 = (int64_t)blockIdx.x * rpb;
  const int64_t rb1 = min(n, rb0 + rpb);
  const int nst = rb0 < rb1 ? (int)((rb1 - rb0 + kLrRows - 1) / kLrRows) : 0;
  {
    const int k = tid >> 3, g = tid & 7;
    ws[tid] = (k < rank && r0 + g < R) ? cu * (float)W[k * R + r0 + g] : 0.0f;
  }
  auto issue = [&](int s) {
    float* d = us + (s % kLrStages) * kLrStage;
    const int64_t i0 = rb0 + (int64_t)s * kLrRows;
    const int rows = (int)min((int64_t)kLrRows, rb1 - i0);
#pragma unroll
    for (int m = 0; m < 4; ++m) {
      const int e = tid + 256 * m, row = e >> 3, j = (e & 7) * 4;
      const bool ok = row < rows && j < rank;
      cp16(d + row * kLrPad + j, ok ? U + (i0 + row) * rank + j : U, ok);
    }
    // right-hand side tid / 32, rows 4 (tid mod 32) .. of each vector (n % 4 == 0)
    const int g = tid >> 5, j = (tid & 31) * 4;
    const bool ok = j < rows && r0 + g < R;
    const int64_t o = ok ? (r0 + g) * n + i0 + j : 0;
    float* v = d + kLrRows * kLrPad + g * kLrRows + j;
    cp16(v, q + o, ok);
    cp16(v + 8 * kLrRows, p + o, ok);
    cp16(v + 16 * kLrRows, r + o, ok);
    cp16(v + 24 * kLrRows, x + o, ok);
  };
#pragma unroll
  for (int s = 0; s < kLrStages - 1; ++s) {
    if (s < nst) issue(s);
    asm volatile("cp.async.commit_group;" ::: "memory");
  }
  const int row = tid & 127, half = tid >> 7;  // this thread's row and 4 right-hand sides
  float al[4];
#pragma unroll
  for (int e = 0; e < 4; ++e) {
    const int64_t v = r0 + half * 4 + e;
    al[e] = v < R ? (float)st[v].alpha : 0.0f;
  }
  float srz[4] = {0.f, 0.f, 0.f, 0.f}, srr[4] = {0.f, 0.f, 0.f, 0.f};
  float acc[4][8];
#pragma unroll
  for (int e = 0; e < 4; ++e)
#pragma unroll
    for (int g = 0; g < 8; ++g) acc[e][g] = 0.f;
  const int c = lane & 7, g4 = lane >> 3, rr = warp * 16 + 4 * g4;
  for (int s = 0; s < nst; ++s) {
    const int64_t i = rb0 + (int64_t)s * kLrRows + row;
    const bool in = i < rb1;
    const float mi = in ? (invd ? __ldg(invd + i) : 1.0f) : 0.0f;
    asm volatile("cp.async.wait_group %0;" ::"n"(kLrStages - 2) : "memory");
    __syncthreads();  // stage s landed; stage s - 1 is no longer read
    if (s + kLrStages - 1 < nst) issue(s + kLrStages - 1);
    asm volatile("cp.async.commit_group;" ::: "memory");
    const float* ut = us + (s % kLrStages) * kLrStage;
    float* zs = us + (s % kLrStages) * kLrStage + kLrRows * kLrPad;  // q, then z
    float qv[4], pv[4], rv[4], xv[4];
#pragma unroll
    for (int e = 0; e < 4; ++e) {
      const int o = (half * 4 + e) * kLrRows + row;
      qv[e] = zs[o];
      pv[e] = zs[o + 8 * kLrRows];
      rv[e] = zs[o + 16 * kLrRows];
      xv[e] = zs[o + 24 * kLrRows];
    }
    float ap[4] = {qv[0], qv[1], qv[2], qv[3]};
#pragma unroll
    for (int k = 0; k < kLrRank; k += 4) {
      const float4 u = ld4f(ut + row * kLrPad + k);
      const float uk[4] = {u.x, u.y, u.z, u.w};
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        const float4 w = ld4f(ws + (k + j) * 8 + half * 4);
        ap[0] = fmaf(uk[j], w.x, ap[0]);
        ap[1] = fmaf(uk[j], w.y, ap[1]);
        ap[2] = fmaf(uk[j], w.z, ap[2]);
        ap[3] = fmaf(uk[j], w.w, ap[3]);
      }
    }
#pragma unroll
    for (int e = 0; e < 4; ++e) {
      const int64_t o = (r0 + half * 4 + e) * n + i;
      const bool ok = in && r0 + half * 4 + e < R;
      float ri = rv[e];
      if (al[e] != 0.0f) {  // a stopped right-hand side keeps x and r as they are
        ri = fmaf(-al[e], ap[e], ri);
        if (ok) {
          x[o] = fmaf(al[e], pv[e], xv[e]);
          r[o] = ri;
        }
      }
      const float z = ri * mi;
      zs[(half * 4 + e) * kLrRows + row] = ok ? z : 0.f;
      if (ok) {
        srz[e] = fmaf(ri, z, srz[e]);
        srr[e] = fmaf(ri, ri, srr[e]);
      }
    }
    __syncthreads();
    float4 v[4];
#pragma unroll
    for (int u = 0; u < 4; ++u) v[u] = ld4f(ut + (rr + u) * kLrPad + 4 * c);
#pragma unroll
    for (int g = 0; g < 8; ++g) {
      const float4 z = ld4f(zs + g * kLrRows + rr);
      const float zq[4] = {z.x, z.y, z.z, z.w};
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        acc[0][g] = fmaf(v[u].x, zq[u], acc[0][g]);
        acc[1][g] = fmaf(v[u].y, zq[u], acc[1][g]);
        acc[2][g] = fmaf(v[u].z, zq[u], acc[2][g]);
        acc[3][g] = fmaf(v[u].w, zq[u], acc[3][g]);
      }
    }
  }
  asm volatile("cp.async.wait_group 0;" ::: "memory");
  const int nb = gridDim.x;
  // r . z and r . r: threads of half h hold right-hand sides 4 h .. + 3 (warps 4 h .. 4 h + 3)
  {
    __shared__ double s2[2][8][4];
#pragma unroll
    for (int e = 0; e < 4; ++e) {
      double a = (double)srz[e], b = (double)srr[e];
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) {
        a += __shfl_xor_sync(0xffffffffu, a, o);
        b += __shfl_xor_sync(0xffffffffu, b, o);
      }
      if (lane == 0) {
        s2[0][warp][e] = a;
        s2[1][warp][e] = b;
      }
    }
    __syncthreads();
    if (tid < 16) {
      const int which = tid >> 3, g = tid & 7, h = g >> 2, e = g & 3;
      double t = 0.0;
      for (int w = 0; w < 4; ++w) t += s2[which][h * 4 + w][e];
      if (r0 + g < R) (which ? part_rr : part_rz)[(r0 + g) * nb + blockIdx.x] = t;
    }
  }
  // U^T z: the 4 row quads of a warp by shuffles, then the 8 warps
  double* red = reinterpret_cast<double*>(smem_raw);  // [8 warps][32][8]
#pragma unroll
  for (int e = 0; e < 4; ++e)
#pragma unroll
    for (int g = 0; g < 8; ++g) {
      double a = (double)acc[e][g];
      a += __shfl_xor_sync(0xffffffffu, a, 8);
      a += __shfl_xor_sync(0xffffffffu, a, 16);
      if (g4 == 0) red[(warp * 32 + 4 * c + e) * 8 + g] = a;
    }
  __syncthreads();
  {
    const int k = tid >> 3, g = tid & 7;
    double t = 0.0;
#pragma unroll
    for (int w = 0; w < 8; ++w) t += red[(w * 32 + k) * 8 + g];
    if (k < rank && r0 + g < R) part_w[((r0 + g) * rank + k) * nb + blockIdx.x] = t;
  }
}

// Wz[k][r] = the ordered sum of the U^T z partials; one warp per (r, k).
__global__ void k_lr_wz(const double* part, int nb, int rank, int64_t R, double* Wz) {
  const int64_t i = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const int lane = threadIdx.x & 31;
  if (i >= rank * R) return;
  double s = 0.0;
  for (int b = lane; b < nb; b += 32) s += part[i * nb + b];
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
  if (lane == 0) Wz[(i % rank) * R + i / rank] = s;
}

__global__ void k_lr_copy(const float* in, double* out, int64_t n) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) out[i] = (double)in[i];
}

inline bool al16(const void* p) { return ((uintptr_t)p & 15u) == 0; }

}  // namespace

bool lr_cg_setup(Ctx* c, const cola_linop* op, int64_t R, LrCg* L) {
  *L = LrCg{};
  if (op->kind != LK_SUM || op->kids.size() < 2 || op->kids.size() > 3) return false;
  const cola_linop *ks = nullptr, *dg = nullptr, *lr = nullptr;
  for (size_t i = 0; i < op->kids.size(); ++i) {
    const cola_linop* k = op->kids[i];
    const float co = (float)op->coeffs[i];
    if (k->kind == LK_KRONSUM && !ks) {
      ks = k;
      L->cs = co;
    } else if (k->kind == LK_DIAG && !dg) {
      dg = k;
      L->cd = co;
    } else if (k->kind == LK_LOWRANK && !lr) {
      lr = k;
      L->cu = op->coeffs[i];
    } else {
      return false;
    }
  }
  if (!ks || !lr || !ks->tridiag || ks->kids.size() != 2 || lr->data2) return false;
  const int64_t n1 = ks->kids[0]->rows, n2 = ks->kids[1]->rows;
  if (n2 % 4 != 0 || n1 * n2 >= ((int64_t)1 << 31) || lr->rank % 4 != 0 || lr->rank > kLrRank ||
      R > 65535)
    return false;
  L->U = leaf_ptr<float>(lr);
  L->bands = (const float*)ks->derived.at(DK_BAND32).p;
  if (dg) {
    L->d = leaf_ptr<float>(dg);
    L->dstride = dg->stride;
  }
  if (!al16(L->U) || (dg && dg->stride && !al16(L->d))) return false;
  L->n1 = (int)n1;
  L->n2 = (int)n2;
  L->rank = (int)lr->rank;
  // strips of up to 32 rows while the threads still fill most of the two blocks
  // an SM holds (2^20 points, 8 vectors: 32 rows, 256 blocks in one wave)
  int S = 32;
  while (S > 1 && (n1 + S - 1) / S * (n2 / 4) * R < (int64_t)c->num_sms * 400) S /= 2;
  L->S = S;
  const int64_t items = (n1 + S - 1) / S * (n2 / 4);
  L->nb_pq = (int)std::min<int64_t>((items + 255) / 256, 1024);
  const int64_t stages = (n1 * n2 + kLrRows - 1) / kLrRows;
  const int64_t want = std::max<int64_t>(1, std::min<int64_t>(stages, 2 * c->num_sms));
  L->rpb = (stages + want - 1) / want * kLrRows;
  L->nb_up = (int)((n1 * n2 + L->rpb - 1) / L->rpb);
  auto& ws = c->ws;
  L->q = (float*)ws.get("lrcg.q", 4 * (size_t)(n1 * n2) * R);
  L->p2 = (float*)ws.get("lrcg.p2", 4 * (size_t)(n1 * n2) * R);
  L->part = (double*)ws.get("lrcg.part", 8 * (size_t)L->nb_pq * R);
  L->part_rz = (double*)ws.get("lrcg.prz", 8 * (size_t)L->nb_up * R);
  L->part_rr = (double*)ws.get("lrcg.prr", 8 * (size_t)L->nb_up * R);
  L->part_w = (double*)ws.get("lrcg.pw", 8 * (size_t)L->nb_up * R * L->rank);
  L->W = (double*)ws.get("lrcg.W", 8 * (size_t)L->rank * R);
  L->Wz = (double*)ws.get("lrcg.Wz", 8 * (size_t)L->rank * R);
  L->w32 = (float*)ws.get("lrcg.w32", 4 * (size_t)L->rank * R);
  L->vtx = (double*)ws.get("lrcg.vtx", 8 * (size_t)kLowRankBlocks * L->rank * R);
  static bool attr[64] = {false};
  if (c->device >= 64 || !attr[c->device]) {
    COLA_CUDA(cudaFuncSetAttribute(k_lr_update, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                   (int)kLrSmem));
    if (c->device < 64) attr[c->device] = true;
  }
  L->on = true;
  return true;
}

// Wz = U^T z after z was replaced from outside the iteration.
void lr_cg_refresh(Ctx* c, const LrCg& L, const float* z, int64_t R) {
  lowrank_vtx<float>(c, L.U, z, (int64_t)L.n1 * L.n2, L.rank, R, L.w32, L.vtx);
  const int64_t n = (int64_t)L.rank * R;
  k_lr_copy<<<(unsigned)((n + 255) / 256), 256, 0, c->s>>>(L.w32, L.Wz, n);
  c->count_launch();
  COLA_CUDA(cudaGetLastError());
}

void lr_cg_step(Ctx* c, const LrCg& L, const float* p_old, float* p_new, float* r, float* x,
                const float* invd, CgState* st, int64_t R) {
  const int64_t N = (int64_t)L.n1 * L.n2;
  k_lr_pq<<<dim3(L.nb_pq, (unsigned)R), 256, 0, c->s>>>(L.n1, L.n2, L.S, L.bands, r, invd, p_old,
                                                        p_new, L.q, L.d, L.dstride, L.cs, L.cd,
                                                        st, L.part);
  c->count_launch();
  k_lr_alpha<<<(unsigned)R, 256, 0, c->s>>>(st, L.part, L.nb_pq, L.rank, R, L.Wz, L.W, L.cu);
  c->count_launch();
  k_lr_update<<<dim3(L.nb_up, (unsigned)((R + 7) / 8)), 256, kLrSmem, c->s>>>(
      L.U, L.rank, N, R, L.rpb, L.W, L.q, p_new, r, x, invd, (float)L.cu, st, L.part_rz,
      L.part_rr, L.part_w);
  c->count_launch();
  k_lr_wz<<<(unsigned)((L.rank * R * 32 + 255) / 256), 256, 0, c->s>>>(L.part_w, L.nb_up, L.rank,
                                                                       R, L.Wz);
  c->count_launch();
  COLA_CUDA(cudaGetLastError());
}

}  // namespace cola
