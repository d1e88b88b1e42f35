// Sum-factorised curved mass term (Sec. 5.2, "mass residual"):
//   v_c = u_{i+1,c} - delta_{i0} u_{0,c},  T_c = (V (x) V (x) V) v_c at the (p+2)^3 Gauss points,
//   W_c = sum_d w_g G_cd T_d,  R_c = mat_f (V^T (x) V^T (x) V^T) W_c,   V[g][j] = L_j(x_g).
//
// One CTA takes a few elements; a job is one (element, field, temporal mode).  Three passes:
//   A  one thread per (job, c, l) plane: x and y contraction of its N x N coefficients in
//      registers, NQ^2 results to shared memory;
//   B  one thread per (job, Gauss column (x, y)): z contraction of the three components, the
//      metric, and the z contraction back, in place;
//   C  one thread per plane: y and x contraction back in registers, then the store.
// So a value crosses shared memory twice on its way instead of seven times (one pass per
// contraction).  Every 1-D contraction is split into even and odd parts: the Gauss points are
// symmetric and L_j(1 - x) = (-1)^j L_j(x), and the odd part is kept relative to L_1, so a forward
// line of N coefficients takes floor(NQ/2) N + ... operations instead of N NQ (N = 4: 9 for 20, N = 8:
// 35 for 72) and a backward line 13 for 20 and 43 for 72.  Shared planes have odd strides: lanes
// on consecutive planes or columns hit different banks.
//
// FP64 is bound by the FP64 pipe (tables from shared memory, sums as three-operand FMAs, see
// PassOps); FP32 by the shared-memory pipe and HBM.  The next batch's coefficients and metric arrive
// by asynchronous copies behind passes B and C.  Against one pass per contraction on the FP64 pipe
// (and 3xTF32 tensor-core products with M = 128, N = 16 tiles in FP32, whose staging through shared
// memory cost more than the products saved), 32^3 elements: FP64 p = 3, q = 2 2.30 -> 1.33 ms; FP32
// p = 5, q = 4 2.88 -> 0.57 ms; FP32 p = 7, q = 6 at 16 x 15 x 17 elements 0.99 -> 0.32 ms.
#include <cuda_runtime.h>
#include <stdint.h>

#include <atomic>

#include "curved.cuh"

namespace stm {

namespace {

template <typename T, int P>
struct MassTab {
  static constexpr int N = P + 1, H = (P + 2) / 2;  // H pairs of Gauss points, then the centre (P odd)
  T L[N][H + 1];  // L_j(x_g), g < H, and at the centre (zero for odd j)
  T r[N][H + 1];  // odd j: L_j(x_g) / L_1(x_g), g < H
};

// CTA shape of degree (P, Q): `epc` elements, `jobs` jobs per batch (all of them when epc > 1) and one
// thread per plane of a batch.
struct MassShape {
  int epc, jobs, threads;
  size_t smem;
};

template <typename T, int P>
struct MassDims {
  static constexpr int N = P + 1, NQ = P + 2, N2 = N * N, N3 = N2 * N, NQ2 = NQ * NQ, NQ3 = NQ2 * NQ;
  static constexpr int PV = N2 | 1, PT = NQ2 | 1;  // plane strides
  // largest block, and the shared memory per CTA that leaves enough CTAs per SM.  Measured at
  // 32^3 elements: FP64 p = 3, q = 2 1.33 ms with 128 threads and 56 KB, 1.41 ms with 256 and 75 KB;
  // FP32 p = 5, q = 4 0.565 ms with 256 and 75 KB, 0.60 ms with 128 and 56 KB
  static constexpr int MAXT = sizeof(T) == 8 ? 128 : 256;
  static constexpr size_t WANT = sizeof(T) == 8 ? 56 * 1024 : 75 * 1024;
  static constexpr int TAB = sizeof(T) == 8 ? 2 * N * (P / 2 + 2) + 4 : 0;  // FP64: tables and constants
};

constexpr int kMassJobs = 64;  // largest batch

// Asynchronous copy of BYTES (4, 8 or 16, both addresses aligned to it) from global to shared memory.
template <int BYTES>
__device__ __forceinline__ void copy_async(void* dst, const void* src) {
  if constexpr (BYTES == 16)
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"((uint32_t)__cvta_generic_to_shared(dst)), "l"(src)
                 : "memory");
  else
    asm volatile("cp.async.ca.shared.global [%0], [%1], %2;\n" ::"r"((uint32_t)__cvta_generic_to_shared(dst)),
                 "l"(src), "n"(BYTES)
                 : "memory");
}
__device__ __forceinline__ void copy_async_wait() { asm volatile("cp.async.wait_all;\n" ::: "memory"); }

template <typename T, int P>
// registers: 128 a thread but for the FP64 planes of N >= 5
__global__ void __launch_bounds__(MassDims<T, P>::MAXT, sizeof(T) == 4 ? 2 : (P <= 3 ? 4 : 1)) k_mass(const T* __restrict__ um, int64_t um_es, int64_t um_cs,
                                              const T* __restrict__ u0, int64_t u0_es, int64_t u0_cs,
                                              const T* __restrict__ Gw, const T* __restrict__ eps,
                                              const T* __restrict__ mu, const MassTab<T, P> tb, int Q, int epc,
                                              int jobs, int64_t ne, T* __restrict__ R, const int32_t* skip) {
  if (skip && *skip) return;
  using D = MassDims<T, P>;
  constexpr int N = D::N, NQ = D::NQ, N2 = D::N2, N3 = D::N3, NQ2 = D::NQ2, NQ3 = D::NQ3, PV = D::PV, PT = D::PT;
  constexpr int H = NQ / 2;
  constexpr bool C = NQ & 1;
  constexpr bool F64 = sizeof(T) == 8;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  T* g6 = reinterpret_cast<T*>(smem_raw);  // [epc][6][NQ3]
  T* vb = g6 + epc * 6 * NQ3;              // planes of the batch, stride PV: coefficients
  T* tb2 = vb + jobs * 3 * N * PV;         // planes of the batch, stride PT: columns (PV: results)
  T* ub = tb2 + jobs * 3 * N * PT;         // planes (element, field, c, l), stride PV: slab start
  T* tab = ub + (u0 ? epc * 6 * N * PV : 0);
  // per job of the batch (double-buffered: the next batch is filled while one runs)
  __shared__ int64_t j_R[2][kMassJobs];
  __shared__ T j_mat[2][kMassJobs];
  __shared__ int j_u0[2][kMassJobs];       // element * 2 + field of a job with i = 0, else -1
  const int tid = threadIdx.x, nt = blockDim.x;
  if constexpr (F64) {
    for (int k = tid; k < N * (H + 1); k += nt) {
      tab[k] = (&tb.L[0][0])[k];
      tab[N * (H + 1) + k] = (&tb.r[0][0])[k];
    }
    if (tid < 3) tab[2 * N * (H + 1) + tid] = tid == 0 ? T(1) : (tid == 1 ? T(-1) : -T(0));
    __syncthreads();
  }
  // coefficients: FP64 from shared memory (a constant-bank operand slows the FP64 pipe), FP32 from
  // the constant bank
  auto L = [&](int j, int g) -> T { return F64 ? tab[j * (H + 1) + g] : tb.L[j][g]; };
  auto Rr = [&](int j, int g) -> T { return F64 ? tab[(N + j) * (H + 1) + g] : tb.r[j][g]; };
  PassOps<T> op{T(1), T(-1), -T(0)};
  if constexpr (F64) op = PassOps<T>{tab[2 * N * (H + 1)], tab[2 * N * (H + 1) + 1], tab[2 * N * (H + 1) + 2]};
  // forward line: values at the pair g (lo at x_g, hi at 1 - x_g) and at the centre
  auto fwd_pair = [&](const T* u, int st, int g, T& lo, T& hi) {
    T e = u[0];
#pragma unroll
    for (int j = 2; j < N; j += 2) e = fma(L(j, g), u[j * st], e);
    if constexpr (N > 1) {
      T o = u[st];
#pragma unroll
      for (int j = 3; j < N; j += 2) o = fma(Rr(j, g), u[j * st], o);
      const T l1 = L(1, g);
      lo = fma(l1, o, e);
      hi = fma(-l1, o, e);
    } else {
      lo = hi = e;
    }
  };
  auto fwd_mid = [&](const T* u, int st) -> T {
    T e = u[0];
#pragma unroll
    for (int j = 2; j < N; j += 2) e = fma(L(j, H), u[j * st], e);
    return e;
  };
  // backward: adds the pair (lo, hi) at g, or the centre value, to the coefficients a[j * st]
  auto bwd_pair = [&](T* a, int st, int g, T lo, T hi, bool first) {
    const T s = op.add(lo, hi), d = op.sub(lo, hi);
    a[0] = first ? s : op.add(a[0], s);
#pragma unroll
    for (int j = 1; j < N; ++j) {
      const T w = (j & 1) ? d : s;
      a[j * st] = first ? op.mul(L(j, g), w) : fma(L(j, g), w, a[j * st]);
    }
  };
  auto bwd_mid = [&](T* a, int st, T v, bool first) {
    a[0] = first ? v : op.add(a[0], v);
#pragma unroll
    for (int j = 1; j < N; ++j) {
      if (j & 1) {
        if (first) a[j * st] = T(0);
      } else {
        a[j * st] = first ? op.mul(L(j, H), v) : fma(L(j, H), v, a[j * st]);
      }
    }
  };
  const int jpe = 2 * Q, lane = tid & 31, warp = tid >> 5, nw = nt >> 5;
  // issues the asynchronous copies of batch b0 of the group at e0 into slot sl; a warp per row of
  // N3 contiguous coefficients, so all its copies are in flight at once
  auto fetch = [&](int64_t e0, int b0, int sl) {
    const int nel = (int)(ne - e0 < epc ? ne - e0 : epc);
    const int nj = nel * jpe - b0 < jobs ? nel * jpe - b0 : jobs;
    auto job = [&](int jl, int64_t& e, int& f, int& i, int& el) {
      const int jg = b0 + jl;
      el = epc > 1 ? jg / jpe : 0;
      const int fi = jg - el * jpe;
      f = fi >= Q ? 1 : 0;
      i = fi - f * Q;
      e = e0 + el;
    };
    int64_t e;
    int f, i, el;
    if (tid < nj) {
      job(tid, e, f, i, el);
      j_R[sl][tid] = (e * 6 + f * 3) * (int64_t)(Q * N3) + (int64_t)i * N3;
      j_mat[sl][tid] = f == 0 ? eps[e] : mu[e];
      j_u0[sl][tid] = (i == 0 && u0) ? el * 2 + f : -1;
    }
    for (int row = warp; row < nj * 3; row += nw) {
      const int jl = row / 3, c = row - 3 * jl;
      job(jl, e, f, i, el);
      const T* src = um + e * um_es + (f * 3 + c) * um_cs + (int64_t)i * N3;
      T* dst = vb + row * N * PV;
#pragma unroll
      for (int k = 0; k < (N3 + 31) / 32; ++k) {
        const int x = lane + 32 * k;
        if (x < N3) copy_async<sizeof(T)>(dst + x + (PV > N2 ? x / N2 : 0), src + x);
      }
      if (u0 && i == 0) {
        const T* s0 = u0 + e * u0_es + (f * 3 + c) * u0_cs;
        T* d0 = ub + ((el * 2 + f) * 3 + c) * N * PV;
#pragma unroll
        for (int k = 0; k < (N3 + 31) / 32; ++k) {
          const int x = lane + 32 * k;
          if (x < N3) copy_async<sizeof(T)>(d0 + x + (PV > N2 ? x / N2 : 0), s0 + x);
        }
      }
    }
  };
  // the metric of the group at e0: pairs of values (6 NQ3 is even, so every block starts aligned)
  auto fetch_metric = [&](int64_t e0) {
    const int nel = (int)(ne - e0 < epc ? ne - e0 : epc);
    const T* src = Gw + e0 * 6 * NQ3;
    for (int k = tid; k < nel * 3 * NQ3; k += nt) copy_async<2 * sizeof(T)>(g6 + 2 * k, src + 2 * k);
  };
  int64_t e0 = (int64_t)blockIdx.x * epc;
  int b0 = 0, sl = 0;
  if (e0 < ne) {
    fetch(e0, 0, 0);
    fetch_metric(e0);
  }
  while (e0 < ne) {
    {
      const int nel = (int)(ne - e0 < epc ? ne - e0 : epc), total = nel * jpe;
      const int nj = total - b0 < jobs ? total - b0 : jobs;
      // the batch after this one
      int64_t e1 = e0;
      int b1 = b0 + jobs;
      if (b1 >= total) {
        b1 = 0;
        e1 = e0 + (int64_t)gridDim.x * epc;
      }
      copy_async_wait();
      __syncthreads();
      const bool plane = tid < nj * 3 * N;  // this thread's plane: (job, c, l) = tid
      {
        T u[N2];
        if (plane) {
#pragma unroll
          for (int k = 0; k < N2; ++k) u[k] = vb[tid * PV + k];
          const int us = j_u0[sl][tid / (3 * N)];
          if (us >= 0) {
            const T* w = ub + (us * 3 * N + tid % (3 * N)) * PV;
#pragma unroll
            for (int k = 0; k < N2; ++k) u[k] = op.sub(u[k], w[k]);
          }
          T* o = tb2 + tid * PT;
          auto column = [&](const T* t, int gx) {  // y contraction of one x column
#pragma unroll
            for (int g = 0; g < H; ++g) {
              T lo, hi;
              fwd_pair(t, 1, g, lo, hi);
              o[g * NQ + gx] = lo;
              o[(NQ - 1 - g) * NQ + gx] = hi;
            }
            if constexpr (C) o[H * NQ + gx] = fwd_mid(t, 1);
          };
#pragma unroll
          for (int g = 0; g < H; ++g) {
            T lo[N], hi[N];
#pragma unroll
            for (int k = 0; k < N; ++k) fwd_pair(u + k * N, 1, g, lo[k], hi[k]);
            column(lo, g);
            column(hi, NQ - 1 - g);
          }
          if constexpr (C) {
            T mid[N];
#pragma unroll
            for (int k = 0; k < N; ++k) mid[k] = fwd_mid(u + k * N, 1);
            column(mid, H);
          }
        }
      }
      __syncthreads();
      if (e1 < ne) fetch(e1, b1, sl ^ 1);
      // z, the metric, z back: one Gauss column, planes (c, l) PT apart
      for (int k = tid; k < nj * NQ2; k += nt) {
        const int jl = k / NQ2, col = k - jl * NQ2;
        const T* G = g6 + (epc > 1 ? (b0 + jl) / jpe : 0) * 6 * NQ3 + col;
        T* B = tb2 + jl * 3 * N * PT + col;
        T v[3][N], a[3][N];
#pragma unroll
        for (int c = 0; c < 3; ++c)
#pragma unroll
          for (int l = 0; l < N; ++l) v[c][l] = B[(c * N + l) * PT];
        auto metric = [&](int gz, const T* t, T* w) {
          const T* Gz = G + gz * NQ2;
          const T gxx = Gz[0], gyy = Gz[NQ3], gzz = Gz[2 * NQ3];
          const T gxy = Gz[3 * NQ3], gxz = Gz[4 * NQ3], gyz = Gz[5 * NQ3];
          w[0] = fma(gxx, t[0], fma(gxy, t[1], op.mul(gxz, t[2])));
          w[1] = fma(gxy, t[0], fma(gyy, t[1], op.mul(gyz, t[2])));
          w[2] = fma(gxz, t[0], fma(gyz, t[1], op.mul(gzz, t[2])));
        };
#pragma unroll
        for (int g = 0; g < H; ++g) {
          T lo[3], hi[3], wl[3], wh[3];
#pragma unroll
          for (int c = 0; c < 3; ++c) fwd_pair(v[c], 1, g, lo[c], hi[c]);
          metric(g, lo, wl);
          metric(NQ - 1 - g, hi, wh);
#pragma unroll
          for (int c = 0; c < 3; ++c) bwd_pair(a[c], 1, g, wl[c], wh[c], g == 0);
        }
        if constexpr (C) {
          T t[3], w[3];
#pragma unroll
          for (int c = 0; c < 3; ++c) t[c] = fwd_mid(v[c], 1);
          metric(H, t, w);
#pragma unroll
          for (int c = 0; c < 3; ++c) bwd_mid(a[c], 1, w[c], H == 0);
        }
#pragma unroll
        for (int c = 0; c < 3; ++c)
#pragma unroll
          for (int l = 0; l < N; ++l) B[(c * N + l) * PT] = a[c][l];
      }
      __syncthreads();
      if (e1 < ne && b1 == 0) fetch_metric(e1);
      {
        T acc[N2];
        if (plane) {
          const T* t = tb2 + tid * PT;
          auto column = [&](int gx, T* r) {  // y contraction back of one x column
#pragma unroll
            for (int g = 0; g < H; ++g) bwd_pair(r, 1, g, t[g * NQ + gx], t[(NQ - 1 - g) * NQ + gx], g == 0);
            if constexpr (C) bwd_mid(r, 1, t[H * NQ + gx], H == 0);
          };
#pragma unroll
          for (int g = 0; g < H; ++g) {
            T lo[N], hi[N];
            column(g, lo);
            column(NQ - 1 - g, hi);
#pragma unroll
            for (int k = 0; k < N; ++k) bwd_pair(acc + k * N, 1, g, lo[k], hi[k], g == 0);
          }
          if constexpr (C) {
            T mid[N];
            column(H, mid);
#pragma unroll
            for (int k = 0; k < N; ++k) bwd_mid(acc + k * N, 1, mid[k], H == 0);
          }
        }
        __syncthreads();
        if (plane) {
          const T mat = j_mat[sl][tid / (3 * N)];
#pragma unroll
          for (int k = 0; k < N2; ++k) tb2[tid * PV + k] = op.mul(acc[k], mat);
        }
      }
      __syncthreads();
      for (int row = warp; row < nj * 3; row += nw) {
        const int jl = row / 3, c = row - 3 * jl;
        T* dst = R + j_R[sl][jl] + (int64_t)c * (Q * N3);
        const T* src = tb2 + row * N * PV;
#pragma unroll
        for (int k = 0; k < (N3 + 31) / 32; ++k) {
          const int x = lane + 32 * k;
          if (x < N3) dst[x] = src[x + (PV > N2 ? x / N2 : 0)];
        }
      }
      e0 = e1;
      b0 = b1;
      sl ^= 1;
    }
  }
}

// Shape with the least idle lanes in passes A/C (one plane per thread) and B (columns over the same
// threads), among those whose shared memory leaves `want` CTAs per SM, else the smallest one.
template <typename T, int P>
MassShape mass_shape(int Q, bool start) {
  using D = MassDims<T, P>;
  auto smem = [&](int epc, int jobs) {
    return sizeof(T) * ((size_t)epc * 6 * (D::NQ3 + (start ? D::N * D::PV : 0)) +
                        (size_t)jobs * 3 * D::N * (D::PT + D::PV) + D::TAB);
  };
  const size_t want = D::WANT, most = 200 * 1024;
  MassShape best{1, 1, 32, smem(1, 1)};
  double best_score = -1.0;
  for (int pass = 0; pass < 2 && best_score < 0; ++pass)
    for (int epc = 1; epc <= 8; ++epc)
      for (int jobs = 1; jobs <= epc * 2 * Q && jobs <= kMassJobs; ++jobs) {
        if (epc > 1 ? jobs != epc * 2 * Q : (2 * Q) % jobs != 0) continue;
        const int planes = 3 * D::N * jobs, threads = (planes + 31) / 32 * 32;
        if (threads > D::MAXT || smem(epc, jobs) > (pass ? most : want)) continue;
        const int cols = D::NQ2 * jobs, rounds = (cols + threads - 1) / threads;
        const double a = (double)planes / threads, b = (double)cols / (rounds * threads);
        // small CTAs spend their time between barriers
        const double score = (0.6 * a + 0.4 * b) * (threads >= 96 ? 1.0 : 0.6 + 0.4 * threads / 96);
        if (score > best_score) {
          best_score = score;
          best = MassShape{epc, jobs, threads, smem(epc, jobs)};
        }
      }
  return best;
}

template <typename T, int P>
int mass_p(int Q, const T* um, int64_t um_es, int64_t um_cs, const T* u0, int64_t u0_es, int64_t u0_cs, const T* Gw,
           const T* eps, const T* mu, const CurvedTables& ct, int64_t ne, T* R, cudaStream_t s, const int32_t* skip) {
  static std::atomic<uint64_t> configured_devices{0};
  once_per_device(configured_devices, [&] {
    cudaFuncSetAttribute(k_mass<T, P>, cudaFuncAttributeMaxDynamicSharedMemorySize, 200 * 1024);
  });
  const MassShape sh = mass_shape<T, P>(Q, u0 != nullptr);
  MassTab<T, P> tb{};
  constexpr int N = P + 1, H = (P + 2) / 2;
  for (int j = 0; j < N; ++j) {
    for (int g = 0; g < H; ++g) {
      tb.L[j][g] = (T)ct.Lq[j][g];
      tb.r[j][g] = (j & 1) ? (T)(ct.Lq[j][g] / ct.Lq[1][g]) : T(0);
    }
    tb.L[j][H] = ((P + 2) & 1) && !(j & 1) ? (T)ct.Lq[j][H] : T(0);
  }
  // grid-stride over elements, one wave of co-resident CTAs (a skipped launch costs one wave)
  static std::atomic<int> cap[2][kMaxQ][64];
  const int grid = wave_grid(k_mass<T, P>, sh.threads, sh.smem, (ne + sh.epc - 1) / sh.epc, cap[u0 ? 1 : 0][Q - 1]);
  k_mass<T, P><<<grid, sh.threads, sh.smem, s>>>(um, um_es, um_cs, u0, u0_es, u0_cs, Gw, eps, mu, tb, Q, sh.epc,
                                                  sh.jobs, ne, R, skip);
  return (int)cudaGetLastError();
}

}  // namespace

template <typename T>
int launch_mass_curved(int P, int Q, const T* um, int64_t um_es, int64_t um_cs, const T* u0, int64_t u0_es,
                       int64_t u0_cs, const T* Gw, const T* eps, const T* mu, const CurvedTables& ct, int64_t ne, T* R,
                       cudaStream_t s, const int32_t* skip) {
  if (Q < 1 || Q > kMaxQ) return (int)cudaErrorInvalidValue;
  switch (P) {
#define STM_MP(p) \
  case p: return mass_p<T, p>(Q, um, um_es, um_cs, u0, u0_es, u0_cs, Gw, eps, mu, ct, ne, R, s, skip);
    STM_MP(0) STM_MP(1) STM_MP(2) STM_MP(3) STM_MP(4) STM_MP(5) STM_MP(6) STM_MP(7)
#undef STM_MP
    default: return (int)cudaErrorInvalidValue;
  }
}

#ifndef STM_MASS_T
#error "compile with -DSTM_MASS_T=float or double"
#endif
template int launch_mass_curved<STM_MASS_T>(int, int, const STM_MASS_T*, int64_t, int64_t, const STM_MASS_T*, int64_t,
                                            int64_t, const STM_MASS_T*, const STM_MASS_T*, const STM_MASS_T*,
                                            const CurvedTables&, int64_t, STM_MASS_T*, cudaStream_t, const int32_t*);

}  // namespace stm
