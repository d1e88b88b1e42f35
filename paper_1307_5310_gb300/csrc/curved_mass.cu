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

#include <algorithm>
#include <atomic>
#include <cmath>

#include "curved.cuh"

namespace stm {

namespace {

template <typename T, int P>
struct MassTab {
  static constexpr int N = P + 1, H = (P + 2) / 2;  // H pairs of Gauss points, then the centre (P odd)
  T L[N][H + 1];  // L_j(x_g), g < H, and at the centre (zero for odd j)
  T r[N][H + 1];  // odd j: L_j(x_g) / L_1(x_g), g < H
};

template <typename T, int P>
struct MassDims {
  static constexpr int N = P + 1, NQ = P + 2, N2 = N * N, N3 = N2 * N, NQ2 = NQ * NQ, NQ3 = NQ2 * NQ;
  static constexpr int PV = N2 | 1, PT = NQ2 | 1;  // plane strides
  // largest block per part, and the shared memory per CTA that leaves enough CTAs per SM on meshes
  // that fill the GPU.  Measured at 32^3 elements: FP64 p = 3, q = 2 1.33 ms with 128 threads and 56 KB, 1.41 ms with 256 and 75 KB;
  // FP32 p = 5, q = 4 0.565 ms with 256 and 75 KB, 0.60 ms with 128 and 56 KB
  static constexpr int MAXT = sizeof(T) == 8 ? 128 : 256;
  static constexpr size_t WANT = sizeof(T) == 8 ? 56 * 1024 : 75 * 1024;
  // threads per Gauss column in pass B, by PARTS: with two threads per plane p <= 4 runs meshes that
  // wait for one CTA's chain, where the extra forward contractions cost less than the chain they cut
  static constexpr int BP[2] = {1, P <= 4 ? 3 : 1};
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

// PARTS: threads per plane in passes A and C.  With two, pass A splits the Gauss columns of a plane
// between them and pass C the coefficient rows by parity (an even row needs only the sums of a pair of
// Gauss points, an odd row only the differences), so no operation is done twice.
// SPLIT: several CTAs may share an element's jobs (FP32 meshes that fill the GPU run without: at p = 0 the
// unit arithmetic costs 6%).
// Registers: 128 a thread but for the FP64 planes of N >= 5.
template <typename T, int P, int PARTS, bool SPLIT>
__global__ void __launch_bounds__(MassDims<T, P>::MAXT * PARTS,
                                  PARTS == 2 ? (P <= 3 ? 2 : 1) : (sizeof(T) == 4 ? 2 : (P <= 3 ? 4 : 1)))
    k_mass(const T* __restrict__ um, int64_t um_es, int64_t um_cs,
                                              const T* __restrict__ u0, int64_t u0_es, int64_t u0_cs,
                                              const T* __restrict__ Gw, const T* __restrict__ eps,
                                              const T* __restrict__ mu, const MassTab<T, P> tb, int Q, int epc,
                                              int jobs, uint32_t split, uint32_t units, int64_t ne, T* __restrict__ R,
                                              const int32_t* skip) {
  if (skip && *skip) return;
  using D = MassDims<T, P>;
  constexpr int N = D::N, NQ = D::NQ, N2 = D::N2, N3 = D::N3, NQ2 = D::NQ2, NQ3 = D::NQ3, PV = D::PV, PT = D::PT;
  constexpr int H = NQ / 2;
  constexpr bool C = NQ & 1;
  constexpr bool F64 = sizeof(T) == 8;
  constexpr int BP = D::BP[PARTS - 1];
  extern __shared__ __align__(16) unsigned char smem_raw[];
  T* g6 = reinterpret_cast<T*>(smem_raw);  // [epc][6][NQ3]
  T* vb = g6 + epc * 6 * NQ3;              // planes of the batch, stride PV: coefficients
  T* tb2 = vb + jobs * 3 * N * PV;         // planes of the batch, stride PT: columns (PV: results)
  T* ub = tb2 + jobs * 3 * N * PT;         // planes (slot, c, l) of the jobs with i = 0, stride PV: slab start
  const bool one_start = jobs <= Q;        // at most one such job in a batch (epc = 1), else slot el * 2 + f
  T* tab = ub + (u0 ? (one_start ? 1 : 2 * epc) * 3 * N * PV : 0);
  // per job of the batch (double-buffered: the next batch is filled while one runs)
  __shared__ int64_t j_R[2][kMassJobs];
  __shared__ T j_mat[2][kMassJobs];
  __shared__ int j_u0[2][kMassJobs];       // slot in ub of a job with i = 0, else -1
  const int tid = threadIdx.x, nt = blockDim.x;
  // coefficients: FP64 from shared memory (a constant-bank operand slows the FP64 pipe), FP32 from
  // the constant bank
  auto L = [&](int j, int g) -> T { return F64 ? tab[j * (H + 1) + g] : tb.L[j][g]; };
  auto Rr = [&](int j, int g) -> T { return F64 ? tab[(N + j) * (H + 1) + g] : tb.r[j][g]; };
  PassOps<T> op{T(1), T(-1), -T(0)};
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
      j_u0[sl][tid] = (i == 0 && u0) ? (one_start ? 0 : el * 2 + f) : -1;
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
        T* d0 = ub + ((one_start ? 0 : el * 2 + f) * 3 + c) * N * PV;
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
  // unit w: batches w % split, w % split + split, ... of the element group w / split (32-bit: element
  // numbers are, and only meshes of few elements are split)
  uint32_t w = blockIdx.x;
  int64_t e0 = (int64_t)w * epc;
  int b0 = 0, sl = 0;
  auto unit = [&](uint32_t u, int64_t& e, int& b) {
    e = (int64_t)(u / split) * epc;
    b = (int)(u % split) * jobs;
  };
  if constexpr (SPLIT) unit(w, e0, b0);
  if (SPLIT ? w < units : e0 < ne) {
    fetch(e0, b0, 0);
    fetch_metric(e0);
  }
  if constexpr (F64) {  // behind the first copies
    for (int k = tid; k < N * (H + 1); k += nt) {
      tab[k] = (&tb.L[0][0])[k];
      tab[N * (H + 1) + k] = (&tb.r[0][0])[k];
    }
    if (tid < 3) tab[2 * N * (H + 1) + tid] = tid == 0 ? T(1) : (tid == 1 ? T(-1) : -T(0));
    __syncthreads();
    op = PassOps<T>{tab[2 * N * (H + 1)], tab[2 * N * (H + 1) + 1], tab[2 * N * (H + 1) + 2]};
  }
  while (SPLIT ? w < units : e0 < ne) {
    {
      const int nel = (int)(ne - e0 < epc ? ne - e0 : epc), total = nel * jpe;
      const int nj = total - b0 < jobs ? total - b0 : jobs;
      // the batch after this one
      uint32_t w1 = w;
      int64_t e1 = e0;
      int b1 = b0 + (SPLIT ? (int)split : 1) * jobs;
      if (b1 >= total) {
        if constexpr (SPLIT) {
          w1 = w + gridDim.x;
          unit(w1, e1, b1);
        } else {
          b1 = 0;
          e1 = e0 + (int64_t)gridDim.x * epc;
        }
      }
      copy_async_wait();
      __syncthreads();
      // this thread's plane: (job, c, l) = pl, and its part of it
      const int np = nj * 3 * N, part = PARTS == 2 && tid >= np ? 1 : 0, pl = tid - part * np;
      const bool plane = pl < np;
      {
        T u[N2];
        if (plane) {
#pragma unroll
          for (int k = 0; k < N2; ++k) u[k] = vb[pl * PV + k];
          const int us = j_u0[sl][pl / (3 * N)];
          if (us >= 0) {
            const T* w = ub + (us * 3 * N + pl % (3 * N)) * PV;
#pragma unroll
            for (int k = 0; k < N2; ++k) u[k] = op.sub(u[k], w[k]);
          }
          T* o = tb2 + pl * PT;
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
          auto pair = [&](int g) {
            T lo[N], hi[N];
#pragma unroll
            for (int k = 0; k < N; ++k) fwd_pair(u + k * N, 1, g, lo[k], hi[k]);
            column(lo, g);
            column(hi, NQ - 1 - g);
          };
          if constexpr (PARTS == 1) {
#pragma unroll
            for (int g = 0; g < H; ++g) pair(g);
          } else {
#pragma unroll 1
            for (int g = part; g < H; g += 2) pair(g);
          }
          if (C && (PARTS == 1 || part == (H & 1))) {
            T mid[N];
#pragma unroll
            for (int k = 0; k < N; ++k) mid[k] = fwd_mid(u + k * N, 1);
            column(mid, H);
          }
        }
      }
      __syncthreads();
      const bool more = SPLIT ? w1 < units : e1 < ne;
      if (more) fetch(e1, b1, sl ^ 1);
      // z, the metric, z back: one Gauss column, planes (c, l) PT apart.  BP = 3: a thread per column
      // and result component (c0), each with its own forward contractions; the column is read by all
      // three before one of them stores
      const int per = nt / BP;
      for (int k0 = 0; k0 < nj * NQ2; k0 += per) {
        const int k = k0 + tid / BP, c0 = BP == 1 ? 0 : tid % BP;
        const bool mine = BP == 1 || (tid < per * BP && k < nj * NQ2);
        if (BP == 1 && k >= nj * NQ2) break;
        const int jl = k / NQ2, col = k - jl * NQ2;
        const T* G = g6 + (epc > 1 ? (b0 + jl) / jpe : 0) * 6 * NQ3 + col;
        T* B = tb2 + jl * 3 * N * PT + col;
        T v[3][N], a[3 / BP][N];
        if (mine) {
#pragma unroll
          for (int c = 0; c < 3; ++c)
#pragma unroll
            for (int l = 0; l < N; ++l) v[c][l] = B[(c * N + l) * PT];
        }
        if constexpr (BP > 1) __syncthreads();
        if (!mine) continue;
        auto metric = [&](int gz, const T* t, T* w) {
          const T* Gz = G + gz * NQ2;
          if constexpr (BP == 1) {
            const T gxx = Gz[0], gyy = Gz[NQ3], gzz = Gz[2 * NQ3];
            const T gxy = Gz[3 * NQ3], gxz = Gz[4 * NQ3], gyz = Gz[5 * NQ3];
            w[0] = fma(gxx, t[0], fma(gxy, t[1], op.mul(gxz, t[2])));
            w[1] = fma(gxy, t[0], fma(gyy, t[1], op.mul(gyz, t[2])));
            w[2] = fma(gxz, t[0], fma(gyz, t[1], op.mul(gzz, t[2])));
          } else {  // row c0
            const int m0 = c0 == 0 ? 0 : c0 + 2, m1 = c0 == 0 ? 3 : (c0 == 1 ? 1 : 5), m2 = c0 == 2 ? 2 : c0 + 4;
            w[0] = fma(Gz[m0 * NQ3], t[0], fma(Gz[m1 * NQ3], t[1], op.mul(Gz[m2 * NQ3], t[2])));
          }
        };
#pragma unroll
        for (int g = 0; g < H; ++g) {
          T lo[3], hi[3], wl[3 / BP], wh[3 / BP];
#pragma unroll
          for (int c = 0; c < 3; ++c) fwd_pair(v[c], 1, g, lo[c], hi[c]);
          metric(g, lo, wl);
          metric(NQ - 1 - g, hi, wh);
#pragma unroll
          for (int c = 0; c < 3 / BP; ++c) bwd_pair(a[c], 1, g, wl[c], wh[c], g == 0);
        }
        if constexpr (C) {
          T t[3], w[3 / BP];
#pragma unroll
          for (int c = 0; c < 3; ++c) t[c] = fwd_mid(v[c], 1);
          metric(H, t, w);
#pragma unroll
          for (int c = 0; c < 3 / BP; ++c) bwd_mid(a[c], 1, w[c], H == 0);
        }
#pragma unroll
        for (int c = 0; c < 3 / BP; ++c)
#pragma unroll
          for (int l = 0; l < N; ++l) B[((c0 + c) * N + l) * PT] = a[c][l];
      }
      __syncthreads();
      if (more && (SPLIT ? w1 != w : b1 == 0)) fetch_metric(e1);
      {
        // rows of this thread: all N, or with two parts k = 2 kk + part
        constexpr int NK = PARTS == 1 ? N : (N + 1) / 2;
        T acc[NK * N];
        if (plane) {
          const T* t = tb2 + pl * PT;
          const T sgn = part ? -op.one : op.one;
          auto column = [&](int gx, T* r) {  // y contraction back of one x column
            if constexpr (PARTS == 1) {
#pragma unroll
              for (int g = 0; g < H; ++g) bwd_pair(r, 1, g, t[g * NQ + gx], t[(NQ - 1 - g) * NQ + gx], g == 0);
              if constexpr (C) bwd_mid(r, 1, t[H * NQ + gx], H == 0);
            } else {
              // even rows take the sums, odd rows the differences (L_k = 0 at the centre for odd
              // k); a row beyond the last (N odd) repeats the last one and is not stored
#pragma unroll
              for (int g = 0; g < H + (C ? 1 : 0); ++g) {
                if (g == H && part) break;
                const T w = g < H ? fma(t[(NQ - 1 - g) * NQ + gx], sgn, t[g * NQ + gx]) : t[g * NQ + gx];
#pragma unroll
                for (int kk = 0; kk < NK; ++kk) {
                  const T l = L(2 * kk + part < N ? 2 * kk + part : N - 1, g);
                  r[kk] = g == 0 ? op.mul(l, w) : fma(l, w, r[kk]);
                }
              }
            }
          };
#pragma unroll
          for (int g = 0; g < H; ++g) {
            T lo[NK], hi[NK];
            column(g, lo);
            column(NQ - 1 - g, hi);
#pragma unroll
            for (int k = 0; k < NK; ++k) bwd_pair(acc + k * N, 1, g, lo[k], hi[k], g == 0);
          }
          if constexpr (C) {
            T mid[NK];
            column(H, mid);
#pragma unroll
            for (int k = 0; k < NK; ++k) bwd_mid(acc + k * N, 1, mid[k], H == 0);
          }
        }
        __syncthreads();
        if (plane) {
          const T mat = j_mat[sl][pl / (3 * N)];
#pragma unroll
          for (int kk = 0; kk < NK; ++kk) {
            const int k = PARTS == 1 ? kk : 2 * kk + part;
            if (PARTS == 2 && k >= N) continue;
#pragma unroll
            for (int j = 0; j < N; ++j) tb2[pl * PV + k * N + j] = op.mul(acc[kk * N + j], mat);
          }
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
      w = w1;
      e0 = e1;
      b0 = b1;
      sl ^= 1;
    }
  }
}

// Launch shape of degree (P, Q) on ne elements.
//
// A mesh that fills at least half of the co-resident CTAs takes the shape with the least idle lanes in
// passes A/C (one plane per thread) and B (columns over the same threads) within a budget of shared
// memory per CTA.  Smaller meshes wait for the chain of one CTA, and the FP64 planes of p >= 5 leave one
// or two CTAs of 32 to 128 threads per SM, with the FP64 pipe idle at every barrier: both (FP32 of p >= 3
// excepted, whose chains are short) take the shape with the least estimated time, over elements per CTA, jobs per batch, units per element,
// threads per plane and block sizes.  The estimate: the busiest SM runs `rounds` times c units of nb
// batches; a batch takes x us alone (FP64: 64 clocks per warp instruction on each of an SM's four
// partitions, plus the rows of the copies) and y us of the SM's shared pipes.  Its constants are fitted
// to 2,028 measured (p, q, elements, start) points (FP64 within 11%, FP32 within 17%); the shape it
// picks is on average 4% (FP32 6%) slower than the best one measured.
// Mass kernel with u0, one pass per contraction / the rule of lanes alone / this rule, us: FP64 125
// elements p = 2, q = 1 8.8 / 18.6 / 10.3, p = 4, q = 1 19.1 / 39.5 / 21.1, p = 6, q = 6 253 / 142 / 130;
// FP64 p = 5, q = 4 2,000 elements 1,193 / 944 / 765, p = 7, q = 6 2,000 elements 4,774 / 4,107 / 2,712,
// p = 7, q = 1 4,000 elements 1,561 / 2,386 / 1,353; FP32 512 elements p = 0, q = 2 6.5 / 12.4 / 6.3.
template <typename T, int P>
MassShape mass_shape_p(int Q, bool start, int64_t ne) {
  using D = MassDims<T, P>;
  constexpr int N = D::N, NQ = D::NQ, H = NQ / 2, C = NQ & 1;
  constexpr bool F64 = sizeof(T) == 8;
  constexpr size_t most = 200 * 1024;
  int dev = 0, sms = 1;
  if (cudaGetDevice(&dev) != cudaSuccess ||
      cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess)
    cudaGetLastError();
  static std::atomic<uint64_t> configured_devices{0};
  once_per_device(configured_devices, [&] {
    cudaFuncSetAttribute(k_mass<T, P, 1, F64>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)most);
    if constexpr (F64)
      cudaFuncSetAttribute(k_mass<T, P, 2, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)most);
    else if constexpr (P <= 2)
      cudaFuncSetAttribute(k_mass<T, P, 1, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)most);
  });
  auto smem = [&](int epc, int jobs) {
    return sizeof(T) * ((size_t)epc * 6 * D::NQ3 + (start ? (size_t)(jobs <= Q ? 1 : 2 * epc) * 3 * N * D::PV : 0) +
                        (size_t)jobs * 3 * N * (D::PT + D::PV) + D::TAB);
  };
  auto resident = [&](int parts, int threads, size_t sm) {
    int occ = 0;
    cudaError_t e;
    if constexpr (F64)
      e = parts == 2 ? cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, k_mass<T, P, 2, true>, threads, sm)
                     : cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, k_mass<T, P, 1, F64>, threads, sm);
    else
      e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, k_mass<T, P, 1, F64>, threads, sm);
    if (e != cudaSuccess) cudaGetLastError();
    return e == cudaSuccess ? occ : 0;
  };
  auto grid = [&](const MassShape& s, int occ) {
    return (int)std::min<int64_t>((ne + s.epc - 1) / s.epc * s.split, (int64_t)std::max(1, occ) * sms);
  };
  auto divides = [&](int epc, int jobs) { return epc > 1 ? jobs == epc * 2 * Q : (2 * Q) % jobs == 0; };
  // least idle lanes
  MassShape best{1, 1, 1, 1, 32, 0, smem(1, 1)};
  double best_score = -1.0;
  for (int epc = 1; epc <= 8; ++epc)
    for (int jobs = 1; jobs <= epc * 2 * Q && jobs <= kMassJobs; ++jobs) {
      const int planes = 3 * N * jobs, threads = (planes + 31) / 32 * 32;
      if (!divides(epc, jobs) || threads > D::MAXT || smem(epc, jobs) > D::WANT) continue;
      if (start && jobs <= Q && smem(epc, jobs) + sizeof(T) * 3 * N * D::PV > D::WANT) continue;  // room for both fields' starts
      const int cols = D::NQ2 * jobs, rounds = (cols + threads - 1) / threads;
      const double a = (double)planes / threads, b = (double)cols / (rounds * threads);
      // small CTAs spend their time between barriers
      const double score = (0.6 * a + 0.4 * b) * (threads >= 96 ? 1.0 : 0.6 + 0.4 * threads / 96);
      if (score > best_score) {
        best_score = score;
        best = MassShape{epc, jobs, 1, 1, threads, 0, smem(epc, jobs)};
      }
    }
  const int occ = resident(1, best.threads, best.smem);
  best.grid = grid(best, occ);
  if (!F64 && P >= 3 && best_score >= 0) return best;
  if (!(F64 && P >= 5) && best_score >= 0 && 2 * ((ne + best.epc - 1) / best.epc) >= (int64_t)occ * sms) return best;
  // least estimated time
  const double fwd = H * N + (N > 1 ? H : 0) + C * ((N + 1) / 2 - 1);  // operations of a line, there and back
  const double bwd = 2 * H + (N - 1) * H + C * ((N - 1) / 2);
  const double ops_ac = (N + NQ) * (fwd + bwd) + N * N;
  double best_t = 1e300;
  for (int epc = 1; epc <= 8; ++epc)
    for (int jobs = 1; jobs <= epc * 2 * Q && jobs <= kMassJobs; ++jobs) {
      if (!divides(epc, jobs) || smem(epc, jobs) > most) continue;
      const int batches = epc > 1 ? 1 : 2 * Q / jobs;
      for (int parts = 1; parts <= (F64 ? 2 : 1); ++parts) {
        const int need = (3 * N * jobs * parts + 31) / 32 * 32, bp = D::BP[parts - 1], cols = D::NQ2 * jobs * bp;
        const double ops_b = bp == 1 ? 3 * (fwd + bwd) + 9 * NQ : 3 * fwd + bwd + 3 * NQ;
        for (int threads : {need, 64, 96, 128, 192, 256}) {
          if (threads < need || threads > D::MAXT * parts || (threads > need && threads > (cols + 31) / 32 * 32)) continue;
          const int occ = resident(parts, threads, smem(epc, jobs));
          if (occ < 1) continue;
          const int w = threads / 32, w_ac = need / 32, w_b = (cols + 31) / 32;
          const double rows = (double)((3 * jobs + w - 1) / w) * ((D::N3 + 31) / 32);
          const double metric = (double)((epc * 3 * D::NQ3 + threads - 1) / threads);
          for (int split = 1; split <= batches; ++split) {
            if (batches % split || (!F64 && P >= 3 && split > 1)) continue;  // (no such instance)
            const MassShape s{epc, jobs, split, parts, threads, 0, smem(epc, jobs)};
            const int64_t units = (ne + epc - 1) / epc * split;
            const int g = grid(s, occ);
            const double rounds = (double)((units + g - 1) / g);
            const double c = (double)std::min<int64_t>(occ, (units + sms - 1) / sms), nb = (double)(batches / split);
            double t;
            if (F64) {
              const double alone = (w_ac + 3) / 4 * ops_ac / parts + (double)((cols + threads - 1) / threads) * ((w + 3) / 4) * ops_b;
              const double pipe = (w_ac * ops_ac / parts + w_b * ops_b) / 4;
              const double kb = sizeof(T) * (epc * 6.0 * D::NQ3 / nb + jobs * 6.0 * D::N3) / 1000;
              const double x = nb * (0.7 + 0.029 * alone + 0.16 * rows) + 0.2 * metric;
              const double y = c * nb * (0.027 * pipe + 0.036 * kb + 0.006 * rows * w);
              t = rounds * std::cbrt(x * x * x + y * y * y);
            } else {
              t = rounds * (nb * (1.1 + 0.037 * rows) + 0.012 * metric + c * nb * 0.011 * rows * w);
            }
            if (t < best_t) {
              best_t = t;
              best = s;
              best.grid = g;
            }
          }
        }
      }
    }
  return best;
}

template <typename T, int P>
int mass_p(const MassShape& sh, int Q, const T* um, int64_t um_es, int64_t um_cs, const T* u0, int64_t u0_es,
           int64_t u0_cs, const T* Gw, const T* eps, const T* mu, const CurvedTables& ct, int64_t ne, T* R,
           cudaStream_t s, const int32_t* skip) {
  MassTab<T, P> tb{};
  constexpr int N = P + 1, H = (P + 2) / 2;
  for (int j = 0; j < N; ++j) {
    for (int g = 0; g < H; ++g) {
      tb.L[j][g] = (T)ct.Lq[j][g];
      tb.r[j][g] = (j & 1) ? (T)(ct.Lq[j][g] / ct.Lq[1][g]) : T(0);
    }
    tb.L[j][H] = ((P + 2) & 1) && !(j & 1) ? (T)ct.Lq[j][H] : T(0);
  }
  const uint32_t units = (uint32_t)((ne + sh.epc - 1) / sh.epc * sh.split);
  // persistent over the units, one wave of co-resident CTAs (a skipped launch costs one wave)
  auto go = [&](auto kernel) {
    kernel<<<sh.grid, sh.threads, sh.smem, s>>>(um, um_es, um_cs, u0, u0_es, u0_cs, Gw, eps, mu, tb, Q, sh.epc, sh.jobs,
                                                (uint32_t)sh.split, units, ne, R, skip);
  };
  if constexpr (sizeof(T) == 8) {
    if (sh.parts == 2) go(k_mass<T, P, 2, true>);
    else go(k_mass<T, P, 1, true>);
  } else if constexpr (P <= 2) {
    if (sh.split > 1) go(k_mass<T, P, 1, true>);
    else go(k_mass<T, P, 1, false>);
  } else {
    go(k_mass<T, P, 1, false>);
  }
  return (int)cudaGetLastError();
}

}  // namespace

template <typename T>
MassShape mass_shape(int P, int Q, bool start, int64_t ne) {
  switch (P) {
#define STM_MP(p) \
  case p: return mass_shape_p<T, p>(Q, start, ne);
    STM_MP(0) STM_MP(1) STM_MP(2) STM_MP(3) STM_MP(4) STM_MP(5) STM_MP(6) STM_MP(7)
#undef STM_MP
    default: return MassShape{};
  }
}

template <typename T>
int launch_mass_curved(const MassShape& sh, int P, int Q, const T* um, int64_t um_es, int64_t um_cs, const T* u0,
                       int64_t u0_es, int64_t u0_cs, const T* Gw, const T* eps, const T* mu, const CurvedTables& ct,
                       int64_t ne, T* R, cudaStream_t s, const int32_t* skip) {
  if (Q < 1 || Q > kMaxQ || !sh.epc) return (int)cudaErrorInvalidValue;
  switch (P) {
#define STM_MP(p) \
  case p: return mass_p<T, p>(sh, Q, um, um_es, um_cs, u0, u0_es, u0_cs, Gw, eps, mu, ct, ne, R, s, skip);
    STM_MP(0) STM_MP(1) STM_MP(2) STM_MP(3) STM_MP(4) STM_MP(5) STM_MP(6) STM_MP(7)
#undef STM_MP
    default: return (int)cudaErrorInvalidValue;
  }
}

#ifndef STM_MASS_T
#error "compile with -DSTM_MASS_T=float or double"
#endif
template MassShape mass_shape<STM_MASS_T>(int, int, bool, int64_t);
template int launch_mass_curved<STM_MASS_T>(const MassShape&, int, int, const STM_MASS_T*, int64_t, int64_t,
                                            const STM_MASS_T*, int64_t, int64_t, const STM_MASS_T*, const STM_MASS_T*,
                                            const STM_MASS_T*, const CurvedTables&, int64_t, STM_MASS_T*, cudaStream_t,
                                            const int32_t*);

}  // namespace stm
