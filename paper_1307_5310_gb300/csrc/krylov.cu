#include "krylov.cuh"

#include <atomic>

#include "residual.cuh"

namespace stm {

namespace {

__device__ __forceinline__ double warp_sum(double v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
  return v;
}

// Block sum in a fixed order: warp shuffles, then warp 0 over the warp totals.
__device__ double block_sum(double v, double* sh) {
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  v = warp_sum(v);
  if (lane == 0) sh[wid] = v;
  __syncthreads();
  double r = 0.0;
  if (wid == 0) {
    r = (lane < (int)(blockDim.x >> 5)) ? sh[lane] : 0.0;
    r = warp_sum(r);
  }
  __syncthreads();
  return r;  // valid in thread 0
}

// Per-thread accumulator: FP64 for double storage; for float storage, FP32
// sums of the 16 products of four 16-byte chunks flushed into an FP64 total
// (the kernels call flush() after every fourth chunk: one conversion and one
// FP64 add per 16 products keeps the FP64 pipe off the critical path).
template <typename S>
struct Acc;
template <>
struct Acc<double> {
  double a = 0.0;
  __device__ __forceinline__ void add(double x, double y) { a = fma(x, y, a); }
  __device__ __forceinline__ void flush() {}
  __device__ __forceinline__ double get() const { return a; }
};
template <>
struct Acc<float> {
  double a = 0.0;
  float f = 0.f;
  __device__ __forceinline__ void add(float x, float y) { f = fmaf(x, y, f); }
  __device__ __forceinline__ void flush() {
    a += (double)f;
    f = 0.f;
  }
  __device__ __forceinline__ double get() const { return a + (double)f; }
};

// 16-byte vectors: float4 / double2.  Basis columns are 16-byte aligned
// (their leading dimension is padded); a scalar loop takes the tail.
template <typename S>
struct Vec;
template <>
struct Vec<float> {
  using T = float4;
  static constexpr int W = 4;
  __device__ static float get(const float4& v, int l) { return l == 0 ? v.x : l == 1 ? v.y : l == 2 ? v.z : v.w; }
  __device__ static void set(float4& v, int l, float x) {
    if (l == 0) v.x = x; else if (l == 1) v.y = x; else if (l == 2) v.z = x; else v.w = x;
  }
};
template <>
struct Vec<double> {
  using T = double2;
  static constexpr int W = 2;
  __device__ static double get(const double2& v, int l) { return l == 0 ? v.x : v.y; }
  __device__ static void set(double2& v, int l, double x) {
    if (l == 0) v.x = x; else v.y = x;
  }
};

// chunks per loop trip: enough independent 16-byte loads in flight per thread
template <int K>
struct Unroll {
  static constexpr int U = K <= 1 ? 4 : (K <= 3 ? 2 : 1);
};

constexpr int kRedWarps = kRedThreads / 32;

constexpr int log2_ceil(int m) { return m <= 1 ? 0 : 1 + log2_ceil((m + 1) / 2); }

// Sums of the M per-thread values get(i) over the block in a fixed order, written to
// partial[i * gridDim.x + blockIdx.x].  Within a warp the values are halved between lane halves at
// each exchange (about M additions a lane instead of 5 M: on small problems these sums are what the
// FP64 pipe does), then the warp totals in groups of eight lanes.
template <int M, typename F>
__device__ __forceinline__ void block_partials(F&& get, double* __restrict__ partial) {
  constexpr int LG = log2_ceil(M), MP = 1 << LG;
  static_assert(M <= 32 && kRedWarps == 8, "one value per lane, eight warps");
  __shared__ double sh[MP][kRedWarps];
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  double v[MP];
#pragma unroll
  for (int i = 0; i < MP; ++i) v[i] = i < M ? get(i) : 0.0;
#pragma unroll
  for (int st = 0; st < 5; ++st) {
    const int o = 16 >> st, cnt = MP >> st;
    if (cnt > 1) {
      const bool up = lane & o;
#pragma unroll
      for (int i = 0; i < cnt / 2; ++i) {
        const double send = up ? v[i] : v[i + cnt / 2], keep = up ? v[i + cnt / 2] : v[i];
        v[i] = keep + __shfl_xor_sync(0xffffffffu, send, o);
      }
    } else {
      v[0] += __shfl_xor_sync(0xffffffffu, v[0], o);
    }
  }
  // lane l holds the total of value l >> (5 - LG)
  if ((lane & ((32 >> LG) - 1)) == 0) sh[lane >> (5 - LG)][wid] = v[0];
  __syncthreads();
  for (int i = (int)threadIdx.x >> 3; i < (M + 3) / 4 * 4; i += kRedThreads / 8) {
    double t = i < M ? sh[i][threadIdx.x & 7] : 0.0;
#pragma unroll
    for (int o = 4; o > 0; o >>= 1) t += __shfl_down_sync(0xffffffffu, t, o, 8);
    if (i < M && (threadIdx.x & 7) == 0) partial[(int64_t)i * gridDim.x + blockIdx.x] = t;
  }
}

// True in every thread of the block that is the last of the grid to arrive (its reads of the other
// blocks' partial sums are then valid); the counter is back at 0 for the next launch.
__device__ bool last_block(GmresState* st) {
  __shared__ bool last;
  __threadfence();
  __syncthreads();
  if (threadIdx.x == 0) {
    last = atomicAdd(&st->ticket, 1) == (int)gridDim.x - 1;
    if (last) st->ticket = 0;
  }
  __syncthreads();
  if (last) __threadfence();
  return last;
}

// The grid's sums of m values in a fixed order (one warp per value: lane-strided, then a shuffle tree).
__device__ void grid_sums(const double* __restrict__ partial, int m, double* out) {
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, nb = gridDim.x;
  for (int i = wid; i < m; i += kRedWarps) {
    double v = 0.0;
#pragma unroll 8
    for (int b = lane; b < nb; b += 32) v += __ldcg(partial + (int64_t)i * nb + b);
    v = warp_sum(v);
    if (lane == 0) out[i] = v;
  }
  __syncthreads();
}

// ---- scalar steps of the device-side GMRES control, run by the last block of a reduction ----

__device__ void outer_check(GmresState* st) {
  st->used = st->k;
  st->k = 0;
  st->skip_reo = 1;
  const double beta = sqrt(st->red[0]);
  const double ref = st->ref;
  st->rel = ref > 0 ? beta / ref : beta;
  if (!isfinite(st->rel)) {
    st->status = -5;  // STM_ENAN
    st->skip = 1;
    st->halt = 1;
    return;
  }
  bool done;
  if (st->inexact) {
    st->phi = sqrt(st->red[1]);
    done = st->phi <= st->tol;
  } else {
    done = st->rel <= st->tol;
  }
  if (done) st->outer_done = 1;
  st->skip = (done || st->iters >= st->max_it || beta == 0.0) ? 1 : 0;
  st->halt = st->skip;
}

__device__ void cycle_init(GmresState* st, int slot_start, double floor_rel) {
  if (st->skip) return;
  const double b0 = sqrt(st->red[slot_start]);
  if (!(b0 > 0.0)) {
    st->skip = 1;
    st->halt = 1;
    return;
  }
  st->cycles += 1;
  // v_0 = V[0] / alpha_0 with V[0] = R = -r: alpha_0 = -|start|
  st->alpha[0] = -b0;
  st->g[0] = b0;
  const double target = st->inexact ? st->tol : st->tol * st->ref;
  st->tol_abs = fmax(target, floor_rel * b0);
}

// Coefficients of one Gram-Schmidt pass over V[0..j] from the dot products v (whole block).
__device__ void gs_step(GmresState* st, const double* v, int j, bool second) {
  if ((int)threadIdx.x <= j) {
    const int i = threadIdx.x;
    const double ai = st->alpha[i], aj = st->alpha[j];
    st->cc[i] = v[i] / (ai * ai);
    const double h = v[i] / (ai * aj);
    st->H[i * kMaxDots + j] = second ? st->H[i * kMaxDots + j] + h : h;
  }
}

// Iteration j's Givens step from |W|^2 after the update; at the end of the cycle also the
// triangular system and the combination coefficients (whole block, on a copy in shared memory).
__device__ void givens_step(GmresState* st, double after, int j, int m) {
  __shared__ double H[kMaxDots * kMaxDots], cs[kMaxDots], sn[kMaxDots], g[kMaxDots + 1], al[kMaxDots + 1];
  __shared__ int stop;
  __syncthreads();  // the column written by gs_step
  const int t = threadIdx.x;
  for (int k = t; k < kMaxDots * kMaxDots; k += blockDim.x) H[k] = st->H[k];
  if (t < kMaxDots) {
    cs[t] = st->cs[t];
    sn[t] = st->sn[t];
  }
  if (t <= kMaxDots) {
    g[t] = st->g[t];
    al[t] = st->alpha[t];
  }
  __syncthreads();
  if (t == 0) {
    stop = 0;
    if (!isfinite(after) || !isfinite(st->before)) {
      st->status = -5;  // STM_ENAN
      st->k = 0;
      st->skip = 1;
      st->halt = 1;
      st->skip_reo = 1;
    } else {
      const double nw = sqrt(after);
      const double aj = al[j];
      st->alpha[j + 1] = aj < 0 ? -nw : nw;
      double y0 = nw / fabs(aj);
      double x0 = H[j];
      for (int i = 0; i < j; ++i) {
        const double x = x0, y = H[(i + 1) * kMaxDots + j];
        H[i * kMaxDots + j] = cs[i] * x + sn[i] * y;
        x0 = -sn[i] * x + cs[i] * y;
      }
      const double r = hypot(x0, y0);
      const double c = r > 0 ? x0 / r : 1.0, s = r > 0 ? y0 / r : 0.0;
      H[j * kMaxDots + j] = r;
      const double g1 = -s * g[j];
      g[j] = c * g[j];
      g[j + 1] = g1;
      st->cs[j] = c;
      st->sn[j] = s;
      st->g[j] = g[j];
      st->g[j + 1] = g1;
      st->iters += 1;
      st->k = j + 1;
      stop = fabs(g1) <= st->tol_abs || nw == 0.0 || st->iters >= st->max_it || j + 1 >= m;
      if (stop) {
        st->skip = 1;
        st->skip_reo = 1;
      }
    }
  }
  __syncthreads();
  if (t <= j) st->H[t * kMaxDots + j] = H[t * kMaxDots + j];
  if (stop && t == 0) {
    const int k = j + 1;
    for (int i = k - 1; i >= 0; --i) {
      double y = g[i];
      for (int l = i + 1; l < k; ++l) y -= H[i * kMaxDots + l] * g[l];
      g[i] = y / H[i * kMaxDots + i];
    }
    for (int i = 0; i < kMaxDots; ++i) st->yc[i] = i < k ? g[i] / al[i] : 0.0;
    st->res = fabs(g[k]);
  }
}

// Dot products of w with V[0..K-1] and |w|^2 (index K).  GS: the last block of the grid turns them
// into iteration j = K - 1's Gram-Schmidt coefficients and Hessenberg column.
template <typename S, int K, bool GS>
__global__ void __launch_bounds__(kRedThreads) k_dots(const S* __restrict__ w, const S* __restrict__ V, int64_t ldv,
                                                      int64_t n, double* __restrict__ partial, GmresState* st) {
  if (GS && st->skip) return;
  using VT = typename Vec<S>::T;
  constexpr int W = Vec<S>::W, U = Unroll<K>::U;
  Acc<S> acc[K + 1];
  const int64_t nv = n / W;
  const int64_t tid = blockIdx.x * (int64_t)blockDim.x + threadIdx.x, nth = (int64_t)gridDim.x * blockDim.x;
  const VT* w4 = reinterpret_cast<const VT*>(w);
  int chunks = 0;
  auto trip = [&](auto uc, int64_t c0) {  // chunks c0, c0 + nth, ...: all their loads first
    constexpr int UU = decltype(uc)::value;
    VT wv[UU], vv[UU][K];
#pragma unroll
    for (int u = 0; u < UU; ++u) {
      const int64_t c = c0 + u * nth;
      wv[u] = w4[c];
#pragma unroll
      for (int i = 0; i < K; ++i) vv[u][i] = reinterpret_cast<const VT*>(V + i * ldv)[c];
    }
#pragma unroll
    for (int u = 0; u < UU; ++u) {
#pragma unroll
      for (int l = 0; l < W; ++l) {
        const S x = Vec<S>::get(wv[u], l);
#pragma unroll
        for (int i = 0; i < K; ++i) acc[i].add(x, Vec<S>::get(vv[u][i], l));
        acc[K].add(x, x);
      }
      if ((++chunks & 3) == 0) {
#pragma unroll
        for (int i = 0; i <= K; ++i) acc[i].flush();
      }
    }
  };
  int64_t c0 = tid;
  for (; c0 + (U - 1) * nth < nv; c0 += nth * U) trip(std::integral_constant<int, U>{}, c0);
  for (; c0 < nv; c0 += nth) trip(std::integral_constant<int, 1>{}, c0);
  for (int64_t j = nv * W + tid; j < n; j += nth) {  // tail
    const S x = w[j];
#pragma unroll
    for (int i = 0; i < K; ++i) acc[i].add(x, V[i * ldv + j]);
    acc[K].add(x, x);
  }
  block_partials<K + 1>([&](int i) { return acc[i].get(); }, partial);
  if constexpr (GS) {
    if (!last_block(st)) return;
    __shared__ double v[K + 1];
    grid_sums(partial, K + 1, v);
    gs_step(st, v, K - 1, false);
    if (threadIdx.x == 0) st->before = v[K];
  }
}

enum UpdateMode { kPlain, kOnly, kFirst, kSecond };

// w -= sum_i c_i V[i] and |w|^2.  kPlain: c from the argument, partial sums only.  The others are the
// update of iteration j = K - 1 with the coefficients of the device state: kOnly ends the iteration
// (no second Gram-Schmidt pass); kFirst also forms the updated w's dot products with the same V chunks
// (the second pass then needs no read of the basis for them) and its last block decides on that pass:
// coefficients for it, or the end of the iteration; kSecond applies it and ends the iteration.  On the
// 32^3 mixed solve both passes run in every iteration: a dot pass, two updates instead of two of each.
template <typename S, int K, int MODE>
__global__ void __launch_bounds__(kRedThreads) k_update(S* __restrict__ w, const S* __restrict__ V, int64_t ldv,
                                                        Coef16 c, int64_t n, double* __restrict__ partial,
                                                        GmresState* st, int m) {
  if (MODE != kPlain && (MODE == kSecond ? st->skip_reo : st->skip)) return;
  using VT = typename Vec<S>::T;
  constexpr int W = Vec<S>::W, U = Unroll<K>::U, ND = MODE == kFirst ? K : 0;
  S cc[K > 0 ? K : 1];
  if constexpr (sizeof(S) == 8 && K > 0) {
    // one copy per lane: the compiler cannot make these uniform, and the FP64 pipe takes FMAs with
    // three vector registers at full rate only
    __shared__ double cl[K][32];
    for (int k = threadIdx.x; k < K * 32; k += blockDim.x) cl[k / 32][k & 31] = MODE != kPlain ? st->cc[k / 32] : c.c[k / 32];
    __syncthreads();
#pragma unroll
    for (int i = 0; i < K; ++i) cc[i] = cl[i][threadIdx.x & 31];
  } else {
#pragma unroll
    for (int i = 0; i < K; ++i) cc[i] = (S)(MODE != kPlain ? st->cc[i] : c.c[i]);
  }
  Acc<S> acc, dot[ND > 0 ? ND : 1];
  const int64_t nv = n / W;
  const int64_t tid = blockIdx.x * (int64_t)blockDim.x + threadIdx.x, nth = (int64_t)gridDim.x * blockDim.x;
  VT* w4 = reinterpret_cast<VT*>(w);
  int chunks = 0;
  auto trip = [&](auto uc, int64_t c0) {  // chunks c0, c0 + nth, ...: all their loads first
    constexpr int UU = decltype(uc)::value;
    VT wv[UU], vv[UU][K > 0 ? K : 1];
#pragma unroll
    for (int u = 0; u < UU; ++u) {
      const int64_t cix = c0 + u * nth;
      wv[u] = w4[cix];
#pragma unroll
      for (int i = 0; i < K; ++i) vv[u][i] = reinterpret_cast<const VT*>(V + i * ldv)[cix];
    }
#pragma unroll
    for (int u = 0; u < UU; ++u) {
#pragma unroll
      for (int l = 0; l < W; ++l) {
        S x = Vec<S>::get(wv[u], l);
#pragma unroll
        for (int i = 0; i < K; ++i) x = fma(-cc[i], Vec<S>::get(vv[u][i], l), x);
        Vec<S>::set(wv[u], l, x);
        acc.add(x, x);
#pragma unroll
        for (int i = 0; i < ND; ++i) dot[i].add(x, Vec<S>::get(vv[u][i], l));
      }
      if ((++chunks & 3) == 0) {
        acc.flush();
#pragma unroll
        for (int i = 0; i < ND; ++i) dot[i].flush();
      }
      if (K > 0) w4[c0 + u * nth] = wv[u];
    }
  };
  int64_t c0 = tid;
  for (; c0 + (U - 1) * nth < nv; c0 += nth * U) trip(std::integral_constant<int, U>{}, c0);
  for (; c0 < nv; c0 += nth) trip(std::integral_constant<int, 1>{}, c0);
  for (int64_t j = nv * W + tid; j < n; j += nth) {  // tail
    S x = w[j];
#pragma unroll
    for (int i = 0; i < K; ++i) x = fma(-cc[i], V[i * ldv + j], x);
    if (K > 0) w[j] = x;
    acc.add(x, x);
#pragma unroll
    for (int i = 0; i < ND; ++i) dot[i].add(x, V[i * ldv + j]);
  }
  block_partials<ND + 1>([&](int i) { return i < ND ? dot[i].get() : acc.get(); }, partial);
  if constexpr (MODE != kPlain) {
    if (!last_block(st)) return;
    __shared__ double v[ND + 1];
    __shared__ int again;
    grid_sums(partial, ND + 1, v);
    const double after = v[ND];
    if constexpr (MODE == kFirst) {
      if (threadIdx.x == 0) {
        again = after < 0.5 * st->before;  // the DGKS test
        st->skip_reo = again ? 0 : 1;
      }
      __syncthreads();
      if (again) {
        gs_step(st, v, K - 1, true);
        return;
      }
    }
    if constexpr (MODE == kSecond) {
      if (threadIdx.x == 0) st->skip_reo = 1;
    }
    givens_step(st, after, K - 1, m);
  }
}

// |v|^2 of an FP64 vector, with the step that follows it in the slab solve (by the last block); CONV
// also rounds the vector to float and takes |v32|^2.
template <bool CONV>
__global__ void __launch_bounds__(kRedThreads) k_norm_step(const double* __restrict__ v, float* __restrict__ v32,
                                                           int64_t n, double* __restrict__ partial, GmresState* st,
                                                           NormStep step) {
  if (step.kind == NormStep::kSlabStart) {
  } else if (CONV) {
    if (st->skip) return;
  } else if (st->halt) {
    // the slab has stopped: this cycle applies nothing
    if (blockIdx.x == 0 && threadIdx.x == 0) {
      st->used = st->k;
      st->k = 0;
      st->skip = 1;
      st->skip_reo = 1;
    }
    return;
  }
  const int64_t nv = n / 4;
  const int64_t tid = blockIdx.x * (int64_t)blockDim.x + threadIdx.x, nth = (int64_t)gridDim.x * blockDim.x;
  const double2* v2 = reinterpret_cast<const double2*>(v);
  Acc<double> acc;
  Acc<float> acc32;
  int chunks = 0;
#pragma unroll 4
  for (int64_t c = tid; c < nv; c += nth) {  // four entries: two 16-byte loads
    const double2 a = v2[2 * c], b = v2[2 * c + 1];
    if constexpr (CONV) {
      const float4 f = make_float4((float)a.x, (float)a.y, (float)b.x, (float)b.y);
      reinterpret_cast<float4*>(v32)[c] = f;
      acc32.add(f.x, f.x);
      acc32.add(f.y, f.y);
      acc32.add(f.z, f.z);
      acc32.add(f.w, f.w);
      if ((++chunks & 3) == 0) acc32.flush();
    } else {
      acc.add(a.x, a.x);
      acc.add(a.y, a.y);
      acc.add(b.x, b.x);
      acc.add(b.y, b.y);
    }
  }
  for (int64_t j = nv * 4 + tid; j < n; j += nth) {  // tail
    if constexpr (CONV) {
      const float f = (float)v[j];
      v32[j] = f;
      acc32.add(f, f);
    } else {
      acc.add(v[j], v[j]);
    }
  }
  block_partials<1>([&](int) { return CONV ? acc32.get() : acc.get(); }, partial);
  if (!last_block(st)) return;
  __shared__ double sum[1];
  grid_sums(partial, 1, sum);
  if (threadIdx.x != 0) return;
  switch (step.kind) {
    case NormStep::kSlabStart:
      st->red[0] = sum[0];
      st->ref = sqrt(sum[0]);
      st->tol = step.tol;
      st->max_it = step.max_it;
      st->inexact = step.inexact;
      st->iters = 0;
      st->cycles = 0;
      st->status = 0;
      st->outer_done = 0;
      st->halt = 0;
      st->skip = 0;
      st->skip_reo = 1;
      st->k = 0;
      st->rel = 0.0;
      st->phi = 0.0;
      st->res = 0.0;
      break;
    case NormStep::kResidual:
      st->red[0] = sum[0];
      break;
    case NormStep::kCheck:
      st->red[step.slot] = sum[0];
      outer_check(st);
      if (step.init) cycle_init(st, step.slot, 0.0);
      break;
    case NormStep::kStart32:
      st->red[2] = sum[0];
      cycle_init(st, 2, 1e-6);
      break;
  }
}

__global__ void k_finish(const double* __restrict__ partial, int m, int nb, double* __restrict__ out) {
  // one warp per result, fixed order: lane-strided partial sums then a shuffle tree
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  for (int i = wid; i < m; i += blockDim.x >> 5) {
    double v = 0.0;
    for (int b = lane; b < nb; b += 32) v += partial[i * nb + b];
    v = warp_sum(v);
    if (lane == 0) out[i] = v;
  }
}

template <bool Small>
__device__ __forceinline__ int64_t block_of(int64_t j, int64_t blk) {
  return Small ? (int64_t)((uint32_t)j / (uint32_t)blk) : j / blk;
}

template <typename S, bool Small>
__global__ void k_precond(S* __restrict__ z, const S* __restrict__ v, const S* __restrict__ inv, int64_t blk,
                          int64_t n, const int32_t* skip) {
  if (skip && *skip) return;
  using VT = typename Vec<S>::T;
  constexpr int W = Vec<S>::W;
  const int64_t nv = n / W;
  const int64_t tid = blockIdx.x * (int64_t)blockDim.x + threadIdx.x, nth = (int64_t)gridDim.x * blockDim.x;
  for (int64_t c = tid; c < nv && blk >= W; c += nth) {  // blocks of at least W entries: <= 2 per vector
    VT x = reinterpret_cast<const VT*>(v)[c];
    const int64_t j0 = c * W, b0 = block_of<Small>(j0, blk), edge = (b0 + 1) * blk;
    const S s0 = inv[b0], s1 = (j0 + W > edge) ? inv[b0 + 1] : s0;
#pragma unroll
    for (int l = 0; l < W; ++l) Vec<S>::set(x, l, Vec<S>::get(x, l) * (j0 + l < edge ? s0 : s1));
    reinterpret_cast<VT*>(z)[c] = x;
  }
  for (int64_t j = (blk >= W ? nv * W : 0) + tid; j < n; j += nth) z[j] = v[j] * inv[block_of<Small>(j, blk)];
}

// Four entries a thread: 16-byte loads of the basis (FP32; two of them in FP64) and of x.  64^3-like
// vectors are far larger than L2, so this is bound by HBM: 32^3 elements, p = 4, q = 3, ten FP32
// columns 1.01 -> 0.64 ms.
template <typename S, typename X, int K, bool Small>
__global__ void k_precond_combine(X* __restrict__ x, const S* __restrict__ V, int64_t ldv,
                                  const S* __restrict__ inv, int64_t blk, int64_t n, const GmresState* st) {
  const int kk = st->k;  // K is the largest
  if (kk <= 0) return;
  S yy[K > 0 ? K : 1];
#pragma unroll
  for (int i = 0; i < K; ++i) yy[i] = (S)st->yc[i];
  using VS = typename Vec<S>::T;
  using VX = typename Vec<X>::T;
  constexpr int WS = Vec<S>::W, WX = Vec<X>::W, GS = 4 / WS, GX = 4 / WX;
  const int64_t n4 = n / 4;
  const int64_t tid = blockIdx.x * (int64_t)blockDim.x + threadIdx.x, nth = (int64_t)gridDim.x * blockDim.x;
  for (int64_t c = tid; c < n4; c += nth) {
    VX xv[GX];
#pragma unroll
    for (int g = 0; g < GX; ++g) xv[g] = reinterpret_cast<const VX*>(x)[c * GX + g];
    S v[4] = {S(0), S(0), S(0), S(0)};
#pragma unroll
    for (int i = 0; i < K; ++i) {
      if (i < kk) {
#pragma unroll
        for (int g = 0; g < GS; ++g) {
          const VS w = reinterpret_cast<const VS*>(V + i * ldv)[c * GS + g];
#pragma unroll
          for (int l = 0; l < WS; ++l) v[g * WS + l] = fma(yy[i], Vec<S>::get(w, l), v[g * WS + l]);
        }
      }
    }
    int64_t b = block_of<Small>(c * 4, blk), edge = (b + 1) * blk;
    S s = inv[b];
#pragma unroll
    for (int l = 0; l < 4; ++l) {
      if (c * 4 + l >= edge) {
        s = inv[++b];
        edge += blk;
      }
      Vec<X>::set(xv[l / WX], l % WX, Vec<X>::get(xv[l / WX], l % WX) + (X)(v[l] * s));
    }
#pragma unroll
    for (int g = 0; g < GX; ++g) reinterpret_cast<VX*>(x)[c * GX + g] = xv[g];
  }
  for (int64_t j = n4 * 4 + tid; j < n; j += nth) {  // tail
    S v = S(0);
#pragma unroll
    for (int i = 0; i < K; ++i)
      if (i < kk) v = fma(yy[i], V[i * ldv + j], v);
    x[j] = x[j] + (X)(v * inv[block_of<Small>(j, blk)]);
  }
}

template <bool Small>
__global__ void __launch_bounds__(kRedThreads) k_energy(const double* __restrict__ u, const double* __restrict__ mass,
                                                        int64_t n3, int64_t n, double* __restrict__ partial) {
  __shared__ double sh[32];
  double acc = 0.0;
  const int64_t tid = blockIdx.x * (int64_t)blockDim.x + threadIdx.x, nth = (int64_t)gridDim.x * blockDim.x;
#pragma unroll 4
  for (int64_t c = tid; c < n / 2; c += nth) {
    const double2 v = reinterpret_cast<const double2*>(u)[c];
    acc = fma(mass[block_of<Small>(2 * c, n3)] * v.x, v.x, acc);
    acc = fma(mass[block_of<Small>(2 * c + 1, n3)] * v.y, v.y, acc);
  }
  if (tid == 0 && (n & 1)) acc = fma(mass[block_of<Small>(n - 1, n3)] * u[n - 1], u[n - 1], acc);
  const double r = block_sum(acc, sh);
  if (threadIdx.x == 0) partial[blockIdx.x] = 0.5 * r;
}

template <typename D, typename S>
__global__ void k_convert(D* __restrict__ d, const S* __restrict__ s, int64_t n, const int32_t* skip) {
  if (skip && *skip) return;
  for (int64_t j = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; j < n; j += (int64_t)gridDim.x * blockDim.x)
    d[j] = (D)s[j];
}


inline int grid_for(int64_t n) {
  int64_t g = (n + kRedThreads - 1) / kRedThreads;
  return (int)(g < 4 * kRedBlocks ? (g < 1 ? 1 : g) : 4 * kRedBlocks);
}

inline bool small(int64_t n) { return n <= (int64_t)0xffffffffLL; }

// Blocks of a reduction over nv vectors: one vector a thread on small problems, else one wave of
// co-resident blocks (at most kRedBlocks).  A fixed 608 ran a second, mostly empty wave where the
// registers hold fewer than four blocks per SM (ten FP32 columns: 618 us against 490 expected).
template <typename F>
inline int red_grid(F kernel, int64_t nv, std::atomic<int>* cache) {
  const int64_t g = (nv + kRedThreads - 1) / kRedThreads;
  return wave_grid(kernel, kRedThreads, 0, g < 1 ? 1 : (g < kRedBlocks ? g : kRedBlocks), cache);
}

template <typename S, typename X, int K>
void combine_k(X* x, const S* V, int64_t ldv, const S* inv, int64_t blk, int64_t n, cudaStream_t s,
               const GmresState* st) {
  const int g = grid_for((n + 3) / 4);
  if (small(n)) k_precond_combine<S, X, K, true><<<g, kRedThreads, 0, s>>>(x, V, ldv, inv, blk, n, st);
  else k_precond_combine<S, X, K, false><<<g, kRedThreads, 0, s>>>(x, V, ldv, inv, blk, n, st);
}

#define STM_SWITCH_K(k, CALL)  \
  switch (k) {                 \
    case 1: CALL(1); break;    \
    case 2: CALL(2); break;    \
    case 3: CALL(3); break;    \
    case 4: CALL(4); break;    \
    case 5: CALL(5); break;    \
    case 6: CALL(6); break;    \
    case 7: CALL(7); break;    \
    case 8: CALL(8); break;    \
    case 9: CALL(9); break;    \
    case 10: CALL(10); break;  \
    case 11: CALL(11); break;  \
    case 12: CALL(12); break;  \
    case 13: CALL(13); break;  \
    case 14: CALL(14); break;  \
    default: CALL(15); break;  \
  }

}  // namespace

void dot(const double* w, const double* v, int64_t n, double* partial, double* out, cudaStream_t s) {
  static std::atomic<int> cap[64];
  const int g = red_grid(k_dots<double, 1, false>, n / Vec<double>::W, cap);
  k_dots<double, 1, false><<<g, kRedThreads, 0, s>>>(w, v, 0, n, partial, nullptr);
  k_finish<<<1, 32, 0, s>>>(partial, 1, g, out);
}

void axpy_norm(double* w, const double* v, double c, int64_t n, double* partial, double* out, cudaStream_t s) {
  static std::atomic<int> cap[64];
  const int g = red_grid(k_update<double, 1, kPlain>, n / Vec<double>::W, cap);
  Coef16 cc{};
  cc.c[0] = c;
  if (v) k_update<double, 1, kPlain><<<g, kRedThreads, 0, s>>>(w, v, 0, cc, n, partial, nullptr, 0);
  else k_update<double, 0, kPlain><<<g, kRedThreads, 0, s>>>(w, w, 0, cc, n, partial, nullptr, 0);
  k_finish<<<1, 32, 0, s>>>(partial, 1, g, out);
}

template <typename S, int K>
void dots_k(const S* w, const S* V, int64_t ldv, int64_t n, double* partial, GmresState* st, cudaStream_t s) {
  static std::atomic<int> cap[64];
  auto k = k_dots<S, K, true>;
  k<<<red_grid(k, n / Vec<S>::W, cap), kRedThreads, 0, s>>>(w, V, ldv, n, partial, st);
}

template <typename S, int K, int MODE>
void update_k(S* w, const S* V, int64_t ldv, int64_t n, double* partial, GmresState* st, int m, cudaStream_t s) {
  static std::atomic<int> cap[64];
  auto k = k_update<S, K, MODE>;
  k<<<red_grid(k, n / Vec<S>::W, cap), kRedThreads, 0, s>>>(w, V, ldv, Coef16{}, n, partial, st, m);
}

template <typename S>
void gmres_dots(const S* w, const S* V, int64_t ldv, int j, int64_t n, double* partial, GmresState* st,
                cudaStream_t s) {
#define STM_MD(K) dots_k<S, K>(w, V, ldv, n, partial, st, s)
  STM_SWITCH_K(j + 1, STM_MD)
#undef STM_MD
}

template <typename S>
void gmres_update(S* w, const S* V, int64_t ldv, int j, int64_t n, double* partial, GmresState* st, int m, bool reorth,
                  cudaStream_t s) {
#define STM_UP(K) update_k<S, K, kOnly>(w, V, ldv, n, partial, st, m, s)
#define STM_UP1(K) update_k<S, K, kFirst>(w, V, ldv, n, partial, st, m, s)
#define STM_UP2(K) update_k<S, K, kSecond>(w, V, ldv, n, partial, st, m, s)
  if (reorth) {
    STM_SWITCH_K(j + 1, STM_UP1)
    STM_SWITCH_K(j + 1, STM_UP2)
  } else {
    STM_SWITCH_K(j + 1, STM_UP)
  }
#undef STM_UP
#undef STM_UP1
#undef STM_UP2
}

void gmres_norm(const double* v, int64_t n, double* partial, GmresState* st, const NormStep& step, cudaStream_t s) {
  static std::atomic<int> cap[64];
  k_norm_step<false><<<red_grid(k_norm_step<false>, n / 4, cap), kRedThreads, 0, s>>>(v, nullptr, n, partial, st, step);
}

void gmres_start32(const double* v, float* v32, int64_t n, double* partial, GmresState* st, cudaStream_t s) {
  NormStep step{};
  step.kind = NormStep::kStart32;
  static std::atomic<int> cap[64];
  k_norm_step<true><<<red_grid(k_norm_step<true>, n / 4, cap), kRedThreads, 0, s>>>(v, v32, n, partial, st, step);
}

template <typename S>
void precond_apply(S* z, const S* v, const S* inv, int64_t blk, int64_t n, cudaStream_t s, const int32_t* skip) {
  if (small(n)) k_precond<S, true><<<grid_for(n), kRedThreads, 0, s>>>(z, v, inv, blk, n, skip);
  else k_precond<S, false><<<grid_for(n), kRedThreads, 0, s>>>(z, v, inv, blk, n, skip);
}

template <typename S, typename X>
void precond_combine(X* x, const S* V, int64_t ldv, int m, const S* inv, int64_t blk, int64_t n, cudaStream_t s,
                     const GmresState* st) {
#define STM_CB(K) combine_k<S, X, K>(x, V, ldv, inv, blk, n, s, st)
  STM_SWITCH_K(m, STM_CB)
#undef STM_CB
}

void energy_brick(const double* u, const double* mass, int64_t n3, int64_t n, double* partial, double* out,
                  cudaStream_t s) {
  if (small(n)) k_energy<true><<<kRedBlocks, kRedThreads, 0, s>>>(u, mass, n3, n, partial);
  else k_energy<false><<<kRedBlocks, kRedThreads, 0, s>>>(u, mass, n3, n, partial);
  k_finish<<<1, 32, 0, s>>>(partial, 1, kRedBlocks, out);
}

template <typename D, typename S>
void convert(D* dst, const S* src, int64_t n, cudaStream_t s, const int32_t* skip) {
  k_convert<D, S><<<grid_for(n), kRedThreads, 0, s>>>(dst, src, n, skip);
}


template void gmres_dots<double>(const double*, const double*, int64_t, int, int64_t, double*, GmresState*, cudaStream_t);
template void gmres_dots<float>(const float*, const float*, int64_t, int, int64_t, double*, GmresState*, cudaStream_t);
template void gmres_update<double>(double*, const double*, int64_t, int, int64_t, double*, GmresState*, int, bool,
                                   cudaStream_t);
template void gmres_update<float>(float*, const float*, int64_t, int, int64_t, double*, GmresState*, int, bool,
                                  cudaStream_t);
template void precond_apply<double>(double*, const double*, const double*, int64_t, int64_t, cudaStream_t,
                                    const int32_t*);
template void precond_apply<float>(float*, const float*, const float*, int64_t, int64_t, cudaStream_t,
                                   const int32_t*);
template void precond_combine<double, double>(double*, const double*, int64_t, int, const double*, int64_t, int64_t,
                                              cudaStream_t, const GmresState*);
template void precond_combine<float, double>(double*, const float*, int64_t, int, const float*, int64_t, int64_t,
                                             cudaStream_t, const GmresState*);
template void convert<float, double>(float*, const double*, int64_t, cudaStream_t, const int32_t*);

}  // namespace stm
