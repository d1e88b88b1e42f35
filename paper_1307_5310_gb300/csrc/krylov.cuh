// Vector kernels of the per-slab GMRES solve (Sec. 5.4) and the discrete
// energy (Eq. stability:energydef).  Storage type S is double or float.
// Reductions use a fixed summation order on a grid that follows from the vector
// length and the device, so results are bitwise reproducible run to run on one
// kind of device.  With S = double every product and sum is FP64.  With
// S = float (the inner solve of the mixed-precision path) each thread sums the 16
// products of four 16-byte chunks, a grid stride apart, in FP32 and accumulates
// those partial sums in FP64; the grid and block reductions are FP64.
//
// The last block of a reduction to arrive sums the grid's partials and takes the scalar step that
// needs them (Gram-Schmidt coefficients, Givens rotation, stop tests, triangular solve), so an
// iteration is two launches besides the operator (three with a second Gram-Schmidt pass) instead of
// four (eight) and no single-thread kernel walks the state in device memory.  4^3 elements, p = 2,
// q = 1, FP64 to 1e-12 (26 iterations, both passes): 2.12 -> 1.15 ms per slab.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

namespace stm {

constexpr int kRedBlocks = 608;   // 4 x 152 SMs
constexpr int kRedThreads = 256;
constexpr int kMaxDots = 16;      // restart <= 15 basis vectors + one norm

struct Coef16 { double c[kMaxDots]; };

// Device-side state of the restarted GMRES slab solve (Sec. 5.4): the Hessenberg
// matrix of the current cycle with its Givens rotations, the basis scales, the stop
// tests and the flags that let a whole restart cycle run without the host.  Every
// kernel of an iteration takes `skip` (a pointer into this struct) and returns at
// once while it is set, so a cycle is a fixed launch sequence (capturable in a CUDA
// graph) whose tail is a no-op after convergence.
struct GmresState {
  double H[kMaxDots * kMaxDots];  // H[i * kMaxDots + j], column j = iteration j
  double cs[kMaxDots], sn[kMaxDots], g[kMaxDots + 1], alpha[kMaxDots + 1];
  double cc[kMaxDots];            // Gram-Schmidt coefficients of the current iteration
  double yc[kMaxDots];            // combination coefficients at the end of the cycle
  double red[4];                  // reduction results: 0 |R|^2, 1 |S R|^2, 2 |start vector|^2
  double before;                  // |W|^2 before the update (DGKS test)
  double ref;                     // |R(U with unknowns 0)| of the slab (stop test R6)
  double tol;                     // relative target (exact solve) or eta budget (inexact)
  double tol_abs;                 // this cycle's stop threshold on |g|
  double rel, phi, res;           // last true relative residual, weighted norm, |g_k|
  int32_t k;                      // basis vectors used in this cycle
  int32_t used;                   // those of the cycle before the last stop test
  int32_t skip;                   // 1: the rest of the cycle is skipped
  int32_t skip_reo;               // 1: no second Gram-Schmidt pass in this iteration
  int32_t iters;                  // GMRES iterations of the slab so far
  int32_t max_it;
  int32_t status;                 // 0, or a negative STM_* code
  int32_t outer_done;             // 1: the slab's stop test holds
  int32_t inexact;                // 1: stop on the weighted norm (eta_it), 0: on rel
  int32_t cycles;                 // restart cycles started
  int32_t ticket;                 // blocks of the running reduction that have arrived (0 between launches)
  int32_t halt;                   // 1: the slab solve has stopped (stop test, cap, zero residual or
                                  //    error); every later kernel of the slab is skipped
};

// partial: kMaxDots * kRedBlocks doubles of scratch for every reduction below.

// out[0] = sum_n w[n] v[n].
void dot(const double* w, const double* v, int64_t n, double* partial, double* out, cudaStream_t s);

// w[n] -= c v[n] (v null: w unchanged), then out[0] = sum_n w[n]^2.
void axpy_norm(double* w, const double* v, double c, int64_t n, double* partial, double* out, cudaStream_t s);

// z[n] = v[n] * inv[n / blk]  (blk = entries per (element, field, component) block).
template <typename S>
void precond_apply(S* z, const S* v, const S* inv, int64_t blk, int64_t n, cudaStream_t s,
                   const int32_t* skip = nullptr);

// x[n] += inv[n / blk] * sum_{i < st->k} st->yc[i] V[i*ldv + n], st->k <= m.
template <typename S, typename X>
void precond_combine(X* x, const S* V, int64_t ldv, int m, const S* inv, int64_t blk, int64_t n, cudaStream_t s,
                     const GmresState* st);

// ---- device-side GMRES: reductions whose last block takes the scalar step that follows ----
// Each launch is skipped on the device once the cycle (st->skip) or the slab (st->halt) has stopped.

// The step after the norm of an FP64 vector.
struct NormStep {
  enum Kind {
    kSlabStart,  // st->ref = norm; iteration count, flags and targets reset (tol, max_it, inexact)
    kResidual,   // red[0] = norm^2 (inexact solve: the weighted norm follows)
    kCheck,      // red[slot] = norm^2, the slab's stop test on the true residual (R6): sets
                 // outer_done, and skip when done, at the iteration cap or at R = 0; then, with
                 // init, the start of the restart cycle: v_0 = start / (-|start|) and its threshold
    kStart32     // red[2] = |v32|^2 and the start of an FP32 cycle (threshold at least 1e-6 |start|)
  } kind = kResidual;
  double tol = 0.0;
  int max_it = 0, inexact = 0, slot = 0, init = 0;
};
void gmres_norm(const double* v, int64_t n, double* partial, GmresState* st, const NormStep& step, cudaStream_t s);
// v32 = (float) v, then the kStart32 step.
void gmres_start32(const double* v, float* v32, int64_t n, double* partial, GmresState* st, cudaStream_t s);
// Iteration j: dot products of w with V[0..j] and |w|^2, the Gram-Schmidt coefficients and H column.
template <typename S>
void gmres_dots(const S* w, const S* V, int64_t ldv, int j, int64_t n, double* partial, GmresState* st,
                cudaStream_t s);
// Iteration j: w -= sum_i cc[i] V[i] and |w|^2; with reorth a second pass where |w| fell below 1/sqrt(2)
// of its value (the DGKS test); then the Givens step, which stops the cycle on |g_{j+1}| <= tol_abs,
// breakdown, the iteration cap or its end (j = m - 1) and there solves for the coefficients yc.
template <typename S>
void gmres_update(S* w, const S* V, int64_t ldv, int j, int64_t n, double* partial, GmresState* st, int m, bool reorth,
                  cudaStream_t s);

// out = 1/2 sum_n mass[n / n3] u[n]^2 (state layout, blocks of n3 per (element, field, component)).
void energy_brick(const double* u, const double* mass, int64_t n3, int64_t n, double* partial, double* out,
                  cudaStream_t s);

// dst[n] = (D) src[n]
template <typename D, typename S>
void convert(D* dst, const S* src, int64_t n, cudaStream_t s, const int32_t* skip = nullptr);

}  // namespace stm
