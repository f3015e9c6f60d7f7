// K-GRAPE evaluation in a parity-excitation (PE) subspace of the XXZ chain (Sec. 3.1), one CTA
// per control pulse, and the host side of the kg_sector_* entry points.
//
// The subspaces of Sec. 3.1 are small (D of a few hundred to a few thousand) and the pulses long
// (M = 4D slices), so a pulse is a long chain of short Krylov steps whose cost is latency.  A CTA
// keeps the whole state in shared memory and runs the forward sweep, the target overlap, the
// co-state sweep with the gradient overlaps and the gradient assembly of one pulse with nothing
// but block barriers; the CTAs of a launch take independent pulses (a batch: line-search
// candidates, restarts, scans).
//
// H0 in the reduced basis.  Basis vector r is |r> = (|s_r> + p |Pi s_r>)/sqrt(n_r) over the orbit
// {s_r, Pi s_r} (n_r = 1 for a palindrome).  Since H0 commutes with Pi,
//   <r'|H0|r> = sqrt(n_r'/n_r) sum_{t in orbit r} phi(t) <t|H0|s_r'>,
// phi(t) = +1 for the smaller member of its orbit, p for the mirrored one (parity 0: one state per
// orbit).  Row r' therefore needs H0 applied to the single state s_r': its diagonal
// (Jz/4)(L-1 - 2 popcount((s ^ s>>1) & mask)), computed on the fly, and one term Jxy/2 per
// antiparallel bond, landing in orbit r(t) with the factor sqrt(n_r'/n_r(t)) phi(t), one of 1, sqrt 2,
// 1/sqrt 2 and -1.  The host splits those terms by weight, so that the kernel decodes no weight: list A
// holds the columns of weight Jxy/2, in an ELL layout [entry][row]; list B those of a second weight
// (even parity: Jxy/(2 sqrt 2), a sqrt 2 listed twice; odd: -Jxy/2), which few rows have, in one ELL
// slice per 32 rows.  Padding points at a zero element behind the vector.  Columns are 16 bits, two
// in a word; the CTA keeps both lists in shared memory.  A row has between 1 and 2 K antiparallel bonds
// (L = 14, K = 4: 5.7 of 8 on average), so the kernel's rows are the basis vectors in order of their lists'
// length, and 32 rows stop at the longest of theirs: with all rows as long as the longest one (us a slice, m =
// 10) complex64 69.0 instead of 64.3 at D = 511, 53.3 instead of 43.4 at D = 1204, 78.5 instead of 76.4 at D = 2445;
// float-float 85.9 instead of 74.3 and 107.8 instead of 96.7; complex128 145 instead of 121 and 325 instead of 274.  Hc is diagonal
// (mirror-symmetric Sz mask): hc_amp (popcount(mask) - 2 popcount(s & mask))/2.
//
// One Lanczos step (App. A, Alg. "Lanczos", Paige's order), thread t owning rows t + NT i, v_{k-1}, v_k
// and w in registers, v_k in shared memory for the gather:
//   w       = H v_k - b_k v_{k-1}
//   alpha_k = <v_k|w>,  b_{k+1}^2 = ||w||^2 - 2 alpha_k <v_k|w> + alpha_k^2 ||v_k||^2   (one block reduction)
//   v_{k+1} = (w - alpha_k v_k) / b_{k+1}               (into shared memory and the basis)
// with two block barriers: every warp adds up the warps' partial sums and forms the scalars for itself.
// Complex64 path: vectors and partial sums in FP32, cross-warp sums, the tridiagonal T, its exponential and the
// norms between slices in float-float (warp 0, once per slice): a step has no FP64 instruction, a slice only
// the conversion of its control.  Complex128 path: FP64 throughout (the error indicator and the breakdown
// test, a comparison with a tolerance, in FP32).
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstring>
#include <string>
#include <unordered_map>
#include <type_traits>
#include <vector>

#include "kg_device.cuh"
#include "kg_launch.h"

namespace kg {

// ---------------------------------------------------------------- float-float vectors (KG_PREC_FF)
// Every amplitude is the unevaluated sum hi + lo of two FP32 numbers (about 44 significant bits),
// and the arithmetic on it is FP32 with error-free transformations (Knuth's TwoSum, the FMA
// TwoProduct: ff_add, ff_mul), so that the rounding of the Krylov vectors -- what limits the
// complex64 path over the 2 x 4D slices of Sec. 3.2's pulses -- shrinks by about 2^20 without one
// FP64 instruction (1/64 of the FP32 rate on this GPU) per amplitude.  alpha and b stay float-float too; the
// norms and overlaps of a slice, T and its exponential are FP64, as on the complex128 path.
struct FFR {
  float hi, lo;
  FFR() = default;
  __device__ __forceinline__ FFR(float h, float l) : hi(h), lo(l) {}
  __device__ __forceinline__ FFR(int a) : hi((float)a), lo(0.f) {}
  __device__ __forceinline__ explicit FFR(double a) : hi((float)a), lo((float)(a - (double)(float)a)) {}
  __device__ __forceinline__ explicit operator double() const { return (double)hi + (double)lo; }
  __device__ __forceinline__ explicit operator float() const { return __fadd_rn(hi, lo); }
};
// A complex amplitude: high parts of (re, im), then low parts, so that the packed FP32x2 instructions work
// on both components at once: half the instructions of two scalar float-float numbers, which the
// kernel's issue slots bound.
struct __align__(16) FFC {
  float2 hi, lo;
};
__device__ __forceinline__ FFR operator+(FFR a, FFR b) {
  const FF s = ff_add(FF{a.hi, a.lo}, FF{b.hi, b.lo});
  return FFR(s.hi, s.lo);
}
__device__ __forceinline__ FFR operator-(FFR a) { return FFR(-a.hi, -a.lo); }
__device__ __forceinline__ FFR operator-(FFR a, FFR b) { return a + (-b); }
__device__ __forceinline__ FFR operator*(FFR a, FFR b) {
  const FF p = ff_mul(FF{a.hi, a.lo}, FF{b.hi, b.lo});
  return FFR(p.hi, p.lo);
}
__device__ __forceinline__ FFR fma(FFR a, FFR b, FFR c) { return a * b + c; }
// 1/sqrt(a) and sqrt(a): the FP32 estimate y refined by r/2 + 3 r^2 / 8, r = 1 - a y^2 formed exactly.
__device__ __forceinline__ void ff_rsqrt(FF a, FF& root, FF& inv) {
  if (!(a.hi > 1e-30f)) {
    root = ff_sqrt(a);
    inv = (root.hi > 0.f) ? ff_rcp(root) : FF{0.f, 0.f};
    return;
  }
  const float y = rsqrtf(a.hi);
  const float p = __fmul_rn(a.hi, y), e = __fmaf_rn(a.hi, y, -p);
  const float q = __fmul_rn(p, y), f = __fmaf_rn(p, y, -q);
  const float r = __fsub_rn(__fsub_rn(__fsub_rn(1.f, q), f), __fmul_rn(__fmaf_rn(a.lo, y, e), y));
  inv = ff_two_sum(y, __fmul_rn(__fmul_rn(y, r), __fmaf_rn(0.375f, r, 0.5f)));
  root = ff_mul(a, inv);
}
// The float-float operations on both components (packed FP32x2; see ff_two_sum, ff_mul, ff_dot3).
__device__ __forceinline__ float2 p2_add(float2 a, float2 b) { return __fadd2_rn(a, b); }
__device__ __forceinline__ float2 p2_sub(float2 a, float2 b) { return __ffma2_rn(b, make_float2(-1.f, -1.f), a); }
__device__ __forceinline__ float2 p2_mul(float2 a, float2 b) { return __fmul2_rn(a, b); }
__device__ __forceinline__ float2 p2_fma(float2 a, float2 b, float2 c) { return __ffma2_rn(a, b, c); }
__device__ __forceinline__ float2 p2_neg(float2 a) { return make_float2(-a.x, -a.y); }
__device__ __forceinline__ FFC ffc_two_sum(float2 a, float2 b) {
  const float2 s = p2_add(a, b), bb = p2_sub(s, a);
  return {s, p2_add(p2_sub(a, p2_sub(s, bb)), p2_sub(b, bb))};
}
__device__ __forceinline__ FFC ffc_close(float2 hi, float2 lo) {  // renormalised hi + lo, |lo| << |hi|
  const float2 h = p2_add(hi, lo);
  return {h, p2_sub(lo, p2_sub(h, hi))};
}
__device__ __forceinline__ FFC ffc_bcast(FFR a) { return {make_float2(a.hi, a.hi), make_float2(a.lo, a.lo)}; }
// a b = p + t: the products by FMA TwoProduct with the cross terms in t
__device__ __forceinline__ void ffc_prod(FFC a, FFC b, float2& p, float2& t) {
  p = p2_mul(a.hi, b.hi);
  t = p2_fma(a.hi, b.lo, p2_fma(a.lo, b.hi, p2_fma(a.hi, b.hi, p2_neg(p))));
}
__device__ __forceinline__ FFC ffc_mul(FFC a, FFC b) {
  float2 p, t;
  ffc_prod(a, b, p, t);
  return ffc_close(p, t);
}
__device__ __forceinline__ FFC ffc_fma(FFC a, FFC b, FFC c) {  // a b + c
  float2 p, t;
  ffc_prod(a, b, p, t);
  const FFC s = ffc_two_sum(c.hi, p);
  return ffc_close(s.hi, p2_add(s.lo, p2_add(t, c.lo)));
}
__device__ __forceinline__ FFC ffc_dot3(FFC a, FFC x, FFC b, FFC y, FFC c, FFC z) {
  float2 p, q, r, tp, tq, tr;
  ffc_prod(a, x, p, tp);
  ffc_prod(b, y, q, tq);
  ffc_prod(c, z, r, tr);
  const FFC s = ffc_two_sum(p, r), u = ffc_two_sum(s.hi, q);
  return ffc_close(u.hi, p2_add(p2_add(p2_add(tp, tr), tq), p2_add(s.lo, u.lo)));
}
// Unevaluated sum of many float-float terms: the high parts by TwoSum, everything below them in one FP32
// accumulator; ffc_close renormalises once at the end.
__device__ __forceinline__ void ffc_acc(FFC& a, FFC v) {
  const FFC s = ffc_two_sum(a.hi, v.hi);
  a.hi = s.hi;
  a.lo = p2_add(a.lo, p2_add(s.lo, v.lo));
}
__device__ __forceinline__ void ffc_acc_mul(FFC& a, FFC x, FFC y) {  // a += x y, by component
  float2 p, t;
  ffc_prod(x, y, p, t);
  const FFC s = ffc_two_sum(a.hi, p);
  a.hi = s.hi;
  a.lo = p2_add(a.lo, p2_add(s.lo, t));
}
__device__ __forceinline__ FF ff_of(FFR a) { return FF{a.hi, a.lo}; }
__device__ __forceinline__ FFR ffr_of(FF a) { return FFR(a.hi, a.lo); }
using ::fma;  // the float and double functions stay visible beside the overload inside namespace kg
template <> struct VecTraits<FFC> { using R = FFR; };
template <> __device__ __forceinline__ FFC vmake<FFC>(FFR a, FFR b) {
  return FFC{make_float2(a.hi, b.hi), make_float2(a.lo, b.lo)};
}
// The components of an amplitude.
__device__ __forceinline__ float vre(float2 a) { return a.x; }
__device__ __forceinline__ float vim(float2 a) { return a.y; }
__device__ __forceinline__ double vre(double2 a) { return a.x; }
__device__ __forceinline__ double vim(double2 a) { return a.y; }
__device__ __forceinline__ FFR vre(FFC a) { return FFR(a.hi.x, a.lo.x); }
__device__ __forceinline__ FFR vim(FFC a) { return FFR(a.hi.y, a.lo.y); }


// Meta word of 32 rows: first word of their list B, words a row of list A, words a row of list B.
__host__ __device__ constexpr unsigned sec_meta(unsigned first, unsigned na, unsigned nb) { return first << 12 | na << 6 | nb; }
__host__ __device__ constexpr unsigned sec_meta_first(unsigned m) { return m >> 12; }
__host__ __device__ constexpr unsigned sec_meta_na(unsigned m) { return (m >> 6) & 63u; }
__host__ __device__ constexpr unsigned sec_meta_nb(unsigned m) { return m & 63u; }

struct SectorParams {
  int D, N, m, B, L1, grad_mode;
  int na2, rows, groups, words;  // list A: words per row, row stride; 32-row groups; words of the whole table
  unsigned maskL1, hc_mask;
  double qz, hc_amp, dt, bd_tol;
  double wa, wb;                 // weights of lists A and B
  float wa_f, wb_f, dt_f, bd_tol_f;  // the same, dt and the breakdown tolerance rounded to FP32
  const unsigned* tab_g;         // [na2][rows] list A, [groups] meta words (sec_meta_*), list B
  const unsigned* states;        // [D] s_r of the kernel's row r
  const unsigned short* perm;    // [D] basis index of the kernel's row r
  const double* u;               // [B][N]
  const double* psi0;            // [2D] complex128
  const double* target;          // [2D] complex128
  double* fid;                   // [B]
  double* grad;                  // [B][N] or null
  void* traj;                    // [grid][N+1][D] psi_0..psi_N of the pulse in hand
  void* basis;                   // [grid][m][D] Lanczos vectors of the slice in hand
  void* tint;                    // [grid][2N][D] interior Gauss-Lobatto states (KG_GRAD_EXACT), or null
  double* G;                     // [grid][N+1]
  double* scal;                  // [B][kScCount]
  int* ctrl;                     // status word
  long long time_limit_ns;       // per pulse
  long long* prof;               // [8] phase cycles of CTA 0 (KG_FLAG_PHASE_TIMING), or null
};

// Block barrier of this kernel.  Several barriers follow work that only thread 0 does (FP64
// square roots and divisions, the failure record, the time check), so lanes of warp 0 may reach
// them apart.  __syncthreads() is PTX's .aligned barrier, whose behaviour is undefined unless every
// warp arrives converged at the same barrier instruction; with it, CTAs that evaluated a second
// pulse came out of step by a barrier.  The barrier without .aligned waits per thread and is
// defined for diverged arrival.
__device__ __forceinline__ void sec_sync() { asm volatile("barrier.sync 0;" ::: "memory"); }

struct SecSmem {
  float red_f[2][16 * 4];   // warp partials by reduction parity: complex64
  float2 red_ff[2][16 * 4]; // float-float
  double red_d[2][16 * 4];  // complex128, and FP64 sums of every path
  double alpha[kMaxM], beta[kMaxM + 1];    // T, FP64
  float alpha_f[kMaxM], beta_f[kMaxM + 1]; // its FP32 copies (norm bounds, Taylor terms)
  float2 ff_a[kMaxM], ff_n[kMaxM], ff_q[kMaxM], ff_e[kMaxM];  // the steps' sums; ff_e: b_{k+1}^2 (complex64),
                                                              // or the explicit one (float-float)
  float2 tau_ff[3];            // complex64: dt and the interior quadrature nodes
  float2 diag_ff[4];           // Jz / 4, hc_amp / 2, weights of lists A and B: float-float
  double diag_d[4];
  float coef_f[3][2][kMaxM];   // [slice end, interior node a, b][re, im][k]
  double coef_d[3][2][kMaxM];
  float err_max;
  unsigned ff_e_set;
  int breakdowns;
  int abort;                    // the pulse in hand is abandoned (status set)
  int fail_step, fail_check;    // where it was abandoned (sec_record)
  long long prof_last, prof_acc[8];  // phase timing (thread 0 of CTA 0)
  unsigned long long t_start;   // globaltimer at the pulse's start
};

// Phase timing (KG_FLAG_PHASE_TIMING, thread 0 of CTA 0): cycles since the last mark go to
// counter `ph`: 0 Lanczos gathers and updates, 1 block reductions, 4 tridiagonal T and small
// exponential, 5 recombination, 6 pulse setup and overlaps.
__device__ __forceinline__ void sec_mark(const SectorParams& p, SecSmem& sm, int ph) {
  if (p.prof && blockIdx.x == 0 && threadIdx.x == 0) {
    const long long now = clock64();
    sm.prof_acc[ph] += now - sm.prof_last;
    sm.prof_last = now;
  }
}

// ---------------------------------------------------------------- block reductions
// Every thread receives the three totals, the same bits in each.  One barrier: the warps' partials, then
// every warp adds them up for itself (the partials alternate between two sets, so that the next
// reduction's do not overwrite what a slow warp still reads).
template <int NT>
__device__ __forceinline__ void sec_reduce(SecSmem& sm, int& par, float v0, float v1, float v2, FF (&out)[3]) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  float* red = sm.red_f[par];
  par ^= 1;
  const float s = warp_sum3(v0, v1, v2);
  if (lane < 4) red[warp * 4 + lane] = s;
  sec_sync();
  warps_sum3<NT / 32, FF>([&](int w, int i) { return FF{red[w * 4 + i], 0.f}; }, out);
}
template <int NT>
__device__ __forceinline__ void sec_reduce(SecSmem& sm, int& par, FF v0, FF v1, FF v2, FF (&out)[3]) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  float2* red = sm.red_ff[par];
  par ^= 1;
  const FF s = warp_sum3(v0, v1, v2);
  if (lane < 4) red[warp * 4 + lane] = make_float2(s.hi, s.lo);
  sec_sync();
  warps_sum3<NT / 32, FF>([&](int w, int i) { return FF{red[w * 4 + i].x, red[w * 4 + i].y}; }, out);
}
template <int NT>
__device__ __forceinline__ void sec_reduce(SecSmem& sm, int& par, double v0, double v1, double v2, double (&out)[3]) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  double* red = sm.red_d[par];
  par ^= 1;
  const double s = warp_sum3(v0, v1, v2);
  if (lane < 4) red[warp * 4 + lane] = s;
  sec_sync();
  warps_sum3<NT / 32, double>([&](int w, int i) { return red[w * 4 + i]; }, out);
}

__device__ __forceinline__ void sec_flag(const SectorParams& p, int code) { atomicCAS(p.ctrl, 0, code); }

// Where a pulse was abandoned, kept in the pulse's scalar block for diagnosis: scal[5] = slice
// (+j forward, -j backward), scal[6] = Lanczos step (-1: after the loop), scal[7] = check
// (1 non-finite step sums, 2 non-finite norm, 3 tridiagonal bound, 4 time limit).  Thread 0 only.
__device__ __forceinline__ void sec_record(SecSmem& sm, int k, int check) {
  if (sm.fail_check == 0) {
    sm.fail_step = k;
    sm.fail_check = check;
  }
}

template <class V> __device__ __forceinline__ V vscale(typename VecTraits<V>::R a, V x) {
  if constexpr (std::is_same<V, FFC>::value) return ffc_mul(ffc_bcast(a), x);
  else return vmake<V>(a * x.x, a * x.y);
}
template <class V> __device__ __forceinline__ V vaxpy(typename VecTraits<V>::R a, V x, V y) {
  if constexpr (std::is_same<V, FFC>::value) return ffc_fma(ffc_bcast(a), x, y);
  else return vmake<V>(fma(a, x.x, y.x), fma(a, x.y, y.y));
}
// (a + ib) x + y, the part with b first
template <class V>
__device__ __forceinline__ V vcaxpy(typename VecTraits<V>::R a, typename VecTraits<V>::R b, V x, V y) {
  if constexpr (std::is_same<V, FFC>::value) {
    const FFC fb{make_float2(-b.hi, b.hi), make_float2(-b.lo, b.lo)};
    const FFC xs{make_float2(x.hi.y, x.hi.x), make_float2(x.lo.y, x.lo.x)}, one = ffc_bcast(FFR(1));
    return ffc_dot3(ffc_bcast(a), x, fb, xs, one, y);
  } else {
    return vmake<V>(fma(a, x.x, fma(-b, x.y, y.x)), fma(a, x.y, fma(b, x.x, y.y)));
  }
}

// ---------------------------------------------------------------- per-precision scalars
// S: a step's sums; N: ||x|| between slices.
template <class V> struct SecPrec;
template <> struct SecPrec<float2> {
  using S = FF;
  using N = FF;
};
template <> struct SecPrec<FFC> {
  using S = FF;
  using N = double;
};
template <> struct SecPrec<double2> {
  using S = double;
  using N = double;
};
// Per-row partial sums: acc += Re(conj(x) y) (float-float: by component, added up in sclose).
__device__ __forceinline__ void sacc(float& a, float2 x, float2 y) { a = fmaf(x.y, y.y, fmaf(x.x, y.x, a)); }
__device__ __forceinline__ void sacc(double& a, double2 x, double2 y) { a = ::fma(x.y, y.y, ::fma(x.x, y.x, a)); }
__device__ __forceinline__ void sacc(FFC& a, FFC x, FFC y) { ffc_acc_mul(a, x, y); }
__device__ __forceinline__ float sclose(float a) { return a; }
__device__ __forceinline__ double sclose(double a) { return a; }
__device__ __forceinline__ FF sclose(FFC a) {
  const FFC c = ffc_close(a.hi, a.lo);
  return ff_add(FF{c.hi.x, c.lo.x}, FF{c.hi.y, c.lo.y});
}
template <class V> struct SecAcc { using T = typename VecTraits<V>::R; };
template <> struct SecAcc<FFC> { using T = FFC; };

// alpha_k, b_{k+1} and 1/b_{k+1} from a step's sums (or from an explicit b_{k+1}^2).
__device__ __forceinline__ FF sec_b2(const FF (&o)[3]) {
  return ff_add(o[1], ff_mul(ff_mul(o[0], o[0]), ff_add(o[2], FF{-2.f, 0.f})));
}
__device__ __forceinline__ double sec_b2(const double (&o)[3]) { return ::fma(o[0] * o[0], o[2] - 2.0, o[1]); }
__device__ __forceinline__ void sec_roots(FF b2, float& b, float& ib) {
  FF r, i;
  ff_rsqrt(b2, r, i);
  b = __fadd_rn(r.hi, r.lo);
  ib = __fadd_rn(i.hi, i.lo);
}
__device__ __forceinline__ void sec_roots(FF b2, FFR& b, FFR& ib) {
  FF r, i;
  ff_rsqrt(b2, r, i);
  b = ffr_of(r);
  ib = ffr_of(i);
}
__device__ __forceinline__ void sec_roots(double b2, double& b, double& ib) {
  if (!(b2 > 1e-30 && b2 < 1e30)) {
    b = ::sqrt(::fmax(b2, 0.0));
    ib = (b > 0.0) ? 1.0 / b : 0.0;
    return;
  }
  const double y = (double)rsqrtf((float)b2);  // one step of Halley's iteration: 2^-22 -> below 2^-60
  const double r = ::fma(-b2 * y, y, 1.0);
  ib = ::fma(y, r * ::fma(0.375, r, 0.5), y);
  b = b2 * ib;
}
__device__ __forceinline__ float sec_top(FF a) { return a.hi; }
__device__ __forceinline__ double sec_top(double a) { return a; }
// The identity for b^2 cancels: near an invariant subspace.
__device__ __forceinline__ bool sec_cancels(FF b2, FF n) { return b2.hi < 1e-3f * n.hi; }
__device__ __forceinline__ bool sec_cancels(double b2, double n) { return b2 < 1e-3 * n; }
__device__ __forceinline__ float sec_real(FF a, float) { return __fadd_rn(a.hi, a.lo); }
__device__ __forceinline__ FFR sec_real(FF a, FFR) { return ffr_of(a); }
__device__ __forceinline__ double sec_real(double a, double) { return a; }
__device__ __forceinline__ float sec_f32(float a) { return a; }
__device__ __forceinline__ float sec_f32(double a) { return (float)a; }
__device__ __forceinline__ float sec_f32(FFR a) { return a.hi; }
// A sum kept in 8 bytes of a double array between slices.
__device__ __forceinline__ double sec_pack(FF a) { return __hiloint2double(__float_as_int(a.hi), __float_as_int(a.lo)); }
__device__ __forceinline__ double sec_pack(double a) { return a; }
template <bool F32>
__device__ __forceinline__ double sec_unpack(double d) {
  if constexpr (F32) return (double)__int_as_float(__double2hiint(d)) + (double)__int_as_float(__double2loint(d));
  else return d;
}

// The diagonals of H0 and of Hc on the row of state st: a weight (float-float, so that FP32 and
// float-float need no FP64 instruction) times a small whole number.
__device__ __forceinline__ float sec_times(const SecSmem& sm, int which, int n, float) {
  const float2 q = sm.diag_ff[which];
  return fmaf(q.x, (float)n, q.y * (float)n);
}
// The weights of lists A (2) and B (3) in the vectors' real type.  Complex64: rounded by the host (the
// conversion of an FP64 parameter is an FP64 instruction, which every warp of every step repeated: D = 511
// 63.0 us a slice instead of 61.7, one pulse at D = 110 16.3 instead of 15.3); float-float and complex128: from
// shared memory, as their conversion or constant operand in the loop costs FP64 issue (2 and 7 % at D = 2445).
__device__ __forceinline__ float sec_weight(const SectorParams& p, const SecSmem&, int which, float) {
  return which == 2 ? p.wa_f : p.wb_f;
}
__device__ __forceinline__ FFR sec_weight(const SectorParams&, const SecSmem& sm, int which, FFR) {
  return FFR(sm.diag_ff[which].x, sm.diag_ff[which].y);
}
__device__ __forceinline__ double sec_weight(const SectorParams&, const SecSmem& sm, int which, double) {
  return sm.diag_d[which];
}
__device__ __forceinline__ FFR sec_times(const SecSmem& sm, int which, int n, FFR) {
  const float2 q = sm.diag_ff[which];
  return ffr_of(ff_mul(FF{q.x, q.y}, FF{(float)n, 0.f}));
}
__device__ __forceinline__ double sec_times(const SecSmem& sm, int which, int n, double) {
  return sm.diag_d[which] * (double)n;
}
template <class R>
__device__ __forceinline__ R sec_d0(const SectorParams& p, const SecSmem& sm, unsigned st) {
  return sec_times(sm, 0, p.L1 - 2 * __popc((st ^ (st >> 1)) & p.maskL1), R());
}
template <class R>
__device__ __forceinline__ R sec_hc(const SectorParams& p, const SecSmem& sm, unsigned st) {
  return sec_times(sm, 1, __popc(p.hc_mask) - 2 * __popc(st & p.hc_mask), R());
}

// ---------------------------------------------------------------- H in the subspace
// h = (diagonal + H0's couplings) x - bk xp on the own rows; S holds x for the gather (element D is 0).
// The words of list A are read row by row in step, so that every thread has its rows' loads in flight
// together; the rows are ordered by the length of their lists, longest first, so that 32 rows read no more
// words than the longest of them has, and a thread's last rows fewer than its first.
// The tables hold 8 x the column (at most 8 x 4096): the byte offset of a complex64 amplitude, which saves the
// shift (D = 511 64.5 -> 63.4 us a slice, D = 1204 43.4 -> 42.1; the 16-byte types shift either way).
template <class V>
__device__ __forceinline__ V sec_elem(const V* S, unsigned at8) {  // element at8 / 8
  return *reinterpret_cast<const V*>(reinterpret_cast<const char*>(S) + at8 * (unsigned)(sizeof(V) / 8));
}
template <class V, int NT, int RPT>
__device__ __forceinline__ void sec_apply(const SectorParams& p, const SecSmem& sm, const V* S, const unsigned* tab,
                                          const typename VecTraits<V>::R (&dj)[RPT], const V (&x)[RPT],
                                          typename VecTraits<V>::R bk, const V (&xp)[RPT], V (&h)[RPT]) {
  using R = typename VecTraits<V>::R;
  constexpr bool FFM = std::is_same<R, FFR>::value;
  const int tid = threadIdx.x, D = p.D;
  const unsigned* ta = tab + min(tid, D);
  const unsigned* meta = tab + p.na2 * p.rows;
  const unsigned* tb = meta + p.groups + (tid & 31);
  const R wa = sec_weight(p, sm, 2, R());
  unsigned mt[RPT];
#pragma unroll
  for (int i = 0; i < RPT; ++i) {
    const int g = (tid >> 5) + (NT / 32) * i;
    mt[i] = (g < p.groups) ? meta[g] : 0u;
  }
  const int na_all = (int)sec_meta_na(mt[RPT - 1]), na = (int)sec_meta_na(mt[0]);
  if constexpr (FFM) {
    FFC acc[RPT];
#pragma unroll
    for (int i = 0; i < RPT; ++i) acc[i] = FFC{make_float2(0.f, 0.f), make_float2(0.f, 0.f)};
    auto entry = [&](int q, int i) {
      const unsigned w = (tid + NT * i <= D) ? ta[q * p.rows + NT * i] : tab[q * p.rows + D];
      ffc_acc(acc[i], sec_elem(S, w & 0xffffu));
      ffc_acc(acc[i], sec_elem(S, w >> 16));
    };
    for (int q = 0; q < na_all; ++q) {
#pragma unroll
      for (int i = 0; i < RPT; ++i) entry(q, i);
    }
    for (int q = na_all; q < na; ++q) {
#pragma unroll
      for (int i = 0; i < RPT; ++i)
        if (i == 0 || q < (int)sec_meta_na(mt[i])) entry(q, i);
    }
    const FFC wf = ffc_bcast(wa), nb = ffc_bcast(-bk);
#pragma unroll
    for (int i = 0; i < RPT; ++i)
      h[i] = ffc_dot3(ffc_bcast(dj[i]), x[i], wf, ffc_close(acc[i].hi, acc[i].lo), nb, xp[i]);
  } else {
#pragma unroll
    for (int i = 0; i < RPT; ++i) h[i] = vscale<V>(dj[i], x[i]);
    auto entry = [&](int q, int i) {
      const unsigned w = (tid + NT * i <= D) ? ta[q * p.rows + NT * i] : tab[q * p.rows + D];
      h[i] = vaxpy<V>(wa, sec_elem(S, w & 0xffffu), h[i]);
      h[i] = vaxpy<V>(wa, sec_elem(S, w >> 16), h[i]);
    };
#pragma unroll 2
    for (int q = 0; q < na_all; ++q) {
#pragma unroll
      for (int i = 0; i < RPT; ++i) entry(q, i);
    }
    for (int q = na_all; q < na; ++q) {
#pragma unroll
      for (int i = 0; i < RPT; ++i)
        if (i == 0 || q < (int)sec_meta_na(mt[i])) entry(q, i);
    }
#pragma unroll
    for (int i = 0; i < RPT; ++i) h[i] = vaxpy<V>(-bk, xp[i], h[i]);
  }
#pragma unroll
  for (int i = 0; i < RPT; ++i) {  // list B: the same number of words for all lanes of a warp
    if (sec_meta_nb(mt[i])) {
      const R wb = sec_weight(p, sm, 3, R());
      for (unsigned q = 0; q < sec_meta_nb(mt[i]); ++q) {
        const unsigned w = tb[sec_meta_first(mt[i]) + 32 * q];
        h[i] = vaxpy<V>(wb, sec_elem(S, w & 0xffffu), h[i]);
        h[i] = vaxpy<V>(wb, sec_elem(S, w >> 16), h[i]);
      }
    }
  }
}

// Taylor-hierarchy terms of backward slice j (App. B, Eq. gradp), this thread's partial sum:
// x was chi_j, psi_end is psi_j, H = H_j, and Im <chi| Hbar_c^[P] |psi> with a_m = H^m chi,
// b_n = H^n psi and Hc diagonal is
//   P = 1: Im M00 - (dt/2) Re(M10 - M01);  P = 2: also - (dt^2/6) Im(M20 - 2 M11 + M02),
// M_mn = <a_m|Hc|b_n>.  The a_m come from the slice's Lanczos vectors (H v_0 = alpha_0 v_0 +
// b_1 v_1, H v_1 = b_1 v_0 + alpha_1 v_1 + b_2 v_2), the b_n from the slice's gather applied to
// psi_j once or twice.  Nothing reads the shared vectors after the Lanczos loop.  Kept out of
// line: it runs once per backward slice and its arrays would crowd the Lanczos loop's registers.
template <class V, int NT, int RPT>
__device__ __noinline__ typename VecTraits<V>::R sec_taylor(const SectorParams& p, SecSmem& sm, V* Sa, V* Sb,
                                                          const unsigned* tab, const V* basis, double uj,
                                                          int meff, typename VecTraits<V>::R nin, int taylor,
                                                          const V* psi_end) {
  using R = typename VecTraits<V>::R;
  constexpr bool F32 = sizeof(R) == 4;
  const int tid = threadIdx.x, D = p.D;
  // the diagonals of H0 and Hc, formed again here from the rows' states
  R dj[RPT], hh[RPT];
#pragma unroll
  for (int i = 0; i < RPT; ++i) {
    const int r = tid + NT * i;
    dj[i] = 0;
    hh[i] = 0;
    if (r < D) {
      const unsigned st = __ldg(p.states + r);
      hh[i] = sec_hc<R>(p, sm, st);
      dj[i] = fma((R)uj, hh[i], sec_d0<R>(p, sm, st));
    }
  }
  R pt = 0;
  V b0[RPT], b1[RPT], b2[RPT];
#pragma unroll
  for (int i = 0; i < RPT; ++i) {
    const int r = tid + NT * i;
    b0[i] = (r < D) ? psi_end[r] : vmake<V>(0, 0);
    b1[i] = b2[i] = vmake<V>(0, 0);
    if (r < D) Sa[r] = b0[i];
  }
  sec_sync();
  sec_apply<V, NT, RPT>(p, sm, Sa, tab, dj, b0, (R)0, b2, b1);
  if (taylor >= 2) {
#pragma unroll
    for (int i = 0; i < RPT; ++i) {
      const int r = tid + NT * i;
      if (r < D) Sb[r] = b1[i];
    }
    sec_sync();
    sec_apply<V, NT, RPT>(p, sm, Sb, tab, dj, b1, (R)0, b0, b2);
  }
  const R al0 = (meff > 0) ? (F32 ? (R)sm.alpha_f[0] : (R)sm.alpha[0]) : (R)0;
  const R al1 = (meff > 1) ? (F32 ? (R)sm.alpha_f[1] : (R)sm.alpha[1]) : (R)0;
  const R be1 = (meff > 1) ? (F32 ? (R)sm.beta_f[1] : (R)sm.beta[1]) : (R)0;
  const R be2 = (meff > 2) ? (F32 ? (R)sm.beta_f[2] : (R)sm.beta[2]) : (R)0;
  const R c0 = al0 * al0 + be1 * be1, c1 = be1 * (al0 + al1), c2 = be1 * be2;
  const R h1 = (R)(0.5 * p.dt), h2 = (R)(p.dt * p.dt / 6.0);
#pragma unroll
  for (int i = 0; i < RPT; ++i) {
    const int r = tid + NT * i;
    if (r < D && meff > 0) {
      const V v0 = basis[r];
      const V v1 = (meff > 1) ? basis[(size_t)D + r] : vmake<V>(0, 0);
      const V v2 = (taylor >= 2 && meff > 2) ? basis[(size_t)2 * D + r] : vmake<V>(0, 0);
      const V a0 = vscale<V>(nin, v0);
      const V a1 = vscale<V>(nin, vaxpy<V>(be1, v1, vscale<V>(al0, v0)));
      // conj(a) b = (a.x b.x + a.y b.y) + i (a.x b.y - a.y b.x)
      R t = a0.x * b0[i].y - a0.y * b0[i].x;                                                   // Im M00
      t -= h1 * ((a1.x * b0[i].x + a1.y * b0[i].y) - (a0.x * b1[i].x + a0.y * b1[i].y));     // Re(M10 - M01)
      if (taylor >= 2) {
        const V a2 = vscale<V>(nin, vaxpy<V>(c2, v2, vaxpy<V>(c1, v1, vscale<V>(c0, v0))));
        const R i20 = a2.x * b0[i].y - a2.y * b0[i].x, i11 = a1.x * b1[i].y - a1.y * b1[i].x;
        const R i02 = a0.x * b2[i].y - a0.y * b2[i].x;
        t -= h2 * (i20 - (R)2 * i11 + i02);
      }
      pt = fma(hh[i], t, pt);
    }
  }
  return pt;
}

// Interior Gauss-Lobatto states of a slice (KG_GRAD_EXACT), from the slice's basis and the
// coefficients warps 1 and 2 formed: forward (lob = 1) psi(t_{j-1} + s) for s = s_a, s_b, stored
// to io[0..D), io[D..2D); backward (lob = 2) chi(t_{j-1} + s), overlapped with those stored states:
// the return value is this thread's share of Im <chi_a|Hc|psi_a> + Im <chi_b|Hc|psi_b>.  Out of line,
// so that its arrays stay out of the Lanczos loop's registers.
template <class V, int NT, int RPT>
__device__ __noinline__ typename VecTraits<V>::R sec_interior(const SectorParams& p, SecSmem& sm, const V* basis,
                                                            int meff, int lob, V* io) {
  using R = typename VecTraits<V>::R;
  constexpr bool F32 = sizeof(R) == 4;
  const int tid = threadIdx.x, D = p.D;
  R pg = 0;
  for (int w = 1; w <= 2; ++w) {
    V y[RPT];
#pragma unroll
    for (int i = 0; i < RPT; ++i) y[i] = vmake<V>(0, 0);
    for (int k = meff - 1; k >= 0; --k) {
      const R a = F32 ? (R)sm.coef_f[w][0][k] : (R)sm.coef_d[w][0][k];
      const R b = F32 ? (R)sm.coef_f[w][1][k] : (R)sm.coef_d[w][1][k];
#pragma unroll
      for (int i = 0; i < RPT; ++i) {
        const int r = tid + NT * i;
        if (r < D) {
          const V q = basis[(size_t)k * D + r];
          y[i].x = fma(a, q.x, fma(-b, q.y, y[i].x));
          y[i].y = fma(a, q.y, fma(b, q.x, y[i].y));
        }
      }
    }
    V* slot = io + (size_t)(w - 1) * D;
#pragma unroll
    for (int i = 0; i < RPT; ++i) {
      const int r = tid + NT * i;
      if (r >= D) continue;
      if (lob == 1) {
        slot[r] = y[i];
      } else {
        const V o = slot[r];
        pg = fma(sec_hc<R>(p, sm, __ldg(p.states + r)), y[i].x * o.y - y[i].y * o.x, pg);  // Im(conj(chi_s) Hc psi_s), Hc diagonal
      }
    }
  }
  return pg;
}

// The small exponentials of a slice and the recombination coefficients, one warp each: the slice end
// (w = 0) and, with lob, the interior nodes s_a, s_b = (1 -+ 1/sqrt 5) dt/2 (forward exp(-i s H) psi_{j-1},
// backward exp(+i (dt - s) H) chi_j, dt - s_a = s_b).  Warp 0 also keeps the error indicator and checks
// the pulse's time limit.
template <class V>
__device__ __forceinline__ void sec_coefficients(const SectorParams& p, SecSmem& sm, int w, bool back, int meff,
                                                 bool broke, float beta_m, typename SecPrec<V>::N nrm, float inv,
                                                 float2 fact) {
  using R = typename VecTraits<V>::R;
  constexpr bool F32 = sizeof(R) == 4;
  const int k = threadIdx.x & 31;
  // The exponential takes ceil(||tau T|| / 4) sub-steps: refuse a T whose Gershgorin bound is not a
  // finite, sane number (it would come from corrupted coefficients) instead of looping on it.
  float row = 0.f;
  if (k < meff) row = p.dt_f * (fabsf(sm.alpha_f[k]) + (k >= 1 ? sm.beta_f[k] : 0.f) + (k + 1 < meff ? sm.beta_f[k + 1] : 0.f));
  row = (row == row) ? row : 3.0e38f;  // NaN -> refused
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) row = fmaxf(row, __shfl_xor_sync(0xffffffffu, row, o));
  const bool sane = row <= 1.0e5f;
  if (w == 0 && k == 0 && !sane) {
    sec_flag(p, KG_ERR_NONFINITE);
    sec_record(sm, -1, 3);
    sm.abort = 1;
  }
  float tnorm = 0.f, cre = 0.f, cim = 0.f, n0;
  if constexpr (F32) {
    const float2 a2 = (k < meff) ? sm.ff_a[k] : make_float2(0.f, 0.f);
    const float2 b2 = (k >= 1 && k < meff) ? sm.ff_e[k - 1] : make_float2(0.f, 0.f);
    const float2 t2 = sm.tau_ff[back && w > 0 ? 3 - w : w];
    const FF t = back ? FF{-t2.x, -t2.y} : FF{t2.x, t2.y};
    FF fr{0.f, 0.f}, fi{0.f, 0.f};
    if (meff > 0 && sane) tridiag_expv_e1_fff(FF{a2.x, a2.y}, ff_sqrt(FF{b2.x, b2.y}), meff, t, 1e-13f, fact, fr, fi, tnorm);
    // v_0 = inv x with inv rounded to FP32: 1 / inv, not ||x||, takes the rounding out again (with ||x||
    // every slice would multiply the state's norm by ||x|| inv)
    const FF sc = (inv > 0.f) ? ff_rcp(FF{inv, 0.f}) : nrm;
    const FF cr = ff_mul(fr, sc), ci = ff_mul(fi, sc);
    cre = __fadd_rn(cr.hi, cr.lo);
    cim = __fadd_rn(ci.hi, ci.lo);
    n0 = nrm.hi;
    if (k < meff) {
      sm.coef_f[w][0][k] = cre;
      sm.coef_f[w][1][k] = cim;
    }
  } else {
    double tw = p.dt;
    if (w > 0) tw = 0.5 * p.dt * (1.0 + ((w == 1) != back ? -1.0 : 1.0) / ::sqrt(5.0));
    if (back) tw = -tw;
    double cr = 0.0, ci = 0.0;
    if (meff > 0 && sane) tridiag_expv_e1(sm.alpha, sm.beta, sm.alpha_f, sm.beta_f, meff, tw, (float)tw, 1e-18, cr, ci, tnorm);
    cr *= nrm;
    ci *= nrm;
    if (k < meff) {
      sm.coef_d[w][0][k] = cr;
      sm.coef_d[w][1][k] = ci;
    }
    cre = (float)cr;
    cim = (float)ci;
    n0 = (float)nrm;
  }
  if (w == 0 && k == meff - 1) {  // a-posteriori indicator ||x|| b_m |c_{m-1}| (0 after a breakdown)
    float cm = hypotf(cre, cim);  // the squares may underflow
    if (cm == 0.f && !broke) {
      cm = n0;
      for (int i = 1; i < meff; ++i) cm *= tnorm * kInvFF[i].x;
    }
    if (broke) sm.breakdowns += 1;
    else sm.err_max = fmaxf(sm.err_max, beta_m * cm);
  }
  __syncwarp();
  if (w == 0 && k == 0) {
    sm.ff_e_set = 0u;
    // time limit of one pulse: a pulse that runs past it ends with KG_ERR_TIMEOUT
    if (sm.abort == 0 && (long long)(globaltimer_ns() - sm.t_start) > p.time_limit_ns) {
      sec_flag(p, KG_ERR_TIMEOUT);
      sec_record(sm, -1, 4);
      sm.abort = 1;
    }
  }
}

// One slice: x (own rows, norm nrm, inv = 1/nrm) -> x = ||x|| V exp(-+i dt T) e_1 (App. A; back: the
// co-state sweep), written to dst (if not null), then ||x||^2 and, back, ex = Im <x| Hc |other> over the
// own rows are reduced.  Returns false after a non-finite coefficient (status set).
template <class V, int NT, int RPT>
__device__ __forceinline__ bool sec_slice(const SectorParams& p, SecSmem& sm, int& par, V* Sa, V* Sb,
                                          const unsigned* tab, V* basis, double uj, bool back, V (&x)[RPT],
                                          typename SecPrec<V>::N& nrm, typename VecTraits<V>::R& inv, const V* other,
                                          V* dst, typename SecPrec<V>::N& ex, int taylor, const V* psi_end,
                                          typename SecPrec<V>::N& tay, int lob, V* tint_io, float2 fact) {
  using R = typename VecTraits<V>::R;
  using S = typename SecPrec<V>::S;
  using A = typename SecAcc<V>::T;
  constexpr bool F32 = sizeof(R) == 4;
  constexpr bool FFM = std::is_same<R, FFR>::value;  // float-float vectors (KG_PREC_FF)
  const int tid = threadIdx.x, D = p.D, m = p.m;
  R dj[RPT];
#pragma unroll
  for (int i = 0; i < RPT; ++i) {
    const int r = tid + NT * i;
    dj[i] = 0;
    if (r < D) {
      const unsigned st = __ldg(p.states + r);
      dj[i] = fma((R)uj, sec_hc<R>(p, sm, st), sec_d0<R>(p, sm, st));
    }
  }
  // ---- v_0 = x / ||x||
  V v[RPT], vp[RPT], w[RPT];
  V* Sc = Sa;
  V* Sn = Sb;
#pragma unroll
  for (int i = 0; i < RPT; ++i) {
    const int r = tid + NT * i;
    v[i] = vscale<V>(inv, x[i]);
    vp[i] = vmake<V>(0, 0);
    if (r < D) {
      Sc[r] = v[i];
      basis[r] = v[i];
    }
  }
  int meff = (sec_top(nrm) > 0) ? m : 0;
  bool broke = false;
  R alpha = 0, bk = 0, ib = 0;
  float amax = 0.f, bmax = 0.f, beta_m = 0.f;
  const float tol = p.bd_tol_f;
  for (int k = 0; k < meff; ++k) {
    const bool last = (k == m - 1);
    sec_sync();  // v_k is in shared memory
    sec_apply<V, NT, RPT>(p, sm, Sc, tab, dj, v, bk, vp, w);
    A pa = A(), pn = A(), pq = A();
#pragma unroll
    for (int i = 0; i < RPT; ++i) {
      sacc(pa, v[i], w[i]);
      sacc(pn, w[i], w[i]);
      sacc(pq, v[i], v[i]);
    }
    sec_mark(p, sm, 0);
    S o[3];
    sec_reduce<NT>(sm, par, sclose(pa), sclose(pn), sclose(pq), o);
    sec_mark(p, sm, 1);
    alpha = sec_real(o[0], R());
    S b2 = sec_b2(o);
    sec_roots(b2, bk, ib);
    const float af = fabsf(sec_f32(alpha));
    const bool usual = isfinite(sec_top(o[0])) && isfinite(sec_top(o[1])) &&
                       !sec_cancels(b2, o[1]) &&
                       sec_f32(bk) > tol * fmaxf(1.f, fmaxf(amax, af) + bmax);
    if (!usual) {
      if (!isfinite(sec_top(o[0])) || !isfinite(sec_top(o[1]))) {
        if (tid == 0) {
          sec_flag(p, KG_ERR_NONFINITE);
          sec_record(sm, k, 1);
        }
        return false;
      }
      if (!last && sec_cancels(b2, o[1])) {
        // near an invariant subspace: ||w - alpha v||^2 explicitly
        A e = A();
#pragma unroll
        for (int i = 0; i < RPT; ++i) {
          const V d = vaxpy<V>(-alpha, v[i], w[i]);
          sacc(e, d, d);
        }
        S oe[3];
        sec_reduce<NT>(sm, par, sclose(e), sclose(A()), sclose(A()), oe);
        b2 = oe[0];
        sec_roots(b2, bk, ib);
        if constexpr (FFM) {
          if (tid == 0) {
            sm.ff_e[k] = make_float2(b2.hi, b2.lo);
            sm.ff_e_set |= 1u << k;
          }
        }
      }
      // Alg. "Lanczos": b_j > 0, with a tolerance
      if (!last) broke = sec_f32(bk) <= tol * fmaxf(1.f, fmaxf(amax, af) + bmax);
    }
    amax = fmaxf(amax, af);
    bmax = fmaxf(bmax, sec_f32(bk));
    if (tid == 0) {
      sm.alpha_f[k] = sec_f32(alpha);
      sm.beta_f[k + 1] = sec_f32(bk);
      if constexpr (F32) {
        sm.ff_a[k] = make_float2(o[0].hi, o[0].lo);
        sm.ff_e[k] = make_float2(b2.hi, b2.lo);
      } else if constexpr (FFM) {
        sm.ff_a[k] = make_float2(o[0].hi, o[0].lo);
        sm.ff_n[k] = make_float2(o[1].hi, o[1].lo);
        sm.ff_q[k] = make_float2(o[2].hi, o[2].lo);
      } else {
        sm.alpha[k] = o[0];
        sm.beta[k + 1] = bk;
      }
    }
    if (last || broke) {
      beta_m = sec_f32(bk);
      meff = k + 1;
      break;
    }
#pragma unroll
    for (int i = 0; i < RPT; ++i) {
      const int r = tid + NT * i;
      vp[i] = v[i];
      v[i] = vscale<V>(ib, vaxpy<V>(-alpha, v[i], w[i]));
      if (r < D) {
        Sn[r] = v[i];
        basis[(size_t)(k + 1) * D + r] = v[i];
      }
    }
    V* t = Sc;
    Sc = Sn;
    Sn = t;
  }
  sec_mark(p, sm, 0);
  // ---- T, exp(-+i dt T) e_1 and the recombination coefficients (warp 0; with lob, warps 1 and 2 form the
  // coefficients of the two interior Gauss-Lobatto nodes at the same time)
  if (tid < 32) {
    __syncwarp();  // thread 0's stores of the step sums are visible to the warp
    if constexpr (FFM) {  // T in FP64 from the float-float sums, lane k for step k
      const int k = tid;
      if (k < meff) {
        const double al = ff_to_double(FF{sm.ff_a[k].x, sm.ff_a[k].y});
        double b2;
        if ((sm.ff_e_set >> k) & 1u) {
          b2 = ff_to_double(FF{sm.ff_e[k].x, sm.ff_e[k].y});
        } else {
          const double nn = ff_to_double(FF{sm.ff_n[k].x, sm.ff_n[k].y});
          const double q = ff_to_double(FF{sm.ff_q[k].x, sm.ff_q[k].y});
          b2 = nn - 2.0 * al * al + al * al * q;
        }
        sm.alpha[k] = al;
        if (k + 1 < meff) sm.beta[k + 1] = ::sqrt(::fmax(b2, 0.0));
      }
      __syncwarp();
    }
  }
  if (lob) sec_sync();  // T is read by warps 1 and 2 as well
  if (tid < (lob ? 96 : 32)) sec_coefficients<V>(p, sm, tid >> 5, back, meff, broke, beta_m, nrm, F32 ? (float)sec_f32(inv) : 0.f, fact);
  sec_sync();
  if (sm.abort) return false;
  sec_mark(p, sm, 4);
  // ---- recombination x = sum_k coef_k v_k (own rows), the small terms first; fused ||x||^2 and overlap.
  // The own rows' basis values come from L2: KB basis vectors' loads are issued together.
  constexpr int KB = (F32 ? 16 : 8) / RPT < 2 ? 2 : (F32 ? 16 : 8) / RPT;
  V y[RPT];
#pragma unroll
  for (int i = 0; i < RPT; ++i) y[i] = vmake<V>(0, 0);
  for (int k0 = meff - 1; k0 >= 0; k0 -= KB) {
    V q[KB][RPT];
#pragma unroll
    for (int u = 0; u < KB; ++u)
#pragma unroll
      for (int i = 0; i < RPT; ++i) {
        const int r = tid + NT * i;
        q[u][i] = (k0 >= u && r < D) ? basis[(size_t)(k0 - u) * D + r] : vmake<V>(0, 0);
      }
#pragma unroll
    for (int u = 0; u < KB; ++u) {
      if (k0 >= u) {
        const int k = k0 - u;
        const R a = F32 ? (R)sm.coef_f[0][0][k] : (R)sm.coef_d[0][0][k];
        const R b = F32 ? (R)sm.coef_f[0][1][k] : (R)sm.coef_d[0][1][k];
#pragma unroll
        for (int i = 0; i < RPT; ++i) {
          y[i] = vcaxpy<V>(a, b, q[u][i], y[i]);
        }
      }
    }
  }
  R pn = 0, pg = 0;
#pragma unroll
  for (int i = 0; i < RPT; ++i) {
    const int r = tid + NT * i;
    if (r < D) {
      if (dst) dst[r] = y[i];
      pn = fma(vre(y[i]), vre(y[i]), fma(vim(y[i]), vim(y[i]), pn));
      if (back) {
        const V o = other[r];
        pg = fma(sec_hc<R>(p, sm, __ldg(p.states + r)), vre(y[i]) * vim(o) - vim(y[i]) * vre(o), pg);  // Im(conj(y) Hc o)
      }
    }
    x[i] = y[i];
  }
  // ---- Taylor hierarchy (App. B, Eq. gradp), backward slice j (sec_taylor)
  R pt = 0;
  if constexpr (!FFM) {  // the float-float path offers the centred and zeroth-order gradients
    if (taylor > 0) {
      R nx;
      if constexpr (F32) nx = __fadd_rn(nrm.hi, nrm.lo);
      else nx = nrm;
      pt = sec_taylor<V, NT, RPT>(p, sm, Sa, Sb, tab, basis, uj, meff, nx, taylor, psi_end);
    }
    if (lob > 0) pt = sec_interior<V, NT, RPT>(p, sm, basis, meff, lob, tint_io);
  }
  sec_mark(p, sm, 5);
  if constexpr (F32) {
    FF o[3];
    sec_reduce<NT>(sm, par, pn, pg, pt, o);
    FF id;
    ff_rsqrt(o[0], nrm, id);
    inv = __fadd_rn(id.hi, id.lo);
    ex = o[1];
    tay = o[2];
    if (!isfinite(o[0].hi)) {
      if (tid == 0) {
        sec_flag(p, KG_ERR_NONFINITE);
        sec_record(sm, -1, 2);
      }
      return false;
    }
  } else {
    double o[3];
    sec_reduce<NT>(sm, par, (double)pn, (double)pg, (double)pt, o);
    if (!isfinite(o[0])) {
      if (tid == 0) {
        sec_flag(p, KG_ERR_NONFINITE);
        sec_record(sm, -1, 2);
      }
      return false;
    }
    double id;
    sec_roots(o[0], nrm, id);
    inv = (R)id;
    ex = o[1];
    tay = o[2];
  }
  sec_mark(p, sm, 1);
  return true;
}

// Thread 0: F = NaN and the failure record of pulse b, abandoned in slice j (negative: backward).
__device__ __forceinline__ void sec_abandon(const SectorParams& p, const SecSmem& sm, int b, int j) {
  p.fid[b] = __longlong_as_double(0x7ff8000000000000LL);
  double* sc = p.scal + (size_t)b * kScCount;
  sc[5] = (double)j;
  sc[6] = (double)sm.fail_step;
  sc[7] = (double)sm.fail_check;
}

__device__ __forceinline__ void sec_norm(double n2, FF& n, float& inv) {
  const double d = ::sqrt(n2);
  n = ff_from_double(d);
  inv = (d > 0.0) ? (float)(1.0 / d) : 0.f;
}
template <class R>
__device__ __forceinline__ void sec_norm(double n2, double& n, R& inv) {
  n = ::sqrt(n2);
  inv = (n > 0.0) ? (R)(1.0 / n) : (R)0;
}
__device__ __forceinline__ double sec_double(FF a) { return ff_to_double(a); }
__device__ __forceinline__ double sec_double(double a) { return a; }

template <class V, int NT, int RPT>
__device__ __forceinline__ void sec_eval(const SectorParams& p, int b, SecSmem& sm, V* S0, V* S1, const unsigned* tab,
                                         float2 fact) {
  using R = typename VecTraits<V>::R;
  using N = typename SecPrec<V>::N;
  constexpr bool F32 = sizeof(R) == 4;
  const int tid = threadIdx.x, D = p.D, NS = p.N;
  V* traj = (V*)p.traj + (size_t)blockIdx.x * (size_t)(NS + 1) * D;
  V* basis = (V*)p.basis + (size_t)blockIdx.x * (size_t)p.m * D;
  double* G = p.G + (size_t)blockIdx.x * (NS + 1);
  double* gb = p.grad ? p.grad + (size_t)b * NS : nullptr;
  const double* u = p.u + (size_t)b * NS;
  const double2* psi0 = reinterpret_cast<const double2*>(p.psi0);
  const double2* tgt = reinterpret_cast<const double2*>(p.target);
  sec_sync();  // the previous pulse (possibly abandoned after a non-finite value) is done with shared memory
  if (tid == 0) {
    sm.err_max = 0.f;
    sm.breakdowns = 0;
    sm.ff_e_set = 0u;
    sm.abort = 0;
    sm.prof_last = clock64();
    sm.fail_step = 0;
    sm.fail_check = 0;
    sm.t_start = globaltimer_ns();
  }
  int par = 0;
  V x[RPT];
  N nrm;
  R inv;
  {  // psi_0 into the trajectory and its norm (FP64)
    double acc = 0.0, o[3];
#pragma unroll
    for (int i = 0; i < RPT; ++i) {
      const int r = tid + NT * i;
      x[i] = vmake<V>(0, 0);
      if (r < D) {
        const double2 q = psi0[p.perm[r]];
        x[i] = vmake<V>((R)q.x, (R)q.y);
        traj[r] = x[i];
        const double re = (double)vre(x[i]), im = (double)vim(x[i]);
        acc = ::fma(re, re, ::fma(im, im, acc));
      }
    }
    sec_reduce<NT>(sm, par, acc, 0.0, 0.0, o);
    sec_norm(o[0], nrm, inv);
  }
  sec_mark(p, sm, 6);
  const bool exact = (p.grad_mode == KG_GRAD_EXACT);
  const int taylor = (p.grad_mode == KG_GRAD_TAYLOR1) ? 1 : (p.grad_mode == KG_GRAD_TAYLOR2) ? 2 : 0;
  V* tint = exact ? (V*)p.tint + (size_t)blockIdx.x * 2 * (size_t)NS * D : nullptr;
  // Forward slices j = 1..N, then the co-state's j = N..1: one loop, one copy of the slice's code.
  double br = 0.0, bi = 0.0, nfin = 0.0;
  bool back = false;
  for (int j = 1;;) {
    N ex, tay;
    if (!sec_slice<V, NT, RPT>(p, sm, par, S0, S1, tab, basis, u[j - 1], back, x, nrm, inv, traj + (size_t)(j - 1) * D,
                               back ? nullptr : traj + (size_t)j * D, ex, back ? taylor : 0, traj + (size_t)j * D, tay,
                               !exact ? 0 : back ? 2 : 1, exact ? tint + (size_t)2 * (j - 1) * D : nullptr, fact)) {
      if (tid == 0) sec_abandon(p, sm, b, back ? -j : j);
      return;
    }
    if (back) {
      if (tid == 0) {
        G[j - 1] = sec_pack(ex);
        if (taylor) G[j] = sec_pack(tay);     // slice j's Taylor-hierarchy value replaces G_j
        if (exact) gb[j - 1] = sec_pack(tay);  // the interior nodes' share, weighted below
      }
      if (--j == 0) break;
      continue;
    }
    if (j < NS) {
      ++j;
      continue;
    }
    // ---- beta = <f|psi_N> (FP64), F = |beta|^2
    nfin = sec_double(nrm);
    {
      double a0 = 0.0, a1 = 0.0, o[3];
#pragma unroll
      for (int i = 0; i < RPT; ++i) {
        const int r = tid + NT * i;
        if (r < D) {
          const double2 f = tgt[p.perm[r]];
          const double xr = (double)vre(x[i]), xi = (double)vim(x[i]);
          a0 = ::fma(f.x, xr, ::fma(f.y, xi, a0));   // Re(conj(f) x)
          a1 = ::fma(f.x, xi, ::fma(-f.y, xr, a1));  // Im(conj(f) x)
        }
      }
      sec_reduce<NT>(sm, par, a0, a1, 0.0, o);
      br = o[0];
      bi = o[1];
    }
    if (p.grad_mode == KG_GRAD_NONE) break;
    {  // chi_N = beta f; G_N = 2 dt Im <chi_N|Hc|psi_N>
      double a0 = 0.0, a1 = 0.0, o[3];
#pragma unroll
      for (int i = 0; i < RPT; ++i) {
        const int r = tid + NT * i;
        V c = vmake<V>(0, 0);
        if (r < D) {
          const double2 f = tgt[p.perm[r]];
          c = vmake<V>((R)(br * f.x - bi * f.y), (R)(br * f.y + bi * f.x));
          const double cr = (double)vre(c), ci = (double)vim(c);
          a0 = ::fma(cr, cr, ::fma(ci, ci, a0));
          a1 = ::fma((double)sec_hc<R>(p, sm, __ldg(p.states + r)), cr * (double)vim(x[i]) - ci * (double)vre(x[i]), a1);
        }
        x[i] = c;
      }
      sec_reduce<NT>(sm, par, a0, a1, 0.0, o);
      sec_norm(o[0], nrm, inv);
      if constexpr (F32) {
        if (tid == 0) G[NS] = sec_pack(ff_from_double(o[1]));
      } else {
        if (tid == 0) G[NS] = o[1];
      }
    }
    sec_mark(p, sm, 6);
    back = true;
  }
  if (back) {
    sec_sync();  // G complete (written by thread 0)
    const double f = 2.0 * p.dt;
    for (int j = tid; j < NS; j += NT) {
      const double gl = f * sec_unpack<F32>(G[j]), gr = f * sec_unpack<F32>(G[j + 1]);
      if (exact)  // 4-point Gauss-Lobatto over slice j: weights 1/12, 5/12, 5/12, 1/12
        gb[j] = (gl + gr) / 12.0 + (5.0 / 12.0) * f * sec_unpack<F32>(gb[j]);
      else
        gb[j] = (p.grad_mode == KG_GRAD_CENTERED) ? 0.5 * (gl + gr) : gr;  // zeroth, Taylor
    }
  }
  if (tid == 0) {
    p.fid[b] = br * br + bi * bi;
    double* sc = p.scal + (size_t)b * kScCount;
    sc[kScBetaRe] = br;
    sc[kScBetaIm] = bi;
    sc[kScErrMax] = (double)sm.err_max;
    sc[kScNormFinal] = nfin;
    sc[kScBreakdowns] = (double)sm.breakdowns;
    sc[5] = sc[6] = sc[7] = 0.0;
  }
  sec_sync();
}

// CTAs (pulses) per SM the register allocation is sized for.  A pulse is a chain of latencies
// (block barriers, FP64 on warp 0), so pulses sharing an SM hide each other's: complex64 blocks of
// 128 threads are held to 64 registers a thread, eight pulses per SM (a few spills; measured 1.9x the
// pulses/s of three per SM at D = 511); float-float blocks of 128 threads to 128 registers, four per
// SM (no spills; 732 against 626 pulses/s at three per SM, D = 511); other blocks of up to 256
// threads to 128 registers, two per SM.
template <class V, int NT>
constexpr int sec_min_blocks() {
  return (NT == 128 && sizeof(V) == sizeof(float2)) ? 8 : (NT == 128 && std::is_same<V, FFC>::value) ? 4
                                                    : (NT <= 256) ? 2 : 1;
}

// Elements of a vector in shared memory: D, the zero element behind it, 16-element steps.
__host__ __device__ constexpr int sec_padded(int D) { return (D + 16) & ~15; }

template <class V, int NT, int RPT>
__global__ void __launch_bounds__(NT, (sec_min_blocks<V, NT>())) kg_sector_kernel(const __grid_constant__ SectorParams p) {
  extern __shared__ __align__(16) unsigned char sec_dyn[];
  __shared__ SecSmem sm;
  const int Dp = sec_padded(p.D);
  V* S0 = reinterpret_cast<V*>(sec_dyn);
  V* S1 = S0 + Dp;
  unsigned* tab = reinterpret_cast<unsigned*>(S1 + Dp);
  for (int i = threadIdx.x; i < p.words; i += NT) tab[i] = p.tab_g[i];
  if (threadIdx.x == 0) {
    S0[p.D] = S1[p.D] = vmake<V>(0, 0);  // what the tables' padding points at
    const double sa = 0.5 * p.dt * (1.0 - 1.0 / ::sqrt(5.0));
    const double w[7] = {p.qz, 0.5 * p.hc_amp, p.wa, p.wb, p.dt, sa, p.dt - sa};
    for (int i = 0; i < 7; ++i) {
      const FF f = ff_from_double(w[i]);
      if (i < 4) {
        sm.diag_d[i] = w[i];
        sm.diag_ff[i] = make_float2(f.hi, f.lo);
      } else {
        sm.tau_ff[i - 4] = make_float2(f.hi, f.lo);
      }
    }
  }
  if (threadIdx.x < 8) sm.prof_acc[threadIdx.x] = 0;
  const long long t0 = clock64();
  const float2 fact = kInvFactFF[min((int)threadIdx.x & 31, 29)];
  sec_sync();
  for (int b = blockIdx.x; b < p.B; b += gridDim.x) sec_eval<V, NT, RPT>(p, b, sm, S0, S1, tab, fact);
  if (p.prof && blockIdx.x == 0 && threadIdx.x == 0) {
    for (int i = 0; i < 7; ++i) p.prof[i] = sm.prof_acc[i];
    p.prof[7] = clock64() - t0;
  }
}

// ---------------------------------------------------------------- launch selection
struct SecKernel {
  const void* fn;
  int threads;
};

template <class V, int NT, int RPT>
static SecKernel sec_choice() {
  return {reinterpret_cast<const void*>(&kg_sector_kernel<V, NT, RPT>), NT};
}

// 128 threads: as many rows a thread as D needs (a row beyond D costs its FP64 or float-float work).
template <class V>
static SecKernel sec_small(int D) {
  if (D <= 128) return sec_choice<V, 128, 1>();
  if (D <= 256) return sec_choice<V, 128, 2>();
  return (D <= 512) ? sec_choice<V, 128, 4>() : SecKernel{nullptr, 0};
}

// Threads and rows per thread by dimension: the smallest block that covers D with <= 8 rows per
// thread (10 for complex64 up to 2560, which keeps two CTAs on an SM); or, with nt = 128, 256 or
// 512 threads, that block with the fewest rows per thread that covers D (nt.threads == 0: none).
static SecKernel sec_pick(int prec, int D, int nt = 0) {
  if (prec == KG_PREC_FF) {  // the complex128 path's shapes (16-byte amplitudes); 512 x 5 up to
                             // D = 2560 holds its arrays in registers (512 x 8 spills)
    if (nt == 128) return sec_small<FFC>(D);
    if (nt == 256) return (D <= 1024) ? sec_choice<FFC, 256, 4>()
                                      : (D <= 2048) ? sec_choice<FFC, 256, 8>() : SecKernel{nullptr, 0};
    if (nt == 512)
      return (D <= 2560) ? sec_choice<FFC, 512, 5>() : (D <= 4096) ? sec_choice<FFC, 512, 8>() : SecKernel{nullptr, 0};
    if (D <= 512) return sec_small<FFC>(D);
    if (D <= 1024) return sec_choice<FFC, 256, 4>();
    if (D <= 2048) return sec_choice<FFC, 256, 8>();
    if (D <= 2560) return sec_choice<FFC, 512, 5>();
    return sec_choice<FFC, 512, 8>();
  }
  if (prec == KG_PREC_C128) {  // 512 x 5 up to D = 2560 spills less than 512 x 8
    if (nt == 128) return sec_small<double2>(D);
    if (nt == 256) return (D <= 1024) ? sec_choice<double2, 256, 4>()
                                      : (D <= 2048) ? sec_choice<double2, 256, 8>() : SecKernel{nullptr, 0};
    if (nt == 512)
      return (D <= 2560) ? sec_choice<double2, 512, 5>()
                         : (D <= 4096) ? sec_choice<double2, 512, 8>() : SecKernel{nullptr, 0};
    if (D <= 512) return sec_small<double2>(D);
    if (D <= 1024) return sec_choice<double2, 256, 4>();
    if (D <= 2048) return sec_choice<double2, 256, 8>();
    if (D <= 2560) return sec_choice<double2, 512, 5>();
    return sec_choice<double2, 512, 8>();
  }
  if (nt == 128) return sec_small<float2>(D);
  if (nt == 256)
    return (D <= 1024) ? sec_choice<float2, 256, 4>()
                       : (D <= 2048) ? sec_choice<float2, 256, 8>()
                                     : (D <= 2560) ? sec_choice<float2, 256, 10>() : SecKernel{nullptr, 0};
  if (nt == 512) return (D <= 4096) ? sec_choice<float2, 512, 8>() : SecKernel{nullptr, 0};
  if (D <= 512) return sec_small<float2>(D);
  if (D <= 1024) return sec_choice<float2, 256, 4>();
  if (D <= 2048) return sec_choice<float2, 256, 8>();
  if (D <= 2560) return sec_choice<float2, 256, 10>();  // two CTAs per SM (registers)
  return sec_choice<float2, 512, 8>();
}

constexpr int kSecMaxRows = 4096;  // 512 threads x 8 rows
// Dynamic shared memory of the largest subspace taken (sector_fits; 202 KB is the most any needs), and
// every kernel's limit: one value, so that no call can lower it between another host thread's setting and
// launch.
constexpr size_t kSecMaxSmem = 216 * 1024;

size_t sector_smem_bytes(int prec, int D, int words) {
  const size_t vb = (prec == KG_PREC_C64_F64REC) ? 8 : 16;
  return 2 * (size_t)sec_padded(D) * vb + (size_t)words * 4;
}

cudaError_t sector_kernel_max_ctas(int prec, int D, int words, int nt, int* out) {
  const SecKernel k = sec_pick(prec, D, nt);
  if (!k.fn) return cudaErrorInvalidValue;
  const size_t smem = sector_smem_bytes(prec, D, words);
  cudaError_t e = cudaFuncSetAttribute(k.fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSecMaxSmem);
  if (e != cudaSuccess) return e;
  int dev = 0, sms = 0, per = 0;
  if ((e = cudaGetDevice(&dev)) != cudaSuccess) return e;
  if ((e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev)) != cudaSuccess) return e;
  if ((e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, k.fn, k.threads, smem)) != cudaSuccess) return e;
  *out = per * sms;
  return cudaSuccess;
}

int sector_threads(int prec, int D, int nt) { return sec_pick(prec, D, nt).threads; }
bool sector_shape_ok(int prec, int D, int nt) { return sec_pick(prec, D, nt).fn != nullptr; }

cudaError_t launch_sector_kernel(int prec, const SectorParams& p, int ctas, int nt, cudaStream_t stream) {
  const SecKernel k = sec_pick(prec, p.D, nt);
  if (!k.fn) return cudaErrorInvalidValue;
  const size_t smem = sector_smem_bytes(prec, p.D, p.words);
  cudaError_t e = cudaFuncSetAttribute(k.fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSecMaxSmem);
  if (e != cudaSuccess) return e;
  void* args[] = {const_cast<SectorParams*>(&p)};
  return cudaLaunchKernel(k.fn, dim3(ctas), dim3(k.threads), args, smem, stream);
}

}  // namespace kg

// ================================================================ host side of the ABI
namespace {

using kg::host_fail;

struct SectorBasis {
  std::vector<uint64_t> states;       // s_r, ascending
  std::vector<unsigned> tab;          // list A, the 32-row groups' meta words, list B (see sec_apply); 8 x columns
  std::vector<unsigned short> perm;   // the tables' row -> basis index
  int D = 0, bonds = 0;               // bonds: most antiparallel bonds of a row
  int na2 = 0, rows = 0, groups = 0;
  int words() const { return (int)tab.size(); }
};

uint64_t mirror_bits(uint64_t s, int L) {
  uint64_t r = 0;
  for (int b = 0; b < L; ++b) r |= ((s >> b) & 1ull) << (L - 1 - b);
  return r;
}

kg_status check_sector(const kg_sector* s) {
  if (!s) return host_fail(KG_ERR_INVALID_ARG, "sector must not be NULL");
  if (s->L < 2 || s->L > kg::kMaxL) return host_fail(KG_ERR_INVALID_ARG, "L must satisfy 2 <= L <= 30");
  if (s->K < 0 || s->K > s->L) return host_fail(KG_ERR_INVALID_ARG, "K must satisfy 0 <= K <= L");
  if (s->parity < -1 || s->parity > 1) return host_fail(KG_ERR_INVALID_ARG, "parity must be -1, 0 or +1");
  if (s->block_threads != 0 && s->block_threads != 128 && s->block_threads != 256 && s->block_threads != 512)
    return host_fail(KG_ERR_INVALID_ARG, "block_threads must be 0, 128, 256 or 512");
  if ((s->hc_site_mask >> s->L) != 0) return host_fail(KG_ERR_INVALID_ARG, "hc_site_mask has bits at or above L");
  if (s->parity != 0 && mirror_bits(s->hc_site_mask, s->L) != s->hc_site_mask)
    return host_fail(KG_ERR_INVALID_ARG, "a parity subspace needs a mirror-symmetric hc_site_mask");
  if (!std::isfinite(s->Jxy) || !std::isfinite(s->Jz) || !std::isfinite(s->hc_amp))
    return host_fail(KG_ERR_INVALID_ARG, "Jxy, Jz and hc_amp must be finite");
  return KG_OK;
}

// Orbits of the K-excitation states under the mirror, in the order of their smaller member.
// orbit[s] for every state s of the sector (via its position in `all`): the row, the member's
// sign phi, and whether the orbit is a palindrome.  Returns false if D would exceed `limit`.
struct OrbitInfo {
  int row;     // -1: no basis vector (a palindrome in the odd subspace)
  int phi;     // +1 smaller member, parity for the mirrored one
  int n;       // orbit size
};

bool build_basis(const kg_sector* s, size_t limit, bool want_ell, SectorBasis& out, std::string& why) {
  const int L = s->L, K = s->K, P = s->parity;
  // the dimension in closed form, to refuse large subspaces before enumerating them: C(L,K) states,
  // pal of them mirror-symmetric (fixed by the first floor(L/2) bits and, for odd L, the middle one);
  // D = C (parity 0), (C + pal)/2 (even), (C - pal)/2 (odd)
  {
    auto binom = [](int n, int k) {
      double c = 1.0;
      for (int i = 0; i < k; ++i) c = c * (double)(n - i) / (double)(i + 1);
      return c;
    };
    const int h = L / 2;
    const double C = binom(L, K);
    const double pal = (L % 2 == 0) ? ((K % 2 == 0) ? binom(h, K / 2) : 0.0) : binom(h, K / 2);
    const double Dd = (P == 0) ? C : 0.5 * (C + (double)P * pal);
    if (Dd > (double)limit + 0.5) {
      why = "subspace dimension " + std::to_string((long long)(Dd + 0.5)) + " exceeds " + std::to_string(limit);
      return false;
    }
  }
  std::vector<uint64_t> all;  // the K-excitation states, ascending (Gosper's next-combination step)
  if (K == 0) {
    all.push_back(0);
  } else {
    uint64_t v = (1ull << K) - 1;
    const uint64_t end = 1ull << L;
    while (v < end) {
      all.push_back(v);
      if (all.size() > 64ull * 1024 * 1024) {
        why = "the K-excitation sector is too large";
        return false;
      }
      const uint64_t c = v & (~v + 1);
      const uint64_t r = v + c;
      v = (((r ^ v) >> 2) / c) | r;
    }
  }
  std::unordered_map<uint64_t, OrbitInfo> orb;
  orb.reserve(all.size() * 2);
  out.states.clear();
  for (const uint64_t st : all) {
    const uint64_t t = (P == 0) ? st : mirror_bits(st, L);
    if (t < st) continue;  // met at its smaller member already
    OrbitInfo oi{-1, 1, (t == st) ? 1 : 2};
    if (!(P == -1 && t == st)) {
      oi.row = (int)out.states.size();
      out.states.push_back(st);
    }
    orb[st] = oi;
    if (t != st) orb[t] = OrbitInfo{oi.row, P, 2};
  }
  out.D = (int)out.states.size();
  if ((size_t)out.D > limit) {
    why = "subspace dimension " + std::to_string(out.D) + " exceeds " + std::to_string(limit);
    return false;
  }
  if (!want_ell) return true;
  // per row: one column per antiparallel bond of s_r whose image has a basis vector, on the list of its weight
  std::vector<std::vector<int>> la(out.D), lb(out.D);
  size_t wide = 0;
  for (int r = 0; r < out.D; ++r) {
    const uint64_t st = out.states[r];
    const int nr = orb[st].n;
    int bonds = 0;
    for (int b = 0; b + 1 < L; ++b) {
      if (((st >> b) & 1ull) == ((st >> (b + 1)) & 1ull)) continue;
      const OrbitInfo& o = orb.at(st ^ (3ull << b));
      if (o.row < 0) continue;
      ++bonds;
      if (P == 1 && nr != o.n) {  // factor sqrt(n_r'/n_r): sqrt 2 = 2 / sqrt 2, or 1 / sqrt 2
        lb[r].push_back(o.row);
        if (nr == 2) lb[r].push_back(o.row);
      } else if (P == -1 && o.phi < 0) {
        lb[r].push_back(o.row);
      } else {
        la[r].push_back(o.row);
      }
    }
    out.bonds = std::max(out.bonds, bonds);
    wide = std::max(wide, la[r].size());
  }
  const int D = out.D;
  // the kernel's rows: longest lists first
  std::vector<int> order(D), row_of(D);
  for (int r = 0; r < D; ++r) order[r] = r;
  std::stable_sort(order.begin(), order.end(), [&](int x, int y) {
    const size_t ax = (la[x].size() + 1) / 2, ay = (la[y].size() + 1) / 2;
    return ax != ay ? ax > ay : (lb[x].size() + 1) / 2 > (lb[y].size() + 1) / 2;
  });
  out.perm.assign(order.begin(), order.end());
  for (int i = 0; i < D; ++i) row_of[order[i]] = i;
  auto word = [&](const std::vector<int>& l, size_t q) {  // entries 2q, 2q + 1; padding: the zero element D
    const unsigned c0 = (2 * q < l.size()) ? 8u * (unsigned)row_of[l[2 * q]] : 8u * (unsigned)D;
    const unsigned c1 = (2 * q + 1 < l.size()) ? 8u * (unsigned)row_of[l[2 * q + 1]] : 8u * (unsigned)D;
    return c0 | (c1 << 16);
  };
  out.na2 = (int)((wide + 1) / 2);
  out.rows = D + 1;  // row D: all padding, for the threads without a row of their own
  out.groups = (D + 31) / 32;
  out.tab.clear();
  const std::vector<int> none;
  for (int q = 0; q < out.na2; ++q)
    for (int r = 0; r <= D; ++r) out.tab.push_back(word(r < D ? la[order[r]] : none, (size_t)q));
  const size_t meta = out.tab.size();
  out.tab.resize(meta + out.groups);
  for (int g = 0; g < out.groups; ++g) {
    size_t na = 0, nb = 0;
    for (int r = 32 * g; r < std::min(D, 32 * g + 32); ++r) {
      na = std::max(na, (la[order[r]].size() + 1) / 2);
      nb = std::max(nb, (lb[order[r]].size() + 1) / 2);
    }
    out.tab[meta + g] = kg::sec_meta((unsigned)(out.tab.size() - meta - out.groups), (unsigned)na, (unsigned)nb);
    for (size_t q = 0; q < nb; ++q)
      for (int i = 0; i < 32; ++i) out.tab.push_back(word(32 * g + i < D ? lb[order[32 * g + i]] : none, q));
  }
  return true;
}

// Weights of the two lists.
void list_weights(const kg_sector* s, double& wa, double& wb) {
  wa = 0.5 * s->Jxy;
  wb = (s->parity > 0) ? wa / std::sqrt(2.0) : (s->parity < 0) ? -wa : 0.0;
}

struct SectorLayout {
  size_t ctrl = 0, scal = 0, prof = 0, G = 0, basis = 0, traj = 0, tint = 0, tab = 0, states = 0, perm = 0, total = 0;
};

size_t align_up(size_t x) { return (x + kg::kAlign - 1) / kg::kAlign * kg::kAlign; }

SectorLayout sector_layout(int D, int words, const kg_options* o, int B, int grid) {
  SectorLayout l;
  const size_t vb = (size_t)D * (o->prec == KG_PREC_C64_F64REC ? 8 : 16);
  size_t off = 0;
  auto take = [&](size_t bytes) {
    const size_t at = off;
    off = align_up(off + bytes);
    return at;
  };
  l.ctrl = take(64);
  l.scal = take(sizeof(double) * kg::kScCount * (size_t)B);
  l.prof = take(sizeof(long long) * 8);
  l.G = take(sizeof(double) * (size_t)(o->N + 1) * grid);
  l.basis = take(vb * (size_t)o->m * grid);
  l.traj = take(vb * (size_t)(o->N + 1) * grid);
  l.tint = take(o->grad == KG_GRAD_EXACT ? vb * 2 * (size_t)o->N * grid : 0);
  l.tab = take((size_t)words * 4);
  l.states = take(sizeof(unsigned) * (size_t)D);
  l.perm = take(sizeof(unsigned short) * (size_t)D);
  l.total = off;
  return l;
}

kg_status check_sector_opts(const kg_options* o, int B) {
  if (!o) return host_fail(KG_ERR_INVALID_ARG, "options must not be NULL");
  if (B < 1) return host_fail(KG_ERR_INVALID_ARG, "B must be >= 1");
  if (o->N < 1) return host_fail(KG_ERR_INVALID_ARG, "N must be >= 1");
  if (o->m < 1 || o->m > kg::kMaxM) return host_fail(KG_ERR_INVALID_ARG, "m must satisfy 1 <= m <= 32");
  if (o->prec != KG_PREC_C128 && o->prec != KG_PREC_C64_F64REC && o->prec != KG_PREC_FF)
    return host_fail(KG_ERR_INVALID_ARG, "prec must be KG_PREC_C128, KG_PREC_C64_F64REC or KG_PREC_FF");
  if (o->grad != KG_GRAD_NONE && o->grad != KG_GRAD_CENTERED && o->grad != KG_GRAD_ZEROTH &&
      o->grad != KG_GRAD_EXACT && o->grad != KG_GRAD_TAYLOR1 && o->grad != KG_GRAD_TAYLOR2)
    return host_fail(KG_ERR_INVALID_ARG, "grad must be KG_GRAD_NONE, _CENTERED, _ZEROTH, _EXACT, _TAYLOR1 or _TAYLOR2");
  if (o->prec == KG_PREC_FF && o->grad != KG_GRAD_NONE && o->grad != KG_GRAD_CENTERED &&
      o->grad != KG_GRAD_ZEROTH)
    return host_fail(KG_ERR_UNSUPPORTED, "KG_PREC_FF offers KG_GRAD_NONE, _CENTERED and _ZEROTH");
  if (o->ckpt_every != 0) return host_fail(KG_ERR_UNSUPPORTED, "subspace evaluations keep every state: ckpt_every must be 0");
  if (o->tile_bits != 0) return host_fail(KG_ERR_INVALID_ARG, "tile_bits must be 0 for subspaces");
  if ((o->flags & ~KG_FLAG_PHASE_TIMING) != 0)
    return host_fail(KG_ERR_INVALID_ARG, "only KG_FLAG_PHASE_TIMING is accepted for subspaces");
  if (o->ctas < 0) return host_fail(KG_ERR_INVALID_ARG, "ctas must be >= 0");
  if (!(o->dt > 0.0) || !std::isfinite(o->dt)) return host_fail(KG_ERR_INVALID_ARG, "dt must be finite and > 0");
  if (std::isnan(o->breakdown_tol)) return host_fail(KG_ERR_INVALID_ARG, "breakdown_tol must not be NaN");
  return KG_OK;
}

// Whether a subspace is taken: two vectors and one 16-bit column per row and antiparallel bond within
// 200 KB (the split lists, which pad and double some entries, then take at most 202 KB: L = 14, K = 7 without
// parity).
bool sector_fits(const kg_options* o, const SectorBasis& b) {
  const size_t vb = (o->prec == KG_PREC_C64_F64REC) ? 8 : 16;
  const size_t Dp = ((size_t)b.D + 15) & ~(size_t)15;
  return 2 * Dp * vb + (size_t)b.bonds * b.D * 2 <= 200 * 1024 &&
         kg::sector_smem_bytes(o->prec, b.D, b.words()) <= kg::kSecMaxSmem;
}

// Grid for B pulses: every CTA that fits co-resident, at most B, at most opts->ctas.
kg_status sector_grid(const kg_options* o, const SectorBasis& b, int nt, int B, int* grid) {
  if (!sector_fits(o, b))
    return host_fail(KG_ERR_UNSUPPORTED, "the subspace's state and tables exceed one CTA's shared memory");
  int maxc = 0;
  cudaError_t e = kg::sector_kernel_max_ctas(o->prec, b.D, b.words(), nt, &maxc);
  if (e != cudaSuccess) {
    return host_fail(KG_ERR_CUDA, std::string("occupancy query: ") + cudaGetErrorName(e));
  }
  if (maxc < 1) return host_fail(KG_ERR_UNSUPPORTED, "the subspace kernel does not fit on this device");
  int g = std::min(B, maxc);
  if (o->ctas > 0) g = std::min(g, o->ctas);
  *grid = g;
  return KG_OK;
}

}  // namespace

struct kg_sector_handle {
  kg_sector sector;
  kg_options opts;
  SectorLayout lay;
  SectorBasis basis;
  char* ws = nullptr;
  cudaStream_t stream = nullptr;
  int device = 0, B = 1, grid = 1;
};

extern "C" {

kg_status kg_sector_dim(const kg_sector* s, int32_t* D) {
  if (!D) return host_fail(KG_ERR_INVALID_ARG, "D must not be NULL");
  kg_status st = check_sector(s);
  if (st != KG_OK) return st;
  SectorBasis b;
  std::string why;
  if (!build_basis(s, (size_t)kg::kSecMaxRows, false, b, why)) return host_fail(KG_ERR_UNSUPPORTED, why);
  *D = b.D;
  return KG_OK;
}

kg_status kg_sector_states(const kg_sector* s, uint64_t* states, int32_t D) {
  if (!states) return host_fail(KG_ERR_INVALID_ARG, "states must not be NULL");
  kg_status st = check_sector(s);
  if (st != KG_OK) return st;
  SectorBasis b;
  std::string why;
  if (!build_basis(s, (size_t)kg::kSecMaxRows, false, b, why)) return host_fail(KG_ERR_UNSUPPORTED, why);
  if (D != b.D) return host_fail(KG_ERR_INVALID_ARG, "D must equal the subspace dimension " + std::to_string(b.D));
  std::copy(b.states.begin(), b.states.end(), states);
  return KG_OK;
}

kg_status kg_sector_apply_h0(const kg_sector* s, const double* v, double* w, int32_t D) {
  if (!v || !w) return host_fail(KG_ERR_INVALID_ARG, "v and w must not be NULL");
  kg_status st = check_sector(s);
  if (st != KG_OK) return st;
  SectorBasis b;
  std::string why;
  if (!build_basis(s, (size_t)kg::kSecMaxRows, true, b, why)) return host_fail(KG_ERR_UNSUPPORTED, why);
  if (D != b.D) return host_fail(KG_ERR_INVALID_ARG, "D must equal the subspace dimension " + std::to_string(b.D));
  double wa, wb;
  list_weights(s, wa, wb);
  const uint64_t maskL1 = (1ull << (s->L - 1)) - 1ull;
  const unsigned* meta = b.tab.data() + (size_t)b.na2 * b.rows;
  for (int i = 0; i < b.D; ++i) {  // the kernel's row i: diagonal from its state, then the two lists
    const int r = b.perm[i];
    const uint64_t x = b.states[r];
    const double d = 0.25 * s->Jz * (double)(s->L - 1 - 2 * __builtin_popcountll((x ^ (x >> 1)) & maskL1));
    double re = d * v[2 * r], im = d * v[2 * r + 1];
    auto add = [&](unsigned word, double wt) {
      for (const int col : {(int)(word & 0xffffu) / 8, (int)(word >> 16) / 8}) {
        if (col >= b.D) continue;  // padding
        const int c = b.perm[col];
        re += wt * v[2 * c];
        im += wt * v[2 * c + 1];
      }
    };
    const unsigned mt = meta[i >> 5];
    for (unsigned q = 0; q < kg::sec_meta_na(mt); ++q) add(b.tab[(size_t)q * b.rows + i], wa);
    for (unsigned q = 0; q < kg::sec_meta_nb(mt); ++q) add(meta[b.groups + kg::sec_meta_first(mt) + 32 * q + (i & 31)], wb);
    w[2 * r] = re;
    w[2 * r + 1] = im;
  }
  return KG_OK;
}

kg_status kg_sector_workspace_bytes(const kg_sector* s, const kg_options* o, int32_t B, size_t* bytes) {
  if (!bytes) return host_fail(KG_ERR_INVALID_ARG, "bytes must not be NULL");
  kg_status st = check_sector(s);
  if (st != KG_OK) return st;
  if ((st = check_sector_opts(o, B)) != KG_OK) return st;
  SectorBasis b;
  std::string why;
  if (!build_basis(s, (size_t)kg::kSecMaxRows, true, b, why)) return host_fail(KG_ERR_UNSUPPORTED, why);
  if (!kg::sector_shape_ok(o->prec, b.D, s->block_threads))
    return host_fail(KG_ERR_INVALID_ARG, "block_threads too few for the subspace's dimension");
  // one trajectory per CTA: size for the grid kg_sector_create will choose on the current device
  // (B CTAs if no device can be queried)
  int grid = B;
  int dev = 0, maxc = 0;
  if (cudaGetDevice(&dev) == cudaSuccess &&
      sector_fits(o, b) &&
      kg::sector_kernel_max_ctas(o->prec, b.D, b.words(), s->block_threads, &maxc) == cudaSuccess && maxc > 0) {
    grid = std::min(B, maxc);
    if (o->ctas > 0) grid = std::min(grid, o->ctas);
  } else {
    cudaGetLastError();  // no device here: clear the error the query left
  }
  *bytes = sector_layout(b.D, b.words(), o, B, grid).total;
  return KG_OK;
}

kg_status kg_sector_create(kg_sector_handle** handle, const kg_sector* s, const kg_options* o, int32_t B,
                           void* workspace, size_t bytes, void* cuda_stream) {
  if (!handle) return host_fail(KG_ERR_INVALID_ARG, "handle must not be NULL");
  *handle = nullptr;
  kg_status st = check_sector(s);
  if (st != KG_OK) return st;
  if ((st = check_sector_opts(o, B)) != KG_OK) return st;
  kg_sector_handle* h = new kg_sector_handle();
  std::string why;
  if (!build_basis(s, (size_t)kg::kSecMaxRows, true, h->basis, why)) {
    delete h;
    return host_fail(KG_ERR_UNSUPPORTED, why);
  }
  if (h->basis.D < 1) {
    delete h;
    return host_fail(KG_ERR_INVALID_ARG, "the subspace is empty");
  }
  if (!kg::sector_shape_ok(o->prec, h->basis.D, s->block_threads)) {
    delete h;
    return host_fail(KG_ERR_INVALID_ARG, "block_threads too few for the subspace's dimension");
  }
  const size_t need1 = sector_layout(h->basis.D, h->basis.words(), o, B, 1).total;  // one CTA
  if (!workspace || ((uintptr_t)workspace % kg::kAlign) != 0 || bytes < need1) {
    delete h;
    return host_fail(KG_ERR_WORKSPACE, "workspace must be 256-byte aligned and hold at least " +
                                           std::to_string(need1) + " bytes");
  }
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) {
    delete h;
    return host_fail(KG_ERR_CUDA, std::string("cudaGetDevice: ") + cudaGetErrorName(e));
  }
  int grid = 1;
  if ((st = sector_grid(o, h->basis, s->block_threads, B, &grid)) != KG_OK) {
    delete h;
    return st;
  }
  const size_t need = sector_layout(h->basis.D, h->basis.words(), o, B, grid).total;
  if (bytes < need) {
    delete h;
    return host_fail(KG_ERR_WORKSPACE, "workspace too small: need " + std::to_string(need) + " bytes, got " +
                                           std::to_string(bytes));
  }
  h->sector = *s;
  h->opts = *o;
  if (!(h->opts.breakdown_tol > 0.0))
    h->opts.breakdown_tol = (o->prec == KG_PREC_C128) ? 1e-12 : (o->prec == KG_PREC_FF) ? 1e-10 : 1e-5;
  h->lay = sector_layout(h->basis.D, h->basis.words(), o, B, grid);
  h->ws = (char*)workspace;
  h->stream = (cudaStream_t)cuda_stream;
  h->device = dev;
  h->B = B;
  h->grid = grid;
  // tables into the workspace (32-bit states: L <= 30)
  std::vector<unsigned> st32;
  for (const unsigned short r : h->basis.perm) st32.push_back((unsigned)h->basis.states[r]);
  e = cudaMemcpyAsync(h->ws + h->lay.states, st32.data(), st32.size() * sizeof(unsigned), cudaMemcpyHostToDevice,
                      h->stream);
  if (e == cudaSuccess)
    e = cudaMemcpyAsync(h->ws + h->lay.perm, h->basis.perm.data(), h->basis.perm.size() * sizeof(unsigned short),
                        cudaMemcpyHostToDevice, h->stream);
  if (e == cudaSuccess)
    e = cudaMemcpyAsync(h->ws + h->lay.tab, h->basis.tab.data(), h->basis.tab.size() * 4, cudaMemcpyHostToDevice,
                        h->stream);
  if (e == cudaSuccess) e = cudaStreamSynchronize(h->stream);
  if (e != cudaSuccess) {
    delete h;
    return host_fail(KG_ERR_CUDA, std::string("upload of the subspace tables: ") + cudaGetErrorName(e));
  }
  *handle = h;
  return KG_OK;
}

kg_status kg_sector_evaluate(kg_sector_handle* h, const double* u, const void* psi0, const void* target, double* fid,
                             double* grad) {
  if (!h) return host_fail(KG_ERR_INVALID_ARG, "handle must not be NULL");
  if (!u || !psi0 || !target || !fid) return host_fail(KG_ERR_INVALID_ARG, "u, psi0, target and fid must not be NULL");
  if (h->opts.grad != KG_GRAD_NONE && !grad) return host_fail(KG_ERR_INVALID_ARG, "grad must not be NULL");
  if (((uintptr_t)psi0 % 16) || ((uintptr_t)target % 16) || ((uintptr_t)u % 8) || ((uintptr_t)fid % 8) ||
      (grad && ((uintptr_t)grad % 8)))
    return host_fail(KG_ERR_INVALID_ARG, "psi0/target must be 16-byte aligned, u/fid/grad 8-byte aligned");
  int dev = -1;
  cudaGetDevice(&dev);
  if (dev != h->device) return host_fail(KG_ERR_INVALID_ARG, "current device differs from the handle's device");
  const kg_sector& s = h->sector;
  const kg_options& o = h->opts;
  kg::SectorParams p{};
  p.D = h->basis.D;
  p.N = o.N;
  p.m = o.m;
  p.na2 = h->basis.na2;
  p.rows = h->basis.rows;
  p.groups = h->basis.groups;
  p.words = h->basis.words();
  p.B = h->B;
  p.L1 = s.L - 1;
  p.grad_mode = o.grad;
  p.maskL1 = (unsigned)((1ull << (s.L - 1)) - 1ull);
  p.hc_mask = (unsigned)s.hc_site_mask;
  p.qz = 0.25 * s.Jz;
  p.hc_amp = s.hc_amp;
  p.dt = o.dt;
  p.bd_tol = o.breakdown_tol;
  list_weights(&s, p.wa, p.wb);
  p.wa_f = (float)p.wa;
  p.wb_f = (float)p.wb;
  p.dt_f = (float)p.dt;
  p.bd_tol_f = (float)p.bd_tol;
  char* ws = h->ws;
  p.tab_g = (const unsigned*)(ws + h->lay.tab);
  p.states = (const unsigned*)(ws + h->lay.states);
  p.perm = (const unsigned short*)(ws + h->lay.perm);
  p.u = u;
  p.psi0 = (const double*)psi0;
  p.target = (const double*)target;
  p.fid = fid;
  p.grad = grad;
  p.traj = ws + h->lay.traj;
  p.basis = ws + h->lay.basis;
  p.tint = (o.grad == KG_GRAD_EXACT) ? (void*)(ws + h->lay.tint) : nullptr;
  p.G = (double*)(ws + h->lay.G);
  p.scal = (double*)(ws + h->lay.scal);
  p.ctrl = (int*)(ws + h->lay.ctrl);
  p.time_limit_ns = kg::sector_time_limit_ns();
  p.prof = (o.flags & KG_FLAG_PHASE_TIMING) ? (long long*)(ws + h->lay.prof) : nullptr;
  cudaError_t e = cudaMemsetAsync(ws + h->lay.ctrl, 0, 64, h->stream);
  if (e != cudaSuccess) return host_fail(KG_ERR_CUDA, std::string("cudaMemsetAsync(control block): ") + cudaGetErrorName(e));
  e = kg::launch_sector_kernel(o.prec, p, h->grid, h->sector.block_threads, h->stream);
  if (e != cudaSuccess) return host_fail(KG_ERR_CUDA, std::string("launch of the subspace kernel: ") + cudaGetErrorName(e));
  return KG_OK;
}

kg_status kg_sector_sync(kg_sector_handle* h, kg_report* rep) {
  if (!h) return host_fail(KG_ERR_INVALID_ARG, "handle must not be NULL");
  cudaError_t e = cudaStreamSynchronize(h->stream);
  if (e != cudaSuccess) return host_fail(KG_ERR_CUDA, std::string("cudaStreamSynchronize: ") + cudaGetErrorName(e));
  int ctrl[2] = {0, 0};
  e = cudaMemcpy(ctrl, h->ws + h->lay.ctrl, sizeof(ctrl), cudaMemcpyDeviceToHost);
  if (e != cudaSuccess) return host_fail(KG_ERR_CUDA, std::string("cudaMemcpy(status): ") + cudaGetErrorName(e));
  if (rep) {
    std::vector<double> sc((size_t)h->B * kg::kScCount);
    e = cudaMemcpy(sc.data(), h->ws + h->lay.scal, sc.size() * sizeof(double), cudaMemcpyDeviceToHost);
    if (e != cudaSuccess) return host_fail(KG_ERR_CUDA, std::string("cudaMemcpy(report): ") + cudaGetErrorName(e));
    std::memset(rep, 0, sizeof(*rep));
    rep->beta_re = sc[kg::kScBetaRe];
    rep->beta_im = sc[kg::kScBetaIm];
    rep->norm_final = sc[kg::kScNormFinal];
    double emax = 0.0, bd = 0.0;
    for (int b = 0; b < h->B; ++b) {
      emax = std::max(emax, sc[(size_t)b * kg::kScCount + kg::kScErrMax]);
      bd += sc[(size_t)b * kg::kScCount + kg::kScBreakdowns];
    }
    rep->krylov_err_max = emax;
    rep->breakdowns = (int32_t)bd;
    rep->status = ctrl[kg::kCtrlStatus];
    rep->launches = 1;
    rep->ctas = h->grid;
    rep->threads = kg::sector_threads(h->opts.prec, h->basis.D, h->sector.block_threads);
    rep->ckpt_every = 0;
    rep->reserved0 = 0;
    if (h->opts.flags & KG_FLAG_PHASE_TIMING) {
      long long pc[8];
      e = cudaMemcpy(pc, h->ws + h->lay.prof, sizeof(pc), cudaMemcpyDeviceToHost);
      if (e != cudaSuccess) return host_fail(KG_ERR_CUDA, std::string("cudaMemcpy(phase timing): ") + cudaGetErrorName(e));
      for (int i = 0; i < 8; ++i) rep->phase_cycles[i] = pc[i];
    }
  }
  const int stv = ctrl[kg::kCtrlStatus];
  if (stv == KG_ERR_TIMEOUT) return host_fail(KG_ERR_TIMEOUT, "a pulse ran past the per-pulse time limit");
  if (stv == KG_ERR_NONFINITE) return host_fail(KG_ERR_NONFINITE, "non-finite Lanczos coefficient or norm");
  if (stv != 0) return host_fail(KG_ERR_CUDA, "device status " + std::to_string(stv));
  return KG_OK;
}

kg_status kg_sector_destroy(kg_sector_handle* h) {
  delete h;
  return KG_OK;
}

}  // extern "C"
