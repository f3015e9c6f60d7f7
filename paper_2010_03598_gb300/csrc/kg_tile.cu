// K-GRAPE evaluation with one tile of amplitudes per CTA, held in registers: the forward Krylov
// sweep, target overlap, co-state sweep and gradient of one pulse, in one launch.
//
// For chains whose amplitudes fit the registers of one CTA (or of the co-resident CTAs with one tile
// each) an evaluation is a chain of short Krylov steps, whose cost is latency: block
// barriers, warp sums, the recurrence's scalars and the small exponential.  This kernel is laid out
// for that chain.  A CTA has as many threads as its tile needs (a thread owns APT amplitudes
// li = tid + NT j), two block barriers per Lanczos step, and on the complex64 path a step has no FP64
// instruction (a slice has a few: the conversions and prefactors of set_control): one FP64 instruction
// occupies a quarter of the SM's FP64 unit for 64 cycles whatever the number of active lanes, so padding
// warps and scalar chains in FP64 are what small chains spend their time on otherwise.
//
// One Lanczos step (App. A, Alg. "Lanczos", Paige's order), v_k in shared memory for the neighbours:
//   W_{k+1} = H v_k - b_k v_{k-1},   H v = diag v + (Jxy/2) sum_{antiparallel bonds} v[partner] (+ control)
//   alpha_k = <v_k|W_{k+1}>,  b_{k+1}^2 = ||W_{k+1}||^2 - 2 alpha_k <v_k|W_{k+1}> + alpha_k^2 ||v_k||^2
//   v_{k+1} = (W_{k+1} - alpha_k v_k) / b_{k+1}
// with the two block barriers (the sums, v_{k+1}); every warp adds up the warps' partial sums and forms the
// scalars for itself.  v_{k-1}, v_k and W stay in registers; the basis holds the v_k (shared memory if
// it fits, else global).
//
// Several CTAs: the stencil acts on the raw vector W_k, which needs none of the step's
// scalars, so that it runs while the group's sums are under way:
//   v_k = (W_k - alpha_{k-1} v_{k-1}) / b_k,   H v_k = (H W_k - alpha_{k-1} H v_{k-1}) / b_k.
// (On one CTA the waits it would hide are short, and H v_k by its recurrence carries more rounding.)  A
// control warp posts the CTA's sums in 16-byte {values, sequence number} messages: every CTA polls the
// other CTAs' messages and adds them up in the same order.  The tiles' W_k are exchanged through global
// memory: complex64 in such messages as well, which their readers poll, so that a step is one trip
// through L2; complex128 (16-byte amplitudes) as plain data, which a fence before the sums' message
// makes visible, and which is copied once the sums have arrived.
#include <cuda_runtime.h>

#include <type_traits>

#include "kg_device.cuh"
#include "kg_launch.h"

namespace kg {
namespace {

// ---------------------------------------------------------------- per-precision arithmetic
// Sum of a reduction, scalar of the recurrence (complex64: float-float sums, FP32 scalars).
template <class V> struct Prec;
template <> struct Prec<float2> {
  using R = float;
  using S = FF;
  static constexpr bool F32 = true;
};
template <> struct Prec<double2> {
  using R = double;
  using S = double;
  static constexpr bool F32 = false;
};

__device__ __forceinline__ float2 vadd(float2 a, float2 b) { return __fadd2_rn(a, b); }
__device__ __forceinline__ double2 vadd(double2 a, double2 b) { return make_double2(a.x + b.x, a.y + b.y); }
__device__ __forceinline__ float2 vmul(float a, float2 x) { return __fmul2_rn(make_float2(a, a), x); }
__device__ __forceinline__ double2 vmul(double a, double2 x) { return make_double2(a * x.x, a * x.y); }
__device__ __forceinline__ float2 vfma(float a, float2 x, float2 y) { return __ffma2_rn(make_float2(a, a), x, y); }
__device__ __forceinline__ double2 vfma(double a, double2 x, double2 y) {
  return make_double2(fma(a, x.x, y.x), fma(a, x.y, y.y));
}
// y + (a + ib) x, the part with b first: a is the larger one where the rounding counts (slot 0)
__device__ __forceinline__ float2 vcfma(float a, float b, float2 x, float2 y) {
  return make_float2(fmaf(a, x.x, fmaf(-b, x.y, y.x)), fmaf(a, x.y, fmaf(b, x.x, y.y)));
}
__device__ __forceinline__ double2 vcfma(double a, double b, double2 x, double2 y) {
  return make_double2(fma(a, x.x, fma(-b, x.y, y.x)), fma(a, x.y, fma(b, x.x, y.y)));
}

__device__ __forceinline__ FF sfrom(double d, FF) { return ff_from_double(d); }
__device__ __forceinline__ double sfrom(double d, double) { return d; }
__device__ __forceinline__ double sdouble(FF a) { return ff_to_double(a); }
__device__ __forceinline__ double sdouble(double a) { return a; }
__device__ __forceinline__ float sround(FF a) { return __fadd_rn(a.hi, a.lo); }
__device__ __forceinline__ double sround(double a) { return a; }
__device__ __forceinline__ bool sfinite(FF a) { return isfinite(a.hi); }
__device__ __forceinline__ bool sfinite(double a) { return isfinite(a); }

// A sum kept in 8 bytes of a double array (G, nrm) between slices; read back by whoever needs it.
__device__ __forceinline__ double spack(FF a) {
  return __hiloint2double(__float_as_int(a.hi), __float_as_int(a.lo));
}
__device__ __forceinline__ double spack(double a) { return a; }
__device__ __forceinline__ FF sunpack(double d, FF) {
  return FF{__int_as_float(__double2hiint(d)), __int_as_float(__double2loint(d))};
}
__device__ __forceinline__ double sunpack(double d, double) { return d; }

__device__ __forceinline__ float sinv(FF n) {
  const float f = sround(n);
  return (f > 0.f) ? __frcp_rn(f) : 0.f;
}
__device__ __forceinline__ double sinv(double n) { return (n > 0.0) ? 1.0 / n : 0.0; }
// ||x|| and 1/||x|| from ||x||^2.
__device__ __forceinline__ void snorm(FF n2, FF& n, float& inv) {
  n = ff_sqrt(n2);
  inv = sinv(n);
}
__device__ __forceinline__ void snorm(double n2, double& n, double& inv) {
  n = sqrt(fmax(n2, 0.0));
  inv = (n > 0.0) ? 1.0 / n : 0.0;
}

// b^2 = n + a^2 (q - 2), b and 1/b
__device__ __forceinline__ FF sb2(FF a, FF n, FF q) { return ff_add(n, ff_mul(ff_mul(a, a), ff_add(q, FF{-2.f, 0.f}))); }
__device__ __forceinline__ double sb2(double a, double n, double q) { return fma(a * a, q - 2.0, n); }
__device__ __forceinline__ bool scancels(FF b2, FF n) { return b2.hi < 1e-3f * n.hi; }
__device__ __forceinline__ bool scancels(double b2, double n) { return b2 < 1e-3 * n; }
// b and 1/b from b^2: the FP32 estimate of 1/sqrt refined by one step of Newton's iteration (complex64:
// the residual 1 - b^2 y^2 formed exactly, so that both results are rounded once) or of Halley's (FP64:
// cubic convergence, 2^-22 -> below 2^-60), then b = b^2 / b.
__device__ __forceinline__ void sroot(FF b2, float& b, float& inv) {
  const float x = b2.hi;
  if (!(x > 1e-30f)) {
    b = __fsqrt_rn(fmaxf(sround(b2), 0.f));
    inv = (b > 0.f) ? __frcp_rn(b) : 0.f;
    return;
  }
  const float y = rsqrtf(x);
  const float p = __fmul_rn(x, y);
  const float e = __fmaf_rn(x, y, -p) + b2.lo * y;  // b2 y = p + e
  const float r = __fmaf_rn(-p, y, 1.f) - e * y;
  inv = fmaf(0.5f * r, y, y);
  const float c = x * inv;
  b = fmaf(0.5f * inv, fmaf(-c, c, x) + b2.lo, c);
}
__device__ __forceinline__ void sroot(double b2, double& b, double& inv) {
  if (!(b2 > 1e-30 && b2 < 1e30)) {
    inv = (b2 > 0.0) ? rsqrt(b2) : 0.0;
    b = fmax(b2, 0.0) * inv;
    return;
  }
  const double y = (double)rsqrtf((float)b2);
  const double r = fma(-b2 * y, y, 1.0);
  inv = fma(y, r * fma(0.375, r, 0.5), y);
  b = b2 * inv;
}

constexpr int kTileSums = 3;  // values of one reduction

struct TileSmem {
  float red_f[2][16][4];     // warp partials (complex64: FP32 sums), by reduction parity
  double red_d[2][16][4];    // warp partials (complex128, and the FP64 overlaps of complex64)
  double tot[2][4];          // group totals (several CTAs), by parity (complex64: packed float-float)
  float2 al_ff[kMaxM], b2_ff[kMaxM];  // complex64: alpha_k, b_{k+1}^2 of the slice (float-float)
  double al[kMaxM], be[kMaxM + 1];    // complex128: alpha_k, b_{k+1}
  double coef_re[3][kMaxM], coef_im[3][kMaxM];
  float coef_re_f[3][kMaxM], coef_im_f[3][kMaxM];
  float2 tau_ff[3];          // complex64: dt and the interior quadrature nodes s_a, s_b of a slice
  float err_max;
  int breakdowns;
  int cmd, ok;               // control warp: hand-over and answer
  int lost;                  // a worker gave up waiting for partner amplitudes
  long long prof_last, prof_acc[8];
};

// ---------------------------------------------------------------- messages between CTAs
// 16-byte accesses at one point of the memory system: value and sequence number travel together.
__device__ __forceinline__ void st_msg(ulonglong2* p, unsigned long long v, unsigned long long seq) {
  asm volatile("{\n .reg .b128 q;\n mov.b128 q, {%1, %2};\n st.relaxed.gpu.global.b128 [%0], q;\n}" ::"l"(p), "l"(v), "l"(seq)
               : "memory");
}
__device__ __forceinline__ ulonglong2 ld_msg(const ulonglong2* p) {
  ulonglong2 r;
  asm volatile("{\n .reg .b128 q;\n ld.relaxed.gpu.global.b128 q, [%2];\n mov.b128 {%0, %1}, q;\n}"
               : "=l"(r.x), "=l"(r.y)
               : "l"(p)
               : "memory");
  return r;
}

// Lighter than __threadfence(), which is sequentially consistent.
__device__ __forceinline__ void fence_acq_rel() { asm volatile("fence.acq_rel.gpu;" ::: "memory"); }

constexpr int kTileBarPost = 2, kTileBarGroup = 3;
constexpr int kTileCmdSums = 1, kTileCmdExit = 2, kTileCmdFp64 = 8, kTileCmdFence = 16;  // bit 2: the reduction's parity

// A 16-byte message of three floats and a sequence number.
struct Atom {
  float f[3];
  unsigned seq;
};
__device__ __forceinline__ void st_atom(ulonglong2* p, float a, float b, float c, unsigned seq) {
  asm volatile("{\n .reg .b128 q;\n .reg .b64 x, y;\n mov.b64 x, {%1, %2};\n mov.b64 y, {%3, %4};\n mov.b128 q, {x, y};\n"
               " st.relaxed.gpu.global.b128 [%0], q;\n}" ::"l"(p), "f"(a), "f"(b), "f"(c), "r"(seq)
               : "memory");
}
__device__ __forceinline__ Atom ld_atom(const ulonglong2* p) {
  Atom a;
  asm volatile("{\n .reg .b128 q;\n .reg .b64 x, y;\n ld.relaxed.gpu.global.b128 q, [%4];\n mov.b128 {x, y}, q;\n"
               " mov.b64 {%0, %1}, x;\n mov.b64 {%2, %3}, y;\n}"
               : "=f"(a.f[0]), "=f"(a.f[1]), "=f"(a.f[2]), "=r"(a.seq)
               : "l"(p)
               : "memory");
  return a;
}

template <class V, int NT, int APT, bool SB, bool MULTI>
struct Tile {
  using P = Prec<V>;
  using R = typename P::R;
  using S = typename P::S;
  static constexpr bool F32 = P::F32;
  static constexpr int NW = NT / 32;
  static constexpr int LT = (NT == 32) ? 5 : (NT == 64) ? 6 : (NT == 128) ? 7 : (NT == 256) ? 8 : 9;
  static constexpr int LA = (APT == 1) ? 0 : (APT == 2) ? 1 : (APT == 4) ? 2 : (APT == 8) ? 3 : 4;
  static constexpr int T = NT * APT;
  static constexpr bool RAW = MULTI || APT == 16;  // the stencil acts on the raw vectors
  static constexpr bool MSG = MULTI && F32;        // W_k travels in messages
  static_assert((1 << LT) == NT && (1 << LA) == APT, "powers of two");

  const EvalParams& p;
  TileSmem& sm;
  V* sw;        // [2][T] the neighbours' vector, by the parity of the step; SB: [m][T], the basis itself
  V* ring;      // MULTI: [RD][T] partner blocks of W_k
  int tid, wid, rank, D1;  // D1: amplitudes of the tile that exist (T, or fewer for chains below 5 spins)
  size_t base, D;
  int nb;       // bonds inside the tile
  int par;      // parity of the next reduction
  R hxy;
  R dj[APT];           // diagonal of H_j
  R cx;                // Sx control weight of the slice
  double hca;          // hc_amp, times 1/2 for an Sx control
  unsigned bonds_hi;   // MULTI: active bonds with both bits above the tile, bit b
  unsigned seq;        // MSG: number of the newest W_k
  V wo[APT];           // own W_k
  float2 fact;         // complex64: this lane's entry of kInvFactFF
  float w1;            // one warp, complex64: its sums (lane i: sum i)
  S nrm;               // ||W_0||
  R inv;               // 1 / ||W_0||

  __device__ __forceinline__ void mark(int ph) {
    if (p.prof != nullptr && rank == 0 && tid == 0) {
      const long long now = clock64();
      sm.prof_acc[ph] += now - sm.prof_last;
      sm.prof_last = now;
    }
  }

  __device__ __forceinline__ void sync() {
    if constexpr (MULTI) asm volatile("barrier.sync 1, %0;" ::"n"(NT) : "memory");
    else if constexpr (NW == 1) __syncwarp();
    else asm volatile("barrier.sync 0;" ::: "memory");  // lanes of warp 0 may arrive apart
  }

  // -------------------------------------------------------------- sums over the block / the group
  // post: this thread's values into the warp partials (and, MULTI, the hand-over to the control
  // warp); collect (after the barrier that follows): the totals, the same bits in every thread.
  // fence: what the CTA stored before is visible to who reads the sums (several CTAs).
  __device__ __forceinline__ void post(const R (&v)[kTileSums], bool fence = true) {
    const int lane = tid & 31, warp = tid >> 5;
    const R s = warp_sum3<R>(v[0], v[1], v[2]);
    if constexpr (F32 && NW == 1) {
      w1 = s;
      return;
    }
    if (lane < 4) {
      if constexpr (F32) sm.red_f[par][warp][lane] = s;
      else sm.red_d[par][warp][lane] = s;
    }
    if constexpr (MULTI) {
      if (tid == 0) sm.cmd = kTileCmdSums | (fence ? kTileCmdFence : 0) | (par << 2);
      nbar_arrive(kTileBarPost, NT + 32);
    }
  }
  __device__ __forceinline__ bool collect(S (&out)[kTileSums]) {
    if constexpr (MULTI) {
      nbar_sync(kTileBarGroup, NT + 32);
#pragma unroll
      for (int i = 0; i < kTileSums; ++i) out[i] = sunpack(sm.tot[par][i], S());
      par ^= 1;
      return sm.ok != 0;
    } else if constexpr (F32 && NW == 1) {
#pragma unroll
      for (int i = 0; i < kTileSums; ++i) out[i] = FF{__shfl_sync(0xffffffffu, w1, i), 0.f};
    } else if constexpr (F32) {
      warps_sum3<NW, FF>([&](int w, int i) { return FF{sm.red_f[par][w][i], 0.f}; }, out);
      par ^= 1;
    } else {
      warps_sum3<NW, double>([&](int w, int i) { return sm.red_d[par][w][i]; }, out);
      par ^= 1;
    }
    return true;
  }
  // Sums of FP64 values whatever the path (overlap with the complex128 target): twice an evaluation.
  __device__ __forceinline__ bool sum_fp64(const double (&v)[kTileSums], double (&out)[kTileSums]) {
    const int lane = tid & 31, warp = tid >> 5;
    if constexpr (!F32) {
      post(v);
      if constexpr (!MULTI) sync();
      return collect(out);
    } else {
#pragma unroll
      for (int i = 0; i < kTileSums; ++i) {
        const double s = warp_sum(v[i]);
        if (lane == 0) sm.red_d[par][warp][i] = s;
      }
      if constexpr (MULTI) {  // the other CTAs' share arrives in float-float
        if (tid == 0) sm.cmd = kTileCmdSums | kTileCmdFence | kTileCmdFp64 | (par << 2);
        nbar_arrive(kTileBarPost, NT + 32);
        S o[kTileSums];
        if (!collect(o)) return false;
#pragma unroll
        for (int i = 0; i < kTileSums; ++i) out[i] = sdouble(o[i]);
        return true;
      }
      sync();
#pragma unroll
      for (int i = 0; i < kTileSums; ++i) {
        double s = sm.red_d[par][lane & (NW - 1)][i];
#pragma unroll
        for (int o = 1; o < NW; o <<= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
        out[i] = s;
      }
      par ^= 1;
      return true;
    }
  }

  // -------------------------------------------------------------- setup
  __device__ __forceinline__ int li(int j) const { return tid + j * NT; }
  __device__ __forceinline__ void init() {
    wid = __shfl_sync(0xffffffffu, tid >> 5, 0);
    hxy = (R)(0.5 * p.Jxy);
    hca = (p.hc_kind == KG_HC_SX_SITE) ? 0.5 * p.hc_amp : p.hc_amp;
    nb = MULTI ? LT + LA - 1 : min(p.L - 1, LT + LA - 1);
    bonds_hi = 0u;
    fact = kInvFactFF[min(tid & 31, 29)];
    if (F32 && tid == 0) {
      const double s = 0.5 * p.dt * (1.0 - 0.4472135954999579);  // 1/sqrt(5)
      const FF t[3] = {ff_from_double(p.dt), ff_from_double(s), ff_from_double(p.dt - s)};
      for (int i = 0; i < 3; ++i) sm.tau_ff[i] = make_float2(t[i].hi, t[i].lo);
    }
    if constexpr (MULTI)
      bonds_hi = (unsigned)((base ^ (base >> 1)) & ((1u << (p.L - 1)) - 1u)) & ~((1u << (LT + LA)) - 1u);
  }
  // Diagonal of Hc = hc_amp sum Sz over the mask, in units of hc_amp.
  __device__ __forceinline__ R zdiag(int j) const {
    const unsigned mk = (unsigned)p.hc_mask, gi = (unsigned)(base + li(j));
    return (R)(0.5f * (float)(__popc(mk) - 2 * __popc(gi & mk)));
  }
  __device__ __forceinline__ void set_control(double uj) {
    const bool sx = (p.hc_kind == KG_HC_SX_SITE);
    const R c = (R)(uj * hca);
    cx = sx ? c : (R)0;
    const unsigned maskL1 = (p.L >= 2) ? ((1u << (p.L - 1)) - 1u) : 0u;
    const R qz = (R)(0.25 * p.Jz);
#pragma unroll
    for (int j = 0; j < APT; ++j) {
      const unsigned gi = (unsigned)(base + li(j));
      dj[j] = qz * (R)((p.L - 1) - 2 * __popc((gi ^ (gi >> 1)) & maskL1));
      if (!sx) dj[j] = fma(c, zdiag(j), dj[j]);
    }
  }

  // -------------------------------------------------------------- H x inside the tile
  // s: the tile's vector in shared memory; x: the own amplitudes of the same vector.
  __device__ __forceinline__ void stencil(const V* s, const V (&x)[APT], V (&h)[APT]) {
#pragma unroll
    for (int j = 0; j < APT; ++j) h[j] = vmake<V>(0, 0);
    const unsigned xt = (unsigned)(tid ^ (tid >> 1));
    // Bonds with a bit inside the warp: every lane loads its partner and adds it times 0 or 1, so that
    // no branch separates the loads (with the loads under the lane's condition each bond's latency was
    // waited for by itself: 24.2 us a slice at L = 10, m = 16 instead of 22.2).
#pragma unroll
    for (int b = 0; b < (LT - 1 < 5 ? LT - 1 : 5); ++b) {
      if (b < nb) {
        const V* q = s + (tid ^ (3 << b));
        const R on = (R)(float)((xt >> b) & 1u);
#pragma unroll
        for (int j = 0; j < APT; ++j) h[j] = vfma(on, q[j * NT], h[j]);
      }
    }
#pragma unroll
    for (int b = 5; b < LT - 1; ++b) {  // both bits in the warp's number: the same for all lanes
      if (((wid >> (b - 5)) ^ (wid >> (b - 4))) & 1) {
        const V* q = s + (tid ^ (3 << b));
#pragma unroll
        for (int j = 0; j < APT; ++j) h[j] = vadd(h[j], q[j * NT]);
      }
    }
    if constexpr (APT > 1) {
      const int tt = (tid >> (LT - 1)) & 1;  // top bit of tid against bit 0 of j
#pragma unroll
      for (int j = 0; j < APT; ++j)
        if (tt != (j & 1)) h[j] = vadd(h[j], s[(tid ^ (NT / 2)) + (j ^ 1) * NT]);
#pragma unroll
      for (int c = 0; c + 1 < LA; ++c)  // both bits in j: registers
#pragma unroll
        for (int j = 0; j < APT; ++j)
          if (((j >> c) ^ (j >> (c + 1))) & 1) h[j] = vadd(h[j], x[j ^ (3 << c)]);
    }
#pragma unroll
    for (int j = 0; j < APT; ++j) h[j] = vfma(dj[j], x[j], vmul(hxy, h[j]));
    if (p.hc_kind == KG_HC_SX_SITE && p.hc_site < LT + LA) {
#pragma unroll
      for (int j = 0; j < APT; ++j) h[j] = vfma(cx, s[li(j) ^ (1 << p.hc_site)], h[j]);
    }
  }

  // MULTI: partner blocks of W_k from the other tiles, through this thread's own slots of the ring.
  // Slot 0: the bond between the tile's top bit and the lowest bit above it (half of the amplitudes);
  // then the bonds above the tile that are antiparallel for the whole tile; then an Sx control above it.
  __device__ __forceinline__ bool top_active(int j) const {
    constexpr int b = LT + LA - 1;
    return ((unsigned)(li(j) >> b) ^ (unsigned)(base >> (b + 1))) & 1u;
  }
  // Blocks in flight: complex128 through a ring in shared memory, complex64 in registers (more of them find
  // more messages that have not arrived: 16 spins 59.4 us a slice with 2, 61.4 with 3, 75.5 with 4; 18
  // spins 89.5 with 1, 98.4 with 2).
  static constexpr int RD = F32 ? (NT <= 128 ? 2 : 1) : (T <= 1024) ? 6 : 4;
  __device__ __forceinline__ int cross_count() const {
    return 1 + __popc(bonds_hi) + ((p.hc_kind == KG_HC_SX_SITE && p.hc_site >= LT + LA) ? 1 : 0);
  }
  // complex64: a thread's amplitudes of W_k travel as messages of three floats and the vector's number,
  // which their readers poll: one trip through L2 for the exchange, where data, a fence and a barrier
  // take three (m = 16: 16 spins 72.8 -> 59.4 us a slice, 13 spins 52 -> 40).  12 bytes an amplitude: two
  // vectors' messages take the three vectors wbuf, xbuf of the workspace.  Every partner amplitude belongs to the same thread of another CTA (all bits
  // of the thread's number lie below those that change), so that a message holds one thread's floats.
  // Two sets, by the number's parity: number n + 2 is stored only after the sums that every CTA posted
  // with n already read.  A message is never read in part: the two halves of the amplitudes (by the top bit of the tile) fill
  // messages of their own, and what is left of the last one of each holds the number too and is checked.
  // (With a component unused the compiler loads the others apart, and number and floats may then
  // belong to different vectors.)
  static constexpr int NH = (APT + 2) / 3, NA = 2 * NH;  // messages of a half, of a thread
  static_assert(!MSG || NA * 16 <= 12 * APT, "the messages of two vectors fit three vectors");
  Atom xa[MSG ? RD : 1][MSG ? NA : 1];
  __device__ __forceinline__ ulonglong2* atoms(unsigned n, int r) const {
    return reinterpret_cast<ulonglong2*>(p.wbuf) + ((size_t)(n & 1u) << (p.L - LT - LA)) * (NA * NT) + (size_t)r * (NA * NT) + tid;
  }
  __device__ __forceinline__ void send() {  // wo as the next number
    if constexpr (MSG) {
      ++seq;
      ulonglong2* q = atoms(seq, rank);
#pragma unroll
      for (int a = 0; a < NA; ++a) {
        float f[3];
#pragma unroll
        for (int i = 0; i < 3; ++i) {
          const int o = 3 * (a % NH) + i, n = a / NH * APT + min(o, APT - 1);  // float n of the thread
          f[i] = (o >= APT) ? __uint_as_float(seq) : (float)(n & 1 ? wo[n / 2].y : wo[n / 2].x);
        }
        st_atom(q + a * NT, f[0], f[1], f[2], seq);
      }
    }
  }
  // The CTA of block n > 0; `act` (the active bonds from block n on) moves on.
  __device__ __forceinline__ int cross_rank(unsigned& act) const {
    const int r = rank ^ (act ? 3 << (__ffs(act) - 1 - LT - LA) : 1 << (p.hc_site - LT - LA));
    act &= act - 1;
    return r;
  }
  __device__ __forceinline__ void recv_issue(int r, int half, Atom (&q)[MSG ? NA : 1]) {
    const ulonglong2* s = atoms(seq, r);
#pragma unroll
    for (int a = 0; a < NA; ++a)
      if (half < 0 || a / NH == half) q[a] = ld_atom(s + a * NT);
  }
  static __device__ __forceinline__ bool is_number(const Atom& q, int a, unsigned n) {
    bool is = q.seq == n;
#pragma unroll
    for (int i = 0; i < 3; ++i)
      if (3 * (a % NH) + i >= APT) is = is && __float_as_uint(q.f[i]) == n;
    return is;
  }
  // Polls until every atom of the block carries the number; gives up like the control warp, which then
  // ends the evaluation (sm.lost).
  __device__ __forceinline__ void recv_wait(int r, int half, Atom (&q)[MSG ? NA : 1]) {
    const ulonglong2* s = atoms(seq, r);
    unsigned polls = 0;
    unsigned long long t0 = 0;
    for (;;) {
      bool open = false;
#pragma unroll
      for (int a = 0; a < NA; ++a) open |= (half < 0 || a / NH == half) && !is_number(q[a], a, seq);
      if (!open) break;
      if ((++polls & 31u) == 0u) {
        bool give_up = ld_volatile_i32(p.ctrl + kCtrlAbort) != 0;
        const unsigned long long now = globaltimer_ns();
        if (t0 == 0) {
          t0 = now;
        } else if ((long long)(now - t0) > p.wait_limit_ns) {
          atomicCAS(p.ctrl + kCtrlStatus, 0, (int)KG_ERR_TIMEOUT);
          atomicExch(p.ctrl + kCtrlAbort, 1);
          give_up = true;
        }
        if (give_up) {
          sm.lost = 1;
          break;
        }
      }
#pragma unroll
      for (int a = 0; a < NA; ++a)
        if ((half < 0 || a / NH == half) && !is_number(q[a], a, seq)) q[a] = ld_atom(s + a * NT);
    }
    __syncwarp();
  }
  static __device__ __forceinline__ float atom_float(const Atom (&q)[MSG ? NA : 1], int n) {
    return q[n / APT * NH + n % APT / 3].f[n % APT % 3];
  }
  static __device__ __forceinline__ V atom_amp(const Atom (&q)[MSG ? NA : 1], int j) {
    if constexpr (MSG) return vmake<V>(atom_float(q, 2 * j), atom_float(q, 2 * j + 1));
    else return vmake<V>(0, 0);
  }
  // Copies of block n into slot n % RD; `act`: the active bonds from block n on.  One commit group per
  // block, empty past the last.
  __device__ __forceinline__ void cross_copy(const V* w, int n, int count, unsigned& act) {
    if constexpr (MULTI && !F32) {
      V* r = ring + (n % RD) * T;
      if (n == 0) {
#pragma unroll
        for (int j = 0; j < APT; ++j)
          if (top_active(j)) cp_async16(r + li(j), w + ((base + li(j)) ^ ((size_t)3 << (LT + LA - 1))));
      } else if (n < count) {
        const V* q = w + (base ^ (act ? (size_t)3 << (__ffs(act) - 1) : (size_t)1 << p.hc_site));
        act &= act - 1;
#pragma unroll
        for (int j = 0; j < APT; ++j) cp_async16(r + li(j), q + li(j));
      }
      cp_async_commit();
    }
  }
  __device__ __forceinline__ void cross_issue(const V* w, unsigned& act) {
    act = bonds_hi;
    const int count = cross_count();
    if constexpr (MSG) {
      if (rank & 1) recv_issue(rank ^ 1, 1, xa[0]);
      else recv_issue(rank ^ 1, 0, xa[0]);
#pragma unroll
      for (int n = 1; n < RD; ++n)
        if (n < count) recv_issue(cross_rank(act), -1, xa[n]);
    } else {
#pragma unroll
      for (int n = 0; n < RD; ++n) cross_copy(w, n, count, act);
    }
  }
  __device__ __forceinline__ void cross_add(const V* w, unsigned act, V (&h)[APT]) {
    const int count = cross_count(), nb1 = 1 + __popc(bonds_hi);
    if constexpr (MSG) {
      auto top = [&](int half) {  // the own amplitudes with the other top bit
        recv_wait(rank ^ 1, half, xa[0]);
#pragma unroll
        for (int j = 0; j < APT / 2; ++j) {
          V& y = h[j + (half ? 0 : APT / 2)];
          y = vfma(hxy, atom_amp(xa[0], j + (half ? APT / 2 : 0)), y);
        }
      };
      if (rank & 1) top(1);
      else top(0);
      auto take = [&](int n, const Atom (&q)[NA]) {
        const R c = (n < nb1) ? hxy : cx;
#pragma unroll
        for (int j = 0; j < APT; ++j) h[j] = vfma(c, atom_amp(q, j), h[j]);
      };
      unsigned a2 = bonds_hi;
#pragma unroll
      for (int n = 1; n < RD; ++n) {
        if (n < count) {
          recv_wait(cross_rank(a2), -1, xa[n]);
          take(n, xa[n]);
        }
      }
      for (int n = RD; n < count; ++n) {
        const int r = cross_rank(act);
        recv_issue(r, -1, xa[0]);
        recv_wait(r, -1, xa[0]);
        take(n, xa[0]);
      }
    }
    if constexpr (!MSG) {
      V x[APT];
#pragma unroll
      for (int j = 0; j < APT; ++j) x[j] = vmake<V>(0, 0);
      for (int n = 0; n < count; ++n) {
        cp_async_wait<RD - 1>();
        const V* r = ring + (n % RD) * T;
        if (n == 0) {
#pragma unroll
          for (int j = 0; j < APT; ++j)
            if (top_active(j)) x[j] = r[li(j)];
        } else if (n < nb1) {
#pragma unroll
          for (int j = 0; j < APT; ++j) x[j] = vadd(x[j], r[li(j)]);
        } else {
#pragma unroll
          for (int j = 0; j < APT; ++j) h[j] = vfma(cx, r[li(j)], h[j]);
        }
        cross_copy(w, n + RD, count, act);
      }
#pragma unroll
      for (int j = 0; j < APT; ++j) h[j] = vfma(hxy, x[j], h[j]);
    }
  }

  __device__ __forceinline__ V* sbasis(int k) const { return sw + k * T; }  // SB: v_k
  __device__ __forceinline__ V* gbasis(int k) const { return (V*)p.basis + (size_t)(k - 1) * D + base; }
  __device__ __forceinline__ V* gw(int k) const { return (V*)p.wbuf + (size_t)(k & 1) * D; }

  __device__ __forceinline__ void fail_nonfinite() {
    if (tid == 0) {
      atomicCAS(p.ctrl + kCtrlStatus, 0, (int)KG_ERR_NONFINITE);
      atomicExch(p.ctrl + kCtrlAbort, 1);
    }
  }

  // Lanczos basis of the slice from wo (||wo|| = nrm): v_k in the basis, alpha_k and b_{k+1} in shared
  // memory, the number of vectors, whether the basis ended early, b_m.  false: aborted.
  __device__ __forceinline__ bool lanczos(int& meff, bool& broke, R& beta_m) {
    const int m = p.m;
    V vp[APT], v[APT], w[APT];
    V* s = sw;  // v_k
#pragma unroll
    for (int j = 0; j < APT; ++j) {
      vp[j] = vmake<V>(0, 0);
      v[j] = vmul(inv, wo[j]);
      s[li(j)] = v[j];
    }
    R alpha = 0, bk = 0, ib = 0;
    float amax = 0.f, bmax = 0.f;
    const float tol = (float)p.bd_tol;
    meff = (sround(nrm) > 0) ? m : 0;
    broke = false;
    beta_m = 0;
    for (int k = 0; k < meff; ++k) {
      const bool last = (k == m - 1);
      sync();  // v_k is in shared memory
      stencil(s, v, w);
      R acc[3] = {0, 0, 0};
#pragma unroll
      for (int j = 0; j < APT; ++j) {
        w[j] = vfma(-bk, vp[j], w[j]);
        acc[0] = fma(v[j].x, w[j].x, fma(v[j].y, w[j].y, acc[0]));
        acc[1] = fma(w[j].x, w[j].x, fma(w[j].y, w[j].y, acc[1]));
        acc[2] = fma(v[j].x, v[j].x, fma(v[j].y, v[j].y, acc[2]));
      }
      post(acc);
      sync();
      S o[kTileSums];
      if (!collect(o)) return false;
      if (!step_scalars(k, last, o, v, w, tol, amax, bmax, alpha, bk, ib, broke)) return false;
      if (last) beta_m = bk;
      if (last || broke) {
        meff = k + 1;
        break;
      }
      s = SB ? sw + (k + 1) * T : sw + ((k + 1) & 1) * T;
#pragma unroll
      for (int j = 0; j < APT; ++j) {
        const V vn = vmul(ib, vfma(-alpha, v[j], w[j]));
        vp[j] = v[j];
        v[j] = vn;
        s[li(j)] = vn;
        if constexpr (!SB) stv(gbasis(k + 1) + li(j), vn);
      }
    }
    return true;
  }
  // The same by the raw vectors (several CTAs, or 16 amplitudes a thread, where the other arrangement's
  // third vector does not fit the registers); src is W_0 in global memory.
  __device__ __forceinline__ bool lanczos_raw(const V* src, int& meff, bool& broke, R& beta_m) {
    const int m = p.m;
    V vp[APT], hp[APT];
#pragma unroll
    for (int j = 0; j < APT; ++j) vp[j] = hp[j] = vmake<V>(0, 0);
    R ap = 0, ib = inv, bk = 0;
    float amax = 0.f, bmax = 0.f;
    const float tol = (float)p.bd_tol;
    meff = (sround(nrm) > 0) ? m : 0;
    broke = false;
    beta_m = 0;
    for (int k = 0; k < meff; ++k) {
      const bool last = (k == m - 1);
      V h[APT];
      const V* wk = (k > 0) ? gw(k) : src;
      unsigned act = 0u;
      stencil(sw + (k & 1) * T, wo, h);
      if constexpr (MSG) {
        cross_issue(wk, act);
        cross_add(wk, act, h);
      }
      if (k > 0) {  // alpha_{k-1}, b_k from the sums of step k - 1
        S o[kTileSums];
        if (!collect(o)) return false;
        if constexpr (MULTI && !MSG) cross_issue(wk, act);
        if (!step_scalars(k - 1, false, o, vp, wo, tol, amax, bmax, ap, bk, ib, broke)) return false;
        if (broke) {
          meff = k;
          if constexpr (MULTI && !MSG) cp_async_wait<0>();
          break;
        }
      } else if constexpr (MULTI && !MSG) {
        cross_issue(wk, act);
      }
      if constexpr (MULTI && !MSG) cross_add(wk, act, h);
      R acc[3] = {0, 0, 0};
      V* sn = sw + ((k + 1) & 1) * T;
      V* vslot = (k > 0) ? gbasis(k) : nullptr;
#pragma unroll
      for (int j = 0; j < APT; ++j) {
        const V v = vmul(ib, vfma(-ap, vp[j], wo[j]));
        const V hv = vmul(ib, vfma(-ap, hp[j], h[j]));
        const V w = vfma(-bk, vp[j], hv);  // b_0 counts as 0: v_{-1} = 0
        acc[0] = fma(v.x, w.x, fma(v.y, w.y, acc[0]));
        acc[1] = fma(w.x, w.x, fma(w.y, w.y, acc[1]));
        acc[2] = fma(v.x, v.x, fma(v.y, v.y, acc[2]));
        vp[j] = v;
        hp[j] = hv;
        wo[j] = w;
        if (!last) {
          sn[li(j)] = w;
          if constexpr (MULTI && !MSG) stv(gw(k + 1) + base + li(j), w);
        }
        if (!MSG && k > 0) stv(vslot + li(j), v);
      }
      if (MSG && !last) send();
      post(acc, !MSG);
      if constexpr (MSG) {
#pragma unroll
        for (int j = 0; j < APT; ++j)
          if (k > 0) stv(vslot + li(j), vp[j]);
      }
      sync();
    }
    if (meff > 0 && !broke) {  // the last step's sums: alpha_{m-1}, b_m of the error indicator
      S o[kTileSums];
      if (!collect(o)) return false;
      bool unused = false;
      if (!step_scalars(m - 1, true, o, vp, wo, tol, amax, bmax, ap, beta_m, ib, unused)) return false;
    }
    return true;
  }

  // One slice, x (own amplitudes in wo) -> exp(-+i dt H_j) x in wo, written to dst.  back: the co-state
  // sweep, whose sums carry Im <dst|Hc|other>.  lob 1: the interior quadrature
  // states of a forward slice go to tint; 2: the sums carry the overlap with the interior states of
  // a backward slice.  On return the new vector's sums are posted (collect gives ||dst||^2 and the
  // overlaps); false: aborted (in every thread alike).
  __device__ __forceinline__ bool slice(bool back, V* dst, const V* src, const V* other, int lob, V* tint) {
    int meff;
    bool broke;
    R beta_m;
    if constexpr (RAW) {
      if (!lanczos_raw(src, meff, broke, beta_m)) return false;
    } else {
      if (!lanczos(meff, broke, beta_m)) return false;
    }
    mark(0);
    // ---- the other vector of the overlap and the newest basis vectors are fetched while the small
    // exponential runs
    V q[APT];
    if (back) load_partner(other, q);
    if (lob) sync();  // thread 0 wrote alpha and b; its warp alone reads them unless lob
    else __syncwarp();
    coefficients(back, meff, broke, beta_m, lob);
    sync();
    mark(4);
    // ---- recombination
    R pgi = 0;
#pragma unroll 1
    for (int a = lob ? 2 : 0; a >= 0; --a) {
      recombine(a, meff, src, wo);
      if (a == 0) break;
      V* t = tint + (size_t)(a - 1) * D;
      if (lob == 1) {
#pragma unroll
        for (int j = 0; j < APT; ++j)
          if (li(j) < D1) stv(t + base + li(j), wo[j]);
      } else {
        V z[APT];
        load_partner(t, z);
        pgi += hc_overlap(wo, z);
      }
    }
    publish(dst);
    R pn = 0;
#pragma unroll
    for (int j = 0; j < APT; ++j) pn = fma(wo[j].x, wo[j].x, fma(wo[j].y, wo[j].y, pn));
    const R vals[3] = {pn, back ? hc_overlap(wo, q) : (R)0, pgi};
    post(vals);
    sync();
    mark(5);
    return true;
  }

  // wo is the next slice's initial vector: into the trajectory (and, RAW, W_0 in shared memory).
  __device__ __forceinline__ void publish(V* dst) {
#pragma unroll
    for (int j = 0; j < APT; ++j) {
      if constexpr (RAW) sw[li(j)] = wo[j];
      if (li(j) < D1) stv(dst + base + li(j), wo[j]);
    }
    send();
  }

  // The amplitudes of vector v that Hc couples to the own ones (Sx: the flipped site; Sz: the same).
  __device__ __forceinline__ void load_partner(const V* v, V (&q)[APT]) const {
    const size_t flip = (p.hc_kind == KG_HC_SX_SITE) ? (size_t)1 << p.hc_site : 0;
#pragma unroll
    for (int j = 0; j < APT; ++j) q[j] = (li(j) < D1) ? ldv(v + ((base + li(j)) ^ flip)) : vmake<V>(0, 0);
  }

  // This thread's share of Im <y|Hc|q> (q already at the partner index for an Sx control).
  __device__ __forceinline__ R hc_overlap(const V (&y)[APT], const V (&q)[APT]) {
    const bool sx = (p.hc_kind == KG_HC_SX_SITE);
    const R amp = (R)p.hc_amp;
    R g = 0;
#pragma unroll
    for (int j = 0; j < APT; ++j) {
      const R w = sx ? (R)0.5 : zdiag(j);
      g = fma(w, fma(y[j].x, q[j].y, -(y[j].y * q[j].x)), g);
    }
    return amp * g;
  }

  // Scalars after step k from its sums o = (<v|W>, ||W||^2, ||v||^2): alpha_k, b_{k+1}, 1/b_{k+1};
  // near an invariant subspace b_{k+1}^2 = ||W_{k+1} - alpha_k v_k||^2 formed explicitly.  broke:
  // b_{k+1} vanishes (Alg. "Lanczos", b_j > 0 with a tolerance).  false: not finite, or aborted.
  __device__ __forceinline__ bool step_scalars(int k, bool last, const S (&o)[kTileSums], const V (&v)[APT],
                                               const V (&w)[APT], float tol,
                                               float& amax, float& bmax, R& alpha, R& beta, R& inv_b, bool& broke) {
    alpha = sround(o[0]);
    S b2 = sb2(o[0], o[1], o[2]);
    sroot(b2, beta, inv_b);
    const float af = fabsf((float)alpha);  // the breakdown test needs no more than FP32
    const bool usual = !scancels(b2, o[1]) && sfinite(o[0]) && sfinite(o[1]) && (float)beta > tol * fmaxf(1.f, fmaxf(amax, af) + bmax);
    if (!usual) {
      if (!sfinite(o[0]) || !sfinite(o[1])) {
        fail_nonfinite();
        return false;
      }
      if (!last && scancels(b2, o[1])) {
        R e[3] = {0, 0, 0};
#pragma unroll
        for (int j = 0; j < APT; ++j) {
          const V d = vfma(-alpha, v[j], w[j]);
          e[0] = fma(d.x, d.x, fma(d.y, d.y, e[0]));
        }
        post(e);
        if constexpr (!MULTI) sync();
        S oe[kTileSums];
        if (!collect(oe)) return false;
        b2 = oe[0];
        sroot(b2, beta, inv_b);
      }
      if (!last) broke = (float)beta <= tol * fmaxf(1.f, fmaxf(amax, af) + bmax);
    }
    amax = fmaxf(amax, af);
    bmax = fmaxf(bmax, (float)beta);
    if (tid == 0) {
      if constexpr (F32) {
        sm.al_ff[k] = make_float2(o[0].hi, o[0].lo);
        sm.b2_ff[k] = make_float2(b2.hi, b2.lo);
      } else {
        sm.al[k] = o[0];
        sm.be[k + 1] = beta;
      }
    }
    return true;
  }

  // Small exponentials: c = exp(-+i t T) e_1 for the slice end (0) and, with lob, the interior
  // quadrature nodes (1, 2), one warp each; times ||x|| for the normalised basis vectors (slot 0 is x).
  __device__ __forceinline__ void coefficients(bool back, int meff, bool broke, R beta_m, int lob) {
    const int lane = tid & 31, warp = tid >> 5;
    const int nc = lob ? 3 : 1;
    for (int a = warp; a < nc; a += NW) {
      R cr = 0, ci = 0;
      float tnorm = 0.f;
      if constexpr (F32) {
        const float2 a2 = (lane < meff) ? sm.al_ff[lane] : make_float2(0.f, 0.f);
        const float2 b2 = (lane >= 1 && lane < meff) ? sm.b2_ff[lane - 1] : make_float2(0.f, 0.f);
        FF fr{0.f, 0.f}, fi{0.f, 0.f};
        // forward exp(-i s T); backward exp(+i (dt - s) T), where dt - s_a = s_b
        const float2 t2 = sm.tau_ff[back && a > 0 ? 3 - a : a];
        const FF t = back ? FF{-t2.x, -t2.y} : FF{t2.x, t2.y};
        if (meff > 0) tridiag_expv_e1_fff(FF{a2.x, a2.y}, ff_sqrt(FF{b2.x, b2.y}), meff, t, 1e-13f, fact, fr, fi, tnorm);
        const FF f = (lane == 0) ? FF{1.f, 0.f} : nrm;
        cr = sround(ff_mul(fr, f));
        ci = sround(ff_mul(fi, f));
        if (lane < meff) {
          sm.coef_re_f[a][lane] = cr;
          sm.coef_im_f[a][lane] = ci;
        }
      } else {
        // FP32 copies for the exponential's norm bound
        if (lane < meff) {
          sm.coef_re_f[a][lane] = (float)sm.al[lane];
          sm.coef_im_f[a][lane] = (lane >= 1) ? (float)sm.be[lane] : 0.f;
        }
        __syncwarp();
        double dr = 0.0, di = 0.0, t = p.dt;
        if (a > 0) t = 0.5 * p.dt * (1.0 + ((a == 1) != back ? -0.4472135954999579 : 0.4472135954999579));  // 1/sqrt(5)
        if (back) t = -t;
        if (meff > 0)
          tridiag_expv_e1(sm.al, sm.be, sm.coef_re_f[a], sm.coef_im_f[a], meff, t, (float)t, 1e-18, dr, di, tnorm);
        const double f = (lane == 0) ? 1.0 : nrm;
        cr = dr * f;
        ci = di * f;
        if (lane < meff) {
          sm.coef_re[a][lane] = cr;
          sm.coef_im[a][lane] = ci;
        }
      }
      if (a == 0 && lane == meff - 1) {
        // a-posteriori indicator ||x|| b_m |c_{m-1}|; where the Taylor series stopped before index
        // m - 1, ||x|| b_m ||tau T||^(m-1)/(m-1)! bounds it
        const float n0 = (float)sround(nrm);
        const float re = (float)cr, im = (float)ci;
        float cm = hypotf(re, im);  // the squares may underflow
        if (lane == 0) cm *= n0;
        if (cm == 0.f) {
          cm = n0;
          for (int i = 1; i < meff; ++i) cm *= tnorm * kInvFF[i].x;
        }
        if (broke) sm.breakdowns += 1;
        else sm.err_max = fmaxf(sm.err_max, (float)beta_m * cm);
      }
    }
  }

  // y = sum_k coef[a]_k (basis vector k), own amplitudes; the small terms (large k) first, so that the
  // sum is rounded at full size only where the largest term, psi's, comes last.
  __device__ __forceinline__ void recombine(int a, int meff, const V* src, V (&y)[APT]) {
    const R* cre = F32 ? (const R*)sm.coef_re_f[a] : (const R*)sm.coef_re[a];
    const R* cim = F32 ? (const R*)sm.coef_im_f[a] : (const R*)sm.coef_im[a];
#pragma unroll
    for (int j = 0; j < APT; ++j) y[j] = vmake<V>(0, 0);
    if constexpr (SB) {
      V x[APT];
#pragma unroll
      for (int j = 0; j < APT; ++j) x[j] = (li(j) < D1) ? ldv(src + base + li(j)) : vmake<V>(0, 0);
      for (int k = meff - 1; k >= 1; --k) {
        const R c0 = cre[k], c1 = cim[k];
        const V* q = sbasis(k);
#pragma unroll
        for (int j = 0; j < APT; ++j) y[j] = vcfma(c0, c1, q[li(j)], y[j]);
      }
      if (meff > 0) {
        const R c0 = cre[0], c1 = cim[0];
#pragma unroll
        for (int j = 0; j < APT; ++j) y[j] = vcfma(c0, c1, x[j], y[j]);
      }
    } else {
      // several basis vectors' loads in flight
      constexpr int KB = (sizeof(V) * APT > 64) ? 2 : 4;
      for (int k0 = meff - 1; k0 >= 0; k0 -= KB) {
        V q[KB][APT];
#pragma unroll
        for (int u = 0; u < KB; ++u) {
          const int k = k0 - u;
          const V* s = (k == 0) ? src + base : gbasis(k);
#pragma unroll
          for (int j = 0; j < APT; ++j) q[u][j] = (k >= 0) ? ldv(s + li(j)) : vmake<V>(0, 0);
        }
#pragma unroll
        for (int u = 0; u < KB; ++u) {
          const int k = k0 - u;
          const R c0 = (k >= 0) ? cre[k] : (R)0, c1 = (k >= 0) ? cim[k] : (R)0;
#pragma unroll
          for (int j = 0; j < APT; ++j) y[j] = vcfma(c0, c1, q[u][j], y[j]);
        }
      }
    }
  }

  // The new vector's sums: its norm (for the next slice) and the overlaps.
  __device__ __forceinline__ bool finish(S& g, S& gi) {
    S o[kTileSums];
    if (!collect(o)) return false;
    if (!sfinite(o[0])) {
      fail_nonfinite();
      return false;
    }
    snorm(o[0], nrm, inv);
    g = o[1];
    gi = o[2];
    return true;
  }

  __device__ __forceinline__ V* fwd_slot(int j) const {  // storage of psi_j (see kg_abi.cu's layout)
    V* traj = (V*)p.traj;
    const int C = p.ckpt;
    if (C == 0) return traj + (size_t)j * D;
    if (j % C == 0) return traj + (size_t)(j / C) * D;
    if (j == p.N) return traj + (size_t)(p.N / C + 1) * D;
    return (V*)p.seg + (size_t)(C - 1 + (j & 1)) * D;
  }

  // The next slice starts from a stored vector.
  __device__ __forceinline__ void load_state(const V* v) {
#pragma unroll
    for (int j = 0; j < APT; ++j) {
      wo[j] = (li(j) < D1) ? ldv(v + base + li(j)) : vmake<V>(0, 0);
      if constexpr (RAW) sw[li(j)] = wo[j];
    }
    send();
  }

  __device__ __forceinline__ bool run() {
    init();
    if constexpr (MSG) {  // before the first reduction: no number of an earlier launch is left
      seq = 0u;
#pragma unroll
      for (int a = 0; a < 2 * NA; ++a) st_atom(atoms(a & 1, rank) + (a >> 1) * NT, 0.f, 0.f, 0.f, 0u);
    }
    S g, gi;
    // ---- psi_0
    {
      double acc[3] = {0.0, 0.0, 0.0};
#pragma unroll
      for (int j = 0; j < APT; ++j) {
        wo[j] = vmake<V>(0, 0);
        if (li(j) < D1) {
          const double2 a = reinterpret_cast<const double2*>(p.psi0)[base + li(j)];
          wo[j] = vmake<V>((R)a.x, (R)a.y);
          acc[0] += (double)wo[j].x * wo[j].x + (double)wo[j].y * wo[j].y;
        }
      }
      publish(fwd_slot(0));
      double o[3];
      if (!sum_fp64(acc, o)) return false;
      if (!isfinite(o[0])) {
        fail_nonfinite();
        return false;
      }
      const double n = sqrt(fmax(o[0], 0.0));
      nrm = sfrom(n, S());
      inv = (n > 0.0) ? (R)(1.0 / n) : (R)0;
      if (F32 && rank == 0 && tid == 0) p.scal[kScInv0] = (double)inv;
    }
    const bool lead = (rank == 0 && tid == 0);
    if (lead) p.nrm[0] = spack(nrm);
    const bool exact = (p.grad_mode == KG_GRAD_EXACT);
    mark(6);
    // The slices in order: the forward sweep, then segment by segment (one segment without
    // checkpoints) the recomputation of psi_{a+1..b-1} and the co-state sweep.  One loop, one copy of
    // the slice's code: three copies miss the instruction cache at every change of direction.
    V* chi[2] = {(V*)p.chi, (V*)p.chi + D};
    const int C = p.ckpt;
    enum { kForward, kRecompute, kBackward };
    int kind = kForward, j = 1, a = 0, b = p.N, cur = 0;
    S nchi = nrm;
    R ichi = inv;
    for (;;) {
      const V* src;
      const V* other = nullptr;
      V* dst;
      if (kind == kForward) {
        src = fwd_slot(j - 1);
        dst = fwd_slot(j);
      } else if (kind == kRecompute) {
        src = seg_slot(a, j - 1);
        dst = (V*)p.seg + (size_t)(j - a - 1) * D;
      } else {
        src = chi[cur];
        dst = chi[cur ^ 1];
        other = (C == 0) ? (V*)p.traj + (size_t)(j - 1) * D : seg_slot(a, j - 1);
      }
      set_control(p.u[j - 1]);
      const bool back = kind == kBackward;
      const int lob = !exact ? 0 : back ? 2 : 1;
      if (!slice(back, dst, src, other, lob, exact ? (V*)p.tint + (size_t)2 * (j - 1) * D : nullptr))
        return false;
      if (!finish(g, gi)) return false;
      // ---- what follows the slice
      if (kind == kForward) {
        if (lead) p.nrm[j] = spack(nrm);
        if (j < p.N) {
          ++j;
          continue;
        }
        if (!turn(lead, chi[0])) return false;
        if (p.grad_mode == KG_GRAD_NONE) break;
        mark(6);
        a = (C > 0) ? (p.N - 1) / C * C : 0;
      } else if (kind == kRecompute) {
        if (j + 1 < b) {
          ++j;
          continue;
        }
        sync();  // every warp is done with W_0 in shared memory
        load_state(chi[cur]);
        nrm = nchi;
        inv = ichi;
        sync();
        kind = kBackward;
        j = b;
        continue;
      } else {
        if (lead) {
          p.G[j - 1] = spack(g);
          if (exact) p.Gi[j - 1] = spack(gi);  // both interior nodes of slice j
        }
        cur ^= 1;
        if (j - 1 > a) {
          --j;
          continue;
        }
        if (a == 0) break;
        b = a;
        a -= C;
      }
      // ---- the next segment (a, b]
      kind = kBackward;
      j = b;
      if (C > 0 && b - a > 1) {
        nchi = nrm;
        ichi = inv;
        sync();
        load_state(seg_slot(a, a));
        nrm = sunpack(__ldcg(p.nrm + a), S());
        inv = (F32 && a == 0) ? (R)__ldcg(p.scal + kScInv0) : sinv(nrm);  // psi_0's was rounded once, from FP64
        sync();
        kind = kRecompute;
        j = a + 1;
      }
    }
    // ---- outputs (rank 0)
    if (rank == 0) {
      sync();
      if (p.grad_mode != KG_GRAD_NONE) {
        const double f = 2.0 * p.dt;
        for (int j = tid; j < p.N; j += NT) {
          const double gl = f * sdouble(sunpack(__ldcg(p.G + j), S())), gr = f * sdouble(sunpack(__ldcg(p.G + j + 1), S()));
          if (exact)  // Gauss-Lobatto weights 1/12, 5/12, 5/12, 1/12
            p.grad[j] = (gl + gr) / 12.0 + 5.0 * (f * sdouble(sunpack(__ldcg(p.Gi + j), S()))) / 12.0;
          else
            p.grad[j] = (p.grad_mode == KG_GRAD_ZEROTH) ? gr : 0.5 * (gl + gr);
        }
      }
      if (tid == 0) {
        p.scal[kScErrMax] = (double)sm.err_max;
        p.scal[kScBreakdowns] = (double)sm.breakdowns;
      }
    }
    return true;
  }

  // psi_j of the segment that starts at checkpoint a.
  __device__ __forceinline__ V* seg_slot(int a, int j) const {
    return (j == a) ? (V*)p.traj + (size_t)(a / p.ckpt) * D : (V*)p.seg + (size_t)(j - 1 - a) * D;
  }

  // The end of the forward sweep: beta = <f|psi_N> (FP64) and F; with a gradient chi_N = beta f (into
  // wo and chi), its norm, and G_N = 2 dt Im <chi_N|Hc|psi_N>.
  __device__ __forceinline__ bool turn(bool lead, V* chi) {
    const double2* f = reinterpret_cast<const double2*>(p.target) + base;
    double acc[3] = {0.0, 0.0, 0.0}, o[3];
#pragma unroll
    for (int j = 0; j < APT; ++j) {
      if (li(j) < D1) {
        const double2 t = f[li(j)];
        const double yr = (double)wo[j].x, yi = (double)wo[j].y;
        acc[0] += t.x * yr + t.y * yi;
        acc[1] += t.x * yi - t.y * yr;
      }
    }
    if (!sum_fp64(acc, o)) return false;
    const double br = o[0], bi = o[1];
    if (lead) {
      p.scal[kScBetaRe] = br;
      p.scal[kScBetaIm] = bi;
      p.scal[kScNormFinal] = sdouble(nrm);
      p.fid[0] = br * br + bi * bi;
    }
    if (p.grad_mode == KG_GRAD_NONE) return true;
    V z[APT];
    load_partner(fwd_slot(p.N), z);
    acc[0] = acc[1] = 0.0;
#pragma unroll
    for (int j = 0; j < APT; ++j) {
      wo[j] = vmake<V>(0, 0);
      if (li(j) < D1) {
        const double2 t = f[li(j)];
        wo[j] = vmake<V>((R)(br * t.x - bi * t.y), (R)(br * t.y + bi * t.x));
        acc[0] += (double)wo[j].x * wo[j].x + (double)wo[j].y * wo[j].y;
      }
    }
    publish(chi);
    const bool sx = (p.hc_kind == KG_HC_SX_SITE);
#pragma unroll
    for (int j = 0; j < APT; ++j) {
      const R w = (R)p.hc_amp * (sx ? (R)0.5 : zdiag(j));
      acc[1] += (double)(w * (wo[j].x * z[j].y - wo[j].y * z[j].x));
    }
    if (!sum_fp64(acc, o)) return false;
    const double n = sqrt(fmax(o[0], 0.0));
    nrm = sfrom(n, S());
    inv = (n > 0.0) ? (R)(1.0 / n) : (R)0;
    if (lead) p.G[p.N] = spack(sfrom(o[1], S()));
    return true;
  }
};

// The control warp of a CTA that is one of several (threads NT .. NT + 31): for every reduction it takes
// the workers' warp partials, makes the CTA's stores visible and posts the CTA's sums with the
// reduction's number, then reads every CTA's message (lane l those of CTAs l, l + 32, ...) until it
// carries that number, adds them up and answers the workers.  Two sets of slots, by the number's
// parity: a CTA posts reduction n + 2 only after every CTA has posted n + 1, so has read n.
template <class V, int NT>
__device__ __forceinline__ void tile_control(const EvalParams& p, TileSmem& sm, int rank, int size) {
  using S = typename Prec<V>::S;
  constexpr bool F32 = Prec<V>::F32;
  constexpr int NW = NT / 32;
  const int lane = threadIdx.x & 31;
  unsigned long long seq = 0;
  for (;;) {
    nbar_sync(kTileBarPost, NT + 32);
    const int cmd = sm.cmd;
    if ((cmd & 3) == kTileCmdExit) return;
    const int par = (cmd >> 2) & 1;
    ++seq;
    ulonglong2* slots = reinterpret_cast<ulonglong2*>(p.red) + (size_t)(seq & 1) * size * kNRed;
    // lane i < 3: the CTA's sum i (FP64 sums of the complex64 path come through the FP64 partials too)
    S c[kTileSums];
    if constexpr (F32) {
      if (cmd & kTileCmdFp64) {
        double d[kTileSums];
        warps_sum3<NW, double>([&](int w, int i) { return sm.red_d[par][w][i]; }, d);
#pragma unroll
        for (int i = 0; i < kTileSums; ++i) c[i] = ff_from_double(d[i]);
      } else {
        warps_sum3<NW, FF>([&](int w, int i) { return FF{sm.red_f[par][w][i], 0.f}; }, c);
      }
    } else {
      warps_sum3<NW, double>([&](int w, int i) { return sm.red_d[par][w][i]; }, c);
    }
    const bool fence = (cmd & kTileCmdFence) != 0;
    if (fence) fence_acq_rel();  // the workers' stores, ordered before this warp by the named barrier
    const bool skip = rank == 0 && ((p.debug_fault == 1 && seq == 1) || (p.debug_fault == 2 && seq == 2));
    ulonglong2* out = slots + rank * kNRed + lane;
    if constexpr (F32) {  // three float-float sums in two messages
      if (lane == 0 && !skip) st_atom(out, c[0].hi, c[0].lo, c[1].hi, (unsigned)seq);
      if (lane == 1 && !skip) st_atom(out, c[1].lo, c[2].hi, c[2].lo, (unsigned)seq);
    } else {
      const double mine = (lane == 0) ? c[0] : (lane == 1) ? c[1] : c[2];
      if (lane < kTileSums && !skip) st_msg(out, (unsigned long long)__double_as_longlong(mine), seq);
    }
    S t[kTileSums] = {S(), S(), S()};
    bool ok = sm.lost == 0;
    unsigned long long t0 = 0;
    unsigned polls = 0;
    using Msg = typename std::conditional<F32, Atom, ulonglong2>::type;
    constexpr int NM = F32 ? 2 : 3;
    auto numbered = [&](const Msg& q) {
      if constexpr (F32) return q.seq == (unsigned)seq;
      else return q.y == seq;
    };
    for (int r = lane; r < size && ok; r += 64) {  // two slots in a round
      Msg q[2][NM];
      unsigned open = (r + 32 < size) ? 3u : 1u;
      const bool two = open == 3u;
      for (;;) {
#pragma unroll
        for (int i = 0; i < 2; ++i) {
          if ((open >> i) & 1u) {
#pragma unroll
            for (int j = 0; j < NM; ++j) {
              if constexpr (F32) q[i][j] = ld_atom(slots + (r + 32 * i) * kNRed + j);
              else q[i][j] = ld_msg(slots + (r + 32 * i) * kNRed + j);
            }
          }
        }
#pragma unroll
        for (int i = 0; i < 2; ++i) {
          bool all = true;
#pragma unroll
          for (int j = 0; j < NM; ++j) all = all && numbered(q[i][j]);
          if (((open >> i) & 1u) && all) open &= ~(1u << i);
        }
        if (!open) break;
        if ((++polls & 31u) == 0u) {
          if (ld_volatile_i32(p.ctrl + kCtrlAbort)) { ok = false; break; }
          const unsigned long long now = globaltimer_ns();
          if (t0 == 0) {
            t0 = now;
          } else if ((long long)(now - t0) > p.wait_limit_ns) {
            atomicCAS(p.ctrl + kCtrlStatus, 0, (int)KG_ERR_TIMEOUT);
            atomicExch(p.ctrl + kCtrlAbort, 1);
            ok = false;
            break;
          }
        }
      }
      if (ok) {
#pragma unroll
        for (int i = 0; i < 2; ++i) {
          if (i == 1 && !two) break;
          if constexpr (F32) {
            const Atom &a = q[i][0], &b = q[i][1];
            t[0] = vx_add(t[0], FF{a.f[0], a.f[1]});
            t[1] = vx_add(t[1], FF{a.f[2], b.f[0]});
            t[2] = vx_add(t[2], FF{b.f[1], b.f[2]});
          } else {
#pragma unroll
            for (int j = 0; j < kTileSums; ++j) t[j] = vx_add(t[j], __longlong_as_double((long long)q[i][j].x));
          }
        }
      }
    }
    ok = __all_sync(0xffffffffu, ok);
    if (fence) fence_acq_rel();  // what the workers read after the barrier was stored before the messages
    const S x = warp_sum3(t[0], t[1], t[2]);
    if (lane < kTileSums) sm.tot[par][lane] = spack(x);
    if (lane == 0) sm.ok = ok ? 1 : 0;
    __syncwarp();
    nbar_arrive(kTileBarGroup, NT + 32);
  }
}

template <class V, int NT, int APT, bool SB, bool MULTI>
__device__ __forceinline__ void tile_cta(const EvalParams& p, TileSmem& sm, V* sw, int rank) {
  using TileT = Tile<V, NT, APT, SB, MULTI>;
  const long long t0 = clock64();
  if (threadIdx.x == 0) {
    sm.err_max = 0.f;
    sm.breakdowns = 0;
    sm.ok = 1;
    sm.lost = 0;
    for (int i = 0; i < 8; ++i) sm.prof_acc[i] = 0;
    sm.prof_last = t0;
  }
  __syncthreads();
  if (MULTI && threadIdx.x >= NT) {
    tile_control<V, NT>(p, sm, rank, (int)gridDim.x);
    return;
  }
  TileT t{p, sm, sw, sw + 2 * TileT::T};
  t.tid = (int)threadIdx.x;
  t.rank = rank;
  t.D = (size_t)1 << p.L;
  t.base = (size_t)rank * TileT::T;
  t.D1 = (int)min((size_t)TileT::T, t.D);
  t.par = 0;
  t.run();
  if constexpr (MULTI) {
    cp_async_wait<0>();  // an abandoned evaluation may have copies under way
    if (threadIdx.x == 0) sm.cmd = kTileCmdExit;
    nbar_arrive(kTileBarPost, NT + 32);
  }
  if (p.prof != nullptr && rank == 0 && threadIdx.x == 0) {
    for (int i = 0; i < 7; ++i) p.prof[i] = sm.prof_acc[i];
    p.prof[7] = clock64() - t0;
  }
}

template <class V, int NT, int APT, bool SB, bool MULTI>
__global__ void __launch_bounds__(MULTI ? NT + 32 : NT, 1) kg_tile_kernel(const __grid_constant__ EvalParams p) {
  extern __shared__ __align__(16) unsigned char tile_dyn[];
  __shared__ TileSmem sm;
  tile_cta<V, NT, APT, SB, MULTI>(p, sm, reinterpret_cast<V*>(tile_dyn), MULTI ? (int)blockIdx.x : 0);
}

// Many problems of one chain length, one CTA each.
template <class V, int NT, int APT, bool SB>
__global__ void __launch_bounds__(NT, 1) kg_tile_list_kernel(const EvalParams* list) {
  extern __shared__ __align__(16) unsigned char tile_dyn[];
  __shared__ TileSmem sm;
  __shared__ EvalParams p;
  if (threadIdx.x == 0) p = list[blockIdx.x];
  __syncthreads();
  tile_cta<V, NT, APT, SB, false>(p, sm, reinterpret_cast<V*>(tile_dyn), 0);
}

// ---------------------------------------------------------------- launch selection
struct TileKernel {
  const void* fn = nullptr;    // one problem (EvalParams by value)
  const void* list = nullptr;  // complex64: a list of problems
  int threads = 0, tile_bits = 0;
  size_t smem = 0;      // of this call (a basis in shared memory grows with m)
  size_t smem_max = 0;  // of any call
  int ctas = 1;
};

// A kernel's limit is shared by the whole process: every call sets the same one, so that none can lower
// it between another host thread's setting and launch.
cudaError_t set_smem_limit(const void* fn, const TileKernel& k) {
  return cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)k.smem_max);
}

// Basis in shared memory up to this size.
constexpr size_t kTileSmemBasis = 100 * 1024;

template <class V, int NT, int APT, bool SB>
TileKernel tile_choice(size_t smem) {
  TileKernel k{reinterpret_cast<const void*>(&kg_tile_kernel<V, NT, APT, SB, false>), nullptr, NT,
               __builtin_ctz(NT * APT), smem, SB ? kTileSmemBasis : smem};
  if constexpr (sizeof(V) == 8) k.list = reinterpret_cast<const void*>(&kg_tile_list_kernel<V, NT, APT, SB>);
  return k;
}
template <class V, int NT, int APT>
TileKernel tile_single(int m) {
  constexpr size_t vec = (size_t)NT * APT * sizeof(V);
  if constexpr (APT < 16 && kMaxM * vec <= kTileSmemBasis) {  // whatever m
    return tile_choice<V, NT, APT, true>(m * vec);
  } else {
    if constexpr (APT < 16)
      if (m * vec <= kTileSmemBasis) return tile_choice<V, NT, APT, true>(m * vec);
    return tile_choice<V, NT, APT, false>(2 * vec);
  }
}

// One of several CTAs: two W_k buffers and (complex128) the ring of partner blocks.
template <class V, int NT, int APT>
TileKernel tile_multi(int L) {
  using TileT = Tile<V, NT, APT, false, true>;
  const int t = __builtin_ctz(NT * APT);
  const size_t smem = (size_t)(2 + (sizeof(V) == 16 ? TileT::RD : 0)) * TileT::T * sizeof(V);
  return {reinterpret_cast<const void*>(&kg_tile_kernel<V, NT, APT, false, true>), nullptr, NT + 32, t, smem, smem,
          1 << (L - t)};
}

// Threads x amplitudes by chain length.  More threads shorten every thread's chain of shared-memory
// loads, fewer make the block's sums cheaper; measured (us per slice, m = 16, complex64):
//   L = 7: 64 x 2 12.7, 32 x 4 12.3;  8: 128 x 2 14.1, 32 x 8 15.3, 64 x 4 15.7;  9: 256 x 2 17.3, 128 x 4
//   17.7, 64 x 8 18.5;  10: 128 x 8 22.2, 256 x 4 22.6;  11: 256 x 8 29.7, 512 x 4 34.8;
//   12: 256 x 16 (raw vectors) 47.7, 512 x 8 61.0 (128 registers), 4 CTAs of 128 x 8 44.7.
// (With three sums by one butterfly since: 8 11.3, 10 20.2, 11 27.3, 12 45.0.)  On several CTAs a step
// costs 2.3 (8 CTAs) to 5.3 us (128), nearly all of it the exchange, so the tiles are as large as the
// registers let them be cheap:
//   13: 128 x 8 40.0;  14: 45.7;  15: 56.9;  16: 59.4;  17: 128 x 8 68.4, 256 x 8 81.4;  18: 256 x 8 89.5.
// At L = 19 the resident loop is the faster one (m = 20: 154.5 us a slice; 128 CTAs of 512 x 8 198.1).
// The kernels that ran these chains before took 100 (L = 5) to 148 us (L = 11), 77 us (L = 12) and, two
// 4096-amplitude tiles per CTA, 128 (L = 13) to 164 us (L = 18).
// complex128 is bound by the FP64 units, one quarter in each quarter of the SM: one warp per quarter
// as soon as there are amplitudes for it, and as many CTAs as there are SMs (us per slice, m = 16):
//   L = 8: 128 x 2 76, 64 x 4 113, 256 x 1 91;  9: 4 CTAs of 128 x 1 76, 2 of 128 x 2 88, one CTA 125;
//   10: 8 CTAs 79, 4 92, one CTA 222;  12: 32 CTAs 100, 16 111, 8 149;  14: 128 CTAs 123, 64 127;
//   15: 128 x 2 146, 256 x 1 162;  16: 128 x 4 180, 256 x 2 219, 64 CTAs 299;  17: 256 x 4 313, 128 x 8 328;
//   18: 256 x 8 588.
// The streaming kernel takes 281 (L = 5) to 496 us (L = 10) for these, 776 at L = 16 and 833 at L = 18.
TileKernel pick_tile(int prec, int L, int m) {
  if (prec == KG_PREC_C64_F64REC) {
    if (L <= 5) return tile_single<float2, 32, 1>(m);
    if (L == 6) return tile_single<float2, 32, 2>(m);
    if (L == 7) return tile_single<float2, 64, 2>(m);
    if (L == 8) return tile_single<float2, 128, 2>(m);
    if (L == 9) return tile_single<float2, 256, 2>(m);
    if (L == 10) return tile_single<float2, 128, 8>(m);
    if (L == 11) return tile_single<float2, 256, 8>(m);
    if (L == 12) return tile_single<float2, 256, 16>(m);
    if (L <= 17) return tile_multi<float2, 128, 8>(L);
    if (L == 18) return tile_multi<float2, 256, 8>(L);
  }
  if (prec == KG_PREC_C128) {
    if (L <= 5) return tile_single<double2, 32, 1>(m);
    if (L == 6) return tile_single<double2, 64, 1>(m);
    if (L == 7) return tile_single<double2, 128, 1>(m);
    if (L == 8) return tile_single<double2, 128, 2>(m);
    if (L <= 14) return tile_multi<double2, 128, 1>(L);
    if (L == 15) return tile_multi<double2, 128, 2>(L);
    if (L == 16) return tile_multi<double2, 128, 4>(L);
    if (L == 17) return tile_multi<double2, 256, 4>(L);
    if (L == 18) return tile_multi<double2, 256, 8>(L);
  }
  return {};
}

}  // namespace

bool tile_kernel_covers(int prec, int L) {
  const TileKernel k = pick_tile(prec, L, 1);
  if (!k.fn || k.ctas == 1) return k.fn != nullptr;
  // the CTAs of a group wait for one another: all of them have to be resident at once
  int per_sm = 0, dev = 0, sms = 0;
  if (set_smem_limit(k.fn, k) != cudaSuccess ||
      cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k.fn, k.threads, k.smem) != cudaSuccess ||
      cudaGetDevice(&dev) != cudaSuccess ||
      cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess)
    return false;
  return per_sm * sms >= k.ctas;
}
int tile_kernel_threads(int prec, int L) { return pick_tile(prec, L, 1).threads; }
int tile_kernel_bits(int prec, int L) { return L < 5 ? L : pick_tile(prec, L, 1).tile_bits; }
int tile_kernel_ctas(int prec, int L) { return pick_tile(prec, L, 1).ctas; }
size_t tile_kernel_clear_bytes(int prec, int L) {
  const int n = pick_tile(prec, L, 1).ctas;
  return n > 1 ? (size_t)2 * n * kNRed * sizeof(ulonglong2) : 0;
}

cudaError_t launch_tile_kernel(int prec, const EvalParams& p, cudaStream_t stream) {
  const TileKernel k = pick_tile(prec, p.L, p.m);
  if (!k.fn) return cudaErrorInvalidValue;
  cudaError_t e = set_smem_limit(k.fn, k);
  if (e != cudaSuccess) return e;
  void* args[] = {const_cast<EvalParams*>(&p)};
  if (k.ctas > 1) return cudaLaunchCooperativeKernel(k.fn, dim3(k.ctas), dim3(k.threads), args, k.smem, stream);
  return cudaLaunchKernel(k.fn, dim3(1), dim3(k.threads), args, k.smem, stream);
}

cudaError_t launch_tile_list(int L, int m, const EvalParams* list, int n, cudaStream_t stream) {
  const TileKernel k = pick_tile(KG_PREC_C64_F64REC, L, m);
  if (!k.list) return cudaErrorInvalidValue;
  cudaError_t e = set_smem_limit(k.list, k);
  if (e != cudaSuccess) return e;
  void* args[] = {const_cast<EvalParams**>(&list)};
  return cudaLaunchKernel(k.list, dim3(n), dim3(k.threads), args, k.smem, stream);
}

}  // namespace kg
