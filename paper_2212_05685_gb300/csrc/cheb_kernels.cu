// Block Chebyshev recursion of the KPM (App. B, Eq. alpha) on slabs of unit
// start vectors, as a fused complex stencil SpMM:
//
//   V_1 = h~ V_0,   V_{m+1} = 2 h~ V_m - V_{m-1},   V_0 = [e_{s0} ... e_{s0+b-1}]
//
// with the moment sums acc[J][s] += a_m V_m[K_s(J), J] over the nine local
// rows K_s(J) of every column (and the grand-potential series on the diagonal)
// fused into the step that reads V_m (Eqs. rho_KPM, F_KPM with unit r).
// Slab column c holds the unit vector of row J = (s0 + c) << js: js = 0 all
// D columns, js = 1 only the columns (j, up) of the particle-hole half pass;
// or (probing, App. B) the vector r_{s0+c} of colour s0 + c, whose entries are
// the phases xi_K on the rows of that colour; then every row J is a source
// whose column estimate conj(xi_J) F_M(h~) r_colour(J) is summed.
//
// Layout: V is row-major, V[K][c] with K = 2 i + alpha the Nambu row and c the
// column inside the slab; the row stride ldv is the slab width rounded up to
// the CTA's column chunk.  FP64 stores interleaved complex (re, im);
// double-float (KPM_DF64) stores (re_hi, im_hi, re_lo, im_lo), each real the
// unevaluated FP32 sum hi + lo, so that a packed f32x2 operation works on both, and runs the FP64 kernel's structure with
// double-float arithmetic.  FP32 stores each column pair (2p, 2p+1) as
// (re_2p, re_2p+1, im_2p, im_2p+1) so that one packed f32x2 FMA advances two
// columns.  h~ is a 13-point stencil per row (diagonal, eight hops, four
// pairings), read from a per-site table of kCoef complex 2h~ entries.
//
// Passes run the march kernel (cheb_march.cuh).  The one-step kernels of this file serve
// FP64 and double-float probing, and slabs narrower than the march kernel's chunk
// (the allocation-free call): each CTA owns a chunk of CB columns and a band
// of lattice rows y0..y1-1 and marches along y keeping lattice rows y-1, y, y+1
// of V_m (all Nx sites, both Nambu components, CB columns) in shared memory, the
// next rows and coefficient rows in flight by cp.async, so every V_m element is
// read from global memory once per CTA while serving the 13 rows that need it;
// V_{m-1} is read ahead and V_{m+1} written in place.
// No tensor cores: the stencil is sparse, not a dense contraction.
#include <cooperative_groups.h>
#include <cuda.h>

#include <string.h>

#include <algorithm>
#include <type_traits>
#include <utility>
#include <vector>

#include "kpm_internal.cuh"

namespace kpm {
namespace {

// local rows of a unit column J = 2 j + beta (slot s): site j + (dx, dy),
// Nambu component beta, or 1 - beta for the pairing slots 5..8; slot 9
// repeats the diagonal for the grand-potential series.
__constant__ int kSlotDx[kSlots] = {0, 1, 0, 1, 1, 1, 0, -1, 0, 0};
__constant__ int kSlotDy[kSlots] = {0, 0, 1, 1, -1, 0, 1, 0, -1, 0};
__constant__ int kSlotFlip[kSlots] = {0, 0, 0, 0, 0, 1, 1, 1, 1, 0};

template <typename Real>
struct CT;
template <>
struct CT<double> {
  using C = double2;
  using V = double2;
  static constexpr int VW = 1;
};

__device__ __forceinline__ void cmac(double2& a, double2 c, double2 v) {
  a.x = fma(c.x, v.x, a.x);
  a.x = fma(-c.y, v.y, a.x);
  a.y = fma(c.x, v.y, a.y);
  a.y = fma(c.y, v.x, a.y);
}
__device__ __forceinline__ void rmac(double2& a, double d, double2 v) {
  a.x = fma(d, v.x, a.x);
  a.y = fma(d, v.y, a.y);
}
__device__ __forceinline__ double2 vneg(double2 v) { return make_double2(-v.x, -v.y); }
__device__ __forceinline__ double2 vscale(double2 v, double s) { return make_double2(s * v.x, s * v.y); }
template <typename V>
__device__ __forceinline__ V vzero();
template <>
__device__ __forceinline__ double2 vzero<double2>() { return make_double2(0.0, 0.0); }
__device__ __forceinline__ double2 vhalf(double2 v) { return vscale(v, 0.5); }
__device__ __forceinline__ void vfinish(double2&) {}
// the two real diagonals packed in table entry 0, and an element as FP64
__device__ __forceinline__ double diag0(double2 d) { return d.x; }
__device__ __forceinline__ double diag1(double2 d) { return d.y; }
__device__ __forceinline__ double cre(double2 v) { return v.x; }
__device__ __forceinline__ double cim(double2 v) { return v.y; }

// Double-float (KPM_DF64): every real is the unevaluated sum hi + lo of two
// FP32 numbers, about 48 significant bits, so the FP64-accurate recursion runs
// on the FP32 pipes.  A complex element of a vector is float4 (re_hi, im_hi, re_lo,
// im_lo), of the table (re_hi, re_lo, im_hi, im_lo); table entry 0 holds the two real diagonals as (d0_hi, d0_lo, d1_hi, d1_lo).
// Products use the exact FMA residual of hi * hi (p + e = xh yh exactly) plus
// the cross terms; sums use Knuth's two-sum, whose error term is exact for any
// ordering of the operands; an accumulator is renormalised once per output.
struct DF {};
template <>
struct CT<DF> {
  using C = float4;
  using V = float4;
  static constexpr int VW = 1;
};
__device__ __forceinline__ void two_sum(float a, float b, float& s, float& e) {
  s = __fadd_rn(a, b);
  const float bb = __fsub_rn(s, a);
  e = __fadd_rn(__fsub_rn(a, __fsub_rn(s, bb)), __fsub_rn(b, bb));
}
// (h, l) += (xh + xl)(yh + yl), dropping xl yl (below 2^-48 of the product)
__device__ __forceinline__ void df_mac(float& h, float& l, float xh, float xl, float yh, float yl) {
  const float p = __fmul_rn(xh, yh);
  float e = __fmaf_rn(xh, yh, -p);
  e = __fmaf_rn(xh, yl, e);
  e = __fmaf_rn(xl, yh, e);
  float s, t;
  two_sum(h, p, s, t);
  h = s;
  l = __fadd_rn(l, __fadd_rn(t, e));
}
__device__ __forceinline__ void cmac(float4& a, float4 c, float4 v) {
  df_mac(a.x, a.z, c.x, c.y, v.x, v.z);
  df_mac(a.x, a.z, -c.z, -c.w, v.y, v.w);
  df_mac(a.y, a.w, c.x, c.y, v.y, v.w);
  df_mac(a.y, a.w, c.z, c.w, v.x, v.z);
}
__device__ __forceinline__ void rmac(float4& a, float2 d, float4 v) {
  df_mac(a.x, a.z, d.x, d.y, v.x, v.z);
  df_mac(a.y, a.w, d.x, d.y, v.y, v.w);
}
__device__ __forceinline__ float4 vneg(float4 v) { return make_float4(-v.x, -v.y, -v.z, -v.w); }
__device__ __forceinline__ float4 vhalf(float4 v) { return make_float4(0.5f * v.x, 0.5f * v.y, 0.5f * v.z, 0.5f * v.w); }
template <>
__device__ __forceinline__ float4 vzero<float4>() { return make_float4(0.f, 0.f, 0.f, 0.f); }
__device__ __forceinline__ void vfinish(float4& v) {
  float h, l;
  two_sum(v.x, v.z, h, l);
  v.x = h;
  v.z = l;
  two_sum(v.y, v.w, h, l);
  v.y = h;
  v.w = l;
}
__device__ __forceinline__ float2 diag0(float4 d) { return make_float2(d.x, d.y); }
__device__ __forceinline__ float2 diag1(float4 d) { return make_float2(d.z, d.w); }
__device__ __forceinline__ double cre(float4 v) { return (double)v.x + (double)v.z; }
__device__ __forceinline__ double cim(float4 v) { return (double)v.y + (double)v.w; }
// FP64 value as hi + lo (the rounding residual of hi is exact in FP64)
__device__ __forceinline__ float2 df_split(double x) {
  const float h = __double2float_rn(x);
  return make_float2(h, __double2float_rn(x - (double)h));
}

__device__ __forceinline__ void cp_async16(void* smem, const void* gmem) {
  const unsigned s = (unsigned)__cvta_generic_to_shared(smem);
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(s), "l"(gmem) : "memory");
}
__device__ __forceinline__ void cp_commit() { asm volatile("cp.async.commit_group;\n" ::: "memory"); }
__device__ __forceinline__ void cp_wait_1() { asm volatile("cp.async.wait_group 1;\n" ::: "memory"); }
__device__ __forceinline__ void cp_wait_0() { asm volatile("cp.async.wait_group 0;\n" ::: "memory"); }

__device__ __forceinline__ int wrapi(int v, int n) {
  v %= n;
  return v < 0 ? v + n : v;
}

// Probing vectors (App. B): colour of Nambu row K = 2 i + alpha, i = (x, y),
// alpha + 2 ((x mod p) + p (y mod p)); phase xi_K = exp(2 pi i u_K) with u_K
// from the counter-based generator SplitMix64 (Steele, Lea and Flood 2014) at
// counter seed * 2^32 + K.
__device__ __forceinline__ uint64_t splitmix64(uint64_t x) {
  x += 0x9E3779B97F4A7C15ull;
  x = (x ^ (x >> 30)) * 0xBF58476D1CE4E5B9ull;
  x = (x ^ (x >> 27)) * 0x94D049BB133111EBull;
  return x ^ (x >> 31);
}
__device__ __forceinline__ double2 probe_xi(uint32_t seed, int64_t K) {
  const double u = (double)(splitmix64(((uint64_t)seed << 32) + (uint64_t)K) >> 11) * 0x1.0p-53;
  double sn, cs;
  sincospi(2.0 * u, &sn, &cs);
  return make_double2(cs, sn);
}
__device__ __forceinline__ int probe_colour(int64_t K, int nx, int p) {
  const int64_t i = K >> 1;
  const int x = (int)(i % nx), y = (int)(i / nx);
  return (int)(K & 1) + 2 * ((x % p) + p * (y % p));
}

// Moment-sum items of lattice row y for the chunk's columns [cb0, cb0 + CB):
// unit vectors: item t = c * kSlots + s over the chunk's columns; probing:
// the row's colours are 2 p (y mod p) + q, q = 2 (x mod p) + alpha in
// [0, 2 p), so the chunk's colours that occur in the row form the range
// [lo, lo + nq) and each has nx / p sources x = q / 2 + p k; item t =
// ((k * nq) + qi) * kSlots + s.  source_item returns false when the item has
// no source here; else the source row J, its chunk column c, the slot s and
// the weight conj(xi_J) (1 for unit vectors).
struct SourceRange {
  int lo, nq;  // probing: first colour and number of the chunk's colours in the row
};
__device__ __forceinline__ int source_items(const ColMap& cm, int nx, int y, int64_t cb0, int CB, SourceRange& sr) {
  if (!cm.probe_p) return CB * kSlots;
  const int p = cm.probe_p;
  const int64_t c0 = cm.s0 + cb0;
  const int64_t base = 2 * (int64_t)p * (y % p);
  const int64_t lo = c0 > base ? c0 : base;
  const int64_t hi = min(c0 + CB, base + 2 * p);
  sr.lo = (int)lo;
  sr.nq = hi > lo ? (int)(hi - lo) : 0;
  return sr.nq * (nx / p) * kSlots;
}
__device__ __forceinline__ bool source_item(const ColMap& cm, const SourceRange& sr, int t, int y, int nx, int64_t D,
                                            int64_t cb0, int CB, int64_t& J, int& c, int& s, double2& wgt) {
  s = t % kSlots;
  const int r = t / kSlots;
  if (cm.probe_p) {
    const int p = cm.probe_p;
    const int qi = r % sr.nq, k = r / sr.nq;
    const int colour = sr.lo + qi;
    const int q = colour - 2 * p * (y % p);
    J = 2 * ((int64_t)y * nx + (q >> 1) + p * k) + (q & 1);
    c = (int)(colour - cm.s0 - cb0);
    wgt = cm.xi[J];
    return true;
  }
  const int64_t col = cm.s0 + cb0 + r;
  if (col >= (D >> cm.js)) return false;
  J = col << cm.js;
  if ((J >> 1) / nx != y) return false;
  c = r;
  wgt = make_double2(1.0, 0.0);
  return true;
}
// acc += coef w v (complex w, v); one explicit FMA per component, so that the
// unit-vector form below (w = 1: the product is v exactly) rounds identically
__device__ __forceinline__ void acc_add(double2* a, double coef, double2 w, double vr, double vi) {
  a->x = __fma_rn(coef, w.x * vr - w.y * vi, a->x);
  a->y = __fma_rn(coef, w.x * vi + w.y * vr, a->y);
}
__device__ __forceinline__ void acc_add_unit(double2* a, double coef, double vr, double vi) {
  a->x = __fma_rn(coef, vr, a->x);
  a->y = __fma_rn(coef, vi, a->y);
}
// diagonal moment [T_m(h~)]_JJ (its estimate for probing) into the record
__device__ __forceinline__ void record_diag(const ColMap& cm, int64_t D, int m, int64_t J, double2 w, double vr,
                                            double vi) {
  cm.rec[(int64_t)m * D + (J & 1) * (D >> 1) + (J >> 1)] = w.x * vr - w.y * vi;
}

// one lattice row of V (2 nx Nambu rows x CB columns) into shared memory
template <typename C, int CB>
__device__ __forceinline__ void stage_row(C* dst, const C* __restrict__ V, int ly, int nx, int64_t ldv,
                                          int64_t cb0) {
  constexpr int per_row = CB * (int)sizeof(C) / 16;
  const int total = 2 * nx * per_row;
  const C* base = V + (int64_t)(2 * nx) * ly * ldv + cb0;
  for (int t = threadIdx.x; t < total; t += blockDim.x) {
    const int r = t / per_row, c = t - r * per_row;
    cp_async16(reinterpret_cast<char*>(dst + r * CB) + 16 * c,
               reinterpret_cast<const char*>(base + (int64_t)r * ldv) + 16 * c);
  }
}

// the 2h~ entries of one lattice row (nx sites x kCoef complex, contiguous)
template <typename C>
__device__ __forceinline__ void stage_coef(C* dst, const C* __restrict__ table, int ly, int nx) {
  const int chunks = nx * kCoef * (int)sizeof(C) / 16;
  const char* src = reinterpret_cast<const char*>(table + (int64_t)ly * nx * kCoef);
  char* d = reinterpret_cast<char*>(dst);
  for (int t = threadIdx.x; t < chunks; t += blockDim.x) cp_async16(d + 16 * t, src + 16 * t);
}

template <typename Real, int CB, int MODE>
__global__ void __launch_bounds__(512, 1)
    cheb_step_kernel(int nx, int ny, int64_t D, int64_t ldv, int ylen, const typename CT<Real>::C* __restrict__ table,
                     const typename CT<Real>::C* __restrict__ Vcur, const typename CT<Real>::C* Vprev,
                     typename CT<Real>::C* Vout, ColMap cmap, double2* __restrict__ acc,
                     const double* __restrict__ am, const double* __restrict__ ao, int m) {
  using C = typename CT<Real>::C;
  using V = typename CT<Real>::V;
  constexpr int VW = CT<Real>::VW;
  constexpr int NV = CB / VW;  // vectors per Nambu row of the chunk

  // shared memory: V_m window [4][2 nx][CB], V_{m-1} rows [2][2 nx][CB]
  // (step mode only), 2h~ rows [2][nx][kCoef]
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int rowsz = 2 * nx * CB;
  C* win = reinterpret_cast<C*>(smem_raw);
  C* prev = win + 4 * rowsz;
  C* coef = prev + (MODE == 1 ? 2 * rowsz : 0);

  const int64_t cb0 = (int64_t)blockIdx.y * CB;
  const int y0 = blockIdx.x * ylen;
  const int y1 = min(ny, y0 + ylen);
  const int nrow = y1 - y0;

  // prologue: V_m rows y0-1, y0, y0+1, V_{m-1} row y0, coefficients of y0;
  // then V_m row y0+2, V_{m-1} row y0+1, coefficients of y0+1
  for (int q = 0; q < 3; ++q) stage_row<C, CB>(win + q * rowsz, Vcur, wrapi(y0 - 1 + q, ny), nx, ldv, cb0);
  if (MODE == 1) stage_row<C, CB>(prev, Vprev, y0, nx, ldv, cb0);
  stage_coef<C>(coef, table, y0, nx);
  cp_commit();
  if (nrow >= 2) {
    stage_row<C, CB>(win + 3 * rowsz, Vcur, wrapi(y0 + 2, ny), nx, ldv, cb0);
    if (MODE == 1) stage_row<C, CB>(prev + rowsz, Vprev, y0 + 1, nx, ldv, cb0);
    stage_coef<C>(coef + nx * kCoef, table, y0 + 1, nx);
  }
  cp_commit();

  for (int q = 0; q < nrow; ++q) {
    const int y = y0 + q;
    cp_wait_1();
    __syncthreads();
    const C* wm = win + (q & 3) * rowsz;        // lattice row y - 1
    const C* w0 = win + ((q + 1) & 3) * rowsz;  // y
    const C* wp = win + ((q + 2) & 3) * rowsz;  // y + 1
    const C* pv = prev + (q & 1) * rowsz;       // V_{m-1}, row y
    const C* cf_row = coef + (q & 1) * nx * kCoef;

    for (int t = threadIdx.x; t < nx * NV; t += blockDim.x) {
      const int x = t / NV, v = t - x * NV;
      const int xr = x + 1 == nx ? 0 : x + 1;
      const int xl = x == 0 ? nx - 1 : x - 1;
      const int64_t K0 = 2 * ((int64_t)y * nx + x);
      const int64_t g0 = K0 * ldv + cb0 + v * VW;
#define KPM_LD(W, XX, AL) (*reinterpret_cast<const V*>((W) + (2 * (XX) + (AL)) * CB + v * VW))
      V a0, a1;
      if (MODE == 1) {
        a0 = vneg(KPM_LD(pv, x, 0));
        a1 = vneg(KPM_LD(pv, x, 1));
      } else {
        a0 = vzero<V>();
        a1 = vzero<V>();
      }
      const C* cf = cf_row + x * kCoef;
      {
        const C d = cf[0];
        rmac(a0, diag0(d), KPM_LD(w0, x, 0));
        rmac(a1, diag1(d), KPM_LD(w0, x, 1));
      }
      // neighbours k = 1..8: (+1,0) (-1,0) (0,+1) (0,-1) (+1,+1) (-1,-1) (+1,-1) (-1,+1)
      const C* wk[8] = {w0, w0, wp, wm, wp, wm, wm, wp};
      const int xk[8] = {xr, xl, x, x, xr, xl, xr, xl};
#pragma unroll
      for (int k = 0; k < 8; ++k) {
        const V u0 = KPM_LD(wk[k], xk[k], 0);
        const V u1 = KPM_LD(wk[k], xk[k], 1);
        cmac(a0, cf[1 + k], u0);
        cmac(a1, cf[9 + k], u1);
        if (k < 4) {
          cmac(a0, cf[17 + k], u1);
          cmac(a1, cf[21 + k], u0);
        }
      }
#undef KPM_LD
      if (MODE == 0) {
        a0 = vhalf(a0);
        a1 = vhalf(a1);
      }
      vfinish(a0);
      vfinish(a1);
      *reinterpret_cast<V*>(Vout + g0) = a0;
      *reinterpret_cast<V*>(Vout + g0 + ldv) = a1;
    }

    if (MODE == 1 && acc != nullptr) {
      // moment sums of the columns whose own site lies in lattice row y
      const double cm = am[m], co = ao[m];
      SourceRange sr;
      const int items = source_items(cmap, nx, y, cb0, CB, sr);
      for (int t = threadIdx.x; t < items; t += blockDim.x) {
        int64_t J;
        int c, s;
        double2 wgt;
        if (!source_item(cmap, sr, t, y, nx, D, cb0, CB, J, c, s, wgt)) continue;
        const int64_t j = J >> 1;
        const int beta = (int)(J & 1);
        const int xs = wrapi((int)(j % nx) + kSlotDx[s], nx);
        const int dy = kSlotDy[s];
        const C* w = dy < 0 ? wm : (dy > 0 ? wp : w0);
        const int al = kSlotFlip[s] ? 1 - beta : beta;
        const C val = w[(2 * xs + al) * CB + c];
        acc_add(acc + J * kSlots + s, s == kSlots - 1 ? co : cm, wgt, cre(val), cim(val));
        if (s == 0 && cmap.rec) record_diag(cmap, D, m, J, wgt, cre(val), cim(val));
      }
    }
    __syncthreads();
    // refill: V_m row y+3 into the buffer of y-1, V_{m-1} row y+2 and
    // coefficients of y+2 into the buffers of row y
    if (y + 3 <= y1) stage_row<C, CB>(win + (q & 3) * rowsz, Vcur, wrapi(y + 3, ny), nx, ldv, cb0);
    if (y + 2 < y1) {
      if (MODE == 1) stage_row<C, CB>(prev + (q & 1) * rowsz, Vprev, y + 2, nx, ldv, cb0);
      stage_coef<C>(coef + (q & 1) * nx * kCoef, table, y + 2, nx);
    }
    cp_commit();
  }
  cp_wait_0();
}

// ------------------------------------------------------------------ FP32 path
typedef unsigned long long u64;
__device__ __forceinline__ u64 f2fma(u64 a, u64 b, u64 c) {
  u64 d;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
  return d;
}
__device__ __forceinline__ u64 f2add(u64 a, u64 b) {
  u64 d;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
  return d;
}
__device__ __forceinline__ u64 f2sub(u64 a, u64 b) {
  u64 d;
  asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
  return d;
}
__device__ __forceinline__ u64 f2mul(u64 a, u64 b) {
  u64 d;
  asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
  return d;
}

// value of column c in an FP32 pair-split row segment
__device__ __forceinline__ float2 pair_elem(const float4* seg, int c) {
  const float4 q = seg[c >> 1];
  return (c & 1) ? make_float2(q.y, q.w) : make_float2(q.x, q.z);
}

// Accumulators of one output row for two columns: P = sum Re(c) v, Q = sum Im(c) v
// (each a (re, im) pair of f32x2); the row value is (P.re - Q.im, P.im + Q.re).
struct Acc2 {
  u64 pr, pi, qr, qi;
};

__device__ __forceinline__ u64 dup2(float a) {
  u64 d;
  asm("mov.b64 %0, {%1, %1};" : "=l"(d) : "f"(a));
  return d;
}
__device__ __forceinline__ void acc_term(Acc2& a, float2 c, ulonglong2 u) {
  const u64 cr = dup2(c.x), ci = dup2(c.y);
  a.pr = f2fma(cr, u.x, a.pr);
  a.pi = f2fma(cr, u.y, a.pi);
  a.qr = f2fma(ci, u.x, a.qr);
  a.qi = f2fma(ci, u.y, a.qi);
}

// 2h~ applied to site x of lattice row y for one column pair, both Nambu
// rows: wm, w0, wp are lattice rows y-1, y, y+1 of a pair-split V in shared
// memory ([nx][2][NV] float4, already offset by the thread's pair), cf_row the
// row's 2h~ entries.  Returns the two output rows as (re pair, im pair).
template <int NV>
__device__ __forceinline__ void stencil_site(const float4* wm, const float4* w0, const float4* wp,
                                             const float2* cf_row, int x, int nx, ulonglong2& o0, ulonglong2& o1) {
  constexpr int RS = 2 * NV;
  const int xr = x + 1 == nx ? 0 : x + 1;
  const int xl = x == 0 ? nx - 1 : x - 1;
  const float2* cf = cf_row + x * kCoef;
#define KPM_L(W, XX, AL) \
  (*reinterpret_cast<const ulonglong2*>((W) + (XX) * RS + (AL) * NV))
  Acc2 a0 = {0ull, 0ull, 0ull, 0ull}, a1 = {0ull, 0ull, 0ull, 0ull};
  {
    const float2 d = cf[0];  // (d0, d1): real diagonals of the two Nambu rows
    const ulonglong2 u0 = KPM_L(w0, x, 0), u1 = KPM_L(w0, x, 1);
    const u64 d0 = dup2(d.x), d1 = dup2(d.y);
    a0.pr = f2fma(d0, u0.x, a0.pr);
    a0.pi = f2fma(d0, u0.y, a0.pi);
    a1.pr = f2fma(d1, u1.x, a1.pr);
    a1.pi = f2fma(d1, u1.y, a1.pi);
  }
  // neighbours k = 1..8: (+1,0) (-1,0) (0,+1) (0,-1) (+1,+1) (-1,-1) (+1,-1) (-1,+1)
  const float4* wk[8] = {w0, w0, wp, wm, wp, wm, wm, wp};
  const int xk[8] = {xr, xl, x, x, xr, xl, xr, xl};
#pragma unroll
  for (int k = 0; k < 8; ++k) {
    const ulonglong2 u0 = KPM_L(wk[k], xk[k], 0);
    const ulonglong2 u1 = KPM_L(wk[k], xk[k], 1);
    acc_term(a0, cf[1 + k], u0);
    acc_term(a1, cf[9 + k], u1);
    if (k < 4) {
      acc_term(a0, cf[17 + k], u1);
      acc_term(a1, cf[21 + k], u0);
    }
  }
#undef KPM_L
  o0 = make_ulonglong2(f2sub(a0.pr, a0.qi), f2add(a0.pi, a0.qr));
  o1 = make_ulonglong2(f2sub(a1.pr, a1.qi), f2add(a1.pi, a1.qr));
}

// The persistent kernel keeps a site's entries in the order stencil_site
// uses them: kCoefOrder[i] = table entry at stored position i (the real
// diagonals, then per neighbour k = 0..7 its hopping entries and, for k < 4,
// its pairing entries; the last position is padding)
__constant__ int kCoefOrder[kCoef] = {0, 1, 9,  17, 21, 2, 10, 18, 22, 3,  11, 19, 23,
                                      4, 12, 20, 24, 5, 13, 6,  14, 7,  15, 8,  16, 25};

// Two neighbouring sites x and x + 1 of one lattice row for one column pair
// (both Nambu rows each), every term in the order of stencil_site (so the
// bits are the same): the twelve V_m positions x-1 .. x+2 of rows y-1, y, y+1
// are loaded once for both sites (24 instead of 36 loads), site B's term k
// following site A's, each position dropped after its last use.  cqA, cqB:
// the sites' entries in kCoefOrder order as 16-byte pairs.
template <int NV>
__device__ __forceinline__ void stencil_2site(const float4* wm, const float4* w0, const float4* wp,
                                              const float4* cqA, const float4* cqB, int x, int nx,
                                              ulonglong2& oA0, ulonglong2& oA1, ulonglong2& oB0, ulonglong2& oB1) {
  constexpr int RS = 2 * NV;
  const int xm = x == 0 ? nx - 1 : x - 1;
  const int x1 = x + 1 >= nx ? x + 1 - nx : x + 1;
  const int x2 = x + 2 >= nx ? x + 2 - nx : x + 2;
  struct Site {
    Acc2 a0, a1;
    float4 q;
    const float4* cq;
  };
  Site A = {{0ull, 0ull, 0ull, 0ull}, {0ull, 0ull, 0ull, 0ull}, make_float4(0.f, 0.f, 0.f, 0.f), cqA};
  Site B = {{0ull, 0ull, 0ull, 0ull}, {0ull, 0ull, 0ull, 0ull}, make_float4(0.f, 0.f, 0.f, 0.f), cqB};
  struct U {
    ulonglong2 e, h;  // Nambu slots 0 and 1 of one position
  };
  auto ld = [&](const float4* W, int xx) {
    U u;
    u.e = *reinterpret_cast<const ulonglong2*>(W + xx * RS);
    u.h = *reinterpret_cast<const ulonglong2*>(W + xx * RS + NV);
    return u;
  };
  // stored entry i of a site, its 16-byte pair loaded when first needed (even i)
  auto cf = [](Site& S, int i) {
    if ((i & 1) == 0) S.q = S.cq[i >> 1];
    return (i & 1) ? make_float2(S.q.z, S.q.w) : make_float2(S.q.x, S.q.y);
  };
  auto diag = [&](Site& S, const U& u) {
    const float2 d = cf(S, 0);
    const u64 d0 = dup2(d.x), d1 = dup2(d.y);
    S.a0.pr = f2fma(d0, u.e.x, S.a0.pr);
    S.a0.pi = f2fma(d0, u.e.y, S.a0.pi);
    S.a1.pr = f2fma(d1, u.h.x, S.a1.pr);
    S.a1.pi = f2fma(d1, u.h.y, S.a1.pi);
  };
  // neighbour k: stored positions 1 + 4k (k < 4, with pairing) or 17 + 2 (k - 4)
  auto nb = [&](Site& S, int k, const U& u) {
    const int i = k < 4 ? 1 + 4 * k : 17 + 2 * (k - 4);
    acc_term(S.a0, cf(S, i), u.e);
    acc_term(S.a1, cf(S, i + 1), u.h);
    if (k < 4) {
      acc_term(S.a0, cf(S, i + 2), u.h);
      acc_term(S.a1, cf(S, i + 3), u.e);
    }
  };
  // k: (+1,0) (-1,0) (0,+1) (0,-1) (+1,+1) (-1,-1) (+1,-1) (-1,+1), as in stencil_site
  const U c0 = ld(w0, x), c1 = ld(w0, x1);
  diag(A, c0);
  diag(B, c1);
  {
    const U c2 = ld(w0, x2);
    nb(A, 0, c1);
    nb(B, 0, c2);
  }
  {
    const U cm = ld(w0, xm);
    nb(A, 1, cm);
    nb(B, 1, c0);
  }
  const U p0 = ld(wp, x), p1 = ld(wp, x1);
  nb(A, 2, p0);
  nb(B, 2, p1);
  const U m0 = ld(wm, x), m1 = ld(wm, x1);
  nb(A, 3, m0);
  nb(B, 3, m1);
  {
    const U p2 = ld(wp, x2);
    nb(A, 4, p1);
    nb(B, 4, p2);
  }
  {
    const U mm = ld(wm, xm);
    nb(A, 5, mm);
    nb(B, 5, m0);
  }
  {
    const U m2 = ld(wm, x2);
    nb(A, 6, m1);
    nb(B, 6, m2);
  }
  {
    const U pm = ld(wp, xm);
    nb(A, 7, pm);
    nb(B, 7, p0);
  }
  oA0 = make_ulonglong2(f2sub(A.a0.pr, A.a0.qi), f2add(A.a0.pi, A.a0.qr));
  oA1 = make_ulonglong2(f2sub(A.a1.pr, A.a1.qi), f2add(A.a1.pi, A.a1.qr));
  oB0 = make_ulonglong2(f2sub(B.a0.pr, B.a0.qi), f2add(B.a0.pi, B.a0.qr));
  oB1 = make_ulonglong2(f2sub(B.a1.pr, B.a1.qi), f2add(B.a1.pi, B.a1.qr));
}

// moment sums acc[J][s] += a V[K_s(J), J] for the columns of the chunk whose
// own site lies in lattice row y; wm, w0, wp hold rows y-1, y, y+1 (unit vectors of a full
// pass: FP32 probing and half passes run the march kernel)
template <int CB>
__device__ __forceinline__ void moment_sums(const float4* wm, const float4* w0, const float4* wp, int nx, int y,
                                            int64_t D, int64_t s0, int m, double cm, double co,
                                            double2* __restrict__ acc) {
  constexpr int NV = CB / 2;
  constexpr int RS = 2 * NV;
  for (int t = threadIdx.x; t < CB * kSlots; t += blockDim.x) {
    const int c = t / kSlots, s = t - c * kSlots;
    const int64_t J = s0 + c, j = J >> 1;
    if (J >= D || j / nx != y) continue;
    const int beta = (int)(J & 1);
    const int xsl = wrapi((int)(j % nx) + kSlotDx[s], nx);
    const int dy = kSlotDy[s];
    const float4* w = dy < 0 ? wm : (dy > 0 ? wp : w0);
    const int al = kSlotFlip[s] ? 1 - beta : beta;
    const float2 val = pair_elem(w + xsl * RS + al * NV, c);
    acc_add_unit(acc + J * kSlots + s, s == kSlots - 1 ? co : cm, (double)val.x, (double)val.y);
  }
}

// FP32 step.  Shared memory: V_m window ring of 5 lattice rows (rows y-1..y+1
// in use, y+2 and y+3 in flight) and a ring of 3 coefficient rows (y in use,
// y+1 and y+2 in flight); V_{m-1} rows are read one row ahead into registers.
template <int CB, int MODE>
__device__ __forceinline__ void f32_step_body(int nx, int ny, int64_t D, int64_t ldv, int ylen,
                                              const float2* __restrict__ table, const float4* __restrict__ Vcur,
                                              const float4* Vprev, float4* Vout, int64_t s0,
                                              double2* __restrict__ acc,
                                              const double* __restrict__ am, const double* __restrict__ ao, int m) {
  constexpr int NV = CB / 2;   // float4 (column pairs) per Nambu row of the chunk
  constexpr int RS = 2 * NV;   // float4 per site of a window row (both Nambu rows)
  const int64_t ldq = ldv / 2; // float4 per slab row

  extern __shared__ __align__(16) unsigned char smem_raw[];
  float4* win = reinterpret_cast<float4*>(smem_raw);  // [5][nx][2][NV]
  float2* coef = reinterpret_cast<float2*>(win + 5 * nx * RS);  // [3][nx][kCoef]
  const int rowsz = nx * RS;
  const int crow = nx * kCoef;

  const int64_t cb0 = (int64_t)blockIdx.y * CB;
  const int64_t q0 = cb0 / 2;
  const int y0 = blockIdx.x * ylen;
  const int y1 = min(ny, y0 + ylen);
  const int nrow = y1 - y0;

  const int v = threadIdx.x % NV;
  const int xs = threadIdx.x / NV;
  const int xstep = blockDim.x / NV;  // sites of a row per thread round; nx <= 2 xstep (planner)
  const bool own0 = xs < nx, own1 = xs + xstep < nx;

  // rows of the chunk's own sites: only there are moment sums due
  int yj_lo = ny, yj_hi = -1;
  {
    const int64_t clo = s0 + cb0, chi = min(D, s0 + cb0 + CB) - 1;
    if (chi >= clo) {
      yj_lo = (int)((clo >> 1) / nx);
      yj_hi = (int)((chi >> 1) / nx);
    }
  }

  // prologue groups: {V rows y0-1..y0+1, coef y0}, {V row y0+2, coef y0+1};
  // iteration q commits {V row y+3, coef y+2} right after its barrier
  for (int q = 0; q < 3; ++q)
    stage_row<float4, NV>(win + q * rowsz, Vcur, wrapi(y0 - 1 + q, ny), nx, ldq, q0);
  stage_coef<float2>(coef, table, y0, nx);
  cp_commit();
  if (nrow >= 2) {
    stage_row<float4, NV>(win + 3 * rowsz, Vcur, wrapi(y0 + 2, ny), nx, ldq, q0);
    stage_coef<float2>(coef + crow, table, y0 + 1, nx);
  }
  cp_commit();

  // V_{m-1} of the thread's sites, one row ahead in registers
  ulonglong2 pc[2][2], pn[2][2];
  const ulonglong2 zero2 = make_ulonglong2(0ull, 0ull);
  auto load_prev = [&](int y, ulonglong2 (&dst)[2][2]) {
    const float4* g = Vprev + (2 * ((int64_t)y * nx + xs)) * ldq + q0 + v;
    const int64_t gstep = 2 * (int64_t)xstep * ldq;
    dst[0][0] = own0 ? *reinterpret_cast<const ulonglong2*>(g) : zero2;
    dst[0][1] = own0 ? *reinterpret_cast<const ulonglong2*>(g + ldq) : zero2;
    dst[1][0] = own1 ? *reinterpret_cast<const ulonglong2*>(g + gstep) : zero2;
    dst[1][1] = own1 ? *reinterpret_cast<const ulonglong2*>(g + gstep + ldq) : zero2;
  };
  if (MODE == 1) load_prev(y0, pc);

  const u64 half2 = 0x3F0000003F000000ull;  // (0.5f, 0.5f)
  int bm = 0;  // ring slot of lattice row y - 1
  int bc = 0;  // ring slot of the coefficients of row y
  for (int q = 0; q < nrow; ++q) {
    const int y = y0 + q;
    if (MODE == 1 && q + 1 < nrow) load_prev(y + 1, pn);
    cp_wait_1();
    __syncthreads();
    // refill (every thread is past row y-1): V_m row y+3 into the slot of
    // y-2, coefficients of y+2 into the slot of y-1
    {
      const int bf = bm == 0 ? 4 : bm - 1;
      const int cfs = bc == 0 ? 2 : bc - 1;
      if (y + 3 <= y1) stage_row<float4, NV>(win + bf * rowsz, Vcur, wrapi(y + 3, ny), nx, ldq, q0);
      if (y + 2 < y1) stage_coef<float2>(coef + cfs * crow, table, y + 2, nx);
      cp_commit();
    }
    const int b0 = bm + 1 == 5 ? 0 : bm + 1;
    const int bp = b0 + 1 == 5 ? 0 : b0 + 1;
    const float4* wm = win + bm * rowsz + v;  // lattice row y - 1
    const float4* w0 = win + b0 * rowsz + v;  // y
    const float4* wp = win + bp * rowsz + v;  // y + 1
    const float2* cf_row = coef + bc * crow;

#pragma unroll
    for (int it = 0; it < 2; ++it) {
      if (!(it == 0 ? own0 : own1)) continue;
      const int x = xs + it * xstep;
      ulonglong2 o0, o1;
      stencil_site<NV>(wm, w0, wp, cf_row, x, nx, o0, o1);
      if (MODE == 1) {
        o0.x = f2sub(o0.x, pc[it][0].x);
        o0.y = f2sub(o0.y, pc[it][0].y);
        o1.x = f2sub(o1.x, pc[it][1].x);
        o1.y = f2sub(o1.y, pc[it][1].y);
      } else {
        o0.x = f2mul(o0.x, half2);
        o0.y = f2mul(o0.y, half2);
        o1.x = f2mul(o1.x, half2);
        o1.y = f2mul(o1.y, half2);
      }
      float4* g = Vout + (2 * ((int64_t)y * nx + x)) * ldq + q0 + v;
      *reinterpret_cast<ulonglong2*>(g) = o0;
      *reinterpret_cast<ulonglong2*>(g + ldq) = o1;
    }

    if (MODE == 1 && acc != nullptr && y >= yj_lo && y <= yj_hi)
      moment_sums<CB>(wm - v, w0 - v, wp - v, nx, y, D, s0 + cb0, m, am[m], ao[m], acc);
    bm = b0;
    bc = bc + 1 == 3 ? 0 : bc + 1;
    if (MODE == 1) {
      pc[0][0] = pn[0][0];
      pc[0][1] = pn[0][1];
      pc[1][0] = pn[1][0];
      pc[1][1] = pn[1][1];
    }
  }
  cp_wait_0();
}

template <int CB, int MODE>
__global__ void __launch_bounds__(512, 1)
    cheb_step_f32_kernel(int nx, int ny, int64_t D, int64_t ldv, int ylen, const float2* __restrict__ table,
                         const float4* __restrict__ Vcur, const float4* Vprev, float4* Vout, int64_t s0,
                         double2* __restrict__ acc, const double* __restrict__ am, const double* __restrict__ ao,
                         int m) {
  f32_step_body<CB, MODE>(nx, ny, D, ldv, ylen, table, Vcur, Vprev, Vout, s0, acc, am, ao, m);
}

// ---- TMA copies and bounded waits (the march kernel) ----------------------
// Waits on mbarriers are bounded in time: a CTA whose copies do not land sets the
// fault word, waits (bounded) for its copies in flight and writes NaN over its
// output rows, so a failed launch shows in the observables instead of hanging the
// device.
__device__ unsigned int g_step_fault;

__device__ __forceinline__ uint32_t smem_u32(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }
__device__ __forceinline__ void mbar_init(uint32_t bar, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;\n" ::"r"(bar), "r"(count) : "memory");
}
__device__ __forceinline__ void mbar_expect_tx(uint32_t bar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;\n" ::"r"(bar), "r"(bytes) : "memory");
}
__device__ __forceinline__ bool mbar_try(uint32_t bar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, p;\n}\n"
      : "=r"(ok)
      : "r"(bar), "r"(parity)
      : "memory");
  return ok != 0;
}
__device__ __forceinline__ uint64_t global_ns() {
  uint64_t t;
  asm volatile("mov.u64 %0, %%globaltimer;\n" : "=l"(t));
  return t;
}
// true once the phase of parity `parity` has completed; false after about
// limit_ns of waiting (or 2^26 polls)
__device__ __noinline__ bool mbar_wait_slow(uint32_t bar, uint32_t parity, uint64_t limit_ns) {
  const uint64_t t0 = global_ns();
  for (uint32_t it = 1; it < (1u << 26); ++it) {
    if (mbar_try(bar, parity)) return true;
    if ((it & 63) == 0 && global_ns() - t0 > limit_ns) return false;
  }
  return false;
}
__device__ __forceinline__ void tma_load_2d(uint32_t dst, const CUtensorMap* tm, int c0, int c1, uint32_t bar) {
  asm volatile(
      "cp.async.bulk.tensor.2d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3}], "
      "[%4];\n" ::"r"(dst),
      "l"(reinterpret_cast<uint64_t>(tm)), "r"(c0), "r"(c1), "r"(bar)
      : "memory");
}
__device__ __forceinline__ void bulk_load(uint32_t dst, const void* src, uint32_t bytes, uint32_t bar) {
  asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];\n" ::"r"(dst),
               "l"(src), "r"(bytes), "r"(bar)
               : "memory");
}

constexpr uint64_t kWaitLimitNs = 2000000000ull;  // 2 s: orders of magnitude above a lattice row's copies
// bounded-wait limit of the march kernel (kWaitLimitNs unless a test shortened it)
// and the number of CTAs that are still to skip one window copy (test hook of
// the failure path: a skipped copy leaves nothing in flight, so only the
// waits on its slot run out)
__device__ unsigned long long g_wait_limit_ns = kWaitLimitNs;
__device__ int g_drop_copy;
__device__ __forceinline__ void mbar_arrive(uint32_t bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];\n" ::"r"(bar) : "memory");
}

#include "cheb_march.cuh"

// V0: entry (K, c) of the start vector held by slab column c (unit vector
// e_{(s0+c) << js}, or probing vector r_{s0+c}); zero in padding columns
__device__ __forceinline__ double2 start_entry(int64_t K, int64_t c, int64_t D, int nx, const ColMap& cm) {
  const int64_t col = cm.s0 + c;
  if (cm.probe_p) {
    if (col >= 2 * (int64_t)cm.probe_p * cm.probe_p || probe_colour(K, nx, cm.probe_p) != col)
      return make_double2(0.0, 0.0);
    return probe_xi(cm.seed, K);
  }
  return make_double2(col < (D >> cm.js) && K == (col << cm.js) ? 1.0 : 0.0, 0.0);
}
__global__ void cheb_init_f64_kernel(int64_t D, int64_t ldv, int nx, double2* __restrict__ V0, ColMap cm) {
  const int64_t total = D * ldv;
  for (int64_t k = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; k < total; k += (int64_t)gridDim.x * blockDim.x) {
    const int64_t K = k / ldv, c = k - K * ldv;
    V0[k] = start_entry(K, c, D, nx, cm);
  }
}
// double-float layout of vectors: float4 (re_hi, im_hi, re_lo, im_lo)
__global__ void cheb_init_df_kernel(int64_t D, int64_t ldv, int nx, float4* __restrict__ V0, ColMap cm) {
  const int64_t total = D * ldv;
  for (int64_t k = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; k < total; k += (int64_t)gridDim.x * blockDim.x) {
    const int64_t K = k / ldv, c = k - K * ldv;
    const double2 e = start_entry(K, c, D, nx, cm);
    const float2 re = df_split(e.x), im = df_split(e.y);
    V0[k] = make_float4(re.x, im.x, re.y, im.y);
  }
}
// FP32 pair-split layout: float4 (re_2p, re_2p+1, im_2p, im_2p+1)
__global__ void cheb_init_f32_kernel(int64_t D, int64_t ldv, int nx, float4* __restrict__ V0, ColMap cm) {
  const int64_t ldq = ldv / 2;
  const int64_t total = D * ldq;
  for (int64_t k = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; k < total; k += (int64_t)gridDim.x * blockDim.x) {
    const int64_t K = k / ldq, c = 2 * (k - K * ldq);
    const double2 e0 = start_entry(K, c, D, nx, cm), e1 = start_entry(K, c + 1, D, nx, cm);
    V0[k] = make_float4((float)e0.x, (float)e1.x, (float)e0.y, (float)e1.y);
  }
}
// the m = 0 moment terms of every source of the slab: a_0 on the own-row slot
// and a^Omega_0 on the diagonal slot (the local rows of a source never share
// its probing colour, so conj(xi_J) V_0 is 1 on row J and 0 on the others)
__global__ void cheb_init_acc_kernel(int64_t D, int64_t ldv, int nx, ColMap cm, double2* __restrict__ acc,
                                     const double* __restrict__ am, const double* __restrict__ ao) {
  const int64_t nsrc = cm.probe_p ? D : ldv;
  for (int64_t k = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; k < nsrc * kSlots;
       k += (int64_t)gridDim.x * blockDim.x) {
    const int64_t r = k / kSlots;
    const int s = (int)(k - r * kSlots);
    int64_t J;
    if (cm.probe_p) {
      const int64_t col = probe_colour(r, nx, cm.probe_p) - cm.s0;
      if (col < 0 || col >= ldv) continue;
      J = r;
    } else {
      if (cm.s0 + r >= (D >> cm.js)) continue;
      J = (cm.s0 + r) << cm.js;
    }
    double2 a = make_double2(0.0, 0.0);
    if (s == 0) a.x = am[0];
    if (s == kSlots - 1) a.x = ao[0];
    if (cm.raw) {  // times xi_J, which the gather takes out again
      const double2 x = cm.xi[J];
      a = make_double2(a.x * x.x, -a.x * x.y);
    }
    acc[J * kSlots + s] = a;
    if (s == 0 && cm.rec) cm.rec[(J & 1) * (D >> 1) + (J >> 1)] = 1.0;  // T_0 = 1
  }
}

__global__ void probe_phase_kernel(int64_t D, uint32_t seed, double2* __restrict__ xi_conj) {
  for (int64_t K = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; K < D; K += (int64_t)gridDim.x * blockDim.x) {
    const double2 x = probe_xi(seed, K);
    xi_conj[K] = make_double2(x.x, -x.y);
  }
}

// Moment sums of a probing slab, V_m = Va and (if given) V_{m+1} = Vb, one thread
// per source and slot.  Every row is a source, and a march CTA meets its share of them in
// bursts (all the sites of every p-th row): in the march's sums warp they held its
// rings up for 6 to 18 us a step.  Here two moments go into one update of the sums, kept
// without the phase conj(xi_J), which the gather multiplies in: four FP64 operations a
// moment and slot pair less than weighting every term (the FP64 pipe is 1/64 of FP32's).
__global__ void probe_sums_kernel(int nx, int ny, int D, int64_t ldv, const float4* __restrict__ Va,
                                  const float4* __restrict__ Vb, ColMap cm, double2* __restrict__ acc,
                                  const double* __restrict__ am, const double* __restrict__ ao, int m) {
  const int p = cm.probe_p;
  const int64_t ldq = ldv / 2;
  for (int t = blockIdx.x * blockDim.x + threadIdx.x; t < D * kSlots; t += gridDim.x * blockDim.x) {
    const int J = t / kSlots, s = t - J * kSlots;
    const int i = J >> 1, y = i / nx, x = i - y * nx;
    const int c = (J & 1) + 2 * (x % p + p * (y % p)) - (int)cm.s0;
    if (c < 0 || c >= ldv) continue;
    int xs = x + kSlotDx[s], ys = y + kSlotDy[s];
    xs = xs < 0 ? xs + nx : xs >= nx ? xs - nx : xs;
    ys = ys < 0 ? ys + ny : ys >= ny ? ys - ny : ys;
    const int64_t K = 2 * (ys * nx + xs) + ((J & 1) ^ kSlotFlip[s]);
    const int64_t at = 4 * (K * ldq + (c >> 1)) + (c & 1);
    double2 a = acc[t];
    const double* const cf = s == kSlots - 1 ? ao : am;
    const float ar = reinterpret_cast<const float*>(Va)[at], ai = reinterpret_cast<const float*>(Va)[at + 2];
    float br = 0.f, bi = 0.f;
    if (Vb) {
      br = reinterpret_cast<const float*>(Vb)[at];
      bi = reinterpret_cast<const float*>(Vb)[at + 2];
    }
    acc_add_unit(&a, cf[m], (double)ar, (double)ai);
    if (Vb) acc_add_unit(&a, cf[m + 1], (double)br, (double)bi);
    acc[t] = a;
    if (s == 0 && cm.rec) {
      record_diag(cm, D, m, J, cm.xi[J], (double)ar, (double)ai);
      if (Vb) record_diag(cm, D, m + 1, J, cm.xi[J], (double)br, (double)bi);
    }
  }
}

// acc += a_m V[local rows] (the last moment, which no step reads again)
// LAY: 0 FP64 interleaved complex, 1 FP32 pair-split, 2 double-float
template <int LAY>
__global__ void cheb_gather_kernel(int nx, int ny, int64_t D, int64_t ldv, int64_t width, const void* __restrict__ V,
                                   ColMap cm, double2* __restrict__ acc, const double* __restrict__ am,
                                   const double* __restrict__ ao, int m) {
  const int64_t total = (cm.probe_p ? D : width) * kSlots;
  for (int64_t k = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; k < total; k += (int64_t)gridDim.x * blockDim.x) {
    const int64_t r = k / kSlots;
    const int s = (int)(k - r * kSlots);
    int64_t J, c;
    double2 wgt = make_double2(1.0, 0.0);
    if (cm.probe_p) {
      J = r;
      c = probe_colour(J, nx, cm.probe_p) - cm.s0;
      if (c < 0 || c >= width) continue;
      wgt = cm.xi[J];
    } else {
      c = r;
      if (cm.s0 + c >= (D >> cm.js)) continue;
      J = (cm.s0 + c) << cm.js;
    }
    const int64_t j = J >> 1;
    const int beta = (int)(J & 1);
    const int xs = wrapi((int)(j % nx) + kSlotDx[s], nx);
    const int ys = wrapi((int)(j / nx) + kSlotDy[s], ny);
    const int al = kSlotFlip[s] ? 1 - beta : beta;
    const int64_t K = 2 * ((int64_t)ys * nx + xs) + al;
    double re, im;
    if (LAY == 1) {
      const float2 val = pair_elem(reinterpret_cast<const float4*>(V) + K * (ldv / 2), (int)c);
      re = val.x;
      im = val.y;
    } else if (LAY == 2) {
      const float4 val = reinterpret_cast<const float4*>(V)[K * ldv + c];
      re = cre(val);
      im = cim(val);
    } else {
      const double2 val = reinterpret_cast<const double2*>(V)[K * ldv + c];
      re = val.x;
      im = val.y;
    }
    double2* const e = acc + J * kSlots + s;
    const double coef = s == kSlots - 1 ? ao[m] : am[m];
    if (cm.raw) {  // sums kept without the phase: conj(xi_J) (sum + the last term)
      double2 t = *e;
      acc_add_unit(&t, coef, re, im);
      *e = make_double2(wgt.x * t.x - wgt.y * t.y, wgt.x * t.y + wgt.y * t.x);
    } else {
      acc_add(e, coef, wgt, re, im);
    }
    if (s == 0 && cm.rec) record_diag(cm, D, m, J, wgt, re, im);
  }
}

// ---- Persistent batched recursion (many cells, one launch per iteration) ----
// A cluster of kPClu CTAs owns one work item, a chunk of kPCB unit columns of
// one cell, for the whole pass: the cell's lattice rows are split into bands
// of R = ceil(ny / kPClu) rows, CTA `rank` of the cluster holds band rank of
// both recursion vectors V_m, V_{m-1} (pair-split FP32, as the step kernels),
// the band's 2h~ entries and the FP64 moment sums of the chunk's columns whose
// own site lies in the band, all in shared memory.  Per Chebyshev step a CTA
// computes its band of V_{m+1} in place over V_{m-1} with the stencil
// arithmetic of the step kernels and adds the moment sums of V_m.  The two
// halo rows of V_m come from the neighbouring bands through a small exchange
// buffer in global memory (L2-resident): every CTA stores the first and last
// row of its band of V_{m+1} there (double-buffered by step parity) and, after
// the cluster barrier that ends the step, fetches its halo rows with cp.async
// while it computes the interior rows of its band, which need no halo.
// (Distributed shared memory carried the halo in a first version; at 32 KB
// per CTA and step its throughput set the step time.)  One cluster barrier per
// step: in step m a CTA writes only its own rows of V_{m+1} and exchange slots
// of parity (m + 1) & 1, which no other CTA reads before that barrier.
// Items come from a device counter in the order of the host's list (longest
// first); rank 0 fetches and publishes each item to the cluster.  Cluster
// barriers are hardware barriers that every CTA of the cluster reaches the
// same number of times (all run the same items and M), so nothing spins.
constexpr int kPCB = 16;  // columns per item
constexpr int kPNV = kPCB / 2;

size_t persist_smem(int nx, int R) {  // V pair + 2 halo rows, coefficients, moment sums
  return sizeof(float4) * (size_t)(2 * R + 2) * nx * 2 * kPNV + sizeof(float2) * (size_t)R * nx * kCoef +
         sizeof(double2) * kPCB * kSlots;
}

__device__ __forceinline__ void cp_async16_cg(void* smem, const void* gmem) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"((uint32_t)__cvta_generic_to_shared(smem)),
               "l"(gmem)
               : "memory");
}

// xbuf: exchange rows of the clusters, xrow float4 each; slot of (cluster c,
// rank k, side h = 0 first / 1 last band row, parity p) is ((c kPClu + k) 2 + h) 2 + p
__global__ void __cluster_dims__(kPClu, 1, 1) __launch_bounds__(512, 1)
    cheb_persist_kernel(const PCell* __restrict__ cells, const PItem* __restrict__ items, int nitems,
                        int* __restrict__ counter, int M, float4* __restrict__ xbuf, int xrow) {
  namespace cg = cooperative_groups;
  cg::cluster_group cluster = cg::this_cluster();
  const int rank = (int)cluster.block_rank();
  const int64_t cbase = (int64_t)(blockIdx.x / kPClu) * kPClu;
  auto xslot = [&](int k, int h, int p) { return xbuf + ((((cbase + k) * 2 + h) * 2 + p) * (int64_t)xrow); };
  extern __shared__ __align__(128) unsigned char smem_p[];
  for (;;) {
    // item fetch: rank 0 takes the next index and publishes it in the first
    // word of its shared memory, which the item's data overwrite only after
    // every CTA of the cluster has read it
    int* slot = reinterpret_cast<int*>(smem_p);
    if (rank == 0 && threadIdx.x == 0) *slot = atomicAdd(counter, 1);
    cluster.sync();
    const int it = *cluster.map_shared_rank(slot, 0);
    cluster.sync();
    if (it >= nitems) break;
    const PItem item = items[it];
    const PCell cell = cells[item.cell];
    const int nx = cell.nx, ny = cell.ny;
    const int64_t D = 2 * (int64_t)nx * ny;
    const int R = (ny + kPClu - 1) / kPClu;
    const int y0 = min(ny, rank * R), y1 = min(ny, y0 + R);
    const int nrow = y1 - y0;
    const int rowsz = nx * 2 * kPNV;  // float4 per lattice row of V
    float4* V0buf = reinterpret_cast<float4*>(smem_p);
    float4* V1buf = V0buf + (size_t)R * rowsz;
    float4* halo = V1buf + (size_t)R * rowsz;  // [2][rowsz]: rows y0 - 1 and y1 of V_m
    float2* coef = reinterpret_cast<float2*>(halo + 2 * rowsz);
    double2* acc = reinterpret_cast<double2*>(coef + (size_t)R * nx * kCoef);
    const int64_t q0 = item.q0;  // first unit column of the chunk
    // bands holding lattice rows y0 - 1 (its last row) and y1 (its first row)
    const int ra = wrapi(y0 - 1, ny) / R, rb = wrapi(y1, ny) / R;

    // coefficients of the band; V_0 = the chunk's unit vectors; a_0 moment terms
    {
      // each site's entries in the order the stencil uses them (kCoefOrder)
      const float2* src = cell.table + (int64_t)y0 * nx * kCoef;
      const int n2 = nrow * nx * kCoef;
      for (int t = threadIdx.x; t < n2; t += blockDim.x) {
        const int site = t / kCoef;
        coef[t] = src[site * kCoef + kCoefOrder[t - site * kCoef]];
      }
      const float4 z4 = make_float4(0.f, 0.f, 0.f, 0.f);
      for (int t = threadIdx.x; t < nrow * rowsz; t += blockDim.x) V0buf[t] = z4;
      if (nrow > 0)
        for (int t = threadIdx.x; t < rowsz; t += blockDim.x) {
          xslot(rank, 0, 0)[t] = z4;
          xslot(rank, 1, 0)[t] = z4;
        }
    }
    __syncthreads();
    if (threadIdx.x < kPCB) {
      const int c = threadIdx.x;
      const int64_t J = q0 + c;
      const int64_t j = J >> 1;
      const int y = (int)(j / nx);
      if (J < D && y >= y0 && y < y1) {
        const int x = (int)(j % nx), be = (int)(J & 1);
        const size_t off = (size_t)x * 2 * kPNV + be * kPNV + (c >> 1);
        float4* e = V0buf + (size_t)(y - y0) * rowsz + off;
        if (c & 1) e->y = 1.0f; else e->x = 1.0f;
        // the boundary rows of V_0 in the exchange buffer as well
        if (y == y0) {
          float4* g = xslot(rank, 0, 0) + off;
          if (c & 1) g->y = 1.0f; else g->x = 1.0f;
        }
        if (y == y1 - 1) {
          float4* g = xslot(rank, 1, 0) + off;
          if (c & 1) g->y = 1.0f; else g->x = 1.0f;
        }
      }
    }
    for (int t = threadIdx.x; t < kPCB * kSlots; t += blockDim.x) {
      const int s = t % kSlots;
      acc[t] = make_double2(s == 0 ? cell.am[0] : (s == kSlots - 1 ? cell.ao[0] : 0.0), 0.0);
    }
    cluster.sync();

    // rows r - 1 and r + 1 of the band (r = 0 .. nrow - 1) in V_m: band rows,
    // or the halo rows y0 - 1 and y1
    auto row_below = [&](const float4* cur, int r) -> const float4* {
      return r > 0 ? cur + (size_t)(r - 1) * rowsz : halo;
    };
    auto row_above = [&](const float4* cur, int r) -> const float4* {
      return r + 1 < nrow ? cur + (size_t)(r + 1) * rowsz : halo + rowsz;
    };
    // halo rows of V_m (exchange parity p) into shared memory, asynchronously
    auto fetch_halo = [&](int p) {
      if (nrow == 0) return;
      const float4* ga = xslot(ra, 1, p);
      const float4* gb = xslot(rb, 0, p);
      for (int t = threadIdx.x; t < 2 * rowsz; t += blockDim.x)
        cp_async16_cg(halo + t, t < rowsz ? ga + t : gb + (t - rowsz));
      cp_commit();
    };
    // moment sums a_m V_m of the chunk's columns whose own site is in the band:
    // thread t < kPCB kSlots owns entry (column c, slot s); where that entry
    // sits in shared memory is the same for every step of the item, so it is
    // worked out once: scode = -1 (column outside the band or the lattice),
    // else (float4 index << 1) | (1 if in the halo rows, 0 if in the V_m band)
    int scode = -1;
    if (threadIdx.x < kPCB * kSlots) {
      const int t = threadIdx.x, c = t / kSlots, s = t - c * kSlots;
      const int64_t J = q0 + c;
      const int64_t j = J >> 1;
      const int y = J < D ? (int)(j / nx) : -1;
      if (y >= y0 && y < y1) {
        const int beta = (int)(J & 1);
        const int xsl = wrapi((int)(j % nx) + kSlotDx[s], nx);
        const int al = kSlotFlip[s] ? 1 - beta : beta;
        const int r = y - y0, dy = kSlotDy[s];
        const int e = xsl * 2 * kPNV + al * kPNV + (c >> 1);
        if (dy < 0 && r == 0) scode = (e << 1) | 1;                   // row y0 - 1: halo row 0
        else if (dy > 0 && r + 1 == nrow) scode = ((rowsz + e) << 1) | 1;  // row y1: halo row 1
        else scode = (((r + dy) * rowsz + e) << 1);
      }
    }
    auto sums = [&](const float4* cur, int m) {
      if (scode < 0) return;
      const int t = threadIdx.x, c = t / kSlots, s = t - c * kSlots;
      const double cm = cell.am[m], co = cell.ao[m];
      const float4 q = ((scode & 1) ? halo : cur)[scode >> 1];
      const float2 val = (c & 1) ? make_float2(q.y, q.w) : make_float2(q.x, q.z);
      acc_add_unit(acc + t, s == kSlots - 1 ? co : cm, (double)val.x, (double)val.y);
    };

    const u64 half2 = 0x3F0000003F000000ull;  // (0.5f, 0.5f)
    const int v = threadIdx.x % kPNV;
    const int gstep = blockDim.x / kPNV;
    // V_{m+1} of site x of band row r from 2h~ V_m (o0, o1): halved at m = 0,
    // else minus V_{m-1} (stored where V_{m+1} goes); boundary rows also go
    // to the exchange slots
    auto emit = [&](float4* out, int m, int r, int x, ulonglong2 o0, ulonglong2 o1) {
      const size_t off = (size_t)x * 2 * kPNV + v;
      ulonglong2* g = reinterpret_cast<ulonglong2*>(out + (size_t)r * rowsz + off);
      if (m == 0) {
        o0.x = f2mul(o0.x, half2);
        o0.y = f2mul(o0.y, half2);
        o1.x = f2mul(o1.x, half2);
        o1.y = f2mul(o1.y, half2);
      } else {
        const ulonglong2 p0 = g[0], p1 = g[kPNV];
        o0.x = f2sub(o0.x, p0.x);
        o0.y = f2sub(o0.y, p0.y);
        o1.x = f2sub(o1.x, p1.x);
        o1.y = f2sub(o1.y, p1.y);
      }
      g[0] = o0;
      g[kPNV] = o1;
      const int p = (m + 1) & 1;
      for (int h = 0; h < 2; ++h)
        if (r == (h == 0 ? 0 : nrow - 1)) {
          ulonglong2* e = reinterpret_cast<ulonglong2*>(xslot(rank, h, p) + off);
          e[0] = o0;
          e[kPNV] = o1;
        }
    };
    // band rows r0, r0 + rstep, ... (< r1) of V_{m+1}, two neighbouring sites
    // of a row per thread and column pair
    const int npair = (nx + 1) >> 1;
    auto rows = [&](const float4* cur, float4* out, int m, int r0, int r1, int rstep) {
      const int nr = (r1 - r0 + rstep - 1) / rstep;
      for (int t = threadIdx.x / kPNV; t < nr * npair; t += gstep) {
        const int ri = t / npair;
        const int r = r0 + ri * rstep, x = 2 * (t - ri * npair);
        const float4* cqA = reinterpret_cast<const float4*>(coef + ((size_t)r * nx + x) * kCoef);
        const float4* cqB = x + 1 < nx ? cqA + kCoef / 2 : cqA;  // odd nx: the last pair has one site
        ulonglong2 oA0, oA1, oB0, oB1;
        stencil_2site<kPNV>(row_below(cur, r) + v, cur + (size_t)r * rowsz + v, row_above(cur, r) + v, cqA, cqB, x,
                            nx, oA0, oA1, oB0, oB1);
        emit(out, m, r, x, oA0, oA1);
        if (x + 1 < nx) emit(out, m, r, x + 1, oB0, oB1);
      }
    };

    for (int m = 0; m + 1 <= M - 1; ++m) {
      // V_m in buffer (m & 1); V_{m+1} over V_{m-1} in buffer ((m + 1) & 1)
      const float4* cur = (m & 1) ? V1buf : V0buf;
      float4* out = (m & 1) ? V0buf : V1buf;
      fetch_halo(m & 1);
      if (nrow > 2) rows(cur, out, m, 1, nrow - 1, 1);  // interior rows while the halo arrives
      cp_wait_0();
      __syncthreads();
      if (nrow > 0) rows(cur, out, m, 0, nrow, nrow > 1 ? nrow - 1 : 1);  // rows 0 and nrow - 1
      if (m >= 1) sums(cur, m);
      cluster.sync();
    }
    if (M >= 2) {  // the last moment, which no step reads
      const int b = (M - 1) & 1;
      fetch_halo(b);
      cp_wait_0();
      __syncthreads();
      sums(b ? V1buf : V0buf, M - 1);
    }
    __syncthreads();
    for (int t = threadIdx.x; t < kPCB * kSlots; t += blockDim.x) {
      const int c = t / kSlots;
      const int64_t J = q0 + c;
      if (J >= D) continue;
      const int y = (int)((J >> 1) / nx);
      if (y >= y0 && y < y1) cell.acc[J * kSlots + (t - c * kSlots)] = acc[t];
    }
    cluster.sync();  // the next item's initial exchange rows follow every read of this item's
  }
}

constexpr size_t kSmemLimit = 227 * 1024;
// host side: launch the test-hook instantiation of the march kernel (set by
// set_step_failure_test; launches enqueued or captured after it)
bool g_step_hook_armed = false;
constexpr int kSMs = 152;

template <int CB>
size_t smem_f32(int nx) {  // V_m window ring of 5 rows + coefficient ring of 3 rows
  return sizeof(float4) * (size_t)5 * nx * CB + sizeof(float2) * (size_t)3 * nx * kCoef;
}
template <int CB>
size_t smem_f64(int nx) {  // V_m window + V_{m-1} rows + coefficient rows
  return sizeof(double2) * ((size_t)6 * 2 * nx * CB + (size_t)2 * nx * kCoef);
}

template <int CB>
cudaError_t set_smem_f32(int nx) {
  cudaError_t e = cudaFuncSetAttribute(cheb_step_f32_kernel<CB, 0>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       (int)kSmemLimit);
  if (e != cudaSuccess) return e;
  e = cudaFuncSetAttribute(cheb_step_f32_kernel<CB, 1>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                           (int)kSmemLimit);
  return e;
}

// cuTensorMapEncodeTiled, resolved once through the runtime's driver entry point
using EncodeTiledFn = CUresult (*)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                                   const cuuint64_t*, const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave,
                                   CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);
EncodeTiledFn encode_tiled() {
  static EncodeTiledFn fn = [] {
    void* f = nullptr;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &f, 12000, cudaEnableDefault, &q) != cudaSuccess ||
        q != cudaDriverEntryPointSuccess) {
      cudaGetLastError();
      return (EncodeTiledFn) nullptr;
    }
    return reinterpret_cast<EncodeTiledFn>(f);
  }();
  return fn;
}

// Tensor map of a slab viewed as D rows of `floats` floats; box: a chunk's elements
// (4 kMarchLanes floats) x brows Nambu rows
cudaError_t encode_slab_map(CUtensorMap* tm, const void* V, int64_t D, int64_t floats, int brows) {
  EncodeTiledFn fn = encode_tiled();
  if (!fn) return cudaErrorNotSupported;
  const cuuint64_t dims[2] = {(cuuint64_t)floats, (cuuint64_t)D};
  const cuuint64_t strides[1] = {(cuuint64_t)(4 * floats)};
  const cuuint32_t box[2] = {4 * kMarchLanes, (cuuint32_t)brows};
  const cuuint32_t estr[2] = {1, 1};
  const CUresult r = fn(tm, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 2, const_cast<void*>(V), dims, strides, box, estr,
                        CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                        CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  return r == CUDA_SUCCESS ? cudaSuccess : cudaErrorInvalidValue;
}
template <int CB>
cudaError_t set_smem_f64(int nx) {
  cudaError_t e = cudaFuncSetAttribute(cheb_step_kernel<double, CB, 0>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       (int)kSmemLimit);
  if (e != cudaSuccess) return e;
  return cudaFuncSetAttribute(cheb_step_kernel<double, CB, 1>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                              (int)kSmemLimit);
}

template <int CB>
cudaError_t launch_f32(const ChebPlan& p, const void* table, const void* Vcur, const void* Vprev, void* Vout,
                       int64_t s0, double2* acc, const double* am, const double* ao, int m, int mode, cudaStream_t s) {
  const dim3 grid((p.ny + p.ylen - 1) / p.ylen, (unsigned)(p.ldv / CB));
  if (mode == 0)
    cheb_step_f32_kernel<CB, 0><<<grid, p.nthreads, p.smem, s>>>(p.nx, p.ny, p.D, p.ldv, p.ylen, (const float2*)table,
                                                                 (const float4*)Vcur, (const float4*)Vprev, (float4*)Vout,
                                                                 s0, acc, am, ao, m);
  else
    cheb_step_f32_kernel<CB, 1><<<grid, p.nthreads, p.smem, s>>>(p.nx, p.ny, p.D, p.ldv, p.ylen, (const float2*)table,
                                                                 (const float4*)Vcur, (const float4*)Vprev, (float4*)Vout,
                                                                 s0, acc, am, ao, m);
  return cudaGetLastError();
}
template <int CB>
cudaError_t set_smem_df(int nx) {
  cudaError_t e = cudaFuncSetAttribute(cheb_step_kernel<DF, CB, 0>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       (int)kSmemLimit);
  if (e != cudaSuccess) return e;
  return cudaFuncSetAttribute(cheb_step_kernel<DF, CB, 1>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                              (int)kSmemLimit);
}
template <int CB>
cudaError_t launch_df(const ChebPlan& p, const void* table, const void* Vcur, const void* Vprev, void* Vout,
                      int64_t s0, double2* acc, const double* am, const double* ao, int m, int mode, cudaStream_t s) {
  const dim3 grid((p.ny + p.ylen - 1) / p.ylen, (unsigned)(p.ldv / CB));
  if (mode == 0)
    cheb_step_kernel<DF, CB, 0><<<grid, p.nthreads, p.smem, s>>>(
        p.nx, p.ny, p.D, p.ldv, p.ylen, (const float4*)table, (const float4*)Vcur, (const float4*)Vprev, (float4*)Vout,
        colmap(p, s0), acc, am, ao, m);
  else
    cheb_step_kernel<DF, CB, 1><<<grid, p.nthreads, p.smem, s>>>(
        p.nx, p.ny, p.D, p.ldv, p.ylen, (const float4*)table, (const float4*)Vcur, (const float4*)Vprev, (float4*)Vout,
        colmap(p, s0), acc, am, ao, m);
  return cudaGetLastError();
}

template <int CB>
cudaError_t launch_f64(const ChebPlan& p, const void* table, const void* Vcur, const void* Vprev, void* Vout,
                       int64_t s0, double2* acc, const double* am, const double* ao, int m, int mode, cudaStream_t s) {
  const dim3 grid((p.ny + p.ylen - 1) / p.ylen, (unsigned)(p.ldv / CB));
  if (mode == 0)
    cheb_step_kernel<double, CB, 0><<<grid, p.nthreads, p.smem, s>>>(
        p.nx, p.ny, p.D, p.ldv, p.ylen, (const double2*)table, (const double2*)Vcur, (const double2*)Vprev, (double2*)Vout,
        colmap(p, s0), acc, am, ao, m);
  else
    cheb_step_kernel<double, CB, 1><<<grid, p.nthreads, p.smem, s>>>(
        p.nx, p.ny, p.D, p.ldv, p.ylen, (const double2*)table, (const double2*)Vcur, (const double2*)Vprev, (double2*)Vout,
        colmap(p, s0), acc, am, ao, m);
  return cudaGetLastError();
}


}  // namespace

namespace {
template <int EL, int NS>
cudaError_t set_smem_march() {
  for (auto fn : {cheb_march_kernel<EL, NS, false, false>, cheb_march_kernel<EL, NS, true, false>,
                  cheb_march_kernel<EL, NS, false, true>, cheb_march_kernel<EL, NS, true, true>}) {
    const cudaError_t e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSmemLimit);
    if (e != cudaSuccess) return e;
  }
  return cudaSuccess;
}
template <int EL, int NS>
cudaError_t march_launch(const MarchPlan& mp, dim3 grid, const MarchMaps& v, const MarchMaps& pr, const MarchArgs& a,
                  const ColMap& cm, bool first, cudaStream_t s) {
  // the failure-path test instantiation only while a test hook is armed
  auto fn = g_step_hook_armed ? (first ? cheb_march_kernel<EL, NS, true, true> : cheb_march_kernel<EL, NS, false, true>)
                              : (first ? cheb_march_kernel<EL, NS, true, false> : cheb_march_kernel<EL, NS, false, false>);
  // Outside graphs the launches are programmatic: a CTA's start runs while the launch
  // before finishes, and the kernel waits for that before it touches anything (37x29,
  // 776 steps: 16.1 -> 14.3 ms; as nodes of a graph, 48x24, the same cost 3%).
  cudaStreamCaptureStatus cap = cudaStreamCaptureStatusNone;
  cudaError_t e = cudaStreamIsCapturing(s, &cap);
  if (e != cudaSuccess) return e;
  cudaLaunchAttribute attr;
  attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr.val.programmaticStreamSerializationAllowed = 1;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = dim3((unsigned)(mp.warps * 32));
  cfg.dynamicSmemBytes = mp.smem;
  cfg.stream = s;
  cfg.attrs = &attr;
  cfg.numAttrs = cap == cudaStreamCaptureStatusNone ? 1 : 0;
  // FP64 rows are bound by the SM's FP64 pipe.  Launched while the grid before finishes, CTAs
  // went two to an SM that was free where others were about to be: with no more CTAs than SMs,
  // each takes more than half of the shared memory, so that they stay apart.  us a step: 24x4
  // 12.8 -> 7.6, 20x5 11.0 -> 7.3, 9x8 10.3 -> 6.2, 8x8 8.4 -> 6.1 (one-step kernel 10.9, 9.1, 8.8, 8.8).
  // (Not in graphs, where they spread by themselves and cells of a batch run side by side.)
  if (EL == kElF64 && cfg.numAttrs == 1 && (int64_t)grid.x * grid.y <= kSMs)
    cfg.dynamicSmemBytes = std::max<size_t>(mp.smem, 116 * 1024);
  return cudaLaunchKernelEx(&cfg, fn, v, pr, a, cm);
}
}  // namespace

namespace {
// band heights of a march launch: as many CTAs per SM as registers and shared memory
// take; a CTA's start (barriers, first copies) costs about five rows (one of double-float),
// and a launch of several steps computes two more rows for every step but the last.
// FP64 rows are bound by the FP64 pipe and long: a start is 0.4 of one (passes of M = 65 with 1.0
// and 0.4, ms: 40x11 5.72 and 4.97, 45x10 6.22 and 5.43, 30x21 11.7 and 10.6, 104x7 14.3 and 13.3).
// Beside the launches of other streams the fewer, higher bands of 1.0 leave room for them:
// batches of 40x11, 45x10, 30x21 cells 18.1 and 19.4 ms, of 45x10 and 36x20 33.2 and 34.2.
int march_per_sm(const MarchPlan& p) {
  return (int)std::max<int64_t>(1, std::min<int64_t>(16 / p.warps, (int64_t)(228 * 1024) / (int64_t)(p.smem + 1024)));
}
int march_bands(const MarchPlan& p, int ny, int64_t ldv, int* out, int maxn) {
  const int per_sm = march_per_sm(p);
  const double start = p.el == kElF32 ? 5.0 + 2.0 * (p.ns - 1) : p.el == kElDF || p.beside ? 1.0 : 0.4;
  return band_rows_candidates(ny, ldv / march_cols(p.el) * p.ntile, out, maxn, per_sm * kSMs, start);
}

// Geometry of a march launch: the whole lattice row per CTA where its threads and rings
// fit, else the fewest equal tiles that do; the deepest rings that fit shared
// memory (several steps: eight rows each), and the band height of the wave model.
// (Two steps in tiles of 26 sites do not fit: 104x104 in five tiles of 21, M = 65, 96.6 ms, one
// step 113.2; 180x60 in eight of 23, M = 33, 53.0 and 56.3.)
MarchPlan plan_march(int nx, int ny, int64_t ldv, int ns, int band_rows, int el = kElF32, bool beside = false) {
  MarchPlan p;
  p.el = el;
  p.beside = beside;
  constexpr int nv = kMarchLanes;
  auto warps = [&](int tx, bool full) {
    int n = 2;  // the producer and the moment sums
    for (int s = 0; s < ns; ++s) n += ((full ? nx : tx + 2 * (ns - 1 - s)) * nv + 31) / 32;
    return n;
  };
  // A set of rows is issued once the last stage has finished the row `lag` before it;
  // single step: row i + 2 of V_m then takes the place of one that the stage and the
  // sums have done with in a ring of lag + 2 rows
  // (a row of double-float or FP64 takes as long as its copy: four are enough)
  auto fits = [&](int tx, bool full) {
    p.warps = warps(tx, full);
    if (p.warps * 32 > kMarchThreads) return false;
    p.wrow = full ? nx : tx + 2 * ns;
    p.crowb = (p.wrow * march_entry_bytes(el) + 127) / 128 * 128;
    for (int lag = el == kElF32 ? 8 : 4; lag >= (ns == 1 ? 2 : 8); --lag) {
      p.lag = lag;
      p.rv = ns == 1 ? lag + 2 : kMarchRows;
      p.rp = p.rc = ns == 1 ? lag : kMarchRows;
      p.rs = kMarchRows;
      p.smem = 32 * (size_t)nv * p.wrow * (p.rv + p.rp + (ns - 1) * p.rs) + (size_t)p.crowb * p.rc +
               8 * (size_t)kMarchBars * (1 + ns) + 16;
      if (p.smem <= kSmemLimit) return true;
    }
    return false;
  };
  if (fits(nx, true)) {
    p.full = 1;
    p.ntile = 1;
    p.tx = nx;
  } else {
    for (int nt = 2; nt <= nx && p.ntile == 0; ++nt) {
      const int tx = (nx + nt - 1) / nt;
      const int last = nx - (nt - 1) * tx;
      if (last < ns || tx < ns || !fits(tx, false)) continue;
      p.ntile = nt;
      p.tx = tx;
    }
    if (p.ntile == 0) return p;
  }
  p.ns = ns;
  int best = ny;
  march_bands(p, ny, ldv, &best, 1);
  p.ylen = band_rows > 0 ? std::min(band_rows, ny) : best;
  return p;
}
}  // namespace

namespace {
cudaError_t march_prepare(const MarchPlan& mp) {
  if (mp.el == kElDF) return set_smem_march<kElDF, 1>();
  if (mp.el == kElF64) return set_smem_march<kElF64, 1>();
  return mp.ns == 1 ? set_smem_march<kElF32, 1>() : mp.ns == 2 ? set_smem_march<kElF32, 2>() : set_smem_march<kElF32, 3>();
}
}  // namespace

cudaError_t encode_slab_maps(const ChebPlan& p, const MarchPlan& mp, const void* V, SlabMaps* out, bool as_v,
                             bool as_p) {
  static_assert(sizeof(MarchMaps) == 3 * 128 && sizeof(SlabMaps::v) == sizeof(MarchMaps), "SlabMaps layout");
  auto encode = [&](unsigned char* to, int halo) {  // boxes of a tile with `halo` sites on each side
    const int sites[3] = {mp.full ? mp.tx : mp.tx + 2 * halo, mp.full ? mp.tx : mp.tx + halo, std::max(1, halo)};
    for (int k = 0; k < (mp.full ? 1 : 3); ++k) {
      CUtensorMap t;
      const cudaError_t e = encode_slab_map(&t, V, p.D, (mp.el == kElF32 ? 2 : 4) * p.ldv, 2 * sites[k]);
      if (e != cudaSuccess) return e;
      memcpy(to + 128 * k, &t, 128);
    }
    return cudaSuccess;
  };
  cudaError_t e = cudaSuccess;
  if (as_v) e = encode(out->v, mp.ns);
  if (as_p && e == cudaSuccess) e = encode(out->p, mp.ns - 1);
  return e;
}

size_t march_table_bytes(const MarchPlan& mp, int ny) { return (size_t)mp.crowb * ny * mp.ntile; }

cudaError_t launch_march(const ChebPlan& p, const MarchPlan& mp, const void* table, const SlabMaps& cur,
                         const SlabMaps& prev, void* outa, void* outb, int64_t s0, double2* acc, const double* am,
                         const double* ao, int m, bool first, cudaStream_t s, int64_t col0, int64_t cols) {
  MarchArgs a;
  a.nx = p.nx;
  a.ny = p.ny;
  a.D = p.D;
  a.ldq = mp.el == kElF32 ? p.ldv / 2 : p.ldv;  // 16-byte elements of a slab row
  a.tx = mp.tx;
  a.ntile = mp.ntile;
  a.full = mp.full;
  a.ylen = mp.ylen;
  a.wrow = mp.wrow;
  a.lag = mp.lag;
  a.rp = mp.rp;
  a.rv = mp.rv;
  a.rs = mp.rs;
  a.rc = mp.rc;
  a.rowb = mp.wrow * 32 * kMarchLanes;
  a.crowb = mp.crowb;
  a.table = (const float4*)table;
  a.outa = (float4*)outa;
  a.outb = (float4*)outb;
  a.acc = acc;
  a.am = am;
  a.ao = ao;
  a.m = m;
  a.chunk0 = (int)(col0 / march_cols(mp.el));
  a.grow = 16 * 2 * (int64_t)p.nx * a.ldq;
  MarchMaps v, pr;
  memcpy(&v, cur.v, sizeof(v));
  memcpy(&pr, prev.p, sizeof(pr));
  const dim3 grid((unsigned)(((p.ny + mp.ylen - 1) / mp.ylen) * mp.ntile), (unsigned)((cols > 0 ? std::min(cols, p.ldv - col0) : p.ldv) / march_cols(mp.el)));
  const ColMap cm = colmap(p, s0);
  if (mp.el == kElDF) return march_launch<kElDF, 1>(mp, grid, v, pr, a, cm, first, s);
  if (mp.el == kElF64) return march_launch<kElF64, 1>(mp, grid, v, pr, a, cm, first, s);
  if (mp.ns == 1) return march_launch<kElF32, 1>(mp, grid, v, pr, a, cm, first, s);
  if (mp.ns == 2) return march_launch<kElF32, 2>(mp, grid, v, pr, a, cm, first, s);
  return march_launch<kElF32, 3>(mp, grid, v, pr, a, cm, first, s);
}

// Wave model of a launch: ctas x nb CTAs (nb bands of ceil(ny/nb) rows) run
// `slots` at a time in ceil(CTAs / slots) waves; a CTA costs its rows and `extra`
// more (two halo rows of V_m, one of the three vectors a row streams; for the
// march kernel its start).  Returns the band heights of the cheapest choices.
int band_rows_candidates(int ny, int64_t ctas, int* out, int maxn, int slots, double extra) {
  std::vector<std::pair<double, int>> cost;
  int last = -1;
  for (int nb = 1; nb <= ny; ++nb) {
    const int rows = (ny + nb - 1) / nb;
    if (rows == last) continue;
    last = rows;
    const int bands = (ny + rows - 1) / rows;
    const int64_t waves = (ctas * bands + slots - 1) / slots;
    cost.push_back({(double)waves * (rows + extra), rows});
  }
  std::stable_sort(cost.begin(), cost.end(), [](const std::pair<double, int>& a, const std::pair<double, int>& b) {
    return a.first < b.first;
  });
  int n = 0;
  for (size_t k = 0; k < cost.size() && n < maxn; ++k) out[n++] = cost[k].second;
  return n;
}

ChebPlan plan_cheb(int nx, int ny, int64_t width, int precision, int cb_request, int band_rows, int steps,
                   bool split, bool beside) {
  ChebPlan p;
  p.nx = nx;
  p.ny = ny;
  p.D = 2 * (int64_t)nx * ny;
  p.nthreads = 512;
  p.cb = 0;
  p.ldv = 0;
  p.sub = 0;
  p.smem = 0;
  p.ylen = ny;
  p.js = 0;
  p.probe_p = 0;
  p.probe_seed = 0;
  p.xi = nullptr;
  p.rec = nullptr;
  p.raw = 0;
  // widest column chunk that fits shared memory (FP32: 16 columns, FP64: 8);
  // FP32 also needs every thread to own at most two sites of a lattice row
  const int cands32[4] = {16, 8, 4, 2};
  const int cands64[4] = {8, 4, 2, 1};
  const int* c = precision == KPM_FP32 ? cands32 : cands64;
  if (cb_request > 0 && cb_request < c[3]) cb_request = c[3];
  for (int k = 0; k < 4; ++k) {
    if (cb_request > 0 && c[k] > cb_request) continue;
    size_t sm;
    if (precision == KPM_FP32) {
      sm = c[k] == 16 ? smem_f32<16>(nx) : c[k] == 8 ? smem_f32<8>(nx) : c[k] == 4 ? smem_f32<4>(nx) : smem_f32<2>(nx);
      const int xstep = p.nthreads / (c[k] / 2);
      if (nx > 2 * xstep) continue;
    } else {
      sm = c[k] == 8 ? smem_f64<8>(nx) : c[k] == 4 ? smem_f64<4>(nx) : c[k] == 2 ? smem_f64<2>(nx) : smem_f64<1>(nx);
    }
    if (sm <= kSmemLimit) {
      p.cb = c[k];
      p.smem = sm;
      break;
    }
  }
  if (steps > 0 && p.cb > 0) {
    // the march kernel, for every lattice whose row the one-step kernels take; its chunks are
    // fixed, cb_request narrows the one-step kernels' only (16x16 FP64, M = 128: 3.56 ms,
    // one-step kernel 4.72 in chunks of 8 columns, 8.82 of 4, 15.3 of 2; 48x24 FP32: 2.27, and
    // 7.85 of 8, 12.3 of 4)
    const int el = precision == KPM_FP32 ? kElF32 : precision == KPM_DF64 ? kElDF : kElF64;
    p.cb = march_cols(el);
    p.ldv = (width + p.cb - 1) / p.cb * p.cb;
    p.sub = split && steps == 1 && el == kElF32 ? march_columns(nx, ny, p.ldv) : p.ldv;
    p.m1 = plan_march(nx, ny, p.sub, 1, band_rows, el, beside);
    p.mk = steps > 1 && el == kElF32 ? plan_march(nx, ny, p.ldv, steps, band_rows) : p.m1;
    if (p.mk.ns == 0) p.mk = p.m1;
    p.ylen = p.mk.ylen;
    p.nthreads = 32 * p.mk.warps;
    p.smem = p.mk.smem;
    return p;
  }
  if (p.cb == 0) return p;
  p.ldv = (width + p.cb - 1) / p.cb * p.cb;
  // band height of the one-step kernels: the caller's, else the best of the
  // wave model (the last wave of a launch as full as the halo rows allow)
  const int64_t chunks = p.ldv / p.cb;
  int best_rows = ny;
  band_rows_candidates(ny, chunks, &best_rows, 1);
  p.ylen = band_rows > 0 ? std::min(band_rows, ny) : best_rows;
  return p;
}


namespace {
// us per step of single steps over the cheapest number of parts of a slab (*cols columns).
// Above L2 the single steps of a whole slab run at the memory's rate (6.3 TB/s of copies).
// Parts that fit L2 do not, but pay the launches' starts, and a part's CTAs fill the SMs
// more or less well: rows of 0.0485 us per stage warp (48x24, 64x32, 64x64: the same within
// 5%).  Measured, whole slab against parts: 40x40 45.9 -> 39 (3 parts), 64x32 75 -> 61 (4),
// 64x64 257 -> 217 (14); up to sixteen parts, beyond which launches only add up
// (80x80 603 -> 601, 27 parts).
double parts_us(int nx, int ny, int64_t width, int64_t* cols) {
  const int64_t D = 2 * (int64_t)nx * ny, cb = march_cols(kElF32), chunks = (width + cb - 1) / cb;
  *cols = chunks * cb;
  double cost = 24.0 * (double)D * (double)width / 6.3e6;
  const MarchPlan p = plan_march(nx, ny, width, 1, 0);
  if (p.ns == 0 || 16 * D * width <= kMarchL2) return cost;
  const int per_sm = march_per_sm(p);
  const double row_us = 0.0485 * (p.warps - 2) * per_sm;
  for (int n = 2; n <= 16 && n <= chunks; ++n) {
    const int64_t c = (chunks + n - 1) / n;
    if (16 * D * cb * c > kMarchL2) continue;
    int rows = ny;
    march_bands(p, ny, c * cb, &rows, 1);
    const int64_t ctas = c * p.ntile * ((ny + rows - 1) / rows);
    const double us = n * row_us * (rows + 5.0) * (double)((ctas + per_sm * kSMs - 1) / (per_sm * kSMs));
    if (us < cost) {
      cost = us;
      *cols = c * cb;
    }
  }
  return cost;
}
}  // namespace

// Two steps per launch where the slabs stream from memory and the tile fills its
// warps: 100x100 (13 or 14 stage warps) 1248 against 1457 us per step, a 2500-column
// slab of it 180 against 213; 64x64, whose tiles of 22 sites fill 11.5, 275 against 266.
// Not where parts that fit L2 are cheaper than its 3.3 ps per row-column (60x60 to
// 100x100: 3.1 to 3.4; 48x48, 3.75: 79.7 against 70 us in four parts).
int march_steps(int nx, int ny, int64_t width) {
  const int64_t D = 2 * (int64_t)nx * ny;
  if (16 * D * width <= kMarchL2) return 1;
  const MarchPlan p = plan_march(nx, ny, width, 2, 0);
  int64_t cols;
  return p.ns == 2 && p.warps >= 15 && 3.3e-6 * (double)D * (double)width < parts_us(nx, ny, width, &cols) ? 2 : 1;
}

int64_t march_columns(int nx, int ny, int64_t width) {
  int64_t cols;
  parts_us(nx, ny, width, &cols);
  return cols;
}

int plan_band_candidates(const ChebPlan& p, int* out, int maxn) {
  if (p.mk.ns) return march_bands(p.mk, p.ny, p.mk.ns == 1 ? p.sub : p.ldv, out, maxn);
  return band_rows_candidates(p.ny, p.ldv / p.cb, out, maxn);
}

size_t table_bytes_per_site(int precision) { return (size_t)kCoef * (precision == KPM_FP32 ? 8 : 16); }

cudaError_t cheb_prepare(const ChebPlan& p, int precision) {
  if (p.mk.ns) {
    cudaError_t e = march_prepare(p.mk);
    if (e == cudaSuccess) e = march_prepare(p.m1);
    return e;
  }
  if (precision == KPM_FP32) {
    switch (p.cb) {
      case 16: return set_smem_f32<16>(p.nx);
      case 8: return set_smem_f32<8>(p.nx);
      case 4: return set_smem_f32<4>(p.nx);
      case 2: return set_smem_f32<2>(p.nx);
    }
  } else if (precision == KPM_DF64) {
    switch (p.cb) {
      case 8: return set_smem_df<8>(p.nx);
      case 4: return set_smem_df<4>(p.nx);
      case 2: return set_smem_df<2>(p.nx);
      case 1: return set_smem_df<1>(p.nx);
    }
  } else {
    switch (p.cb) {
      case 8: return set_smem_f64<8>(p.nx);
      case 4: return set_smem_f64<4>(p.nx);
      case 2: return set_smem_f64<2>(p.nx);
      case 1: return set_smem_f64<1>(p.nx);
    }
  }
  return cudaErrorInvalidValue;
}

cudaError_t launch_cheb_init(const ChebPlan& p, int precision, void* V0, int64_t s0, double2* acc, const double* am,
                             const double* ao, cudaStream_t s) {
  const int64_t total = p.D * p.ldv;
  const int grid = (int)std::min<int64_t>((total + 255) / 256, 8 * kSMs * 4);
  if (precision == KPM_FP32)
    cheb_init_f32_kernel<<<grid, 256, 0, s>>>(p.D, p.ldv, p.nx, (float4*)V0, colmap(p, s0));
  else if (precision == KPM_DF64)
    cheb_init_df_kernel<<<grid, 256, 0, s>>>(p.D, p.ldv, p.nx, (float4*)V0, colmap(p, s0));
  else
    cheb_init_f64_kernel<<<grid, 256, 0, s>>>(p.D, p.ldv, p.nx, (double2*)V0, colmap(p, s0));
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  const int ga = (int)std::max<int64_t>(1, std::min<int64_t>((p.ldv * kSlots + 255) / 256, 4 * kSMs));
  cheb_init_acc_kernel<<<ga, 256, 0, s>>>(p.D, p.ldv, p.nx, colmap(p, s0), acc, am, ao);
  return cudaGetLastError();
}

cudaError_t launch_cheb_step(const ChebPlan& p, int precision, const void* table, const void* Vcur, void* Vout,
                             int64_t s0, double2* acc, const double* am, const double* ao, int m, int mode,
                             cudaStream_t s, const void* Vprev) {
  if (!Vprev) Vprev = Vout;
  if (p.m1.ns) {
    SlabMaps cur, prev;
    cudaError_t e = encode_slab_maps(p, p.m1, Vcur, &cur, true, false);
    if (e == cudaSuccess) e = encode_slab_maps(p, p.m1, Vprev, &prev, false, true);
    if (e != cudaSuccess) return e;
    return launch_march(p, p.m1, table, cur, prev, nullptr, Vout, s0, acc, am, ao, m, mode == 0, s);
  }
  if (precision == KPM_FP32) {
    switch (p.cb) {
      case 16: return launch_f32<16>(p, table, Vcur, Vprev, Vout, s0, acc, am, ao, m, mode, s);
      case 8: return launch_f32<8>(p, table, Vcur, Vprev, Vout, s0, acc, am, ao, m, mode, s);
      case 4: return launch_f32<4>(p, table, Vcur, Vprev, Vout, s0, acc, am, ao, m, mode, s);
      case 2: return launch_f32<2>(p, table, Vcur, Vprev, Vout, s0, acc, am, ao, m, mode, s);
    }
  } else if (precision == KPM_DF64) {
    switch (p.cb) {
      case 8: return launch_df<8>(p, table, Vcur, Vprev, Vout, s0, acc, am, ao, m, mode, s);
      case 4: return launch_df<4>(p, table, Vcur, Vprev, Vout, s0, acc, am, ao, m, mode, s);
      case 2: return launch_df<2>(p, table, Vcur, Vprev, Vout, s0, acc, am, ao, m, mode, s);
      case 1: return launch_df<1>(p, table, Vcur, Vprev, Vout, s0, acc, am, ao, m, mode, s);
    }
  } else {
    switch (p.cb) {
      case 8: return launch_f64<8>(p, table, Vcur, Vprev, Vout, s0, acc, am, ao, m, mode, s);
      case 4: return launch_f64<4>(p, table, Vcur, Vprev, Vout, s0, acc, am, ao, m, mode, s);
      case 2: return launch_f64<2>(p, table, Vcur, Vprev, Vout, s0, acc, am, ao, m, mode, s);
      case 1: return launch_f64<1>(p, table, Vcur, Vprev, Vout, s0, acc, am, ao, m, mode, s);
    }
  }
  return cudaErrorInvalidValue;
}

cudaError_t read_step_fault(unsigned int* out) {
  return cudaMemcpyFromSymbol(out, g_step_fault, sizeof(unsigned int));
}

cudaError_t clear_step_fault() {
  const unsigned int zero = 0u;
  return cudaMemcpyToSymbol(g_step_fault, &zero, sizeof(zero));
}

cudaError_t set_step_failure_test(int drop_copies, uint64_t wait_limit_ns) {
  cudaError_t e = cudaMemcpyToSymbol(g_drop_copy, &drop_copies, sizeof(int));
  if (e != cudaSuccess) return e;
  const unsigned long long lim = wait_limit_ns ? wait_limit_ns : kWaitLimitNs;
  e = cudaMemcpyToSymbol(g_wait_limit_ns, &lim, sizeof(lim));
  g_step_hook_armed = drop_copies > 0 || wait_limit_ns != 0;
  return e;
}

cudaError_t launch_probe_phases(const ChebPlan& p, double2* xi_conj, cudaStream_t s) {
  const int grid = (int)std::max<int64_t>(1, std::min<int64_t>((p.D + 255) / 256, 4 * kSMs));
  probe_phase_kernel<<<grid, 256, 0, s>>>(p.D, p.probe_seed, xi_conj);
  return cudaGetLastError();
}

cudaError_t launch_probe_sums(const ChebPlan& p, const void* Va, const void* Vb, int64_t s0, double2* acc,
                              const double* am, const double* ao, int m, cudaStream_t s) {
  const int64_t n = p.D * kSlots;
  const int grid = (int)std::max<int64_t>(1, std::min<int64_t>((n + 255) / 256, 8 * kSMs));
  probe_sums_kernel<<<grid, 256, 0, s>>>(p.nx, p.ny, (int)p.D, p.ldv, (const float4*)Va, (const float4*)Vb,
                                         colmap(p, s0), acc, am, ao, m);
  return cudaGetLastError();
}

cudaError_t launch_cheb_gather(const ChebPlan& p, int precision, const void* V, int64_t s0, double2* acc,
                               const double* am, const double* ao, int m, cudaStream_t s) {
  const int64_t width = p.ldv;
  const int grid = (int)std::max<int64_t>(1, std::min<int64_t>((width * kSlots + 255) / 256, 4 * kSMs));
  if (precision == KPM_FP32)
    cheb_gather_kernel<1><<<grid, 256, 0, s>>>(p.nx, p.ny, p.D, p.ldv, width, V, colmap(p, s0), acc, am, ao, m);
  else if (precision == KPM_DF64)
    cheb_gather_kernel<2><<<grid, 256, 0, s>>>(p.nx, p.ny, p.D, p.ldv, width, V, colmap(p, s0), acc, am, ao, m);
  else
    cheb_gather_kernel<0><<<grid, 256, 0, s>>>(p.nx, p.ny, p.D, p.ldv, width, V, colmap(p, s0), acc, am, ao, m);
  return cudaGetLastError();
}

size_t persist_smem_bytes(int nx, int ny) { return persist_smem(nx, (ny + kPClu - 1) / kPClu); }
int persist_columns() { return kPCB; }

cudaError_t persist_prepare(size_t smem, int* max_clusters) {
  if (smem > kSmemLimit) return cudaErrorInvalidValue;
  cudaError_t e = cudaFuncSetAttribute(cheb_persist_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       (int)kSmemLimit);
  if (e != cudaSuccess) return e;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(kPClu, 1, 1);
  cfg.blockDim = dim3(512, 1, 1);
  cfg.dynamicSmemBytes = smem;
  int n = 0;
  e = cudaOccupancyMaxActiveClusters(&n, cheb_persist_kernel, &cfg);
  if (e != cudaSuccess) return e;
  *max_clusters = n;
  return n > 0 ? cudaSuccess : cudaErrorInvalidConfiguration;
}

size_t persist_exchange_bytes(int nclusters, int nx_max) {
  return sizeof(float4) * (size_t)nclusters * kPClu * 4 * (size_t)nx_max * 2 * kPNV;
}

cudaError_t launch_cheb_persist(const PCell* cells, const PItem* items, int nitems, int* counter, int M, int nclusters,
                                size_t smem, void* xbuf, int nx_max, cudaStream_t s) {
  cheb_persist_kernel<<<dim3(kPClu * nclusters), 512, smem, s>>>(cells, items, nitems, counter, M, (float4*)xbuf,
                                                                 nx_max * 2 * kPNV);
  return cudaGetLastError();
}

}  // namespace kpm

