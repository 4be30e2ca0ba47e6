// Fused stream-collide kernel of the MRT path, written around opposite-velocity
// pairs.
//
// The collisions reduce to moments (see kernels.cuh): with degree-2 moments
// relaxed at omega and all higher ones at 1 (g), or degrees 1 and 2 at
// omega_phi and higher at 1 (h), every post-collision population is a
// quadratic polynomial of its velocity,
//   f+_i / w_i = alpha + beta . c_i + c_i . Gamma . c_i,
// so a pair (c, -c) shares E = alpha + c.Gamma.c and differs only in the sign
// of L = beta . c.
//   g:  alpha = p* - 3/2 u.u - a2 tr(Pi^d)/3,  beta = 3 u + 3/2 F / rho,
//       Gamma = 9/2 u u^T + a2 Pi^d,           a2 = 9/2 (1 - omega)
//   h:  alpha = phi - a2 tr(Pi^dh)/3,           beta = 3 phi u + a1 J^d + (1 - omega_phi/2) theta n,
//       Gamma = a2 Pi^dh,                       a1 = 3 (1 - omega_phi), a2 = 9/2 (1 - omega_phi)
// For the shifted FP16 format the coefficients are pre-scaled by the format's
// power-of-two factor and alpha_h carries the shift, so a stored value is
// E +- L without a per-population multiply by 1 / w.
//
// Neighbour addressing: per cell, the cell-index offsets of the -1 / +1
// neighbours along each axis (periodic wrap folded in) and whether the link
// crosses a no-slip face; offsets of a direction are sums of these, fixed at
// compile time inside the unrolled loops.
#pragma once

#include "kernels.cuh"
#include "tma.cuh"
#include "vec.cuh"

#ifndef PFL_STEP_THREADS
#define PFL_STEP_THREADS 128
#endif
#ifndef PFL_STEP_MINB
#define PFL_STEP_MINB 4
#endif
// Resident blocks of 256 threads per SM the fused step is compiled for.  Three
// (80 registers) against two (128) and four (64, with spills) on a 256x192x256
// impact: FP16S 15.7, 14.5 and 14.5 GLUPS; FP32 14.4, 14.4 and 6.2 (its L1
// prefetch then overflows).  FP64, bound by the FP64 units, keeps two.
#ifndef PFL_ZM_MINB
#define PFL_ZM_MINB 3
#endif
#ifndef PFL_ZM_MINB_FP64
#define PFL_ZM_MINB_FP64 2
#endif
// L1 prefetch of the g populations of the plane the fused FP32 step collides
// next, issued one plane ahead right after the plane barrier (1; 0 = none), in
// tiles without tensor copies.  us per step with and without: drop 96^3 (32 x 8)
// 59.7 and 61.7, bubble 96x250x99 169.3 and 177.4; bubble 61x183x61 and the Taylor
// tubes equal within 0.5 %; drop 32^3, in L2 anyway, 5.71 and 5.01.  FP16S (issue
// bound) lost 5 %, single-plane lattices 8-10 % and the D3Q27 phase field 1 %, so
// they take none.  (The h populations of the plane filled next as well: 15.0 ->
// 12.5 GLUPS on a 256x192x256 impact.)
#ifndef PFL_ZM_PREFETCH
#define PFL_ZM_PREFETCH 1
#endif
// Programmatic dependent launch of the fused step (1; 0 = plain launches):
// the host launches each step with programmatic stream serialisation, so the
// next step's blocks are scheduled while the last blocks of the previous one
// finish; every block waits (griddepcontrol.wait, a no-op without the launch
// attribute) for the previous grid's completion before its first global access.
// 200x400 wave: FP16S 11.3 -> 12.0 GLUPS, FP32 11.6 -> 12.3; the 3-D bubble is
// unchanged.  Releasing the dependents early (launch_dependents right after
// the wait) lost 6-13 %: waiting blocks then hold the SMs' block slots.
#ifndef PFL_ZM_PDL
#define PFL_ZM_PDL 1
#endif
namespace pfl {

// Exact q = n / d for 32-bit unsigned n and a divisor fixed for the launch
// (division by an invariant integer using multiplication, Granlund and
// Montgomery 1994, round-up multiplier form): with l = ceil(log2 d) and
// m = floor(2^32 (2^l - d) / d) + 1, t = mulhi(m, n), q = (t + ((n - t) >> s1)) >> s2,
// s1 = min(l, 1), s2 = max(l - 1, 0).
struct FastDiv {
  unsigned d, m;
  int s1, s2;
};

inline FastDiv make_fastdiv(unsigned d) {
  FastDiv f;
  f.d = d;
  int l = 0;
  while ((1ull << l) < d) ++l;
  f.m = (unsigned)(((1ull << 32) * ((1ull << l) - d)) / d + 1);
  f.s1 = l < 1 ? l : 1;
  f.s2 = l - 1 > 0 ? l - 1 : 0;
  return f;
}

__host__ __device__ __forceinline__ unsigned fdiv(unsigned n, const FastDiv& f) {
#ifdef __CUDA_ARCH__
  const unsigned t = __umulhi(n, f.m);
#else
  const unsigned t = (unsigned)(((unsigned long long)n * f.m) >> 32);
#endif
  return (t + ((n - t) >> f.s1)) >> f.s2;
}

// Host check of the divider on the boundary cases and a spread of numerators.
inline bool fastdiv_ok(unsigned d, unsigned nmax) {
  const FastDiv f = make_fastdiv(d);
  const unsigned probe[] = {0u, 1u, d - 1, d, d + 1, 2 * d - 1, 2 * d, nmax - 1, nmax};
  for (unsigned n : probe)
    if (n <= nmax && fdiv(n, f) != n / d) return false;
  unsigned long long x = 0x9e3779b97f4a7c15ull;
  for (int k = 0; k < 4096; ++k) {
    x ^= x << 13;
    x ^= x >> 7;
    x ^= x << 17;
    const unsigned n = (unsigned)(x % ((unsigned long long)nmax + 1));
    if (fdiv(n, f) != n / d) return false;
  }
  return true;
}

// Launch geometry of the 32-bit-indexed kernels (27 N < 2^32).
struct Geo32 {
  unsigned nx, ny, nz, N;
  FastDiv dx, dy;   // division by nx and by ny
  int wall[3];
};

struct AxisOff {
  int om, op;    // population neighbour offsets of x-1, x+1
  bool vm, vp;   // the link to x-1 / x+1 stays inside (false behind a wall)
  int sm, sp;    // phi-stencil offsets (mirror at walls)
};

__device__ __forceinline__ AxisOff axis_off(unsigned x, unsigned n, int stride, int wall) {
  AxisOff a;
  if (wall) {
    a.vm = x > 0;
    a.vp = x + 1 < n;
    a.om = -stride;
    a.op = stride;
    a.sm = a.vm ? a.om : 0;
    a.sp = a.vp ? a.op : 0;
  } else {
    a.vm = a.vp = true;
    a.om = x > 0 ? -stride : (int)(n - 1) * stride;
    a.op = x + 1 < n ? stride : -(int)(n - 1) * stride;
    a.sm = a.om;
    a.sp = a.op;
  }
  return a;
}


// Blocked links of a cell next to solid cells: bit (cx+1) + 3(cy+1) + 9(cz+1)
// is set when the neighbour in direction c is solid; bit 13 (the rest
// direction) marks the cell itself solid.  Zero away from solids, and a
// compile-time zero in kernels built without solids.
__host__ __device__ constexpr unsigned link_bit(int cx, int cy, int cz) {
  return 1u << ((cx + 1) + 3 * (cy + 1) + 9 * (cz + 1));
}
constexpr unsigned SOLID_SELF = 1u << 13;

// seed of the FP16 stochastic rounding of step t (Fibonacci hashing of t)
__host__ __device__ __forceinline__ unsigned step_seed_of(unsigned long long t) {
  return (unsigned)(t * 0x9E3779B97F4A7C15ull >> 32);
}

struct CellOff {
  AxisOff X, Y, Z;
  unsigned blk = 0;  // blocked links (solid neighbours)
  // population offset and validity of direction (cx, cy, cz): a link leaving
  // through a no-slip face or into a solid cell is bounced back half-way
  __device__ __forceinline__ int off(int cx, int cy, int cz) const {
    return (cx < 0 ? X.om : cx > 0 ? X.op : 0) + (cy < 0 ? Y.om : cy > 0 ? Y.op : 0) +
           (cz < 0 ? Z.om : cz > 0 ? Z.op : 0);
  }
  __device__ __forceinline__ bool valid(int cx, int cy, int cz) const {
    return (cx < 0 ? X.vm : cx > 0 ? X.vp : true) && (cy < 0 ? Y.vm : cy > 0 ? Y.vp : true) &&
           (cz < 0 ? Z.vm : cz > 0 ? Z.vp : true) && !(blk & link_bit(cx, cy, cz));
  }
  __device__ __forceinline__ int soff(int cx, int cy, int cz) const {
    return (cx < 0 ? X.sm : cx > 0 ? X.sp : 0) + (cy < 0 ? Y.sm : cy > 0 ? Y.sp : 0) +
           (cz < 0 ? Z.sm : cz > 0 ? Z.sp : 0);
  }
};

// Raw stored value as the arithmetic type (FP16: the stored number, unscaled).
template <int PREC>
__device__ __forceinline__ typename Store<PREC>::R raw(typename Store<PREC>::S v) {
  if constexpr (PREC == 2)
    return __half2float(v);
  else
    return v;
}
template <int PREC>
__device__ __forceinline__ typename Store<PREC>::S pack(typename Store<PREC>::R v) {
  if constexpr (PREC == 2)
    return __float2half_rn(v);
  else
    return v;
}

// Stochastic rounding for the FP16 stores of the step.  Round-to-nearest
// repeats the same error every step where a field changes slowly, and those
// errors add up linearly in time (mass drift of phi); rounding up with the
// probability given by the discarded bits makes every store unbiased.  The
// random bits come from a per-cell stream: the 32-bit hash of (cell, step)
// (lowbias32 by C. Wellons) seeds a linear congruential sequence (Numerical
// Recipes constants), whose top 13 bits are added below the FP16 mantissa of
// the FP32 value before truncation toward zero.
__device__ __forceinline__ unsigned hash32(unsigned x) {
  x ^= x >> 16;
  x *= 0x7feb352du;
  x ^= x >> 15;
  x *= 0x846ca68bu;
  x ^= x >> 16;
  return x;
}

struct Dither {
  unsigned r;
  __device__ __forceinline__ unsigned next() {
    r = r * 1664525u + 1013904223u;
    return r >> 19;
  }
  // 32 bits for a pair: the state's high half, and the low half xor-ed with
  // the high one (the low bits of a power-of-two LCG have short periods)
  __device__ __forceinline__ unsigned next32() {
    r = r * 1664525u + 1013904223u;
    return r ^ (r >> 16);
  }
};

// Stochastic rounding of a pair in one conversion (sm_100-family
// cvt.rs.f16x2.f32): A lands in the high half and is rounded with the high 16
// random bits, B in the low half with the low 16; each rounds away from zero
// with the probability of its discarded fraction (an unbiased rounding, like
// pack_sr).  PFL_FP16S_HWSR = 0 keeps pack_sr for every store.
#ifndef PFL_FP16S_HWSR
#define PFL_FP16S_HWSR 1
#endif
__device__ __forceinline__ void pack2_sr(float A, float B, unsigned bits, __half& a, __half& b) {
  unsigned d;
  asm("cvt.rs.f16x2.f32 %0, %1, %2, %3;" : "=r"(d) : "f"(A), "f"(B), "r"(bits));
  a = __ushort_as_half((unsigned short)(d >> 16));
  b = __ushort_as_half((unsigned short)(d & 0xffffu));
}

template <int PREC>
__device__ __forceinline__ typename Store<PREC>::S pack_sr(typename Store<PREC>::R v, Dither& d) {
  if constexpr (PREC == 2) {
    const unsigned b = __float_as_uint(v) + d.next();
    return __float2half_rz(__uint_as_float(b));
  } else {
    return v;
  }
}

__device__ __forceinline__ void cell_off(const Geo32& geo, unsigned c, CellOff& o) {
  const unsigned yz = fdiv(c, geo.dx);
  const unsigned x = c - yz * geo.nx;
  const unsigned z = fdiv(yz, geo.dy);
  const unsigned y = yz - z * geo.ny;
  o.X = axis_off(x, geo.nx, 1, geo.wall[0]);
  o.Y = axis_off(y, geo.ny, (int)geo.nx, geo.wall[1]);
  o.Z = axis_off(z, geo.nz, (int)(geo.nx * geo.ny), geo.wall[2]);
}

// Load the pair (i: direction c, oi: direction -c) arriving at `cell`.
// a, b: raw stored values; fa, fb: the cells that wrote them.  Indices are
// 32-bit (unsigned wrap-around arithmetic; the final index is in range).
template <int PREC, int READ_ODD, class Off>
__device__ __forceinline__ void load_pair(const typename Store<PREC>::S* __restrict__ f, unsigned N, unsigned cell,
                                          const Off& o, int i, int oi, int cx, int cy, int cz,
                                          typename Store<PREC>::R& a, typename Store<PREC>::R& b, unsigned& fa,
                                          unsigned& fb) {
  const bool vmc = o.valid(-cx, -cy, -cz), vc = o.valid(cx, cy, cz);
  const unsigned nm = cell + (unsigned)o.off(-cx, -cy, -cz), np = cell + (unsigned)o.off(cx, cy, cz);
  fa = vmc ? nm : cell;
  fb = vc ? np : cell;
  if (!READ_ODD) {
    a = raw<PREC>(f[(unsigned)i * N + cell]);
    b = raw<PREC>(f[(unsigned)oi * N + cell]);
  } else {
    a = raw<PREC>(f[vmc ? (unsigned)oi * N + nm : (unsigned)i * N + cell]);
    b = raw<PREC>(f[vc ? (unsigned)i * N + np : (unsigned)oi * N + cell]);
  }
}


// ---------------------------------------------------------------------------
// Moments (FP64).  A population set is a tensor product (D3Q27, D2Q9) or its axis
// and corner part (D3Q15), so the moments up to second order fall out of sums and
// differences along x, then y, then z: 66 operations for the ten moments of
// D3Q27 against 111 by opposite pairs, 39 against 63 for D3Q15.  The first moments
// along y and z are differences of sums at the size of p*, so by themselves they
// round at that size (5e-17 off at p* = 5, |u| = 1e-3) where those along x, and
// all three by pairs, are exact.  The populations they are made of are rounded
// at that size already: against 80-bit arithmetic a step's u is nearer than with the
// moments by pairs one by one (walled pool, x, y, z: 3.7, 6.9, 6.1e-17 and 4.8, 9.4,
// 7.1e-17; drop 4.8e-19 and 5.0 to 5.2e-19), phi and p are the same to 2 %.  Sums
// and differences of the pairs first, with shared partial sums (81 operations),
// gave the same errors within 5 % for 3 to 5 % more time (drop 32^3 43.5 and
// 44.9 us per step, bubble 61x183x61 728 and 753).
// ld(cx, cy, cz) gives the population of direction c.
template <class V>
struct Mom {
  V s, x, y, z, xx, yy, zz, xy, yz, xz;  // sum f, sum c f, sum c c f
};
// index of direction c in the lattice's order
template <int Q>
__host__ __device__ constexpr int lq_index(int cx, int cy, int cz) {
  const int i = 9 * (cz + 1) + 3 * (cy + 1) + cx + 1;
  return Q == 27 ? i : (Q == 9 ? i - 9 : (i < 13 ? i / 2 : (i == 13 ? 7 : i / 2 + 1)));
}

template <class V>
__device__ __forceinline__ V sum3(V a, V b, V c) {
  return (a + c) + b;
}

template <class V>
struct PlaneMom {
  V m00, m10, m20, m01, m11, m02;  // x-order, y-order within one z plane
};
template <class V, class LD>
__device__ __forceinline__ PlaneMom<V> plane_mom(const LD& ld, int cz) {
  V a0[3], a1[3], a2[3];
#pragma unroll
  for (int j = 0; j < 3; ++j) {
    const V l = ld(-1, j - 1, cz), c = ld(0, j - 1, cz), r = ld(1, j - 1, cz);
    a0[j] = sum3(l, c, r);
    a1[j] = r - l;
    a2[j] = l + r;
  }
  PlaneMom<V> p;
  p.m00 = sum3(a0[0], a0[1], a0[2]);
  p.m01 = a0[2] - a0[0];
  p.m02 = a0[0] + a0[2];
  p.m10 = sum3(a1[0], a1[1], a1[2]);
  p.m11 = a1[2] - a1[0];
  p.m20 = sum3(a2[0], a2[1], a2[2]);
  return p;
}

template <int Q, class V, class LD>
__device__ __forceinline__ Mom<V> moments(const LD& ld) {
  Mom<V> m;
  if constexpr (Q == 27) {
    const PlaneMom<V> a = plane_mom<V>(ld, -1), b = plane_mom<V>(ld, 0), c = plane_mom<V>(ld, 1);
    m.s = sum3(a.m00, b.m00, c.m00);
    m.z = c.m00 - a.m00;
    m.zz = a.m00 + c.m00;
    m.x = sum3(a.m10, b.m10, c.m10);
    m.xz = c.m10 - a.m10;
    m.y = sum3(a.m01, b.m01, c.m01);
    m.yz = c.m01 - a.m01;
    m.xx = sum3(a.m20, b.m20, c.m20);
    m.yy = sum3(a.m02, b.m02, c.m02);
    m.xy = sum3(a.m11, b.m11, c.m11);
  } else if constexpr (Q == 9) {
    const PlaneMom<V> b = plane_mom<V>(ld, 0);
    m.s = b.m00;
    m.x = b.m10;
    m.y = b.m01;
    m.xx = b.m20;
    m.yy = b.m02;
    m.xy = b.m11;
    m.z = m.zz = m.yz = m.xz = vbc<V>(0.0);
  } else {
    PlaneMom<V> p[2];  // corners of the planes cz = -1, 1: m00, m10, m01, m11
#pragma unroll
    for (int k = 0; k < 2; ++k) {
      const V a = ld(-1, -1, 2 * k - 1), b = ld(1, -1, 2 * k - 1), c = ld(-1, 1, 2 * k - 1), d = ld(1, 1, 2 * k - 1);
      const V r0 = a + b, r1 = c + d, e0 = b - a, e1 = d - c;
      p[k].m00 = r0 + r1;
      p[k].m01 = r1 - r0;
      p[k].m10 = e0 + e1;
      p[k].m11 = e1 - e0;
    }
    const V c0 = p[0].m00 + p[1].m00;
    const V xm = ld(-1, 0, 0), xp = ld(1, 0, 0), ym = ld(0, -1, 0), yp = ld(0, 1, 0), zm = ld(0, 0, -1),
            zp = ld(0, 0, 1), r = ld(0, 0, 0);
    const V sx = xm + xp, sy = ym + yp, sz = zm + zp, dx = xp - xm, dy = yp - ym, dz = zp - zm;
    const V cx = p[0].m10 + p[1].m10, cy = p[0].m01 + p[1].m01, cz = p[1].m00 - p[0].m00;
    m.s = (c0 + ((sx + sy) + sz)) + r;
    m.x = cx + dx;
    m.y = cy + dy;
    m.z = cz + dz;
    m.xx = c0 + sx;
    m.yy = c0 + sy;
    m.zz = c0 + sz;
    m.xy = p[0].m11 + p[1].m11;
    m.xz = p[1].m10 - p[0].m10;
    m.yz = p[1].m01 - p[0].m01;
  }
  return m;
}

// FP32 moments by opposite pairs, in the order of the set's members: S = f_c +
// f_-c feeds the even moments, D = f_c - f_-c the odd ones (see collide_pairs).
template <int Q, class LD>
__device__ __forceinline__ Mom<F1> moments_pairs(const LD& ld) {
  float s = ld(0, 0, 0).v, x = 0, y = 0, z = 0, xx = 0, yy = 0, zz = 0, xy = 0, yz = 0, xz = 0;
#pragma unroll
  for (int i = 0; i < (Q - 1) / 2; ++i) {
    const int cx = q27_cx(lq_to27<Q>(i)), cy = q27_cy(lq_to27<Q>(i)), cz = q27_cz(lq_to27<Q>(i));
    const float a = ld(cx, cy, cz).v, b = ld(-cx, -cy, -cz).v;
    const float S = a + b, D = a - b;
    s += S;
    if (cx) x += cx > 0 ? D : -D;
    if (cy) y += cy > 0 ? D : -D;
    if (cz) z += cz > 0 ? D : -D;
    if (cx) xx += S;
    if (cy) yy += S;
    if (cz) zz += S;
    if (cx && cy) xy += (cx * cy > 0) ? S : -S;
    if (cy && cz) yz += (cy * cz > 0) ? S : -S;
    if (cx && cz) xz += (cx * cz > 0) ? S : -S;
  }
  return Mom<F1>{F1{s}, F1{x}, F1{y}, F1{z}, F1{xx}, F1{yy}, F1{zz}, F1{xy}, F1{yz}, F1{xz}};
}

// FP16S moments, f_i = w_i (s_i / K + shift of its writer), by opposite pairs in
// the same order: the stored and the shift part of a pair's sum and difference
// are formed apart (the difference of two near shifts is exact), joined once, and
// weighted by the fused multiply-add of each moment.
template <int Q, class LD, class SH>
__device__ __forceinline__ Mom<F1> moments_shifted(const LD& ld, const SH& sh, double K) {
  const F1 k = vbc<F1>(1.0 / K);
  Mom<F1> m = {};
  const F1 rest = vfma(ld(0, 0, 0), k, sh(0, 0, 0));
  bool fx = true, fy = true, fz = true, fxy = true, fyz = true, fxz = true;  // first term of a moment
  auto add = [](bool& first, F1& acc, F1 w, F1 t) {
    acc = first ? w * t : vfma(w, t, acc);
    first = false;
  };
#pragma unroll
  for (int i = 0; i < (Q - 1) / 2; ++i) {
    const int cx = q27_cx(lq_to27<Q>(i)), cy = q27_cy(lq_to27<Q>(i)), cz = q27_cz(lq_to27<Q>(i));
    const F1 a = ld(cx, cy, cz), b = ld(-cx, -cy, -cz), pa = sh(cx, cy, cz), pb = sh(-cx, -cy, -cz);
    const F1 w = vbc<F1>(lq_w<Q>(i)), S = vfma(a + b, k, pa + pb), D = vfma(a - b, k, pa - pb);
    m.s = i ? vfma(w, S, m.s) : vfma(vbc<F1>(lq_w<Q>((Q - 1) / 2)), rest, w * S);
    if (cx) m.xx = fx ? w * S : vfma(w, S, m.xx);
    if (cy) m.yy = fy ? w * S : vfma(w, S, m.yy);
    if (cz) m.zz = fz ? w * S : vfma(w, S, m.zz);
    if (cx) add(fx, m.x, cx > 0 ? w : -w, D);
    if (cy) add(fy, m.y, cy > 0 ? w : -w, D);
    if (cz) add(fz, m.z, cz > 0 ? w : -w, D);
    if (cx && cy) add(fxy, m.xy, cx * cy > 0 ? w : -w, S);
    if (cy && cz) add(fyz, m.yz, cy * cz > 0 ? w : -w, S);
    if (cx && cz) add(fxz, m.xz, cx * cz > 0 ? w : -w, S);
  }
  return m;
}

// The moments of a set of a cell: ld gives the raw stored value arriving by
// direction c, sh (FP16S; K the format's factor) the shift of its writer.  m.s is
// phi (h) or p* (g).  Everything that forms phi goes through here (a caller that
// uses m.s alone leaves the rest to dead-code elimination), so all phi of a
// state agree bitwise.
template <int PREC, int Q, class LD, class SH>
__device__ __forceinline__ auto set_moments(const LD& ld, const SH& sh, double K) {
  if constexpr (PREC == 2)
    return moments_shifted<Q>(ld, sh, K);
  else if constexpr (PREC == 1)
    return moments_pairs<Q>(ld);
  else
    return moments<Q, D1>(ld);
}

// ---------------------------------------------------------------------------
// The phi stencil.  The weights factor per axis, w1 = (1/6, 2/3, 1/6) =
// 1 + delta^2 / 6 with delta^2 f = (f(-1) - f) + (f(+1) - f), so
//   grad_x = 1/2 (1 + delta_y^2 / 6)(1 + delta_z^2 / 6)(phi(x+1) - phi(x-1)),
//   lap    = 6 [(1 + delta_x^2 / 6)(1 + delta_y^2 / 6)(1 + delta_z^2 / 6) - 1] phi
//          = q + delta_z^2 phi + delta_z^2 q / 6,  q = dx + delta_y^2 phi + delta_y^2 dx / 6,
//            dx = delta_x^2 phi,
// all in differences that are exact for nearby values.  The in-plane part (28
// operations on nine values) is formed once per plane and kept while the march
// passes; joining three planes takes 22 more: 50 per cell and nine reads
// against about 130 and 27 by opposite pairs.  On one z plane (its own
// neighbour) the z part vanishes exactly.
template <class V>
struct PhiPlane {
  V c, q, gx, gy;
};
template <class V, class AT>
__device__ __forceinline__ PhiPlane<V> phi_plane(const AT& at) {  // at(cx, cy)
  const V w6 = vbc<V>(1.0 / 6.0);
  V c[3], d[3], g[3];
#pragma unroll
  for (int j = 0; j < 3; ++j) {
    const V l = at(-1, j - 1), r = at(1, j - 1);
    c[j] = at(0, j - 1);
    d[j] = (l - c[j]) + (r - c[j]);
    g[j] = r - l;
  }
  PhiPlane<V> p;
  p.c = c[1];
  p.gx = vfma(w6, (g[0] - g[1]) + (g[2] - g[1]), g[1]);
  p.gy = vfma(w6, d[2] - d[0], c[2] - c[0]);
  p.q = vfma(w6, (d[0] - d[1]) + (d[2] - d[1]), d[1] + ((c[0] - c[1]) + (c[2] - c[1])));
  return p;
}
template <class V>
struct Grad {
  V x, y, z, lap;
};
template <class V>
__device__ __forceinline__ Grad<V> phi_grad(const PhiPlane<V>& m, const PhiPlane<V>& o, const PhiPlane<V>& p) {
  const V w6 = vbc<V>(1.0 / 6.0), half = vbc<V>(0.5);
  Grad<V> r;
  r.x = half * vfma(w6, (m.gx - o.gx) + (p.gx - o.gx), o.gx);
  r.y = half * vfma(w6, (m.gy - o.gy) + (p.gy - o.gy), o.gy);
  r.z = half * vfma(w6, p.q - m.q, p.c - m.c);
  r.lap = o.q + vfma(w6, (m.q - o.q) + (p.q - o.q), (m.c - o.c) + (p.c - o.c));
  return r;
}
template <class V>
__device__ __forceinline__ Grad<V> phi_grad_flat(const PhiPlane<V>& o) {  // phi_grad(o, o, o)
  const V half = vbc<V>(0.5);
  return Grad<V>{half * o.gx, half * o.gy, vbc<V>(0.0), o.q};
}
// The same stencil over the D3Q27 (or D2Q9) weights by opposite pairs, in the
// order of FP32 and FP16S (see collide_pairs).  phi_at(cx, cy, cz): phi^t at a
// stencil neighbour.
template <int QG, class PhiAt>
__device__ __forceinline__ Grad<F1> phi_grad_pairs(const PhiAt& phi_at) {
  typedef F1 V;
  const V pc{phi_at(0, 0, 0)};
  V gx = {}, gy = {}, gz = {}, lap = {};
#pragma unroll
  for (int i = 0; i < (QG - 1) / 2; ++i) {
    const int cx = q27_cx(lq_to27<QG>(i)), cy = q27_cy(lq_to27<QG>(i)), cz = q27_cz(lq_to27<QG>(i));
    const V a{phi_at(cx, cy, cz)}, b{phi_at(-cx, -cy, -cz)};
    const V w = vbc<V>(lq_w<QG>(i)), d = a - b;
    const V t = (a - pc) + (b - pc);  // differences first: exact for nearby values
    // (member 0 has every component of the lattice)
    if (cx) gx = i ? vfma(cx > 0 ? w : -w, d, gx) : (cx > 0 ? w : -w) * d;
    if (cy) gy = i ? vfma(cy > 0 ? w : -w, d, gy) : (cy > 0 ? w : -w) * d;
    if (cz) gz = i ? vfma(cz > 0 ? w : -w, d, gz) : (cz > 0 ? w : -w) * d;
    lap = i ? vfma(w, t, lap) : w * t;
  }
  const V three = vbc<V>(3.0);
  return Grad<V>{gx * three, gy * three, gz * three, lap * vbc<V>(6.0)};
}

// ---------------------------------------------------------------------------
// The FP64 step's parameters, formed once on the host.
template <class V>
struct PhysV {
  V rho_l, drho, tau_l, dtau, beta4, mkappa, mdrho3, gx, gy, gz;
  V c4;          // 4 (1 - omega_phi / 2) / xi
  V a1;          // 3 (1 - omega_phi)
  V a2, a2_3;    // 9 (1 - omega_phi), 3/2 (1 - omega_phi): 2 a2 and a2 / 3 of the h collision
};
template <class V>
inline PhysV<V> phys_v(const Phys& p) {
  PhysV<V> q;
  q.rho_l = vbc<V>(p.rho_l);
  q.drho = vbc<V>(p.rho_h - p.rho_l);
  q.tau_l = vbc<V>(p.tau_l);
  q.dtau = vbc<V>(p.tau_h - p.tau_l);
  q.beta4 = vbc<V>(4.0 * p.beta);
  q.mkappa = vbc<V>(-p.kappa);
  q.mdrho3 = vbc<V>(-(p.rho_h - p.rho_l) / 3.0);
  q.gx = vbc<V>(p.gx);
  q.gy = vbc<V>(p.gy);
  q.gz = vbc<V>(p.gz);
  q.c4 = vbc<V>(4.0 * (1.0 - 0.5 * p.omega_phi) * p.inv_xi);
  q.a1 = vbc<V>(3.0 * (1.0 - p.omega_phi));
  q.a2 = vbc<V>(9.0 * (1.0 - p.omega_phi));
  q.a2_3 = vbc<V>(1.5 * (1.0 - p.omega_phi));
  return q;
}

// The same without the combined factors, in the arithmetic type R (the FP32 and
// FP16S steps and the adjoint).
template <typename R>
struct PhysR {
  R rho_l, drho, tau_l, dtau, beta, kappa, inv_xi, omega_phi, gx, gy, gz;
};

template <typename R>
inline PhysR<R> phys_r(const Phys& p) {
  PhysR<R> q;
  q.rho_l = (R)p.rho_l;
  q.drho = (R)(p.rho_h - p.rho_l);
  q.tau_l = (R)p.tau_l;
  q.dtau = (R)(p.tau_h - p.tau_l);
  q.beta = (R)p.beta;
  q.kappa = (R)p.kappa;
  q.inv_xi = (R)p.inv_xi;
  q.omega_phi = (R)p.omega_phi;
  q.gx = (R)p.gx;
  q.gy = (R)p.gy;
  q.gz = (R)p.gz;
  return q;
}

// Arithmetic type of a cell, and the parameters its collision takes.
template <int PREC>
struct StepV {
  typedef F1 T;
  typedef PhysR<float> Par;
};
template <>
struct StepV<0> {
  typedef D1 T;
  typedef PhysV<D1> Par;
};
template <int PREC>
inline typename StepV<PREC>::Par step_par(const Phys& p) {
  if constexpr (PREC == 0)
    return phys_v<D1>(p);
  else
    return phys_r<float>(p);
}

// Emits the post-collision pairs of a quadratic polynomial of the velocity,
//   E = al + c . G . c (off-diagonal G doubled), L = b . c,
// sharing the partial sums between directions: 21 additions for the even parts
// and 10 for the odd ones of D3Q27 instead of 45 and 27.  put(i, oi, cx, cy,
// cz, A, B): A for direction c (member i), B for -c (member oi).
// The stored value is w (s + E +- L) with s the large part added last, one
// rounding at its size.
template <int Q, class V, class PUT>
__device__ __forceinline__ void emit_pairs(V s, V al, V bx, V by, V bz, V Gxx, V Gyy, V Gzz, V Gxy, V Gyz, V Gxz,
                                           const PUT& put) {
  const V Ex = al + Gxx, Ey = al + Gyy, Ez = al + Gzz;
  const V Exy = Ex + Gyy, Exz = Ex + Gzz, Eyz = Ey + Gzz, E3 = Exy + Gzz;
  const V p = E3 + Gxy, m = E3 - Gxy, sg = Gyz + Gxz, dg = Gyz - Gxz;
  const V bxy = bx + by, bxny = bx - by;
#pragma unroll
  for (int i = 0; i < (Q - 1) / 2; ++i) {
    const int cx = q27_cx(lq_to27<Q>(i)), cy = q27_cy(lq_to27<Q>(i)), cz = q27_cz(lq_to27<Q>(i));
    const int n2 = cx * cx + cy * cy + cz * cz;
    // (qx, qy, qz) = +-c with its first non-zero component positive
    const int sgn = cx ? cx : (cy ? cy : cz);
    const int qy = sgn * cy, qz = sgn * cz;
    V E, L;
    if (n2 == 1) {
      E = cx ? Ex : (cy ? Ey : Ez);
      L = cx ? bx : (cy ? by : bz);
    } else if (n2 == 2) {
      if (cx && cy) {
        E = qy > 0 ? Exy + Gxy : Exy - Gxy;
        L = qy > 0 ? bxy : bxny;
      } else if (cx) {
        E = qz > 0 ? Exz + Gxz : Exz - Gxz;
        L = qz > 0 ? bx + bz : bx - bz;
      } else {
        E = qz > 0 ? Eyz + Gyz : Eyz - Gyz;
        L = qz > 0 ? by + bz : by - bz;
      }
    } else {
      E = qy > 0 ? (qz > 0 ? p + sg : p - sg) : (qz > 0 ? m - dg : m + dg);
      const V b2 = qy > 0 ? bxy : bxny;
      L = qz > 0 ? b2 + bz : b2 - bz;
    }
    const double w = lq_w<Q>(i);
    const V e = vbc<V>(w) * E;
    const V A = vfma(vbc<V>(w), s, vfma(vbc<V>(w), L, e)), B = vfma(vbc<V>(w), s, vfma(vbc<V>(-w), L, e));  // of +q and -q
    if (sgn > 0)
      put(i, Q - 1 - i, cx, cy, cz, A, B);
    else
      put(i, Q - 1 - i, cx, cy, cz, B, A);
  }
}
// the rest population of the same polynomial
template <int Q, class V>
__device__ __forceinline__ V emit_rest(V s, V al) {
  const double w = lq_w<Q>((Q - 1) / 2);
  return vfma(vbc<V>(w), s, vbc<V>(w) * al);
}

// The collision of both sets (moments to post-collision populations) of FP64,
// shared by every stream-collide kernel.
//   pc, gr: phi^t of the cell and its stencil; gm: the g moments;
//   hmom(): the h moments, read when their turn comes;
//   out.grest(v), out.g_(i, oi, cx, cy, cz, A, B), out.hrest(v), out.h_(...).
template <int QH, class V, class HM, class OUT>
__device__ __forceinline__ void collide(const PhysV<V>& ph, V pc, const Grad<V>& gr, const Mom<V>& gm, const HM& hmom,
                                        OUT& out) {
  constexpr int QG = qg_of<QH>();  // D2Q9 with the 2-D phase field, else D3Q27
  const V third = vbc<V>(1.0 / 3.0), one = vbc<V>(1.0), half = vbc<V>(0.5);
  const V pst = gm.s;
  V ux, uy, uz;
  {
    // ---- forces and velocity
    const V rho = vfma(pc, ph.drho, ph.rho_l);
    const V tau = vfma(pc, ph.dtau, ph.tau_l);
    const V omega = vrcp(tau), rinv = vrcp(rho);
    const V hr = half * rinv;
    const V mu = vfma(ph.mkappa, gr.lap, ((ph.beta4 * pc) * (pc - one)) * (pc - half));
    const V mc = vfma(pst, ph.mdrho3, mu);
    V Fx = vfma(mc, gr.x, rho * ph.gx), Fy = vfma(mc, gr.y, rho * ph.gy), Fz = vfma(mc, gr.z, rho * ph.gz);
    const V p3 = pst * third;
    {
      const V ax = vfma(Fx, hr, gm.x), ay = vfma(Fy, hr, gm.y), az = vfma(Fz, hr, gm.z);
      const V nx = -ax, ny = -ay, nz = -az;
      const V nxx = vfma(nx, ax, gm.xx - p3), nyy = vfma(ny, ay, gm.yy - p3), nzz = vfma(nz, az, gm.zz - p3);
      const V nxy = vfma(nx, ay, gm.xy), nyz = vfma(ny, az, gm.yz), nxz = vfma(nx, az, gm.xz);
      // -3 nu omega drho = -(1 - omega / 2) drho, since 3 nu = tau - 1/2
      const V cm = vfma(half, omega, -one) * ph.drho;
      Fx = vfma(cm, vfma(nxz, gr.z, vfma(nxy, gr.y, nxx * gr.x)), Fx);
      Fy = vfma(cm, vfma(nyz, gr.z, vfma(nyy, gr.y, nxy * gr.x)), Fy);
      Fz = vfma(cm, vfma(nzz, gr.z, vfma(nyz, gr.y, nxz * gr.x)), Fz);
    }
    ux = vfma(Fx, hr, gm.x);
    uy = vfma(Fy, hr, gm.y);
    uz = vfma(Fz, hr, gm.z);

    // ---- g post-collision coefficients and pair stores
    const V mx = -ux, my = -uy, mz = -uz;
    const V qx = mx * ux, qy = my * uy, qz = mz * uz;  // -u_a^2
    // deviatoric second moments, (3 P_aa - p*) / 3 with one rounding: p* (1/3)
    // would carry the rounded constant 1/3, a bias of 3e-8 p* that repeats
    // every step
    const V mp = -pst, three = vbc<V>(3.0);
    const V dxx = vfma(vfma(three, gm.xx, mp), third, qx), dyy = vfma(vfma(three, gm.yy, mp), third, qy);
    const V dzz = QG == 9 ? vbc<V>(0.0) : vfma(vfma(three, gm.zz, mp), third, qz);  // 2-D: the trace runs over x and y
    const V a2 = vfma(vbc<V>(-4.5), omega, vbc<V>(4.5));
    const V al = vfma(vbc<V>(1.5), (qx + qy) + qz, (a2 * vbc<V>(-1.0 / 3.0)) * ((dxx + dyy) + dzz));
    const V fr = vbc<V>(1.5) * rinv, k3 = three;
    const V bx = vfma(fr, Fx, k3 * ux), by = vfma(fr, Fy, k3 * uy), bz = vfma(fr, Fz, k3 * uz);
    const V k45 = vbc<V>(-4.5), k9 = vbc<V>(-9.0), a22 = a2 + a2;
    const V Gxx = vfma(k45, qx, a2 * dxx), Gyy = vfma(k45, qy, a2 * dyy), Gzz = vfma(k45, qz, a2 * dzz);
    const V qxy = mx * uy, qyz = my * uz, qxz = mx * uz;
    const V Gxy = vfma(k9, qxy, a22 * (gm.xy + qxy)), Gyz = vfma(k9, qyz, a22 * (gm.yz + qyz)),
            Gxz = vfma(k9, qxz, a22 * (gm.xz + qxz));
    out.grest(emit_rest<QG>(pst, al));
    emit_pairs<QG>(pst, al, bx, by, bz, Gxx, Gyy, Gzz, Gxy, Gyz, Gxz,
                   [&](int i, int oi, int cx, int cy, int cz, V A, V B) { out.g_(i, oi, cx, cy, cz, A, B); });
  }

  // ---- h post-collision coefficients and pair stores
  {
    const Mom<V> h = hmom();
    const V gn = vsqrt(vfma(gr.z, gr.z, vfma(gr.y, gr.y, gr.x * gr.x)));
    // (1 - omega_phi / 2) theta / |grad phi|, theta = 4 phi (1 - phi) / xi
    const V tn = vdiv((ph.c4 * pc) * (one - pc), gn + vbc<V>(1e-6));
    // deviatoric second moments as (3 H_aa - phi) / 3 and the non-equilibrium
    // flux J - phi u, one rounding each
    const V mphi = -h.s, three = vbc<V>(3.0);
    const V Gxx = ph.a2_3 * vfma(three, h.xx, mphi), Gyy = ph.a2_3 * vfma(three, h.yy, mphi);
    const V Gzz = QG == 9 ? vbc<V>(0.0) : ph.a2_3 * vfma(three, h.zz, mphi);
    const V al = vbc<V>(-1.0 / 3.0) * ((Gxx + Gyy) + Gzz);
    const V p3 = three * h.s;
    const V bx = vfma(p3, ux, vfma(ph.a1, vfma(mphi, ux, h.x), tn * gr.x));
    const V by = vfma(p3, uy, vfma(ph.a1, vfma(mphi, uy, h.y), tn * gr.y));
    const V bz = vfma(p3, uz, vfma(ph.a1, vfma(mphi, uz, h.z), tn * gr.z));
    out.hrest(emit_rest<QH>(h.s, al));
    emit_pairs<QH>(h.s, al, bx, by, bz, Gxx, Gyy, Gzz, ph.a2 * h.xy, ph.a2 * h.yz, ph.a2 * h.xz,
                   [&](int i, int oi, int cx, int cy, int cz, V A, V B) { out.h_(i, oi, cx, cy, cz, A, B); });
  }
}

// w (s + r) for a lattice weight w, s the large part of a stored population
// (phi or p*) and r the small rest.  FP32 carries w as hi + lo: the FP32
// roundings of the D3Q15 weights alone sum to 1 + 7.5e-9 (D3Q27 likewise),
// a bias of the zeroth and second moments that repeats every step and, over
// 1000 steps, was the largest FP32 error of phi and u.
__device__ __forceinline__ F1 wsum(double w, F1 s, F1 r) {
  const float hi = (float)w, lo = (float)(w - (double)hi);
  return vfma(F1{hi}, s, vfma(F1{lo}, s, F1{hi} * r));
}

// The collision of both sets in FP32 and FP16S, written around opposite-velocity
// pairs.  It keeps the operation order, each fused multiply-add included, that
// these formats' runs have had throughout, so their results stay as they are:
// where the flow amplifies FP32's rounding (the normal of a nearly uniform phi)
// another order moves single cells by 1e-3 within 64 steps of a Taylor bubble, with
// no smaller error against FP64; in FP16S it moves last bits in front of the
// stochastic rounding, which then rounds other values up (the sums of FP64,
// collide(), put FP16S fields 5e-4 to 1e-3 apart and 1-3 % further from FP64 on
// impact, bubble and wave).
//   Arguments as in collide(), gr from phi_grad_pairs();
//   out.shift(pst): FP16S, stores P = fp16(p*) of the cell and returns it.
// FP32 stores add the small terms first and the large part once.  FP16S stores
// K (f / w - shift), K the format's power of two (folded into the coefficients,
// which it scales exactly) and the shift the cell's own (P, phi): E +- L as is.
template <int PREC, int QH, class HM, class OUT>
__device__ __forceinline__ void collide_pairs(const PhysR<float>& par, F1 pc, const Grad<F1>& gr, const Mom<F1>& gm,
                                              const HM& hmom, OUT& out) {
  typedef F1 V;
  constexpr bool F16 = PREC == 2;
  constexpr int QG = qg_of<QH>();   // D2Q9 with the 2-D phase field, else D3Q27
  constexpr int GR = (QG - 1) / 2;  // rest index of g
  const V third = vbc<V>(1.0 / 3.0), one = vbc<V>(1.0), half = vbc<V>(0.5), three = vbc<V>(3.0), zero = vbc<V>(0.0);
  const V rho_l{par.rho_l}, drho{par.drho}, tau_l{par.tau_l}, dtau{par.dtau}, beta{par.beta}, kappa{par.kappa};

  const V gx = gr.x, gy = gr.y, gz = gr.z, lap = gr.lap;

  // ---- forces and velocity
  const V pst = gm.s;
  const V rho = vfma(pc, drho, rho_l), tau = vfma(pc, dtau, tau_l);
  const V omega = vrcp(tau);
  const V nu = (tau - half) * third;
  const V mu = vfma(((vbc<V>(4.0) * beta) * pc) * (pc - one), pc - half, -(kappa * lap));
  const V inv2rho = vdiv(half, rho);
  const V mc = vfma((-pst) * third, drho, mu);
  V Fx = vfma(rho, V{par.gx}, mc * gx), Fy = vfma(rho, V{par.gy}, mc * gy), Fz = vfma(rho, V{par.gz}, mc * gz);
  const V p3 = pst * third;
  {
    const V ax = vfma(Fx, inv2rho, gm.x), ay = vfma(Fy, inv2rho, gm.y), az = vfma(Fz, inv2rho, gm.z);
    const V nxx = vfma(-ax, ax, gm.xx - p3), nyy = vfma(-ay, ay, gm.yy - p3), nzz = vfma(-az, az, gm.zz - p3);
    const V nxy = vfma(-ax, ay, gm.xy), nyz = vfma(-ay, az, gm.yz), nxz = vfma(-ax, az, gm.xz);
    const V cm = ((vbc<V>(-3.0) * nu) * omega) * drho;
    Fx = vfma(cm, vfma(nxz, gz, vfma(nxx, gx, nxy * gy)), Fx);
    Fy = vfma(cm, vfma(nyz, gz, vfma(nxy, gx, nyy * gy)), Fy);
    Fz = vfma(cm, vfma(nzz, gz, vfma(nxz, gx, nyz * gy)), Fz);
  }
  const V ux = vfma(Fx, inv2rho, gm.x), uy = vfma(Fy, inv2rho, gm.y), uz = vfma(Fz, inv2rho, gm.z);

  // ---- g post-collision coefficients and pair stores
  {
    constexpr double K = F16 ? KG16 : 1.0;
    const V y2 = uy * uy;
    V dxx, dyy, dzz, uu;
    if constexpr (F16) {
      uu = vfma(uz, uz, vfma(ux, ux, y2));
      dxx = vfma(-ux, ux, gm.xx - p3);
      dyy = (gm.yy - p3) - y2;
      dzz = vfma(-uz, uz, gm.zz - p3);
    } else {
      // deviatoric second moments, (3 P_aa - p*) / 3 with one rounding: p* (1/3)
      // would carry the rounded constant 1/3, a bias of 3e-8 p* that repeats
      // every step
      const V x2 = ux * ux, z2 = uz * uz;
      uu = (x2 + y2) + z2;
      dxx = vfma(vfma(three, gm.xx, -pst), third, -x2);
      dyy = vfma(vfma(three, gm.yy, -pst), third, -y2);
      dzz = vfma(vfma(three, gm.zz, -pst), third, -z2);
    }
    if (QG == 9) dzz = zero;  // 2-D: the trace runs over x and y
    const V a2 = (one - omega) * vbc<V>(4.5 * K), k45 = vbc<V>(4.5 * K), k3 = vbc<V>(3.0 * K);
    const V tr = a2 * ((dxx + dyy) + dzz);
    V als;  // alpha less the large part
    if constexpr (F16)
      als = vfma(-tr, third, vfma(vbc<V>(-1.5 * K), uu, vbc<V>(K) * (pst - V{out.shift(pst.v)})));
    else
      als = vfma(vbc<V>(-1.5), uu, -(tr * third));
    const V fr = vdiv(vbc<V>(1.5 * K), rho);
    const V bx = vfma(fr, Fx, k3 * ux), by = vfma(fr, Fy, k3 * uy), bz = vfma(fr, Fz, k3 * uz);
    const V tx = k45 * ux, ty = k45 * uy, tz = k45 * uz;
    const V Gxx = vfma(tx, ux, a2 * dxx), Gyy = vfma(ty, uy, a2 * dyy), Gzz = vfma(tz, uz, a2 * dzz);
    const V two = vbc<V>(2.0);
    const V Gxy = two * vfma(tx, uy, a2 * vfma(-ux, uy, gm.xy));
    const V Gyz = two * vfma(ty, uz, a2 * vfma(-uy, uz, gm.yz));
    const V Gxz = two * vfma(tx, uz, a2 * vfma(-ux, uz, gm.xz));
    out.grest(F16 ? als : wsum(lq_w<QG>(GR), pst, als));
#pragma unroll
    for (int i = 0; i < GR; ++i) {
      const int cx = q27_cx(lq_to27<QG>(i)), cy = q27_cy(lq_to27<QG>(i)), cz = q27_cz(lq_to27<QG>(i));
      V E = cx ? Gxx : (cy ? Gyy : Gzz);
      if (F16) E = als + E;
      if (cx && cy) E = E + Gyy;
      if ((cx || cy) && cz) E = E + Gzz;
      if (cx && cy) E = E + ((cx * cy > 0) ? Gxy : -Gxy);
      if (cy && cz) E = E + ((cy * cz > 0) ? Gyz : -Gyz);
      if (cx && cz) E = E + ((cx * cz > 0) ? Gxz : -Gxz);
      V L = cx ? (cx > 0 ? bx : -bx) : (cy ? (cy > 0 ? by : -by) : (cz > 0 ? bz : -bz));
      if (cx && cy) L = L + (cy > 0 ? by : -by);
      if ((cx || cy) && cz) L = L + (cz > 0 ? bz : -bz);
      if constexpr (F16)
        out.g_(i, QG - 1 - i, cx, cy, cz, E + L, E - L);
      else
        out.g_(i, QG - 1 - i, cx, cy, cz, wsum(lq_w<QG>(i), pst, als + (E + L)), wsum(lq_w<QG>(i), pst, als + (E - L)));
    }
  }

  // ---- h post-collision coefficients and pair stores
  {
    constexpr double K = F16 ? KH16 : 1.0;
    const Mom<F1> h = hmom();
    const V phl = h.s, omp{par.omega_phi};
    const V gn = vsqrt(vfma(gz, gz, vfma(gy, gy, gx * gx)));
    const V theta = ((vbc<V>(4.0) * pc) * (one - pc)) * V{par.inv_xi};
    // (1 - omega_phi/2) theta / |grad phi|
    const V tn = vdiv(theta, gn + vbc<V>(1e-6)) * (vbc<V>(K) * (one - half * omp));
    const V a1 = (one - omp) * vbc<V>(3.0 * K), a2 = (one - omp) * vbc<V>(4.5 * K);
    V dxx, dyy, dzz;
    if constexpr (F16) {
      dxx = vfma(-phl, third, h.xx);
      dyy = vfma(-phl, third, h.yy);
      dzz = vfma(-phl, third, h.zz);
    } else {
      // deviatoric second moments as (3 H_aa - phi) / 3, one rounding each
      dxx = vfma(three, h.xx, -phl) * third;
      dyy = vfma(three, h.yy, -phl) * third;
      dzz = vfma(three, h.zz, -phl) * third;
    }
    if (QG == 9) dzz = zero;
    V als;
    if constexpr (F16)  // phi of the cell is the shift of everything it writes
      als = vfma(-(a2 * ((dxx + dyy) + dzz)), third, vbc<V>(K) * (phl - pc));
    else
      als = ((-a2) * ((dxx + dyy) + dzz)) * third;
    // (the non-equilibrium flux J - phi u with one rounding)
    const V p3 = vbc<V>(3.0 * K) * phl;
    const V bx = vfma(tn, gx, vfma(p3, ux, a1 * vfma(-phl, ux, h.x)));
    const V by = vfma(tn, gy, vfma(p3, uy, a1 * vfma(-phl, uy, h.y)));
    const V bz = vfma(tn, gz, vfma(p3, uz, a1 * vfma(-phl, uz, h.z)));
    const V a22 = vbc<V>(2.0) * a2;
    const V Hxx = a2 * dxx, Hyy = a2 * dyy, Hzz = a2 * dzz;
    out.hrest(F16 ? als : wsum(hq_w<QH>(hq_rest<QH>()), phl, als));
#pragma unroll
    for (int k = 0; k < hq_rest<QH>(); ++k) {
      const int cx = hq_cx<QH>(k), cy = hq_cy<QH>(k), cz = hq_cz<QH>(k);
      V E;
      if constexpr (F16)
        E = vfma(a2, cx ? dxx : (cy ? dyy : dzz), als);
      else
        E = cx ? Hxx : (cy ? Hyy : Hzz);
      if (cx && cy) E = vfma(a2, dyy, E);
      if ((cx || cy) && cz) E = vfma(a2, dzz, E);
      if (cx && cy) E = vfma((cx * cy > 0) ? a22 : -a22, h.xy, E);
      if (cy && cz) E = vfma((cy * cz > 0) ? a22 : -a22, h.yz, E);
      if (cx && cz) E = vfma((cx * cz > 0) ? a22 : -a22, h.xz, E);
      V L = cx ? (cx > 0 ? bx : -bx) : (cy ? (cy > 0 ? by : -by) : (cz > 0 ? bz : -bz));
      if (cx && cy) L = L + (cy > 0 ? by : -by);
      if ((cx || cy) && cz) L = L + (cz > 0 ? bz : -bz);
      if constexpr (F16)
        out.h_(k, QH - 1 - k, cx, cy, cz, E + L, E - L);
      else
        out.h_(k, QH - 1 - k, cx, cy, cz, wsum(hq_w<QH>(k), phl, als + (E + L)), wsum(hq_w<QH>(k), phl, als + (E - L)));
    }
  }
}

// Store the post-collision pair (A: direction c, B: direction -c) of `cell`.
template <int PREC, int ODD>
__device__ __forceinline__ void store_pair(typename Store<PREC>::S* __restrict__ f, unsigned N, unsigned cell,
                                           const CellOff& o, int i, int oi, int cx, int cy, int cz,
                                           typename Store<PREC>::R A, typename Store<PREC>::R B, Dither& d) {
  typename Store<PREC>::S a, b;
  if constexpr (PREC == 2 && PFL_FP16S_HWSR) {
    pack2_sr(A, B, d.next32(), a, b);
  } else {
    a = pack_sr<PREC>(A, d);
    b = pack_sr<PREC>(B, d);
  }
  if (!ODD) {
    f[(unsigned)oi * N + cell] = a;
    f[(unsigned)i * N + cell] = b;
  } else {
    const bool vc = o.valid(cx, cy, cz), vmc = o.valid(-cx, -cy, -cz);
    f[vc ? (unsigned)i * N + cell + (unsigned)o.off(cx, cy, cz) : (unsigned)oi * N + cell] = a;
    f[vmc ? (unsigned)oi * N + cell + (unsigned)o.off(-cx, -cy, -cz) : (unsigned)i * N + cell] = b;
  }
}

// Stored value of direction c arriving at `cell`, raw; `from` the cell that
// wrote it.  READ_ODD: the state left by an even in-place step.
template <int PREC, int Q, int READ_ODD>
__device__ __forceinline__ typename Store<PREC>::R load_dir(const typename Store<PREC>::S* f, unsigned N, unsigned cell,
                                                            const CellOff& o, int cx, int cy, int cz) {
  const int i = lq_index<Q>(cx, cy, cz);
  if (!READ_ODD || (!cx && !cy && !cz)) return raw<PREC>(f[(unsigned)i * N + cell]);
  const bool v = o.valid(-cx, -cy, -cz);
  return raw<PREC>(f[v ? (unsigned)(Q - 1 - i) * N + cell + (unsigned)o.off(-cx, -cy, -cz) : (unsigned)i * N + cell]);
}
// the cell that wrote the population of direction c arriving at `cell`
__device__ __forceinline__ unsigned writer(unsigned cell, const CellOff& o, int cx, int cy, int cz) {
  return o.valid(-cx, -cy, -cz) ? cell + (unsigned)o.off(-cx, -cy, -cz) : cell;
}

// The h moments of one cell of a state in memory.
template <int PREC, int QH, int READ_ODD>
__device__ __forceinline__ Mom<typename StepV<PREC>::T> h_moments_cell(
    unsigned N, const typename Store<PREC>::S* h, const typename Store<PREC>::PhiT* __restrict__ shift, unsigned cell,
    const CellOff& o) {
  typedef typename StepV<PREC>::T V;
  return set_moments<PREC, QH>(
      [&](int cx, int cy, int cz) { return V{load_dir<PREC, QH, READ_ODD>(h, N, cell, o, cx, cy, cz)}; },
      [&](int cx, int cy, int cz) { return V{(typename V::R)__ldg(shift + writer(cell, o, cx, cy, cz))}; }, KH16);
}

// Destination of one cell's collision: the pairs go to (h, g) in the layout
// ODD; FP16S: its p* shift to pg_out.
template <int PREC, int QH, int ODD>
struct CellOut {
  typedef typename StepV<PREC>::T V;
  typename Store<PREC>::S *h, *g;
  unsigned N, cell;
  const CellOff& o;
  __half* pg_out;
  Dither dith;
  __device__ __forceinline__ float shift(float pst) {
    const __half q = __float2half_rn(pst);
    pg_out[cell] = q;
    return __half2float(q);
  }
  __device__ __forceinline__ void grest(V v) { g[(unsigned)((qg_of<QH>() - 1) / 2) * N + cell] = pack_sr<PREC>(v.v, dith); }
  __device__ __forceinline__ void hrest(V v) { h[(unsigned)hq_rest<QH>() * N + cell] = pack_sr<PREC>(v.v, dith); }
  __device__ __forceinline__ void g_(int i, int oi, int cx, int cy, int cz, V A, V B) {
    store_pair<PREC, ODD>(g, N, cell, o, i, oi, cx, cy, cz, A.v, B.v, dith);
  }
  __device__ __forceinline__ void h_(int i, int oi, int cx, int cy, int cz, V A, V B) {
    store_pair<PREC, ODD>(h, N, cell, o, i, oi, cx, cy, cz, A.v, B.v, dith);
  }
};

// In-place AA update of one cell with the stencil read from the phi buffer.
// pg_in / pg_out: the p* shifts of the stored g (FP16S; NULL otherwise),
// read for the populations loaded and written for those stored.
template <int PREC, int QH, int ODD>
__device__ __forceinline__ void step_cell(const Geo32& geo, const typename StepV<PREC>::Par& ph,
                                          typename Store<PREC>::S* __restrict__ h,
                                          typename Store<PREC>::S* __restrict__ g,
                                          const typename Store<PREC>::PhiT* __restrict__ phi,
                                          const typename Store<PREC>::PhiT* __restrict__ shift, unsigned cell,
                                          unsigned seed, const __half* __restrict__ pg_in, __half* __restrict__ pg_out) {
  typedef typename StepV<PREC>::T V;
  typedef typename V::R R;
  constexpr int QG = qg_of<QH>();
  CellOff o;
  cell_off(geo, cell, o);
  auto at = [&](int cx, int cy, int cz) { return (R)__ldg(phi + cell + o.soff(cx, cy, cz)); };
  const Mom<V> gm = set_moments<PREC, QG>(
      [&](int cx, int cy, int cz) { return V{load_dir<PREC, QG, ODD>(g, geo.N, cell, o, cx, cy, cz)}; },
      [&](int cx, int cy, int cz) { return V{(R)__half2float(__ldg(pg_in + writer(cell, o, cx, cy, cz)))}; }, KG16);
  CellOut<PREC, QH, ODD> out{h, g, geo.N, cell, o, pg_out, Dither{PREC == 2 ? hash32(cell * 0x9E3779B1u + seed) : 0u}};
  auto hm = [&] { return h_moments_cell<PREC, QH, ODD>(geo.N, h, shift, cell, o); };
  if constexpr (PREC != 0) {
    collide_pairs<PREC, QH>(ph, F1{at(0, 0, 0)}, phi_grad_pairs<QG>(at), gm, hm, out);
  } else {
    auto plane = [&](int cz) { return phi_plane<V>([&](int cx, int cy) { return V{at(cx, cy, cz)}; }); };
    const PhiPlane<V> p0 = plane(0);
    const Grad<V> gr = QG == 9 ? phi_grad_flat(p0) : phi_grad(plane(-1), p0, plane(1));
    collide<QH, V>(ph, p0.c, gr, gm, hm, out);
  }
}

template <int PREC, int QH, int ODD>
__global__ void __launch_bounds__(PFL_STEP_THREADS, PFL_STEP_MINB)
    k_step_mrt(Geo32 geo, typename StepV<PREC>::Par ph, typename Store<PREC>::S* __restrict__ h,
               typename Store<PREC>::S* __restrict__ g, const typename Store<PREC>::PhiT* __restrict__ phi,
               const typename Store<PREC>::PhiT* __restrict__ shift, unsigned seed,
               const __half* __restrict__ pg_in = nullptr, __half* __restrict__ pg_out = nullptr) {
  const unsigned cell = blockIdx.x * blockDim.x + threadIdx.x;
  if (cell >= geo.N) return;
  step_cell<PREC, QH, ODD>(geo, ph, h, g, phi, shift, cell, seed, pg_in, pg_out);
}

// phi = sum_i h_i of the state left by the last step (READ_ODD after an even
// step); `shift` holds the shifts of the stored populations (FP16S).  With
// `links` (a lattice with solid cells) blocked links bounce and solid cells
// hold phi = 0.
template <int PREC, int QH, int READ_ODD>
__global__ void __launch_bounds__(256) k_phi32(Geo32 geo, const typename Store<PREC>::S* __restrict__ h,
                                               const typename Store<PREC>::PhiT* __restrict__ shift,
                                               typename Store<PREC>::PhiT* __restrict__ phi,
                                               const unsigned* __restrict__ links = nullptr) {
  typedef typename Store<PREC>::PhiT PhiT;
  const unsigned cell = blockIdx.x * blockDim.x + threadIdx.x;
  if (cell >= geo.N) return;
  CellOff o;
  cell_off(geo, cell, o);
  o.blk = links ? __ldg(links + cell) : 0u;  // a bounced population was written by this cell
  phi[cell] = (o.blk & SOLID_SELF) ? (PhiT)0 : (PhiT)h_moments_cell<PREC, QH, READ_ODD>(geo.N, h, shift, cell, o).s.v;
}

// ---------------------------------------------------------------------------
// Fused two-array step: stream-collide and the phi stencil in one launch.
//
// The populations live in two array pairs; a step reads the current pair in
// its own cell (every slot local, coalesced) and pushes the post-collision
// populations to the other pair (x + c, or the opposite slot of x behind a
// wall).  Nothing a step reads is overwritten during that step, so a block may
// read its neighbours' populations: each block owns an xy tile of TX x TY
// columns and marches through a chunk of z planes, computing phi^t = sum_i h_i
// for its tile plus a one-cell ring of the next plane into shared memory before
// colliding a plane.  phi^t of every cell is written once (the FP16S shift of
// the populations written this step and the phi output), so the separate phi
// pass and its re-read of h disappear.  Ring and z-halo planes repeat the phi
// sum of neighbouring tiles (from L2).
// A single-plane lattice (FLAT) has no z march to hide latency behind; its
// tiles are 32 x 4, so that a small lattice spreads over more blocks (and the
// SMs' loads even out) for a slightly larger share of ring cells.
constexpr int ZM_TX = 32;
constexpr int ZM_TY = 8;
constexpr int ZM_TY_FLAT = 4;
__host__ __device__ constexpr int zm_ty(int flat) { return flat ? ZM_TY_FLAT : ZM_TY; }
// resident blocks per SM a block of nt threads is compiled for
__host__ __device__ constexpr int zm_minb(int prec, int nt) {
  return (prec == 0 ? PFL_ZM_MINB_FP64 : PFL_ZM_MINB) * 256 / nt;
}

__device__ __forceinline__ void prefetch_l1(const void* p) {
  asm volatile("{\n\t.reg .u64 ga;\n\tcvta.to.global.u64 ga, %0;\n\tprefetch.global.L1 [ga];\n\t}" ::"l"(p));
}

// v one step outside [0, n) brought inside (wrapped, or clamped at walls);
// positions further out, which nothing uses, to the last cell
__device__ __forceinline__ int wrap_or_clamp(int v, int n, int wall) {
  if (v < 0) return wall ? 0 : n - 1;
  if (v < n) return v;
  return wall ? n - 1 : min(v - n, n - 1);
}

// position r in [0, 2 (W + H) - 4) of the frame of a W x H plane -> (i, j)
__device__ __forceinline__ void frame_pos(int r, int W, int H, int& i, int& j) {
  if (r < W) {
    i = r;
    j = 0;
  } else if (r < 2 * W) {
    i = r - W;
    j = H - 1;
  } else if (r < 2 * W + (H - 2)) {
    i = 0;
    j = 1 + (r - 2 * W);
  } else {
    i = W - 1;
    j = 1 + (r - 2 * W - (H - 2));
  }
}

__device__ __forceinline__ CellOff off_xyz(const Geo32& geo, unsigned x, unsigned y, unsigned z, unsigned blk) {
  CellOff o;
  o.X = axis_off(x, geo.nx, 1, geo.wall[0]);
  o.Y = axis_off(y, geo.ny, (int)geo.nx, geo.wall[1]);
  o.Z = axis_off(z, geo.nz, (int)(geo.nx * geo.ny), geo.wall[2]);
  o.blk = blk;
  return o;
}

// One tile of the fused step: the xy tile (bx, by) of TX x TY columns and
// the z chunk bz of zc planes (the grid of k_step_zm, or an entry of the
// batched engine's work list), run by a block of TX x TY threads.  The caller
// has waited for the previous step.  SOLID: the lattice holds solid cells, given
// by `links` (one word per cell).
// TM: the tile's own populations come by tensor copies into dynamic shared
// memory, one box of every member of h and of g per plane, issued as soon as the
// plane before is read; `mbar` holds the two barriers (h, g).  Returns false if
// a copy did not arrive within its wait's limit.
template <int PREC, int QH, int TY, int FLAT, int SOLID, int TX = ZM_TX, int TM = 0>
__device__ __forceinline__ bool zm_tile(const Geo32& geo, const typename StepV<PREC>::Par& ph,
                                        const typename Store<PREC>::S* __restrict__ hA,
                                        const typename Store<PREC>::S* __restrict__ gA,
                                        typename Store<PREC>::S* __restrict__ hB, typename Store<PREC>::S* __restrict__ gB,
                                        const typename Store<PREC>::PhiT* __restrict__ phi_shift,
                                        typename Store<PREC>::PhiT* __restrict__ phi_out, int zc, unsigned seed,
                                        const unsigned* __restrict__ links, const __half* __restrict__ pg_in,
                                        __half* __restrict__ pg_out, int bx, int by, int bz,
                                        const StepMaps* maps = nullptr, unsigned mbar = 0) {
  typedef typename Store<PREC>::PhiT PhiT;
  typedef typename Store<PREC>::S S;
  typedef typename Store<PREC>::R R;
  typedef typename StepV<PREC>::T V;
  constexpr int NT = TX * TY;
  constexpr int PW = TX + 2, PH = TY + 2, PS = PW * PH;
  constexpr int NRING = 2 * (PW + PH) - 4;
  constexpr bool F16 = PREC == 2;
  constexpr int QG = qg_of<QH>();
  // phi planes.  MARCH (FP64): the one being filled and the one being read, whose
  // in-plane stencil part is kept in registers (two slots, one barrier per
  // plane: a slot is refilled only after the barrier that follows its last
  // read).  FP32 and FP16S, and solid cells, whose stencil reads depend on the
  // reading cell: all three planes of the stencil and the one being filled (FP64:
  // three slots, within 48 KB of static shared memory, and a second barrier).  The
  // p* shifts are read for three planes as well.  The h moments are per thread.
  constexpr bool MARCH = PREC == 0 && !SOLID;
  constexpr int NS = FLAT ? 1 : (MARCH ? 2 : (sizeof(R) == 8 ? 3 : 4));
  constexpr int NSP = FLAT ? 1 : 4;
  // FP32 gathers the g populations of the plane about to collide before the next
  // plane's h: both sets of loads are in flight together (bubble 186x378x153, no
  // copies: 13.9 -> 14.5 GLUPS), and with copies one barrier per plane frees both
  // buffers.  FP16S (15.6 -> 14.3), single planes (12.5 -> 12.2) and solid cells
  // (Taylor tube 66x640x66: 9.7 -> 9.6) lose by it.
  constexpr bool EARLY = PREC == 1 && !FLAT && !SOLID;
  // FP32 loads the h populations of the ring (of its first NT cells) before those
  // of the tile, so that both, or the copy, are in flight together: bubble
  // 128x384x128 17.0 -> 17.3 GLUPS and D3Q27 12.3 -> 12.55 (copies), bubble
  // 186x378x153 14.5 -> 14.65, a 200x400 plane 5.97 -> 5.79 us per step and 3.87 ->
  // 3.55 in D2Q9.  FP64 (0.92 -> 0.90, bound by its units) and FP16S planes (D2Q9
  // 4.06 -> 4.14 us) lose: every thread computes, ring cell or not.
  constexpr bool RING1ST = PREC == 1;
  __shared__ PhiT ring[NS][PS];
  __shared__ V hmom[FLAT ? 1 : 2][10 * NT];
  __shared__ float pring[F16 ? NSP : 1][F16 ? PS : 1];  // FP16S: p* shifts of the stored g, ring like phi
  const int tx = threadIdx.x, ty = threadIdx.y, tid = ty * TX + tx;
  const int x0 = bx * TX, y0 = by * TY;
  const int z0 = bz * zc;
  const int z1 = min(z0 + zc, (int)geo.nz);
  const unsigned N = geo.N;
  const int x = x0 + tx, y = y0 + ty;
  const bool active = x < (int)geo.nx && y < (int)geo.ny;
  const int i0 = (ty + 1) * PW + tx + 1;  // ring position of the own cell
  const unsigned xq = (unsigned)wrap_or_clamp(x, (int)geo.nx, geo.wall[0]);
  const unsigned yq = (unsigned)wrap_or_clamp(y, (int)geo.ny, geo.wall[1]);

  // L1 prefetch of the g populations plane zp's collision will read
  auto prefetch_plane = [&](int zp) {
    if (!(PFL_ZM_PREFETCH && !TM && PREC == 1 && QH == 15 && !FLAT) || !active || zp >= z1) return;
    const unsigned c = (unsigned)x + geo.nx * ((unsigned)y + geo.ny * (unsigned)zp);
#pragma unroll
    for (int i = 0; i < QG; ++i) prefetch_l1(gA + (unsigned)i * N + c);
  };
  // tensor copies: h of plane zp (wrapped or clamped), g of plane z
  extern __shared__ __align__(128) unsigned char dyn[];
  S* sG = (S*)dyn;
  S* sH = sG + QG * NT;
  const unsigned mbar_h = mbar, mbar_g = mbar + 8;
  bool ok = true;
  auto issue_h = [&](int zp) {
    if (tid == 0) {
      mbar_expect(mbar_h, QH * NT * sizeof(S));
      tma4(smem_u32(sH), &maps->h, x0, y0, wrap_or_clamp(zp, (int)geo.nz, geo.wall[2]), 0, mbar_h);
    }
  };
  auto issue_g = [&](int z) {
    if (tid == 0) {
      mbar_expect(mbar_g, QG * NT * sizeof(S));
      tma4(smem_u32(sG), &maps->g, x0, y0, z, 0, mbar_g);
    }
  };

  // phi of cell (qx, qy, zq) from memory
  auto phi_at = [&](unsigned qx, unsigned qy, unsigned zq) {
    const unsigned c = qx + geo.nx * (qy + geo.ny * zq);
    CellOff o;
    if (F16) o = off_xyz(geo, qx, qy, zq, SOLID ? __ldg(links + c) : 0u);
    return (PhiT)h_moments_cell<PREC, QH, 0>(N, hA, phi_shift, c, o).s.v;
  };
  // ring cell r of a plane: its place in the ring, its column
  struct RingCell {
    int at;
    unsigned x, y;
  };
  auto ring_cell = [&](int r) {
    int i, j;
    frame_pos(r, PW, PH, i, j);
    return RingCell{j * PW + i, (unsigned)wrap_or_clamp(x0 - 1 + i, (int)geo.nx, geo.wall[0]),
                    (unsigned)wrap_or_clamp(y0 - 1 + j, (int)geo.ny, geo.wall[1])};
  };
  // FP16S finds its ring cell once (bubble 128x384x128: 410 -> 398 us per step; FP64
  // is indifferent, and FP32 planes lose, 5.65 -> 5.84 us on 200x400).
  static_assert(!F16 || NRING <= NT, "one ring cell per thread");
  const RingCell own_ring = F16 ? ring_cell(min(tid, NRING - 1)) : RingCell{};
  // phi of plane zp over the tile (with the h moments of the own cells) and its ring
  auto fill = [&](int zp, int slot, int pslot, int mslot) {
    const unsigned zq = (unsigned)wrap_or_clamp(zp, (int)geo.nz, geo.wall[2]);
    const unsigned c = xq + geo.nx * (yq + geo.ny * zq);
    CellOff o;
    if (F16) o = off_xyz(geo, xq, yq, zq, SOLID ? __ldg(links + c) : 0u);
    // phi of ring cell r and its place
    auto ring_phi = [&](int r, int& at, PhiT& v) {
      const RingCell q = F16 ? own_ring : ring_cell(r);
      at = q.at;
      v = phi_at(q.x, q.y, zq);
      if constexpr (F16) pring[pslot][at] = ld_pshift(pg_in, q.x + geo.nx * (q.y + geo.ny * zq));
    };
    int rat = 0;
    PhiT rv = 0;
    if constexpr (RING1ST) ring_phi(NRING < NT ? min(tid, NRING - 1) : tid, rat, rv);
    if constexpr (TM != 0) ok = copy_wait(mbar_h, zp - (z0 - 1)) && ok;
    if (PREC == 0 && !FLAT && (zp < z0 || zp >= z1)) {
      // FP64, the planes beside the chunk: their cells collide in other blocks, so
      // phi alone (14 additions instead of 39): drop 32^3, one plane per chunk,
      // 47.7 -> 43.9 us per step, 64^3 295 -> 288, bubble 61x183x61 742 -> 728, D3Q27
      // drop 48^3 190 -> 178.  FP32 and FP16S do not wait for the additions and
      // lose 3 % by the second code site.
      ring[slot][i0] = phi_at(xq, yq, zq);
    } else {
      const Mom<V> m = set_moments<PREC, QH>(
          [&](int cx, int cy, int cz) {
            const unsigned i = (unsigned)lq_index<QH>(cx, cy, cz);
            if constexpr (TM != 0) return V{raw<PREC>(sH[i * NT + tid])};
            return V{raw<PREC>(hA[i * N + c])};
          },
          [&](int cx, int cy, int cz) { return V{(R)__ldg(phi_shift + writer(c, o, cx, cy, cz))}; }, KH16);
      // (tile positions outside the lattice serve as ring cells; the copy does not hold them)
      ring[slot][i0] = TM && !active ? phi_at(xq, yq, zq) : (PhiT)m.s.v;
      V* hm = &hmom[mslot][tid];
      hm[0] = m.s;
      hm[NT] = m.x;
      hm[2 * NT] = m.y;
      hm[3 * NT] = m.z;
      hm[4 * NT] = m.xx;
      hm[5 * NT] = m.yy;
      hm[6 * NT] = m.zz;
      hm[7 * NT] = m.xy;
      hm[8 * NT] = m.yz;
      hm[9 * NT] = m.xz;
    }
    if constexpr (F16) pring[pslot][i0] = ld_pshift(pg_in, c);
    if (RING1ST && tid < NRING) ring[slot][rat] = rv;
#pragma unroll
    for (int r0 = RING1ST ? NT : 0; r0 < NRING; r0 += NT) {
      if (r0 + tid < NRING) {
        ring_phi(r0 + tid, rat, rv);
        ring[slot][rat] = rv;
      }
    }
  };
  // in-plane part of the stencil of the plane in a ring slot
  auto plane = [&](int slot) {
    return phi_plane<V>([&](int cx, int cy) { return V{(R)ring[slot][i0 + cy * PW + cx]}; });
  };

  // g moments of the own cell of plane z (plane count b)
  unsigned cell = 0;
  CellOff o;
  Mom<V> gm = {};
  auto gather_g = [&](int b) {
    gm = set_moments<PREC, QG>(
        [&](int cx, int cy, int cz) {
          const unsigned i = (unsigned)lq_index<QG>(cx, cy, cz);
          if constexpr (TM != 0) return V{raw<PREC>(sG[i * NT + tid])};
          return V{raw<PREC>(gA[i * N + cell])};
        },
        [&](int cx, int cy, int cz) {
          // p* of the writer x - c, or of the cell itself after a bounce-back
          // (solid cells: one index from the start of the planes; Taylor tube 62x600x62
          // 206 -> 199 us per step, but bubble 128x384x128 without solids 398 -> 419)
          if constexpr (SOLID && F16) {
            const int own = (FLAT ? 0 : (b & 3) * PS) + i0, at = (FLAT ? 0 : ((b - cz) & 3) * PS) + i0 - cy * PW - cx;
            return V{(&pring[0][0])[o.valid(-cx, -cy, -cz) ? at : own]};
          }
          const float* p0 = pring[FLAT ? 0 : b % NSP];
          const float* pz = FLAT ? p0 : pring[(b - cz) % NSP];
          return V{o.valid(-cx, -cy, -cz) ? (R)pz[i0 - cy * PW - cx] : (R)p0[i0]};
        },
        KG16);
  };

  // Planes z0 - 1 .. z1 are filled in turn; once plane z + 1 is, plane z
  // collides (a single plane: filled and collided at once).
  PhiPlane<V> pm = {}, po = {}, pp = {};
  if (TM) issue_h(z0 - 1);
  prefetch_plane(z0);
  for (int zp = FLAT ? z0 : z0 - 1; zp <= (FLAT ? z0 : z1); ++zp) {
    const int z = FLAT ? zp : zp - 1;
    const int bp = zp - (z0 - 1), b = bp - 1;  // plane counts from z0 - 1
    cell = (unsigned)x + geo.nx * ((unsigned)y + geo.ny * (unsigned)z);
    if (TM) ok = copy_wait(mbar_g, z - z0) && ok;
    if (EARLY && z >= z0 && (TM || active)) gather_g(b);
    fill(FLAT ? 0 : zp, FLAT ? 0 : bp % NS, FLAT ? 0 : bp % NSP, FLAT ? 0 : bp & 1);
    if constexpr (TM != 0) {
      if (!__syncthreads_and(ok)) {
        copy_wait(mbar_h, bp);  // (no other copy has been issued)
        copy_wait(mbar_g, z - z0);
        return false;
      }
      if (zp < z1) issue_h(zp + 1);
      if (zp < z1 && zp >= z0) issue_g(zp);
    } else {
      __syncthreads();
    }
    if (!FLAT && z >= z0) prefetch_plane(z + 1);
    if (MARCH) (FLAT ? po : pp) = plane(FLAT ? 0 : bp % NS);
    if (!FLAT && z < z0) {
      pm = po;
      po = pp;
      continue;
    }
    const unsigned blk = (SOLID && active) ? __ldg(links + cell) : 0u;
    o = off_xyz(geo, (unsigned)x, (unsigned)y, (unsigned)z, blk);
    if (SOLID && active && (blk & SOLID_SELF)) {
      phi_out[cell] = (PhiT)0;  // solid cells are not updated; their populations stay zero
    } else if (active) {
      const PhiT* at0 = ring[FLAT ? 0 : b % NS];
      phi_out[cell] = at0[i0];
      // phi around the cell; a solid neighbour reads as the cell itself (neutral wetting)
      auto at = [&](int cx, int cy, int cz) {
        if (blk & link_bit(cx, cy, cz)) return (R)at0[i0];
        return (R)(FLAT ? at0 : ring[(b + cz) % NS])[i0 + cy * PW + cx];
      };
      // FP64 and FP16S: the stencil before g, whose moments then hold no registers
      // meanwhile
      if (PREC == 1 && !EARLY) gather_g(b);
      const V pc = MARCH ? po.c : V{(R)at0[i0]};
      Grad<V> gr;
      if constexpr (PREC != 0) {
        gr = phi_grad_pairs<QG>(at);
      } else if constexpr (MARCH) {
        gr = FLAT ? phi_grad_flat(po) : phi_grad(pm, po, pp);
      } else {
        auto splane = [&](int cz) { return phi_plane<V>([&](int cx, int cy) { return V{at(cx, cy, cz)}; }); };
        const PhiPlane<V> p0 = splane(0);
        gr = QG == 9 ? phi_grad_flat(p0) : phi_grad(splane(-1), p0, splane(1));
      }
      if (PREC != 1) gather_g(b);
      CellOut<PREC, QH, 1> out{hB, gB, N, cell, o, pg_out, Dither{F16 ? hash32(cell * 0x9E3779B1u + seed) : 0u}};
      const V* hp = &hmom[FLAT ? 0 : b & 1][tid];
      auto hm = [&] {
        return Mom<V>{hp[0], hp[NT], hp[2 * NT], hp[3 * NT], hp[4 * NT], hp[5 * NT], hp[6 * NT], hp[7 * NT], hp[8 * NT], hp[9 * NT]};
      };
      if constexpr (PREC != 0)
        collide_pairs<PREC, QH>(ph, pc, gr, gm, hm, out);
      else
        collide<QH, V>(ph, pc, gr, gm, hm, out);
    }
    if (!FLAT) {
      pm = po;
      po = pp;
    }
    if (NS == 3) __syncthreads();
  }
  return true;
}

// grid: (ceil(nx / TX), ceil(ny / TY), ceil(nz / zc)), block TX x TY.
// tclock (launches replayed from a CUDA graph): the FP16 rounding seed comes
// from the step count *tclock + tofs in device memory instead of `seed`, the
// same function of the step count as the host's.
template <int PREC, int QH, int FLAT, int SOLID = 0, int TX = ZM_TX, int TY = zm_ty(FLAT)>
__global__ void __launch_bounds__(TX* TY, zm_minb(PREC, TX* TY))
    k_step_zm(Geo32 geo, typename StepV<PREC>::Par ph, const typename Store<PREC>::S* __restrict__ hA,
              const typename Store<PREC>::S* __restrict__ gA, typename Store<PREC>::S* __restrict__ hB,
              typename Store<PREC>::S* __restrict__ gB, const typename Store<PREC>::PhiT* __restrict__ phi_shift,
              typename Store<PREC>::PhiT* __restrict__ phi_out, int zc, unsigned seed,
              const unsigned* __restrict__ links = nullptr, const unsigned long long* tclock = nullptr,
              int tofs = 0, const __half* __restrict__ pg_in = nullptr, __half* __restrict__ pg_out = nullptr) {
  // global memory only after the previous step has completed
  if (PFL_ZM_PDL) asm volatile("griddepcontrol.wait;" ::: "memory");
  if (PREC == 2 && tclock) seed = step_seed_of(*tclock + (unsigned long long)tofs);
  zm_tile<PREC, QH, TY, FLAT, SOLID, TX>(geo, ph, hA, gA, hB, gB, phi_shift, phi_out, zc, seed, links, pg_in, pg_out,
                                         blockIdx.x, blockIdx.y, blockIdx.z);
}

// The same with the populations read by tensor copies (3-D lattices without
// solid cells whose rows are whole 16-byte units), in tiles of TX x TY.  err: set
// when a copy did not arrive; the state is lost then, and blocks that find it set
// return at once, so that later waves, steps and graph replays do not each wait for
// their copies' limit.  (Read before the wait for the previous step, whose time
// hides it: bubble 128x384x128 365.0 us per step without, 365.6 with.)
template <int PREC, int QH, int TX, int TY>
__global__ void __launch_bounds__(TX* TY, zm_minb(PREC, TX* TY))
    k_step_tma(const __grid_constant__ StepMaps maps, Geo32 geo, typename StepV<PREC>::Par ph,
               const typename Store<PREC>::S* __restrict__ hA, const typename Store<PREC>::S* __restrict__ gA,
               typename Store<PREC>::S* __restrict__ hB, typename Store<PREC>::S* __restrict__ gB,
               typename Store<PREC>::PhiT* __restrict__ phi_out, int zc, volatile int* err) {
  static_assert(PREC != 2, "FP16S is bound by instruction issue and takes no copies");
  __shared__ unsigned long long mbar[2];
  const unsigned bar = smem_u32(mbar);
  if (threadIdx.x == 0 && threadIdx.y == 0) {
    mbar_init(bar);
    mbar_init(bar + 8);
  }
  const int lost = __syncthreads_or(*err);
  if (PFL_ZM_PDL) asm volatile("griddepcontrol.wait;" ::: "memory");
  if (lost) return;
  if (!zm_tile<PREC, QH, TY, 0, 0, TX, 1>(geo, ph, hA, gA, hB, gB, nullptr, phi_out, zc, 0u, nullptr, nullptr, nullptr,
                                          blockIdx.x, blockIdx.y, blockIdx.z, &maps, bar) &&
      threadIdx.x == 0 && threadIdx.y == 0)
    *err = 1;
}

}  // namespace pfl
