// Moments up to second order of a population set, in the FP64 step's form.
//
// S_c = f_c + f_-c and D_c = f_c - f_-c of the opposite pairs come first, then
// partial sums that the moments share: 81 operations for the ten moments of
// D3Q27 (26 for the pairs, 22 for the first moments, 33 for the even ones)
// against 111 with every moment summed by itself; 39 against 63 for D3Q15.  The
// difference of two near populations is exact, so a first moment carries the
// rounding of its small differences only, on every axis.  (Sums along x, then y,
// then z take 66 operations for D3Q27, but subtract sums at the size of p* for y
// and z: with p* = 5 and |u| = 1e-3 the first moments along y and z were 5e-17
// off, those along x exact.  FP64, us per step, by axes and by pairs: drop 32^3
// 43.5 and 44.9, bubble 61x183x61 728 and 753, D3Q27 drop 48^3 178 and 187.)
#pragma once
#include "vec.cuh"

namespace pfl {

template <class V>
struct Mom {
  V s, x, y, z, xx, yy, zz, xy, yz, xz;  // sum f, sum c f, sum c c f
};

template <class V>
struct PairSD {
  V s, d;
};

// The moments of the lattice Q = 27 (D3Q27), 15 (D3Q15) or 9 (D2Q9); ld(cx, cy,
// cz) gives the population of direction c.
template <int Q, class V, class LD>
__device__ __forceinline__ Mom<V> moments(const LD& ld) {
  auto pair = [&](int cx, int cy, int cz) {
    const V a = ld(cx, cy, cz), b = ld(-cx, -cy, -cz);
    return PairSD<V>{a + b, a - b};
  };
  Mom<V> m;
  const PairSD<V> x = pair(1, 0, 0), y = pair(0, 1, 0);
  V s = x.s + y.s;  // the sum of all but the rest population
  m.x = x.d;
  m.y = y.d;
  m.xx = x.s;
  m.yy = y.s;
  m.z = m.zz = m.xy = m.yz = m.xz = vbc<V>(0.0);
  if constexpr (Q != 9) {
    const PairSD<V> z = pair(0, 0, 1);
    s = s + z.s;
    m.z = z.d;
    m.zz = z.s;
  }
  // pairs along the diagonals of the xy, xz and yz planes
  if constexpr (Q != 15) {
    const PairSD<V> p = pair(1, 1, 0), q = pair(1, -1, 0);
    const V t = p.s + q.s;
    s = s + t;
    m.x = m.x + (p.d + q.d);
    m.y = m.y + (p.d - q.d);
    m.xx = m.xx + t;
    m.yy = m.yy + t;
    m.xy = p.s - q.s;
  }
  if constexpr (Q == 27) {
    const PairSD<V> p = pair(1, 0, 1), q = pair(1, 0, -1);
    const V t = p.s + q.s;
    s = s + t;
    m.x = m.x + (p.d + q.d);
    m.z = m.z + (p.d - q.d);
    m.xx = m.xx + t;
    m.zz = m.zz + t;
    m.xz = p.s - q.s;
  }
  if constexpr (Q == 27) {
    const PairSD<V> p = pair(0, 1, 1), q = pair(0, 1, -1);
    const V t = p.s + q.s;
    s = s + t;
    m.y = m.y + (p.d + q.d);
    m.z = m.z + (p.d - q.d);
    m.yy = m.yy + t;
    m.zz = m.zz + t;
    m.yz = p.s - q.s;
  }
  // pairs towards the corners
  if constexpr (Q != 9) {
    const PairSD<V> a = pair(1, 1, 1), b = pair(1, 1, -1), c = pair(1, -1, 1), d = pair(1, -1, -1);
    const V ps = a.s + b.s, qs = c.s + d.s, pm = a.s - b.s, qm = c.s - d.s;
    const V pd = a.d + b.d, qd = c.d + d.d, t = ps + qs;
    s = s + t;
    m.x = m.x + (pd + qd);
    m.y = m.y + (pd - qd);
    m.z = m.z + ((a.d - b.d) + (c.d - d.d));
    m.xx = m.xx + t;
    m.yy = m.yy + t;
    m.zz = m.zz + t;
    m.xy = Q == 15 ? ps - qs : m.xy + (ps - qs);
    m.xz = Q == 15 ? pm + qm : m.xz + (pm + qm);
    m.yz = Q == 15 ? pm - qm : m.yz + (pm - qm);
  }
  m.s = s + ld(0, 0, 0);
  return m;
}

}  // namespace pfl
