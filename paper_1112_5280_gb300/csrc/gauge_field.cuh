// SU(3) helpers shared by the pure-gauge kernels (heatbath.cu) and the HMC kernels
// (hmc.cu): complex 3x3 matrices in registers, site coordinates of the even-odd index,
// and loads / stores of links in the FP64 18-real layout [parity][mu][word][V/2] of
// double2 (word = row * 3 + column).
#pragma once

#include "dslash.cuh"

namespace lqcd {
namespace gf {

struct C2 {
  double re, im;
};
__device__ __forceinline__ C2 cmul(C2 a, C2 b) { return {a.re * b.re - a.im * b.im, a.re * b.im + a.im * b.re}; }

struct M3 {
  C2 e[9];
};

// ---------------------------------------------------------------- geometry and links

struct Site {
  int c[4];
};

__device__ __forceinline__ Site site_of(const Geom& g, int par, int h) {
  Site s;
  const unsigned r0 = geom_div(g, 0, (unsigned)h);
  const int xh = h - (int)r0 * g.Lxh;
  const unsigned r1 = geom_div(g, 1, r0);
  s.c[1] = (int)r0 - (int)r1 * g.L[1];
  const unsigned r2 = geom_div(g, 2, r1);
  s.c[2] = (int)r1 - (int)r2 * g.L[2];
  s.c[3] = (int)r2;
  s.c[0] = 2 * xh + ((par + s.c[1] + s.c[2] + s.c[3]) & 1);
  return s;
}
__device__ __forceinline__ Site shifted(const Geom& g, Site s, int mu, int d) {
  int v = s.c[mu] + d;
  v = v < 0 ? v + g.L[mu] : (v >= g.L[mu] ? v - g.L[mu] : v);
  s.c[mu] = v;
  return s;
}
// double2 index of word 0 of link (site, mu) in the FP64 18-real layout
__device__ __forceinline__ size_t link_base(const Geom& g, const Site& s, int mu) {
  const int par = (s.c[0] + s.c[1] + s.c[2] + s.c[3]) & 1;
  const int h = (s.c[0] >> 1) + g.Lxh * (s.c[1] + g.L[1] * (s.c[2] + g.L[2] * s.c[3]));
  return (size_t)(par * 4 + mu) * 9 * g.Vh + h;
}
__device__ __forceinline__ M3 load_link(const double2* U, const Geom& g, const Site& s, int mu) {
  const size_t b = link_base(g, s, mu);
  M3 m;
#pragma unroll
  for (int w = 0; w < 9; ++w) {
    const double2 d = U[b + (size_t)w * g.Vh];
    m.e[w] = {d.x, d.y};
  }
  return m;
}
// a + b c, four multiply-adds
__device__ __forceinline__ C2 cmac(C2 a, C2 b, C2 c) {
  return {fma(-b.im, c.im, fma(b.re, c.re, a.re)), fma(b.im, c.re, fma(b.re, c.im, a.im))};
}
// ---------------------------------------------------------------- double-float matrices
// The FP64 pipes of this part run at 1/64 of the FP32 rate, so the SU(3) products of the
// gauge kernels run in double-float (pairs of FP32, 48-bit significand) on the FP32 pipes,
// reading the gauge field's double-float copy (float4 = (re.hi, re.lo, im.hi, im.lo) per
// complex entry, the same word layout as the FP64 master). Products accumulate unnormalised
// and each entry is normalised once.

// A double as an (unnormalised) double-float pair by integer operations on its bits, for
// kernels where the conversion instructions would load the FP64 pipe (1/64 of the FP32
// rate on this part): hi keeps the top 24 significant bits (truncated), lo the next 24 of
// the remaining 29 (truncated), so hi + lo is within 2^-47 relative of x and |lo| < ulp(hi).
// Exponents outside +-60 (including zero, subnormals, inf and NaN) take the FP64 path.
__device__ __forceinline__ df64 df_split_bits(double x) {
  const unsigned long long b = (unsigned long long)__double_as_longlong(x);
  const unsigned hw = (unsigned)(b >> 32), lw = (unsigned)b;
  const int E = (int)((hw >> 20) & 0x7ffu);
  if (E < 1023 - 60 || E > 1023 + 60) return df64(x);
  const unsigned sign = hw & 0x80000000u;
  const float hi = __uint_as_float(sign | ((unsigned)(E - 896) << 23) | ((hw & 0xfffffu) << 3) | (lw >> 29));
  const unsigned rem = lw & 0x1fffffffu;  // weight 2^(E - 1075) per unit
  if (rem == 0u) return df64(hi, 0.0f);
  const int top = 31 - __clz((int)rem);  // leading bit, <= 28
  const unsigned m = top >= 23 ? rem >> (top - 23) : rem << (23 - top);
  const float lo = __uint_as_float(sign | ((unsigned)(top + E - 948) << 23) | (m & 0x7fffffu));
  return df64(hi, lo);
}

struct C2d {
  df64 re, im;
};
struct M3d {
  C2d e[9];
};

__device__ __forceinline__ M3d load_link_df(const float4* U, const Geom& g, const Site& s, int mu) {
  const size_t b = link_base(g, s, mu);
  M3d m;
#pragma unroll
  for (int w = 0; w < 9; ++w) {
    const float4 d = U[b + (size_t)w * g.Vh];
    m.e[w] = {df64(d.x, d.y), df64(d.z, d.w)};
  }
  return m;
}
__device__ __forceinline__ void store_link_df(float4* U, const Geom& g, const Site& s, int mu, const M3d& m) {
  const size_t b = link_base(g, s, mu);
#pragma unroll
  for (int w = 0; w < 9; ++w) U[b + (size_t)w * g.Vh] = make_float4(m.e[w].re.hi, m.e[w].re.lo, m.e[w].im.hi, m.e[w].im.lo);
}
// Complex double-float scalars and matrices in packed arithmetic: the lanes are the real
// and the imaginary part, so c += x y takes two packed multiply-accumulates, x.re (y.re, y.im)
// and x.im (-y.im, y.re), in the order of the scalar form's four.
__device__ __forceinline__ df64x2 c_pack(const C2d& a) { return df2_pack(a.re, a.im); }
__device__ __forceinline__ df64x2 c_rot(const C2d& a) { return df2_pack(-a.im, a.re); }  // i a
__device__ __forceinline__ df64x2 c_dup(df64 a) { return df2_pack(a, a); }
__device__ __forceinline__ C2d c_unpack(df64x2 v) {
  C2d r;
  df2_unpack(v, r.re, r.im);
  return r;
}
__device__ __forceinline__ df64x2 c_zero() { return {0ull, 0ull}; }
__device__ __forceinline__ df64x2 c_mul(const C2d& x, const C2d& y) {  // x y
  df64x2 s = df2_mul_u(c_dup(x.re), c_pack(y));
  df2_mac_u(s, c_dup(x.im), c_rot(y));
  return s;
}
__device__ __forceinline__ void c_mac(df64x2& acc, const C2d& x, const C2d& y) {  // acc += x y
  df2_mac_u(acc, c_dup(x.re), c_pack(y));
  df2_mac_u(acc, c_dup(x.im), c_rot(y));
}

__device__ __forceinline__ C2d cmul_d(const C2d& a, const C2d& b) {
  return c_unpack(df2_norm(c_mul(a, b)));
}
__device__ __forceinline__ C2d cadd_d(const C2d& a, const C2d& b) {
  return c_unpack(df2_norm(df2_add_u(c_pack(a), c_pack(b))));
}
__device__ __forceinline__ C2d csub_d(const C2d& a, const C2d& b) { return cadd_d(a, {-b.re, -b.im}); }
__device__ __forceinline__ C2d cscale_d(df64 f, const C2d& a) { return {f * a.re, f * a.im}; }

// a x + b y in double-float
__device__ __forceinline__ C2d cmix_d(const C2d& a, const C2d& x, const C2d& b, const C2d& y) {
  df64x2 s = c_mul(a, x);
  c_mac(s, b, y);
  return c_unpack(df2_norm(s));
}

// 1/sqrt(n) for n > 0 in double-float: the FP32 estimate and two Newton-Raphson steps
// y <- y + y (1 - n y^2) / 2, each of which squares the relative error
__device__ __forceinline__ df64 df_rsqrt(df64 n) {
  df64 y(rsqrtf(n.hi), 0.0f);
#pragma unroll
  for (int it = 0; it < 2; ++it) {
    const df64 r = df64(1.0f, 0.0f) - n * (y * y);
    y = y + y * r * df64(0.5f, 0.0f);
  }
  return y;
}

// op(a) op(b) with op the adjoint where asked: each entry accumulates unnormalised over k and
// is normalised once. Per k, an entry of b serves the three rows i at once.
template <bool DAGA, bool DAGB>
__device__ __forceinline__ M3d mul_d(const M3d& a, const M3d& b) {
  df64x2 s[9];
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    df64x2 xr[3], xi[3];
#pragma unroll
    for (int i = 0; i < 3; ++i) {
      const C2d x = DAGA ? a.e[k * 3 + i] : a.e[i * 3 + k];
      xr[i] = c_dup(x.re);
      xi[i] = c_dup(DAGA ? -x.im : x.im);
    }
#pragma unroll
    for (int j = 0; j < 3; ++j) {
      C2d y = DAGB ? b.e[j * 3 + k] : b.e[k * 3 + j];
      if (DAGB) y.im = -y.im;
      const df64x2 yp = c_pack(y), yr = c_rot(y);
#pragma unroll
      for (int i = 0; i < 3; ++i) {
        if (k == 0) s[i * 3 + j] = df2_mul_u(xr[i], yp);
        else df2_mac_u(s[i * 3 + j], xr[i], yp);
        df2_mac_u(s[i * 3 + j], xi[i], yr);
      }
    }
  }
  M3d c;
#pragma unroll
  for (int i = 0; i < 9; ++i) c.e[i] = c_unpack(df2_norm(s[i]));
  return c;
}

// coordinate nu of s and the site shifted by d in direction nu, for a direction known only
// at run time (selects, so that the site stays in registers)
__device__ __forceinline__ int coord(const Site& s, int nu) {
  return nu == 0 ? s.c[0] : (nu == 1 ? s.c[1] : (nu == 2 ? s.c[2] : s.c[3]));
}
__device__ __forceinline__ Site shifted_rt(const Geom& g, Site s, int nu, int d) {
  const int L = nu == 0 ? g.L[0] : (nu == 1 ? g.L[1] : (nu == 2 ? g.L[2] : g.L[3]));
  int v = coord(s, nu) + d;
  v = v < 0 ? v + L : (v >= L ? v - L : v);
#pragma unroll
  for (int k = 0; k < 4; ++k) s.c[k] = (nu == k) ? v : s.c[k];
  return s;
}

// ---------------------------------------------------------------- row-split products
// Three threads per link, thread i holding row i of the matrix that is built up. A row of
// a b needs row i of a and all of b, so a chain of products splits over rows without extra
// arithmetic, and a thread needs a third of the accumulators: 24 warps per SM can be
// resident where one thread per link took 254 registers (8 warps), which left the loads and
// the chains of dependent operations uncovered (FMA pipe 60% busy). Entries are packed
// (lanes re, im), each accumulated in the same order as in mul_d.
struct RowD {
  df64x2 e[3];
};
constexpr int SPLIT_LINKS = 64;                 // links per CTA
constexpr int SPLIT_THREADS = 3 * SPLIT_LINKS;  // thread 64 i + j: row (or column) i of link j

// one entry (re.hi, re.lo, im.hi, im.lo) as a packed pair, its imaginary part's sign flipped
// by flip (0 or 0x80000000)
__device__ __forceinline__ df64x2 c_entry(const float4& d, unsigned flip) {
  const float ih = __uint_as_float(__float_as_uint(d.z) ^ flip), il = __uint_as_float(__float_as_uint(d.w) ^ flip);
  return {p_pack(d.x, ih), p_pack(d.y, il)};
}
__device__ __forceinline__ df64x2 c_times_i(df64x2 a) {
  C2d c = c_unpack(a);
  return c_rot(c);
}
__device__ __forceinline__ void c_dups(df64x2 a, df64x2& re, df64x2& im) {
  const C2d c = c_unpack(a);
  re = c_dup(c.re);
  im = c_dup(c.im);
}

// Row i of the staple sum
//   W_mu(x) = sum_{nu != mu} U_nu(x+mu) U_mu(x+nu)^dag U_nu(x)^dag
//                          + U_nu(x+mu-nu)^dag U_mu(x-nu)^dag U_nu(x-nu)
// for a direction mu known at run time, from the double-float copy Ud. The six staples run
// through one loop body of two products
//   up (nu):   T = U_nu(x+mu) U_mu(x+nu)^dag,          W += T U_nu(x)^dag
//   down (nu): T = U_nu(x+mu-nu)^dag U_mu(x-nu)^dag,   W += T U_nu(x-nu)
// so that its instructions stay in the instruction cache; an adjoint is a choice of the
// words read and of the sign of the imaginary parts.
__device__ __forceinline__ RowD staple_row(const float4* Ud, const Geom& g, const Site& x, int mu, int i) {
  RowD W;
#pragma unroll
  for (int c = 0; c < 3; ++c) W.e[c] = c_zero();
  const Site xp = shifted_rt(g, x, mu, 1);
  const size_t vh = (size_t)g.Vh;
#pragma unroll 1
  for (int t = 0; t < 6; ++t) {
    const int k0 = t >> 1, nu = k0 + (k0 >= mu ? 1 : 0);
    const bool up = (t & 1) == 0;
    const Site s0 = up ? xp : shifted_rt(g, xp, nu, -1);
    const Site s1 = shifted_rt(g, x, nu, up ? 1 : -1);
    const Site s2 = up ? x : s1;
    const unsigned flip_a = up ? 0u : 0x80000000u, flip_c = up ? 0x80000000u : 0u;
    const size_t row = vh * 3, one = vh;
    const float4* a = Ud + link_base(g, s0, nu) + (size_t)i * (up ? row : one);
    const float4* b = Ud + link_base(g, s1, mu);
    const float4* c = Ud + link_base(g, s2, nu);
    const size_t a_step = up ? one : row;                        // over k
    const size_t c_row = up ? one : row, c_col = up ? row : one;  // over k and over the column
    RowD T;
    {
      df64x2 xr[3], xi[3];
#pragma unroll
      for (int k = 0; k < 3; ++k) c_dups(c_entry(a[k * a_step], flip_a), xr[k], xi[k]);
#pragma unroll
      for (int j = 0; j < 3; ++j) {
        df64x2 s;
#pragma unroll
        for (int k = 0; k < 3; ++k) {
          const df64x2 y = c_entry(b[(size_t)(3 * j + k) * vh], 0x80000000u);
          if (k == 0) s = df2_mul_u(xr[k], y);
          else df2_mac_u(s, xr[k], y);
          df2_mac_u(s, xi[k], c_times_i(y));
        }
        T.e[j] = df2_norm(s);
      }
    }
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      df64x2 xr, xi;
      c_dups(T.e[k], xr, xi);
#pragma unroll
      for (int q = 0; q < 3; ++q) {
        const df64x2 y = c_entry(c[k * c_row + q * c_col], flip_c);
        df2_mac_u(W.e[q], xr, y);
        df2_mac_u(W.e[q], xi, c_times_i(y));
      }
    }
#pragma unroll
    for (int q = 0; q < 3; ++q) W.e[q] = df2_norm(W.e[q]);
  }
  return W;
}

// A CTA's matrices in shared memory, one per link: entry [row][column][link]
struct SplitM {
  ulonglong2 e[3][3][SPLIT_LINKS];
  __device__ __forceinline__ void put(int r, int c, int j, df64x2 v) { e[r][c][j] = make_ulonglong2(v.hi, v.lo); }
  __device__ __forceinline__ df64x2 get(int r, int c, int j) const {
    const ulonglong2 v = e[r][c][j];
    return {v.x, v.y};
  }
};

// row i of U W for the thread's link j: U's words from u (stride vh), W in shared memory
__device__ __forceinline__ RowD split_row_times(const float4* u, size_t vh, int i, const SplitM& w, int j) {
  RowD r;
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    df64x2 xr, xi;
    c_dups(c_entry(u[(size_t)(3 * i + k) * vh], 0u), xr, xi);
#pragma unroll
    for (int q = 0; q < 3; ++q) {
      const df64x2 y = w.get(k, q, j);
      if (k == 0) r.e[q] = df2_mul_u(xr, y);
      else df2_mac_u(r.e[q], xr, y);
      df2_mac_u(r.e[q], xi, c_times_i(y));
    }
  }
#pragma unroll
  for (int q = 0; q < 3; ++q) r.e[q] = df2_norm(r.e[q]);
  return r;
}

}  // namespace gf
}  // namespace lqcd
