// Meson two-point functions from a point-source propagator (paper Section 4,
// eq. 4.1):  C_Gamma(x) = - Tr[ S^dag(x) g5 Gamma S(x) Gamma g5 ],  trace over
// spin and colour, S(x) the 12 x 12 matrix whose column (beta, b) is the
// solution for the point source of spin beta, colour b, read at site x; and
// C_Gamma(t) = sum of C_Gamma(x) over the spatial sites of time slice t.
//
// In the chiral basis every Gamma used here, and so A = g5 Gamma and
// B = Gamma g5, has one non-zero per row and column, in the columns al ^ x for one
// x of {0, 2, 3} (0 for 1 and g5, 3 for g_x, g_y, 2 for g_z, g_t and their g5
// partners): A[al][al ^ x] = a_al, B[be ^ x][be] = b_be. Then
//   C(x) = - sum_{al, be} a_al b_be G_x[al][be],
//   G_x[al][be] = sum_{a, b} conj(S[al a][be b]) S[al^x a][be^x b],
// and since G_x[al^x][be^x] = conj(G_x[al][be]), the sixteen G_0 are real and eight
// complex entries (be = 0, 1) hold the others. C is linear in them, so the 48 real
// numbers are summed over the sites of a time slice first and every Gamma is formed
// once per slice.
#include <array>
#include <complex>
#include <cstring>
#include <vector>

#include "kernels.cuh"
#include "runtime.h"

namespace lqcd {

namespace {

constexpr int CTHREADS = 128;
constexpr int MAXG = 16;
constexpr int NGRAM = 48;  // 16 G_0, then 8 complex G_3, then 8 complex G_2

struct Monomial {  // one non-zero per row: M[r][col[r]] = (re[r], im[r])
  int col[4];
  double re[4], im[4];
};
struct GammaTab {      // a kernel argument
  double2 a[MAXG][4];  // A = g5 Gamma by rows
  double2 b[MAXG][4];  // Gamma g5 by columns
  int x[MAXG];         // the Gamma's x
  int use;             // bit x set: some Gamma has this x
};
struct Props {
  const double2* half[2][12];  // [parity][source]
};

using cd = std::complex<double>;
using M4 = std::array<std::array<cd, 4>, 4>;

M4 mat_mul(const M4& a, const M4& b) {
  M4 c{};
  for (int i = 0; i < 4; ++i)
    for (int j = 0; j < 4; ++j)
      for (int k = 0; k < 4; ++k) c[i][j] += a[i][k] * b[k][j];
  return c;
}

// chiral basis: g_k = [[0, -i s_k], [i s_k, 0]] (k = x, y, z), g_t = [[0, 1], [1, 0]]
M4 chiral_gamma(int mu) {
  const cd I(0, 1);
  const cd s[3][2][2] = {{{0, 1}, {1, 0}}, {{0, -I}, {I, 0}}, {{1, 0}, {0, -1}}};
  M4 g{};
  for (int a = 0; a < 2; ++a)
    for (int b = 0; b < 2; ++b) {
      if (mu < 3) {
        g[a][2 + b] = -I * s[mu][a][b];
        g[2 + a][b] = I * s[mu][a][b];
      } else if (a == b) {
        g[a][2 + b] = 1;
        g[2 + a][b] = 1;
      }
    }
  return g;
}

M4 gamma_of(int code) {
  M4 g5 = mat_mul(mat_mul(chiral_gamma(0), chiral_gamma(1)), mat_mul(chiral_gamma(2), chiral_gamma(3)));
  if (code == 0) {
    M4 one{};
    for (int i = 0; i < 4; ++i) one[i][i] = 1;
    return one;
  }
  if (code == 1) return g5;
  if (code >= 2 && code <= 5) return chiral_gamma(code - 2);
  return mat_mul(g5, chiral_gamma(code - 6));
}

bool monomial_rows(const M4& m, Monomial& out) {
  for (int r = 0; r < 4; ++r) {
    int n = 0;
    for (int c = 0; c < 4; ++c)
      if (std::abs(m[r][c]) > 1e-12) {
        out.col[r] = c;
        out.re[r] = m[r][c].real();
        out.im[r] = m[r][c].imag();
        ++n;
      }
    if (n != 1) return false;
  }
  return true;
}

// Sums of the 48 numbers over the sites of one CTA, a contiguous range of one parity's
// sites of one time slice (in the half-lattice index a slice is one range per parity).
//
// Bound by the FP64 pipe: 864 FMAs per site (288 for each x), 0.93 ms at 24^3x48 against
// 0.23 ms of HBM. For one colour pair (a, b) everything above involves only the 4 x 4
// spin matrix S[.. a][.. b], so a thread takes whole sites, one colour pair at a time:
// 16 coalesced 16-byte loads, each used in 6 FMAs, no shared memory, and the 48 sums stay
// in registers over the thread's sites. (The form before it staged each site's 144 numbers
// in shared memory at a 2304-byte stride, an eight-way bank conflict, formed all 48 complex
// Gram entries and combined the Gammas at every site: ten Gammas at 24^3x48 took 5.87 ms a
// call, this form 1.09 ms.)
__global__ void __launch_bounds__(CTHREADS, 2) k_meson(const Props p, int Vh, int slice, int nb, int use,
                                                       double* partials) {
  __shared__ double sm[16][CTHREADS + 1];
  const int blk = blockIdx.x % (2 * nb);
  const int t = blockIdx.x / (2 * nb);
  const int par = blk / nb, k = blk % nb;
  const int chunk = (slice + nb - 1) / nb;
  const int lo = t * slice + k * chunk, hi = min((t + 1) * slice, lo + chunk);
  double g0[16], g3[16], g2[16];
#pragma unroll
  for (int q = 0; q < 16; ++q) g0[q] = g3[q] = g2[q] = 0.0;
  for (int h = lo + (int)threadIdx.x; h < hi; h += CTHREADS) {
    for (int a = 0; a < 3; ++a) {
#pragma unroll 1
      for (int b = 0; b < 3; ++b) {
        double2 s[4][4];  // S[al a][be b]; component a * 4 + al of source 3 be + b
#pragma unroll
        for (int be = 0; be < 4; ++be) {
          const double2* base = p.half[par][3 * be + b] + h;
#pragma unroll
          for (int al = 0; al < 4; ++al) s[al][be] = __ldcs(base + (size_t)(a * 4 + al) * Vh);
        }
        if (use & 1) {
#pragma unroll
          for (int al = 0; al < 4; ++al)
#pragma unroll
            for (int be = 0; be < 4; ++be)
              g0[al * 4 + be] = fma(s[al][be].x, s[al][be].x, fma(s[al][be].y, s[al][be].y, g0[al * 4 + be]));
        }
        // conj(u) v for be = 0, 1
        auto cross = [&](double (&g)[16], int x) {
#pragma unroll
          for (int al = 0; al < 4; ++al)
#pragma unroll
            for (int be = 0; be < 2; ++be) {
              const double2 u = s[al][be], v = s[al ^ x][be ^ x];
              double& re = g[(al * 2 + be) * 2];
              double& im = g[(al * 2 + be) * 2 + 1];
              re = fma(u.x, v.x, fma(u.y, v.y, re));
              im = fma(u.x, v.y, fma(-u.y, v.x, im));
            }
        };
        if (use & 8) cross(g3, 3);
        if (use & 4) cross(g2, 2);
      }
    }
  }
  // fixed-order sum over the CTA: eight threads add sixteen values each of one number
  auto reduce = [&](const double (&g)[16], int first) {
    __syncthreads();
#pragma unroll
    for (int q = 0; q < 16; ++q) sm[q][threadIdx.x] = g[q];
    __syncthreads();
    const int q = threadIdx.x >> 3, l = threadIdx.x & 7;
    double v = 0.0;
#pragma unroll
    for (int i = 0; i < CTHREADS / 8; ++i) v += sm[q][i * 8 + l];
#pragma unroll
    for (int o = 4; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o, 8);
    if (l == 0) partials[(size_t)blockIdx.x * NGRAM + first + q] = v;
  };
  if (use & 1) reduce(g0, 0);
  if (use & 8) reduce(g3, 16);
  if (use & 4) reduce(g2, 32);
}

// One CTA per time slice: the slice's 48 numbers (its nblk partials added in a fixed order,
// four interleaved sums each), then C(t) for every Gamma.
__global__ void __launch_bounds__(4 * NGRAM) k_meson_slices(const double* partials, int ngam, int nblk, int lt,
                                                            const GammaTab tab, double* corr) {
  __shared__ double part[4][NGRAM], g[NGRAM];
  const int t = blockIdx.x, q = threadIdx.x % NGRAM, w = threadIdx.x / NGRAM;
  const int x = q < 16 ? 0 : (q < 32 ? 3 : 2);
  double v = 0.0;
  if ((tab.use >> x) & 1)
    for (int k = w; k < nblk; k += 4) v += partials[((size_t)t * nblk + k) * NGRAM + q];
  part[w][q] = v;
  __syncthreads();
  if (w == 0) g[q] = (part[0][q] + part[1][q]) + (part[2][q] + part[3][q]);
  __syncthreads();
  const int gm = threadIdx.x;
  if (gm >= ngam) return;
  double cr = 0.0, ci = 0.0;
  const int xg = tab.x[gm];
  auto add = [&](double2 a, double2 b, double re, double im) {  // a b (re + i im)
    const double pr = a.x * b.x - a.y * b.y, pi = a.x * b.y + a.y * b.x;
    cr += pr * re - pi * im;
    ci += pr * im + pi * re;
  };
  for (int al = 0; al < 4; ++al) {
    if (xg == 0) {
      for (int be = 0; be < 4; ++be) add(tab.a[gm][al], tab.b[gm][be], g[al * 4 + be], 0.0);
    } else {
      const double* gx = g + (xg == 3 ? 16 : 32);
      for (int be = 0; be < 2; ++be) {
        const double re = gx[(al * 2 + be) * 2], im = gx[(al * 2 + be) * 2 + 1];
        add(tab.a[gm][al], tab.b[gm][be], re, im);
        add(tab.a[gm][al ^ xg], tab.b[gm][be ^ xg], re, -im);
      }
    }
  }
  corr[((size_t)gm * lt + t) * 2] = -cr;
  corr[((size_t)gm * lt + t) * 2 + 1] = -ci;
}

}  // namespace
}  // namespace lqcd

using namespace lqcd;

extern "C" int lqcd_meson_correlator(const lqcd_field* const* props, int ngamma, const int* gammas,
                                     double* host_corr) {
  LQCD_TRACE("lqcd_meson_correlator");
  clear_error();
  if (!props || !gammas || !host_corr || ngamma < 1 || ngamma > MAXG)
    return set_error(LQCD_EINVAL, "bad arguments (ngamma = %d, at most %d)", ngamma, MAXG);
  const lqcd_field* f0 = props[0];
  if (!f0) return set_error(LQCD_EINVAL, "NULL propagator field");
  for (int i = 0; i < 12; ++i) {
    const lqcd_field* f = props[i];
    if (!f || f->prec != LQCD_F64 || f->subset != LQCD_FULL || f->ctx != f0->ctx ||
        memcmp(f->g.L, f0->g.L, sizeof f->g.L))
      return set_error(LQCD_EINVAL, "propagator %d: need 12 FULL FP64 fields of one lattice", i);
  }
  GammaTab tab;
  memset(&tab, 0, sizeof tab);
  const M4 g5 = gamma_of(1);
  for (int i = 0; i < ngamma; ++i) {
    if (gammas[i] < 0 || gammas[i] > 9) return set_error(LQCD_EINVAL, "gamma code %d", gammas[i]);
    const M4 G = gamma_of(gammas[i]);
    const M4 A = mat_mul(g5, G), B = mat_mul(G, g5);
    M4 Bt{};
    for (int r = 0; r < 4; ++r)
      for (int c = 0; c < 4; ++c) Bt[c][r] = B[r][c];
    Monomial ma, mb;
    if (!monomial_rows(A, ma) || !monomial_rows(Bt, mb))
      return set_error(LQCD_EINVAL, "gamma code %d is not monomial", gammas[i]);
    const int x = ma.col[0];
    for (int r = 0; r < 4; ++r) {
      if ((x != 0 && x != 2 && x != 3) || ma.col[r] != (r ^ x) || mb.col[r] != (r ^ x))
        return set_error(LQCD_EINVAL, "gamma code %d: unexpected spin structure", gammas[i]);
      tab.a[i][r] = make_double2(ma.re[r], ma.im[r]);
      tab.b[i][r] = make_double2(mb.re[r], mb.im[r]);
    }
    tab.x[i] = x;
    tab.use |= 1 << x;
  }
  lqcd_ctx* c = f0->ctx;
  LQCD_TRY(ctx_enter(c));
  const Geom& g = f0->g;
  Props props_arg;
  for (int i = 0; i < 12; ++i)
    for (int p = 0; p < 2; ++p) props_arg.half[p][i] = static_cast<const double2*>(props[i]->half[p]);
  // Two sites per thread: the 48 sums' reduction costs about 3% of the site work, and CTAs
  // stay small enough for even waves; one site per thread while that fills no more than the
  // resident CTAs.
  const int lt = g.L[3], slice = g.Vh / lt;
  int nb = (slice + CTHREADS - 1) / CTHREADS;
  if ((long long)2 * nb * lt > 2 * device_sm_count()) nb = (slice + 2 * CTHREADS - 1) / (2 * CTHREADS);
  const int nblk = 2 * nb;  // per slice
  const size_t npart = (size_t)nblk * lt * NGRAM;
  const int nout = 2 * ngamma * lt;
  LQCD_TRY(ctx_staging(c, (npart + nout) * sizeof(double)));
  double* d_part = c->staging;
  double* d_corr = d_part + npart;  // ngamma x Lt complex, after the partials
  k_meson<<<(unsigned)(nblk * lt), CTHREADS, 0, c->stream>>>(props_arg, g.Vh, slice, nb, tab.use, d_part);
  k_meson_slices<<<lt, 4 * NGRAM, 0, c->stream>>>(d_part, ngamma, nblk, lt, tab, d_corr);
  LQCD_CK(cudaGetLastError());
  c->launches += 2;
  LQCD_CK(cudaMemcpyAsync(host_corr, d_corr, (size_t)nout * sizeof(double), cudaMemcpyDeviceToHost, c->stream));
  LQCD_CK(cudaStreamSynchronize(c->stream));
  return LQCD_OK;
}
