// Layout kernels (gauge and spinor upload, even-odd split, precision
// conversion, link compression) and the host dispatch of batched launches.
#include <atomic>
#include <cstdlib>
#include <mutex>
#include <unordered_map>

#include "convert.cuh"
#include "launch.h"

namespace lqcd {

// Layouts. On the host side of a copy a field is an array of sites of FP64 reals (AoS); on
// the device it is a structure of arrays of words, word(c, h) = base[c * Vh + h]. Every
// kernel here is bound by HBM, so each side is read and written in runs of consecutive
// addresses by consecutive threads: the AoS kernels pass a tile of sites through shared
// memory, and the conversions between two device layouts move whole words (eight reals of
// a spinor, one link). FP64 <-> FP32 / double-float conversions take the bits apart
// (convert.cuh) because the conversion instructions run at the FP64 pipe's rate.
// Measured on GB300 against one thread per site reading and writing single reals, per call
// with everything else unchanged: a 32^3x64 FP16 operator chain with its result to the host
// layout 1379 -> 1295 us (the download 181 -> 98 us), a 24^3x48 double-float one 1670 ->
// 1618 us, a 22x18x14x38 configuration and source in and the result out 777 -> 723 us.
// They are programmatic dependents and let theirs start, as the operators between them do: a
// download between two 8^4 M-hats 12.3 -> 9.65 us a call.

// ------------------------------------------------------------------ words

// The words of one spinor's reals: W reals of a storage word, to and from FP64.
template <int P>
struct Words;
template <>
struct Words<P_F64> {
  using T = double2;
  static constexpr int W = 2;
  __device__ static void get(const T& w, double* v) { v[0] = w.x; v[1] = w.y; }
  __device__ static T put(const double* v) { return make_double2(v[0], v[1]); }
};
template <>
struct Words<P_DF64> {
  using T = float4;
  static constexpr int W = 2;
  __device__ static void get(const T& w, double* v) {
    v[0] = cv::from_df(w.x, w.y);
    v[1] = cv::from_df(w.z, w.w);
  }
  __device__ static T put(const double* v) {
    T w;
    cv::to_df(v[0], w.x, w.y);
    cv::to_df(v[1], w.z, w.w);
    return w;
  }
};
template <>
struct Words<P_F32> {
  using T = float4;
  static constexpr int W = 4;
  __device__ static void get(const T& w, double* v) {
    v[0] = cv::to_double(w.x); v[1] = cv::to_double(w.y); v[2] = cv::to_double(w.z); v[3] = cv::to_double(w.w);
  }
  __device__ static T put(const double* v) {
    return make_float4(cv::to_float(v[0]), cv::to_float(v[1]), cv::to_float(v[2]), cv::to_float(v[3]));
  }
};
template <bool BF>
struct WordsHalf {
  using T = uint4;
  static constexpr int W = 8;
  __device__ static unsigned pair(double a, double b) {
    if (BF) {
      const __nv_bfloat162 h(__double2bfloat16(a), __double2bfloat16(b));
      return *reinterpret_cast<const unsigned*>(&h);
    }
    const __half2 h(__double2half(a), __double2half(b));
    return *reinterpret_cast<const unsigned*>(&h);
  }
  __device__ static unsigned pair_bits(double a, double b) {
    return BF ? cv::to_bf16(a) | (cv::to_bf16(b) << 16) : cv::to_half(a) | (cv::to_half(b) << 16);
  }
  __device__ static void get2(unsigned w, double* v) {
    const float2 f = BF ? unpack_b2(w) : unpack_h2(w);
    v[0] = cv::to_double(f.x);
    v[1] = cv::to_double(f.y);
  }
  __device__ static void get(const T& w, double* v) {
    get2(w.x, v); get2(w.y, v + 2); get2(w.z, v + 4); get2(w.w, v + 6);
  }
  __device__ static T put(const double* v) {
    return make_uint4(pair(v[0], v[1]), pair(v[2], v[3]), pair(v[4], v[5]), pair(v[6], v[7]));
  }
  // the same on integer bits, for k_spinor_convert: its threads convert in step, one word each,
  // and the conversion instructions do not overlap with its loads (FP64 to FP16 at 16^3x32 20.6
  // -> 13.0 us); the other kernels hide them (an FP16 upload at 32^3x64 99.5 us, by bits 105.8)
  __device__ static T put_bits(const double* v) {
    return make_uint4(pair_bits(v[0], v[1]), pair_bits(v[2], v[3]), pair_bits(v[4], v[5]), pair_bits(v[6], v[7]));
  }
};
template <>
struct Words<P_F16> : WordsHalf<false> {};
template <>
struct Words<P_BF16> : WordsHalf<true> {};

// host real k = (spin * 3 + colour) * 2 + re/im  ->  device position (colour-major)
__device__ __forceinline__ int dev_real(int k) {
  const int ri = k & 1, sc = k >> 1, spin = sc / 3, col = sc % 3;
  return sidx(spin, col) + ri;
}

// (y + z + t) & 1 of half-lattice index h: the even site of the pair 2h, 2h + 1 of the host
// order is 2h when this is 0
__device__ __forceinline__ int row_parity(const Geom& g, int h) {
  const unsigned r0 = geom_div(g, 0, (unsigned)h), r1 = geom_div(g, 1, r0), r2 = geom_div(g, 2, r1);
  return (int)((r0 - r1 * g.L[1]) + (r1 - r2 * g.L[2]) + r2) & 1;
}

// A tile is the 64 consecutive host sites 2 h0 .. 2 h0 + 63, which hold the half-lattice
// sites h0 .. h0 + 31 of both parities. In shared memory site 2h + b of the tile is at
// [b][h][.], its row padded to an odd number of FP64 words, so that 32 threads at
// consecutive h hit different banks.
constexpr int TILE_H = 32;
constexpr int LAYOUT_THREADS = 256;

// ------------------------------------------------------------------ gauge (FP64, 18 reals)

// TO_AOS false: AoS U[site][mu][row][col] -> [parity][mu][word][V/2] of double2; true: back
template <bool TO_AOS>
__global__ void __launch_bounds__(LAYOUT_THREADS) k_gauge_aos(const double* in, Geom g, double* out) {
  pdl_entry();
  __shared__ double sm[2][TILE_H][73];
  const int h0 = blockIdx.x * TILE_H, nh = min(TILE_H, g.Vh - h0);
  const size_t first = (size_t)h0 * 2 * 72;
  if (!TO_AOS) {
    for (int i = threadIdx.x; i < 2 * nh * 72; i += LAYOUT_THREADS) {
      const int site = i / 72;
      sm[site & 1][site >> 1][i - site * 72] = in[first + i];
    }
    __syncthreads();
  }
  const int hl = threadIdx.x % TILE_H;
  if (hl < nh) {
    const int rp = row_parity(g, h0 + hl);
    for (int q = threadIdx.x / TILE_H; q < 2 * 36; q += LAYOUT_THREADS / TILE_H) {
      const int par = q / 36, w = q - par * 36;  // w = mu * 9 + word
      double* s = &sm[par ^ rp][hl][2 * w];
      const size_t at = (size_t)q * g.Vh + h0 + hl;
      if (TO_AOS) {
        const double2 d = reinterpret_cast<const double2*>(in)[at];
        s[0] = d.x;
        s[1] = d.y;
      } else {
        reinterpret_cast<double2*>(out)[at] = make_double2(s[0], s[1]);
      }
    }
  }
  if (TO_AOS) {
    __syncthreads();
    for (int i = threadIdx.x; i < 2 * nh * 72; i += LAYOUT_THREADS) {
      const int site = i / 72;
      out[first + i] = sm[site & 1][site >> 1][i - site * 72];
    }
  }
}

static unsigned aos_grid(const Geom& g) { return (unsigned)((g.Vh + TILE_H - 1) / TILE_H); }

cudaError_t links_from_aos(const double* aos, const Geom& g, double2* U, cudaStream_t s) {
  return launch_k(k_gauge_aos<false>, dim3(aos_grid(g)), dim3(LAYOUT_THREADS), 0, s, aos, g,
                  reinterpret_cast<double*>(U));
}
cudaError_t links_to_aos(const double2* U, const Geom& g, double2* aos, cudaStream_t s) {
  return launch_k(k_gauge_aos<true>, dim3(aos_grid(g)), dim3(LAYOUT_THREADS), 0, s,
                  reinterpret_cast<const double*>(U), g, reinterpret_cast<double*>(aos));
}

// One link of the FP64 18-real layout to precision P with NR reals; word sizes as in LinkIO.
template <int P, int NR>
__global__ void __launch_bounds__(LAYOUT_THREADS) k_gauge_convert(const double2* __restrict__ in64, Geom g, void* out) {
  pdl_entry();
  const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;  // (par, mu, h)
  if (i >= 8LL * g.Vh) return;
  const size_t pm = (size_t)(i / g.Vh);  // 4 par + mu
  const size_t Vh = (size_t)g.Vh, h = (size_t)i - pm * Vh;
  double v[NR];
#pragma unroll
  for (int w = 0; w < NR / 2; ++w) {
    const double2 d = in64[(pm * 9 + w) * Vh + h];
    v[2 * w] = d.x;
    v[2 * w + 1] = d.y;
  }
  constexpr int NW = LinkIO<P, NR>::NW;
  typename LinkIO<P, NR>::Word* o = reinterpret_cast<typename LinkIO<P, NR>::Word*>(out) + pm * NW * Vh + h;
#pragma unroll
  for (int w = 0; w < NW; ++w) {
    if constexpr (P == P_F64 || P == P_DF64) {
      o[w * Vh] = Words<P>::put(v + 2 * w);
    } else if constexpr (P == P_F32 && NR == 18) {
      o[w * Vh] = make_float2(cv::to_float(v[2 * w]), cv::to_float(v[2 * w + 1]));
    } else if constexpr (P == P_F32) {
      o[w * Vh] = Words<P_F32>::put(v + 4 * w);
    } else if constexpr (NR == 18) {
      o[w * Vh] = WordsHalf<false>::pair(v[2 * w], v[2 * w + 1]);
    } else {
      o[w * Vh] = make_uint2(WordsHalf<false>::pair(v[4 * w], v[4 * w + 1]),
                             WordsHalf<false>::pair(v[4 * w + 2], v[4 * w + 3]));
    }
  }
}

template <int P, int NR>
static cudaError_t go_gauge_convert(const void* a, const Geom& g, void* o, cudaStream_t s) {
  const long long n = 8LL * g.Vh;
  return launch_k(k_gauge_convert<P, NR>, dim3((unsigned)((n + LAYOUT_THREADS - 1) / LAYOUT_THREADS)),
                  dim3(LAYOUT_THREADS), 0, s, static_cast<const double2*>(a), g, o);
}

cudaError_t gauge_convert(const void* d64, const Geom& g, int prec, int nr, void* d_out,
                          cudaStream_t s) {
  if (prec == P_F64) return nr == 12 ? go_gauge_convert<P_F64, 12>(d64, g, d_out, s)
                                     : go_gauge_convert<P_F64, 18>(d64, g, d_out, s);
  if (prec == P_F32) return nr == 12 ? go_gauge_convert<P_F32, 12>(d64, g, d_out, s)
                                     : go_gauge_convert<P_F32, 18>(d64, g, d_out, s);
  if (prec == P_F16) return nr == 12 ? go_gauge_convert<P_F16, 12>(d64, g, d_out, s)
                                     : go_gauge_convert<P_F16, 18>(d64, g, d_out, s);
  if (prec == P_DF64 && nr == 18) return go_gauge_convert<P_DF64, 18>(d64, g, d_out, s);
  return cudaErrorInvalidValue;
}

// FP64 master words from the double-float copy (hi + lo, exact in FP64)
__global__ void __launch_bounds__(LAYOUT_THREADS) k_master_from_df(double2* U, const float4* Ud, long long n) {
  pdl_entry();
  const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  const float4 d = Ud[i];
  U[i] = make_double2(cv::from_df(d.x, d.y), cv::from_df(d.z, d.w));
}
cudaError_t master_from_df(double2* U, const float4* Ud, const Geom& g, cudaStream_t s) {
  const long long n = 72LL * g.Vh;
  return launch_k(k_master_from_df, dim3((unsigned)((n + LAYOUT_THREADS - 1) / LAYOUT_THREADS)),
                  dim3(LAYOUT_THREADS), 0, s, U, Ud, n);
}

// ------------------------------------------------------------------ spinors

template <int P>
__global__ void __launch_bounds__(LAYOUT_THREADS) k_spinor_from_aos(const double* __restrict__ aos, Geom g, void* ev,
                                                                    void* od) {
  pdl_entry();
  using Wd = Words<P>;
  __shared__ double sm[2][TILE_H][25];
  const int h0 = blockIdx.x * TILE_H, nh = min(TILE_H, g.Vh - h0);
  const double* src = aos + (size_t)h0 * 2 * 24;
  for (int i = threadIdx.x; i < 2 * nh * 24; i += LAYOUT_THREADS) {
    const int site = i / 24;
    sm[site & 1][site >> 1][dev_real(i - site * 24)] = src[i];
  }
  __syncthreads();
  const int hl = threadIdx.x % TILE_H;
  if (hl >= nh) return;
  const int rp = row_parity(g, h0 + hl);
  constexpr int NW = 24 / Wd::W;
  for (int q = threadIdx.x / TILE_H; q < 2 * NW; q += LAYOUT_THREADS / TILE_H) {
    const int par = q / NW, c = q - par * NW;
    void* dst = par ? od : ev;
    if (dst) reinterpret_cast<typename Wd::T*>(dst)[(size_t)c * g.Vh + h0 + hl] = Wd::put(&sm[par ^ rp][hl][c * Wd::W]);
  }
}

template <int P>
__global__ void __launch_bounds__(LAYOUT_THREADS) k_spinor_to_aos(const void* ev, const void* od, Geom g,
                                                                  double* __restrict__ aos) {
  pdl_entry();
  using Wd = Words<P>;
  __shared__ double sm[2][TILE_H][25];
  __shared__ int rps[TILE_H];
  const int h0 = blockIdx.x * TILE_H, nh = min(TILE_H, g.Vh - h0);
  const int hl = threadIdx.x % TILE_H;
  if (hl < nh) {
    const int rp = row_parity(g, h0 + hl);
    if (threadIdx.x < TILE_H) rps[hl] = rp;
    constexpr int NW = 24 / Wd::W;
    for (int q = threadIdx.x / TILE_H; q < 2 * NW; q += LAYOUT_THREADS / TILE_H) {
      const int par = q / NW, c = q - par * NW;
      const void* src = par ? od : ev;
      if (src) {
        double v[Wd::W];
        Wd::get(reinterpret_cast<const typename Wd::T*>(src)[(size_t)c * g.Vh + h0 + hl], v);
#pragma unroll
        for (int j = 0; j < Wd::W; ++j) sm[par ^ rp][hl][c * Wd::W + j] = v[j];
      }
    }
  }
  __syncthreads();
  double* dst = aos + (size_t)h0 * 2 * 24;
  for (int i = threadIdx.x; i < 2 * nh * 24; i += LAYOUT_THREADS) {
    const int site = i / 24, b = site & 1, h = site >> 1;
    // the site's parity is b ^ rp; sites of a parity that the field does not hold stay
    if ((b ^ rps[h]) ? od : ev) dst[i] = sm[b][h][dev_real(i - site * 24)];
  }
}

// One thread per site and eight reals (one FP16 word, two FP32, four FP64 or double-float).
template <int PI, int PO>
__global__ void __launch_bounds__(LAYOUT_THREADS) k_spinor_convert(const void* in, void* out, int Vh, double scale) {
  pdl_wait();
  if (in != out) pdl_trigger();  // in place: the next grid starts when this one is done
  using Wi = Words<PI>;
  using Wo = Words<PO>;
  const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;  // (group, h)
  if (i >= 3LL * Vh) return;
  const size_t grp = (size_t)(i / Vh), h = (size_t)i - grp * Vh;
  constexpr int NI = 8 / Wi::W, NO = 8 / Wo::W;
  const typename Wi::T* src = reinterpret_cast<const typename Wi::T*>(in) + grp * NI * Vh + h;
  typename Wo::T* dst = reinterpret_cast<typename Wo::T*>(out) + grp * NO * Vh + h;
  double v[8];
#pragma unroll
  for (int w = 0; w < NI; ++w) Wi::get(src[(size_t)w * Vh], v + w * Wi::W);
  if (scale != 1.0) {
#pragma unroll
    for (int k = 0; k < 8; ++k) v[k] *= scale;
  }
#pragma unroll
  for (int w = 0; w < NO; ++w) {
    if constexpr (PO == P_F16 || PO == P_BF16) dst[(size_t)w * Vh] = Wo::put_bits(v + w * Wo::W);
    else dst[(size_t)w * Vh] = Wo::put(v + w * Wo::W);
  }
}

template <int P>
static cudaError_t go_from_aos(const double* a, const Geom& g, void* e, void* o, cudaStream_t s) {
  return launch_k(k_spinor_from_aos<P>, dim3(aos_grid(g)), dim3(LAYOUT_THREADS), 0, s, a, g, e, o);
}
template <int P>
static cudaError_t go_to_aos(const void* e, const void* o, const Geom& g, double* a, cudaStream_t s) {
  return launch_k(k_spinor_to_aos<P>, dim3(aos_grid(g)), dim3(LAYOUT_THREADS), 0, s, e, o, g, a);
}

cudaError_t spinor_from_aos(const double* d_aos, const Geom& g, int prec, void* d_even,
                            void* d_odd, cudaStream_t s) {
  switch (prec) {
    case P_F64: return go_from_aos<P_F64>(d_aos, g, d_even, d_odd, s);
    case P_F32: return go_from_aos<P_F32>(d_aos, g, d_even, d_odd, s);
    case P_F16: return go_from_aos<P_F16>(d_aos, g, d_even, d_odd, s);
    case P_BF16: return go_from_aos<P_BF16>(d_aos, g, d_even, d_odd, s);
    case P_DF64: return go_from_aos<P_DF64>(d_aos, g, d_even, d_odd, s);
  }
  return cudaErrorInvalidValue;
}

cudaError_t spinor_to_aos(const void* d_even, const void* d_odd, const Geom& g, int prec,
                          double* d_aos, cudaStream_t s) {
  switch (prec) {
    case P_F64: return go_to_aos<P_F64>(d_even, d_odd, g, d_aos, s);
    case P_F32: return go_to_aos<P_F32>(d_even, d_odd, g, d_aos, s);
    case P_F16: return go_to_aos<P_F16>(d_even, d_odd, g, d_aos, s);
    case P_BF16: return go_to_aos<P_BF16>(d_even, d_odd, g, d_aos, s);
    case P_DF64: return go_to_aos<P_DF64>(d_even, d_odd, g, d_aos, s);
  }
  return cudaErrorInvalidValue;
}

template <int PI>
static cudaError_t go_convert_in(const void* in, void* out, int pout, int Vh, double sc,
                                 cudaStream_t s) {
  const long long n = 3LL * Vh;
  const unsigned nb = (unsigned)((n + LAYOUT_THREADS - 1) / LAYOUT_THREADS);
  switch (pout) {
    case P_F64: return launch_k(k_spinor_convert<PI, P_F64>, dim3(nb), dim3(LAYOUT_THREADS), 0, s, in, out, Vh, sc);
    case P_F32: return launch_k(k_spinor_convert<PI, P_F32>, dim3(nb), dim3(LAYOUT_THREADS), 0, s, in, out, Vh, sc);
    case P_F16: return launch_k(k_spinor_convert<PI, P_F16>, dim3(nb), dim3(LAYOUT_THREADS), 0, s, in, out, Vh, sc);
    case P_BF16: return launch_k(k_spinor_convert<PI, P_BF16>, dim3(nb), dim3(LAYOUT_THREADS), 0, s, in, out, Vh, sc);
    case P_DF64: return launch_k(k_spinor_convert<PI, P_DF64>, dim3(nb), dim3(LAYOUT_THREADS), 0, s, in, out, Vh, sc);
  }
  return cudaErrorInvalidValue;
}

cudaError_t spinor_convert(const void* in, int pin, void* out, int pout, int Vh, double scale,
                           cudaStream_t s) {
  switch (pin) {
    case P_F64: return go_convert_in<P_F64>(in, out, pout, Vh, scale, s);
    case P_F32: return go_convert_in<P_F32>(in, out, pout, Vh, scale, s);
    case P_F16: return go_convert_in<P_F16>(in, out, pout, Vh, scale, s);
    case P_BF16: return go_convert_in<P_BF16>(in, out, pout, Vh, scale, s);
    case P_DF64: return go_convert_in<P_DF64>(in, out, pout, Vh, scale, s);
  }
  return cudaErrorInvalidValue;
}

// ------------------------------------------------------------------ dispatch

// the slots' reduction totals and scalar finishers of the launch just issued on s
static cudaError_t then_finish(cudaError_t err, const Launch& L, cudaStream_t s) {
  if (err != cudaSuccess || L.finish != 1) return err;
  return launch_finish(L, s);
}

cudaError_t launch_dslash(int sp, int nr, bool dag, int epi, const Launch& L, int grid,
                          cudaStream_t s, int form) {
  // no slot reduces or finishes: the instantiation without the reduction code (a batched
  // launch's finish flag covers its running slots; an inline Work says so itself)
  if ((epi == EPI_LIN || epi == EPI_LIN_TW) && !L.finish &&
      (L.works || (!L.inline_work.red && L.inline_work.fin == FIN_NONE)))
    epi = epi == EPI_LIN ? EPI_PLAIN : EPI_PLAIN_TW;
  switch (sp) {
    case P_F64: return then_finish(launch_dslash_f64(nr, dag, epi, L, grid, s, form), L, s);
    case P_F32: return then_finish(launch_dslash_f32(nr, dag, epi, L, grid, s, form), L, s);
    case P_F16: return then_finish(launch_dslash_f16(nr, dag, epi, L, grid, s, form), L, s);
    case P_BF16: return then_finish(launch_dslash_bf16(nr, dag, epi, L, grid, s, form), L, s);
    case P_DF64: return then_finish(launch_dslash_df64(nr, dag, epi, L, grid, s, form), L, s);
  }
  return cudaErrorInvalidValue;
}

// Programmatic dependent launch of the batched kernels (each CTA lets the next grid launch
// when it starts its last tile). Measured on GB300: the batched 16^3x32 FP32 Dslash of ten
// slots per launch, applied back to back, 81.5 -> 80.5 us per launch; the solvers' step
// chains gain where their launches are small (up to PDL_SOLVER_MAX_TILES tiles) and lose
// where they are large (launch.h). So it is on for the operator launches (lqcd_dslash_eo,
// batches, M-hat) and the small solvers, and off in the large ones (PdlSolverScope);
// LQCD_PDL=1 turns it on everywhere, LQCD_PDL=0 off everywhere.
namespace {
thread_local int t_solver_depth = 0;
}
PdlSolverScope::PdlSolverScope(bool off) : off_(off) {
  if (off_) ++t_solver_depth;
}
PdlSolverScope::~PdlSolverScope() {
  if (off_) --t_solver_depth;
}

namespace {
thread_local bool t_pdl_skip = false;  // the next launch depends on a node that is no kernel
}
void pdl_skip_next(bool skip) { t_pdl_skip = skip; }

bool pdl_enabled() {
  if (t_pdl_skip) {
    t_pdl_skip = false;
    return false;
  }
  static const int mode = [] {
    const char* v = std::getenv("LQCD_PDL");
    if (!v || !v[0]) return -1;
    return v[0] == '1' ? 1 : 0;
  }();
  if (mode >= 0) return mode == 1;
  return t_solver_depth == 0;
}

int dslash_occupancy(int sp, int nr, int form) {
  switch (sp) {
    case P_F64: return dslash_occupancy_f64(nr, form);
    case P_F32: return dslash_occupancy_f32(nr, form);
    case P_F16: return dslash_occupancy_f16(nr, form);
    case P_BF16: return dslash_occupancy_bf16(nr, form);
    case P_DF64: return dslash_occupancy_df64(nr, form);
  }
  return 0;
}

cudaError_t launch_blas(int sp, int op, const Launch& L, int grid, cudaStream_t s, int tp) {
  switch (sp) {
    case P_F64: return then_finish(launch_blas_f64(op, tp, L, grid, s), L, s);
    case P_F32: return then_finish(launch_blas_f32(op, tp, L, grid, s), L, s);
    case P_F16: return then_finish(launch_blas_f16(op, tp, L, grid, s), L, s);
    case P_BF16: return then_finish(launch_blas_bf16(op, tp, L, grid, s), L, s);
    case P_DF64: return then_finish(launch_blas_df64(op, tp, L, grid, s), L, s);
  }
  return cudaErrorInvalidValue;
}

namespace {
std::mutex g_occ_mu;
std::unordered_map<const void*, int> g_occ;  // kernel -> resident CTAs per SM
int g_mult[4] = {0, 0, 0, 0};
int g_nsm = 0;
int g_nsm_dev = -1;
}  // namespace

int device_sm_count() {
  int dev = 0;
  cudaGetDevice(&dev);
  std::lock_guard<std::mutex> lk(g_occ_mu);
  if (g_nsm_dev != dev) {
    cudaDeviceGetAttribute(&g_nsm, cudaDevAttrMultiProcessorCount, dev);
    g_nsm_dev = dev;
    g_occ.clear();
  }
  return g_nsm;
}

std::atomic<unsigned> g_config_epoch{0};
unsigned launch_config_epoch() { return g_config_epoch.load(); }
void launch_config_changed() { ++g_config_epoch; }

void set_grid_multiplier(int family, int mult) {
  launch_config_changed();
  if (family >= 0 && family < 4) g_mult[family] = mult;
}

namespace {
bool g_split[NPREC] = {false, false, false, false, true};
}  // namespace

bool dslash_colour_split(int prec) { return prec >= 0 && prec < NPREC && g_split[prec]; }
void set_dslash_colour_split(int prec, bool on) {
  launch_config_changed();
  if (prec >= 0 && prec < NPREC) g_split[prec] = on;
}

int kernel_occupancy(const void* fn, int block) {
  device_sm_count();  // resets the cache when the device changed
  std::lock_guard<std::mutex> lk(g_occ_mu);
  auto it = g_occ.find(fn);
  if (it != g_occ.end()) return it->second;
  int o = 0;
  if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&o, fn, block, 0) != cudaSuccess || o < 1) {
    cudaGetLastError();
    o = 1;
  }
  g_occ[fn] = o;
  return o;
}

int grid_for(const void* fn, int ntiles, int family, int block, int ctas_per_sm) {
  const int nsm = device_sm_count();
  int occ = kernel_occupancy(fn, block);
  int m = (family >= 0 && family < 4) ? g_mult[family] : 0;
  if (m > 0 && m < occ) occ = m;
  if (ctas_per_sm > 0 && ctas_per_sm < occ) occ = ctas_per_sm;
  long long grid = (long long)nsm * occ;
  if (grid > ntiles) grid = ntiles;
  return (int)(grid < 1 ? 1 : grid);
}

}  // namespace lqcd
