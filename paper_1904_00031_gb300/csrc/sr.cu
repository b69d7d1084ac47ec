// K5-K7: energy statistics and stochastic reconfiguration (Sec. 2.2.5; update
// rule Eq. 2), and K8: the backward of ln psi.
//
// The SR system (S + eps I) delta = F is solved by conjugate gradient with S
// never formed.  All algebra runs on "augmented" operands: T' = [T | 1],
// sigma' = [sigma | 1], and a parameter vector as an (m+1) x (n+1) array X'
// (X'[j][i] = x_W[j][i], X'[j][n] = x_b[j], X'[m][i] = x_a[i], X'[m][n] = 0):
//   (O x)_s         = sum_j T'_sj (X' sigma'_s)_j           (forward contraction)
//   sum_s conj(O_s) v_s = T'^H diag(v) sigma'               (adjoint contraction)
//   S x             = adjoint(w o (O x - <O x>)),  <y> = sum_s w_s y_s.
// The two contractions run at the requested precision: FP32 CUDA-core kernels
// here, or the tensor-core kernels of tc.cu (BF16 hi + lo split); CG vectors,
// inner products and every reduction are FP64, and every reduction has a fixed
// order (no atomics), so a step is bitwise reproducible.
#include <math.h>
#include <string.h>

#include <vector>

#include "common.cuh"
#include "internal.h"
#include "bf16split.cuh"
#include "fgemm.cuh"
#include "status.cuh"
#include "tc.cuh"

namespace nk {

constexpr int kVecBlocks = 1024;  // largest grid of the CG vector kernels

// Blocks of a CG vector kernel over `elems` elements: about 1024 elements per
// 256-thread block, at most kVecBlocks (the partial-sum slots of `red`).  This count
// fixes the order of the FP64 sums, which 50 CG iterations amplify (another count
// moved a 20x20 step's parameters by 5e-8): the fused, the single-problem and the
// batched launches all use it, whatever grid they run on.
static int sr_vec_blocks(int64_t elems) {
  return (int)std::min<int64_t>(kVecBlocks, std::max<int64_t>(1, (elems + 1023) / 1024));
}
constexpr int kVecThreads = 256;

// Centring partials written by the SR forward (one per CTA: sample tiles x
// hidden-tile halves), or 0 when they would not fit the partials buffer.
static int fwd_centring_parts(int64_t ns, int mt) {
  const int64_t parts = ((ns + 127) / 128) * fwd_tc_nseg(ns, mt);
  return parts <= kVecBlocks ? (int)parts : 0;
}

// Whether the SR adjoint centres the forward's output itself (v = w (y - mean)
// formed while loading): every parameter tile's CTAs repeat that FP64 work, so
// only for at most four tiles, where the launch it saves costs more.
static bool adj_centres(int m, int cplx) {
  return (m + 1 + tc_hidden_per_tile(cplx) - 1) / tc_hidden_per_tile(cplx) <= 4;
}
// Elements per thread whose loads are issued together in the vector kernels
// (a thread's elements are still visited, and summed, in grid-stride order).
constexpr int kVecUnroll = 2;
constexpr int kAdjBK = 16;  // granularity of the FP32 adjoint's sample splits

// scalars in the scratch `scal` block
enum {
  SC_RS0 = 0, SC_RS1 = 1,   // r^H r, double-buffered by iteration parity
  SC_DONE = 2,              // converged flag
  SC_ITERS = 3,             // completed iterations
  SC_FNORM = 4,             // ||F||
  SC_EBAR_RE = 5, SC_EBAR_IM = 6,
  SC_NONFINITE = 7,
  SC_ERR = 8,               // int: a bounded wait gave up
  SC_BAR = 9,               // unsigned: arrivals at the fused CG kernel's grid barriers
  SC_LEN = 16
};

SrLayout::SrLayout(int n_, int m_, int cplx_, int64_t ns_) : n(n_), m(m_), cplx(cplx_), ns(ns_) {
  ma = m + 1;
  na = n + 1;
  pa = (int64_t)ma * na;
  int tiles = ceil_div(na, 64) * ceil_div(ma, 64);
  int64_t sp = (2 * 152 + tiles - 1) / tiles;
  sp = std::min<int64_t>(sp, std::max<int64_t>(1, ns / 256));
  splits_fp32 = (int)std::max<int64_t>(1, std::min<int64_t>(sp, 64));
  splits_tc = adj_tc_splits(n, m, cplx, ns);
  const int tiles_tc = (m + 1 + tc_hidden_per_tile(cplx) - 1) / tc_hidden_per_tile(cplx);
  splits = std::min(64, std::max(2 * std::max(splits_fp32, splits_tc), (4 * 152) / tiles_tc));
  na64 = (int)round_up(n + 1, 64);
  mt1 = (m + 1 + tc_hidden_per_tile(cplx) - 1) / tc_hidden_per_tile(cplx);
  ns8 = round_up(std::max<int64_t>(ns, 1), 8);
  size_t d = cplx ? 16 : 8;  // F64 element
  size_t f = cplx ? 8 : 4;   // F32 element
  size_t off = 0;
  auto take = [&](size_t bytes) {
    size_t o = off;
    off += (size_t)round_up((int64_t)bytes, 256);
    return o;
  };
  x = take(pa * d);
  r = take(pa * d);
  p = take(pa * d);
  ap = take(pa * d);
  xf = take(pa * f);
  part = take((size_t)splits * pa * f);
  y = take((size_t)std::max<int64_t>(ns, 1) * 16);
  v = take((size_t)std::max<int64_t>(ns, 1) * 16);
  red = take(4 * kVecBlocks * sizeof(double));
  scal = take(SC_LEN * sizeof(double));
  sigt = take((size_t)na64 * ns8 * 2);
  sigr = take((size_t)std::max<int64_t>(ns, 1) * na64 * 2);
  xbf = take((size_t)2 * mt1 * 128 * na64 * 2);
  total = off;
}

size_t sr_scratch_bytes(int n, int m, int cplx, int64_t ns) {
  return SrLayout(n, m, cplx, ns).total;
}

int sr_choose_splits(const SrLayout& L, int prec, int requested) {
  const int h = prec == NK_PREC_BF16X2 ? L.splits_tc : L.splits_fp32;
  int s = requested > 0 ? requested : h;
  const int64_t max_useful = std::max<int64_t>(1, (L.ns + 63) / 64);
  s = (int)std::min<int64_t>(s, max_useful);
  return std::max(1, std::min(s, L.splits));
}

// ------------------------------------------------------------------ helpers

template <bool CPLX>
struct D;  // F64 element
template <>
struct D<true> {
  using T = double2;
  static __device__ __forceinline__ double2 zero() { return make_double2(0.0, 0.0); }
};
template <>
struct D<false> {
  using T = double;
  static __device__ __forceinline__ double zero() { return 0.0; }
};

__device__ __forceinline__ double re(double x) { return x; }
__device__ __forceinline__ double re(double2 x) { return x.x; }
__device__ __forceinline__ double im(double) { return 0.0; }
__device__ __forceinline__ double im(double2 x) { return x.y; }

// Where the CG's p update also writes what the next forward contraction reads: the
// BF16 hi/lo planes [2][mt*128][na64] of p (tensor-core path) or its F32 copy xf
// (FP32 path), p in the augmented [m+1][na] layout.  The first iteration's come from
// bplanes or to_f32.
struct PlaneOut {
  uint16_t* planes = nullptr;
  int na = 1, mt = 0, na64 = 64;
  void* xf = nullptr;
};
// s + |x|^2 and s + Re conj(a) b, every rounding written out: the fused, the single
// and the batched kernels have to agree bit for bit whatever the compiler would fuse
__device__ __forceinline__ double add_norm2(double s, double x) { return __fma_rn(x, x, s); }
__device__ __forceinline__ double add_norm2(double s, double2 x) {
  return __dadd_rn(s, __fma_rn(x.x, x.x, __dmul_rn(x.y, x.y)));
}
__device__ __forceinline__ double add_cdot(double s, double a, double b) { return __fma_rn(a, b, s); }
__device__ __forceinline__ double add_cdot(double s, double2 a, double2 b) {
  return __dadd_rn(s, __fma_rn(a.x, b.x, __dmul_rn(a.y, b.y)));
}
__device__ __forceinline__ double vadd(double a, double b) { return a + b; }
__device__ __forceinline__ double2 vadd(double2 a, double2 b) {
  return make_double2(a.x + b.x, a.y + b.y);
}
__device__ __forceinline__ double axpy(double a, double x, double y) { return fma(a, x, y); }
__device__ __forceinline__ double2 axpy(double a, double2 x, double2 y) {
  return make_double2(fma(a, x.x, y.x), fma(a, x.y, y.y));
}

// Deterministic block reduction of one double; warp 0 gets the result (an SM does 1.6
// FP64 operations per clock: eight warps repeating the last sum or a division cost a
// microsecond or two, so scalars are one thread's work here and below).
__device__ __forceinline__ double block_sum(double v) {
  __shared__ double sh[32];
  for (int off = 16; off >= 1; off >>= 1) v += __shfl_xor_sync(0xffffffffu, v, off);
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  __syncthreads();
  if (lane == 0) sh[w] = v;
  __syncthreads();
  double t = 0.0;
  const int nw = (blockDim.x + 31) >> 5;
  if (w == 0)
    for (int u = 0; u < nw; ++u) t += sh[u];
  return t;
}

// fn of the sum of nb block partials in a fixed order (every block gets the same
// value; one thread evaluates fn, which may write shared memory that every thread reads
// when this returns).
template <class Fn>
__device__ __forceinline__ double sum_partials(const double* red, int nb, const Fn& fn) {
  __shared__ double tot;
  __syncthreads();  // an earlier call's readers of tot are done
  if (threadIdx.x < 32) {
    double v = 0.0;
#pragma unroll 8
    for (int u = threadIdx.x; u < nb; u += 32) v += red[u];
    for (int off = 16; off >= 1; off >>= 1) v += __shfl_xor_sync(0xffffffffu, v, off);
    if (threadIdx.x == 0) tot = fn(v);
  }
  __syncthreads();
  return tot;
}
__device__ __forceinline__ double sum_partials(const double* red, int nb) {
  return sum_partials(red, nb, [](double v) { return v; });
}

// v_s, the vector an adjoint contraction is taken of, as F32: formed in FP64 and
// rounded once (the contractions multiply it with FP32 values).
template <bool CPLX>
__device__ __forceinline__ void store_v(void* v, int64_t s, double r, double i) {
  if constexpr (CPLX) reinterpret_cast<float2*>(v)[s] = make_float2((float)r, (float)i);
  else reinterpret_cast<float*>(v)[s] = (float)r;
}

// ------------------------------------------------------------------ K7 statistics

// Three passes over the samples in nb blocks (sums of per-block partials in a
// fixed order, so the result does not depend on scheduling):
//   mean:   per-block partials of sum w E_s                 -> red[2K + b], red[3K + b]
//   dev:    E = sum of those; v_s = w_s (E_s - E); per-block partials of
//           sum w |E_s - E|^2 -> red[b] and, over whole chains, of
//           sum_c (mean_c Re E - Re E)^2 -> red[K + b]      (K = kVecBlocks)
//   finish: info {E, var, error from chain means} and the scalars the CG reads.
// v_s is the vector whose adjoint contraction is F.
template <bool CPLX>
__device__ __forceinline__ void stats_mean_body(int bx, int gx, const double* __restrict__ eloc,
                                                const double* __restrict__ weights, int64_t ns,
                                                double* red) {
  const double invn = 1.0 / (double)ns;
  double sr = 0.0, si = 0.0;
  for (int64_t s = bx * (int64_t)blockDim.x + threadIdx.x; s < ns;
       s += (int64_t)gx * blockDim.x) {
    const double w = weights ? weights[s] : invn;
    sr += w * eloc[2 * s];
    si += w * eloc[2 * s + 1];
  }
  const double br = block_sum(sr);
  const double bi = block_sum(si);
  if (threadIdx.x == 0) {
    red[2 * kVecBlocks + bx] = br;
    red[3 * kVecBlocks + bx] = bi;
  }
}

template <bool CPLX>
__device__ __forceinline__ void stats_dev_body(int bx, int gx, const double* __restrict__ eloc,
                                               const double* __restrict__ weights, int64_t ns,
                                               int n_chains, double* red, void* vout, int nb) {
  const double er = sum_partials(red + 2 * kVecBlocks, nb);
  const double ei = sum_partials(red + 3 * kVecBlocks, nb);
  const double invn = 1.0 / (double)ns;
  double vv = 0.0;
  for (int64_t s = bx * (int64_t)blockDim.x + threadIdx.x; s < ns;
       s += (int64_t)gx * blockDim.x) {
    const double w = weights ? weights[s] : invn;
    const double dr = eloc[2 * s] - er, di = eloc[2 * s + 1] - ei;
    vv += w * (dr * dr + di * di);
    store_v<CPLX>(vout, s, w * dr, w * di);
  }
  double ce = 0.0;
  const int64_t spc = n_chains > 0 ? ns / n_chains : 0;
  if (!weights && n_chains > 1 && spc > 0) {
    // one warp per chain (its lanes stride the chain's samples)
    const int lane = threadIdx.x & 31, nw = blockDim.x >> 5;
    for (int64_t c = bx * (int64_t)nw + (threadIdx.x >> 5); c < n_chains; c += (int64_t)gx * nw) {
      double mc = 0.0;
      for (int64_t u = lane; u < spc; u += 32) mc += eloc[2 * (c * spc + u)];
#pragma unroll
      for (int off = 16; off >= 1; off >>= 1) mc += __shfl_xor_sync(0xffffffffu, mc, off);
      mc /= (double)spc;
      if (lane == 0) ce += (mc - er) * (mc - er);
    }
  }
  const double bv = block_sum(vv);
  const double bc = block_sum(ce);
  if (threadIdx.x == 0) {
    red[bx] = bv;
    red[kVecBlocks + bx] = bc;
  }
}

__device__ __forceinline__ void stats_finish_body(const double* __restrict__ weights, int64_t ns,
                                                  int n_chains, const double* red, int nb,
                                                  double* info, double* scal) {
  const double er = sum_partials(red + 2 * kVecBlocks, nb);
  const double ei = sum_partials(red + 3 * kVecBlocks, nb);
  const double var = sum_partials(red, nb);
  const double ce = sum_partials(red + kVecBlocks, nb);
  const int64_t spc = n_chains > 0 ? ns / n_chains : 0;
  if (threadIdx.x == 0) {
    info[NK_INFO_E_RE] = er;
    info[NK_INFO_E_IM] = ei;
    info[NK_INFO_VAR] = var;
    info[NK_INFO_ERR] =
        (!weights && n_chains > 1 && spc > 0) ? sqrt(ce / ((double)n_chains * (n_chains - 1))) : 0.0;
    scal[SC_EBAR_RE] = er;
    scal[SC_EBAR_IM] = ei;
    scal[SC_NONFINITE] = (isfinite(er) && isfinite(ei) && isfinite(var)) ? 0.0 : 1.0;
  }
}

template <bool CPLX>
__global__ void __launch_bounds__(kVecThreads) stats_mean_kernel(const double* __restrict__ eloc,
                                                                 const double* __restrict__ weights,
                                                                 int64_t ns, double* red) {
  stats_mean_body<CPLX>(blockIdx.x, gridDim.x, eloc, weights, ns, red);
}

template <bool CPLX>
__global__ void __launch_bounds__(kVecThreads) stats_dev_kernel(const double* __restrict__ eloc,
                                                                const double* __restrict__ weights,
                                                                int64_t ns, int n_chains,
                                                                double* red, void* vout, int nb) {
  stats_dev_body<CPLX>(blockIdx.x, gridDim.x, eloc, weights, ns, n_chains, red, vout, nb);
}

__global__ void stats_finish_kernel(const double* __restrict__ weights, int64_t ns, int n_chains,
                                    const double* red, int nb, double* info, double* scal) {
  stats_finish_body(weights, ns, n_chains, red, nb, info, scal);
}

// ------------------------------------------------------------------ adjoint contraction
// part[z][j][i] = sum_{s in split z} conj(T'_sj) v_s sigma'_si   (FP32 CUDA cores)

// The centring of an adjoint's input: v_s = w_s (y_s - mean), mean = the fixed-order
// sum of `parts` partials at mean_part (Re) and mean_part + kVecBlocks (Im).
struct CentreArgs {
  const void* y = nullptr;  // F64 [ns]; null: v is read from memory
  const double* mean_part = nullptr;
  int parts = 0;
  const double* weights = nullptr;
  double invn = 0.0;  // 1 / samples
};

// A operand of the adjoint: conj(T'_sj) v_s, formed when it is staged.
template <bool CPLX, int EXT, int N, int kFK>
struct ConjTV {
  using F = typename std::conditional<CPLX, float2, float>::type;
  struct Set {
    F t[N], v[N];
  };
  const F* p;
  const F* vp;   // v of the chunk's first sample (global or shared memory)
  int64_t ld;
  bool in, one;
  int k, left;
  static constexpr int KU = kFThreads / EXT;
  static __device__ __forceinline__ int row(int) { return threadIdx.x % EXT; }
  __device__ __forceinline__ void init(const F* T, int m, int j0, const F* v, int64_t kb,
                                       int64_t ke) {
    left = (int)(ke > kb ? ke - kb : 0);
    k = threadIdx.x / EXT;
    const int j = j0 + row(0);
    in = j < m;
    one = j == m;
    ld = m;
    p = T + (kb + k) * ld + j;
    vp = v;
  }
  __device__ __forceinline__ void load(Set& s) {
#pragma unroll
    for (int u = 0; u < N; ++u) {
      const int ku = k + u * KU;
      s.t[u] = {};
      s.v[u] = {};
      if (ku < left) {
        // (1 before the load: written after it, it would wait for it)
        if (one) fg_one(s.t[u]);
        if (in) s.t[u] = ld_here(p + u * KU * ld);
        s.v[u] = vp[ku];
      }
    }
    p += kFK * ld;
    vp += kFK;
    left -= kFK;
  }
  __device__ __forceinline__ F get(const Set& s, int u) const {
    const F t = s.t[u], v = s.v[u];
    if constexpr (CPLX) {
      const float vr = v.x, vi = v.y;
      // conj(t) * v
      return make_float2(t.x * vr + t.y * vi, t.x * vi - t.y * vr);
    } else {
      return t * v;
    }
  }
};

// Samples of a split that the adjoint centres itself (into shared memory).
constexpr int kAdjCentre = 1024;

template <bool CPLX, int TR>
using AdjTile = Tile<CPLX ? kMulRealB : kMulReal, TR, false, TR == 8 ? 8 : 16>;

// 16 TR parameter rows x 64 (complex) or 128 (real) sites per CTA and sample split
// (fgemm.cuh).  CENTRE: v of the CTA's split is formed from y into shared memory
// first (a launch and a pass over v saved; only for splits of at most kAdjCentre
// samples).  10x10 real, m = 400, 16,384 samples: 81 us (183 with scalar 4 x 4 blocks
// whose loads waited on one another).
template <bool CPLX, int TR, bool CENTRE>
__global__ void __launch_bounds__(kFThreads, 2)
    adjoint_fp32_kernel(const int8_t* __restrict__ sigma, const void* __restrict__ Tv,
                        const void* __restrict__ vv, int64_t ns, int n, int m, int64_t chunk,
                        void* partv, const double* scal, CentreArgs ca) {
  if (scal && scal[SC_DONE] != 0.0) return;
  using L = AdjTile<CPLX, TR>;
  using F = typename std::conditional<CPLX, float2, float>::type;
  extern __shared__ __align__(16) unsigned char smraw[];
  const F* T = reinterpret_cast<const F*>(Tv);
  const int ma = m + 1, na = n + 1;
  const int i0 = blockIdx.x * L::BC, j0 = blockIdx.y * L::BR;
  const int64_t sb = (int64_t)blockIdx.z * chunk;
  const int64_t se = std::min<int64_t>(ns, sb + chunk);
  const F* v = reinterpret_cast<const F*>(vv) + sb;
  if constexpr (CENTRE) {
    F* vs = reinterpret_cast<F*>(smraw + L::STAGE_BYTES);
    const double mr = sum_partials(ca.mean_part, ca.parts);
    const double mi = CPLX ? sum_partials(ca.mean_part + kVecBlocks, ca.parts) : 0.0;
    for (int64_t s = sb + threadIdx.x; s < se; s += kFThreads) {
      const double w = ca.weights ? ca.weights[s] : ca.invn;
      if constexpr (CPLX) {
        const double2 y = reinterpret_cast<const double2*>(ca.y)[s];
        store_v<true>(vs, s - sb, w * (y.x - mr), w * (y.y - mi));
      } else {
        store_v<false>(vs, s - sb, w * (reinterpret_cast<const double*>(ca.y)[s] - mr), 0.0);
      }
    }
    __syncthreads();
    v = vs;
  }
  ConjTV<CPLX, L::BR, L::NA, L::kFK> oa;
  Operand<int8_t, true, L::BC, L::NB, false, true, false, false, L::kFK> ob;
  oa.init(T, m, j0, v, sb, se);
  ob.init(sigma, n, i0, na, sb, se);
  L acc;
  acc.zero();
  acc.bounds(ma - j0, na - i0);
  acc.template run<TR == 8 ? 1 : 2>(smraw, se > sb ? (int)((se - sb + L::kFK - 1) / L::kFK) : 0, oa,
                                    ob, [](int) {});
  F* part = reinterpret_cast<F*>(partv) + (int64_t)blockIdx.z * ma * na;
#pragma unroll
  for (int p = 0; p < L::TP; ++p)
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const int j = j0 + L::row(p) + h;
      if (j >= ma) continue;
#pragma unroll
      for (int q = 0; q < L::TC; ++q) {
        const int i = i0 + L::col(q);
        if (i >= na) continue;
        F& d = part[(int64_t)j * na + i];
        if constexpr (CPLX)
          d = h ? make_float2(acc.x[p][q].y, acc.y[p][q].y) : make_float2(acc.x[p][q].x, acc.y[p][q].x);
        else
          d = h ? acc.x[p][q].y : acc.x[p][q].x;
      }
    }
}

// Samples per split (whole 16-sample steps).
static int64_t adjoint_chunk(int64_t ns, int splits) {
  return round_up((ns + splits - 1) / splits, kAdjBK);
}

// Whether the FP32 adjoint centres its input itself: its splits fit the shared-
// memory v, and few enough tiles repeat the FP64 work on a sample.
static bool adjoint_centres(int64_t ns, int n, int m, int cplx, int splits) {
  const int tiles = ceil_div(m + 1, 64) * ceil_div(n + 1, cplx ? 64 : 128);
  return adjoint_chunk(ns, splits) <= kAdjCentre && tiles <= 16;
}

template <bool CPLX>
static void launch_adjoint_fp32(const int8_t* sigma, const void* T, const void* v, int64_t ns,
                                int n, int m, int splits, void* part, const double* scal,
                                cudaStream_t st, const CentreArgs& ca = CentreArgs{}) {
  const int64_t chunk = adjoint_chunk(ns, splits);
  const int ct = ceil_div(n + 1, AdjTile<CPLX, 8>::BC), t8 = ceil_div(m + 1, 128), t4 = ceil_div(m + 1, 64);
  // 128-row tiles when they fill every SM's two CTAs and pad little more
  const bool big = (int64_t)t8 * ct * splits >= 2 * 152 && 8 * t8 * 128 <= 9 * t4 * 64;
  auto go = [&](auto kern, int rows, size_t smem) {
    kern<<<dim3(ct, rows, splits), kFThreads, smem, st>>>(sigma, T, v, ns, n, m, chunk, part, scal,
                                                          ca);
  };
  const size_t vb = kAdjCentre * (CPLX ? 8 : 4);
  const size_t s8 = AdjTile<CPLX, 8>::STAGE_BYTES, s4 = AdjTile<CPLX, 4>::STAGE_BYTES;
  static_assert(AdjTile<CPLX, 8>::STAGE_BYTES + kAdjCentre * 8 <= 48 * 1024 &&
                    AdjTile<CPLX, 4>::STAGE_BYTES + kAdjCentre * 8 <= 48 * 1024, "shared memory");
  if (ca.y) {
    if (big) go(adjoint_fp32_kernel<CPLX, 8, true>, t8, s8 + vb);
    else go(adjoint_fp32_kernel<CPLX, 4, true>, t4, s4 + vb);
  } else {
    if (big) go(adjoint_fp32_kernel<CPLX, 8, false>, t8, s8);
    else go(adjoint_fp32_kernel<CPLX, 4, false>, t4, s4);
  }
}

// ------------------------------------------------------------------ forward contraction
// y_s = sum_j T'_sj (X' sigma'_s)_j   (FP32 CUDA cores, FP64 row sums)

// 16 TR samples per CTA, all parameter rows in tiles of 64 (complex) or 128 (real);
// a row's products with T' are folded four columns (x + 16 q of 64) at a time in
// FP32, then in FP64.  With mean_part, also the CTA's partial of the centring mean
// sum_s w_s y_s (mean_part[b], Re, and mean_part[kVecBlocks + b], Im).  10x10 real,
// m = 400, 16,384 samples: 73 us (149 with scalar 4 x 4 blocks).
template <bool CPLX, int TR>
__global__ void __launch_bounds__(kFThreads, 2)
    forward_fp32_kernel(const int8_t* __restrict__ sigma, int64_t ns, int n, int m,
                        const void* __restrict__ xf, const void* __restrict__ Tv, void* yv,
                        const double* scal, const double* __restrict__ weights, double invn,
                        double* mean_part) {
  if (scal && scal[SC_DONE] != 0.0) return;
  using L = Tile<CPLX ? kMulRealA : kMulReal, TR, true, TR == 8 ? 8 : 16>;
  using F = typename std::conditional<CPLX, float2, float>::type;
  __shared__ __align__(16) unsigned char smem[L::STAGE_BYTES];
  const F* T = reinterpret_cast<const F*>(Tv);
  const int64_t s0 = (int64_t)blockIdx.x * L::BR;
  const int K = n + 1;
  double2 part[TR];
#pragma unroll
  for (int r = 0; r < TR; ++r) part[r] = make_double2(0.0, 0.0);
  Operand<int8_t, false, L::BR, L::NA, false, false, true, false, L::kFK> oa;
  Operand<F, false, L::BC, L::NB, false, false, false, true, L::kFK> ob;
  oa.init(sigma, n, s0, ns, 0, K);
  ob.init(reinterpret_cast<const F*>(xf), K, 0, m + 1, 0, K);
  L acc;
  acc.zero();
  acc.bounds(ns - s0, m + 1);
  const int nk = (K + L::kFK - 1) / L::kFK;  // chunks per tile of parameter rows
  int kc = 0, j0 = 0;
  acc.template run<1>(smem, nk * ((m + L::BC) / L::BC), oa, ob, [&](int) {
    if (++kc < nk) return;
#pragma unroll
    for (int r = 0; r < TR; ++r) {
      const int64_t s = s0 + L::lr() + r;
      if (s >= ns) continue;
#pragma unroll
      for (int g = 0; g < L::TC / 4; ++g) {
        float pr = 0.f, pi = 0.f;
#pragma unroll
        for (int qq = 0; qq < 4; ++qq) {
          const int q = 4 * g + qq, j = j0 + L::col(q);
          if (j > m) continue;
          const float ar = (r & 1) ? acc.x[r / 2][q].y : acc.x[r / 2][q].x;
          if constexpr (CPLX) {
            const float ai = (r & 1) ? acc.y[r / 2][q].y : acc.y[r / 2][q].x;
            const float2 t = j < m ? T[s * m + j] : make_float2(1.f, 0.f);
            pr += t.x * ar - t.y * ai;
            pi += t.x * ai + t.y * ar;
          } else {
            const float t = j < m ? T[s * m + j] : 1.f;
            pr += t * ar;
          }
        }
        part[r].x += (double)pr;
        part[r].y += (double)pi;
      }
    }
    acc.zero();
    kc = 0;
    j0 += L::BC;
  });
  const bool first = (threadIdx.x & 15) == 0;  // of the 16 lanes that share the rows
  double wr = 0.0, wi = 0.0;
#pragma unroll
  for (int r = 0; r < TR; ++r) {
#pragma unroll
    for (int off = 8; off >= 1; off >>= 1) {
      part[r].x += __shfl_xor_sync(0xffffffffu, part[r].x, off);
      if (CPLX) part[r].y += __shfl_xor_sync(0xffffffffu, part[r].y, off);
    }
    const int64_t s = s0 + L::lr() + r;
    if (first && s < ns) {
      if (CPLX) reinterpret_cast<double2*>(yv)[s] = part[r];
      else reinterpret_cast<double*>(yv)[s] = part[r].x;
      if (mean_part) {
        const double w = weights ? weights[s] : invn;
        wr += w * part[r].x;
        wi += w * part[r].y;
      }
    }
  }
  if (mean_part) {
    const double br = block_sum(wr), bi = CPLX ? block_sum(wi) : 0.0;
    if (threadIdx.x == 0) {
      mean_part[blockIdx.x] = br;
      mean_part[kVecBlocks + blockIdx.x] = bi;
    }
  }
}

// Rows per thread of the FP32 forward: 8 when 128-sample CTAs fill every SM twice.
static int forward_rows(int64_t ns) { return ns >= 2 * 152 * 128 ? 8 : 4; }
static int64_t forward_blocks(int64_t ns) {
  const int bs = 16 * forward_rows(ns);
  return (ns + bs - 1) / bs;
}

template <bool CPLX>
static void launch_forward_fp32(const int8_t* sigma, int64_t ns, int n, int m, const void* xf,
                                const void* T, void* y, const double* scal, const double* weights,
                                double* mean_part, cudaStream_t st) {
  auto go = [&](auto kern) {
    kern<<<(unsigned)forward_blocks(ns), kFThreads, 0, st>>>(sigma, ns, n, m, xf, T, y, scal, weights,
                                                             1.0 / (double)ns, mean_part);
  };
  if (forward_rows(ns) == 8) go(forward_fp32_kernel<CPLX, 8>);
  else go(forward_fp32_kernel<CPLX, 4>);
}

// ------------------------------------------------------------------ CG vector kernels

// X' (FP64) -> FP32 copy for the forward contraction
template <bool CPLX>
__global__ void to_f32_kernel(const void* __restrict__ src, void* dst, int64_t pa,
                              const double* scal) {
  if (scal[SC_DONE] != 0.0) return;
  for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < pa;
       e += (int64_t)gridDim.x * blockDim.x) {
    if (CPLX) {
      double2 v = reinterpret_cast<const double2*>(src)[e];
      reinterpret_cast<float2*>(dst)[e] = make_float2((float)v.x, (float)v.y);
    } else {
      reinterpret_cast<float*>(dst)[e] = (float)reinterpret_cast<const double*>(src)[e];
    }
  }
}

// y~ = w o (y - <y>): pass 1 writes per-block partial sums of w y (fixed grid),
// pass 2 adds them in a fixed order (every block gets the same mean) and
// writes y~.
template <bool CPLX>
__device__ __forceinline__ void center_partial_body(int bx, int gx, 
    const void* __restrict__ yv, const double* __restrict__ weights, int64_t ns, double* red,
    const double* scal) {
  if (scal[SC_DONE] != 0.0) return;
  const double invn = 1.0 / (double)ns;
  double sr = 0.0, si = 0.0;
  const int64_t stride = (int64_t)gx * blockDim.x;
  for (int64_t s0 = bx * (int64_t)blockDim.x + threadIdx.x; s0 < ns;
       s0 += kVecUnroll * stride) {
    double w[kVecUnroll];
    double2 y[kVecUnroll];
#pragma unroll
    for (int u = 0; u < kVecUnroll; ++u) {
      const int64_t s = s0 + u * stride;
      if (s < ns) {
        w[u] = weights ? weights[s] : invn;
        y[u] = CPLX ? reinterpret_cast<const double2*>(yv)[s]
                    : make_double2(reinterpret_cast<const double*>(yv)[s], 0.0);
      }
    }
#pragma unroll
    for (int u = 0; u < kVecUnroll; ++u) {
      if (s0 + u * stride < ns) {
        sr += w[u] * y[u].x;
        if (CPLX) si += w[u] * y[u].y;
      }
    }
  }
  const double br = block_sum(sr);
  const double bi = block_sum(si);
  if (threadIdx.x == 0) {
    red[2 * kVecBlocks + bx] = br;
    red[3 * kVecBlocks + bx] = bi;
  }
}

template <bool CPLX>
__global__ void __launch_bounds__(kVecThreads) center_partial_kernel(
    const void* __restrict__ yv, const double* __restrict__ weights, int64_t ns, double* red,
    const double* scal) {
  center_partial_body<CPLX>(blockIdx.x, gridDim.x, yv, weights, ns, red, scal);
}

template <bool CPLX>
__device__ __forceinline__ void center_apply_body(int bx, int gx, 
    const void* __restrict__ yv, void* vout, const double* __restrict__ weights, int64_t ns,
    const double* red, const double* scal, int nb) {
  if (scal[SC_DONE] != 0.0) return;
  __shared__ double s_invn;
  const double mr = sum_partials(red + 2 * kVecBlocks, nb, [&](double v) {
    s_invn = 1.0 / (double)ns;
    return v;
  });
  const double mi = CPLX ? sum_partials(red + 3 * kVecBlocks, nb) : 0.0;
  const double invn = s_invn;
  const int64_t stride = (int64_t)gx * blockDim.x;
  for (int64_t s0 = bx * (int64_t)blockDim.x + threadIdx.x; s0 < ns;
       s0 += kVecUnroll * stride) {
    double w[kVecUnroll];
    double2 y[kVecUnroll];
#pragma unroll
    for (int u = 0; u < kVecUnroll; ++u) {
      const int64_t s = s0 + u * stride;
      if (s < ns) {
        w[u] = weights ? weights[s] : invn;
        y[u] = CPLX ? reinterpret_cast<const double2*>(yv)[s]
                    : make_double2(reinterpret_cast<const double*>(yv)[s], 0.0);
      }
    }
#pragma unroll
    for (int u = 0; u < kVecUnroll; ++u) {
      const int64_t s = s0 + u * stride;
      if (s < ns) store_v<CPLX>(vout, s, w[u] * (y[u].x - mr), w[u] * (y[u].y - mi));
    }
  }
}

template <bool CPLX>
__global__ void __launch_bounds__(kVecThreads) center_apply_kernel(
    const void* __restrict__ yv, void* vout, const double* __restrict__ weights, int64_t ns,
    const double* red, const double* scal, int nb) {
  center_apply_body<CPLX>(blockIdx.x, gridDim.x, yv, vout, weights, ns, red, scal, nb);
}

// s + e = a + b exactly (Knuth's TwoSum in FP32)
__device__ __forceinline__ void two_sum(float a, float b, float& s, float& e) {
  s = a + b;
  const float bb = s - a;
  e = (a - (s - bb)) + (b - bb);
}

// out = sum_z part[z] (+ eps * p);  red[b] = sum conj(p) . out (if p given).
// The FP32 partials of the splits are added in split order as an unevaluated
// FP32 pair (running sum and running error of TwoSum), converted to FP64 once:
// FP64 arithmetic is a small fraction of the FP32 rate on this GPU.
// The element X'[m][n] (no parameter) is forced to 0.
template <bool CPLX, int KZ, int UN>
__device__ __forceinline__ void reduce_parts_loop(int bx, int gx, 
    const void* __restrict__ partv, int splits, int64_t pa, int64_t corner, void* outv,
    const void* __restrict__ pv, double eps, double* red, const double* scal) {
  if (scal && scal[SC_DONE] != 0.0) return;
  using DT = typename D<CPLX>::T;
  DT* out = reinterpret_cast<DT*>(outv);
  const DT* p = reinterpret_cast<const DT*>(pv);
  double dot = 0.0;
  const int64_t stride = (int64_t)gx * blockDim.x;
  for (int64_t e0 = bx * (int64_t)blockDim.x + threadIdx.x; e0 < pa;
       e0 += UN * stride) {
    float2 hi[UN], lo[UN];
    DT pp[UN];
#pragma unroll
    for (int u = 0; u < UN; ++u) {
      hi[u] = make_float2(0.f, 0.f);
      lo[u] = make_float2(0.f, 0.f);
      pp[u] = D<CPLX>::zero();
      if (p && e0 + u * stride < pa) pp[u] = p[e0 + u * stride];
    }
    // the partials of KZ splits are loaded together, then added in split order
    for (int z0 = 0; z0 < splits; z0 += KZ) {
      float2 v[KZ][UN];
#pragma unroll
      for (int zz = 0; zz < KZ; ++zz)
#pragma unroll
        for (int u = 0; u < UN; ++u) {
          const int64_t e = e0 + u * stride;
          v[zz][u] = make_float2(0.f, 0.f);
          if (z0 + zz < splits && e < pa) {
            const int64_t o = (int64_t)(z0 + zz) * pa + e;
            if constexpr (CPLX) v[zz][u] = reinterpret_cast<const float2*>(partv)[o];
            else v[zz][u].x = reinterpret_cast<const float*>(partv)[o];
          }
        }
#pragma unroll
      for (int zz = 0; zz < KZ; ++zz)
#pragma unroll
        for (int u = 0; u < UN; ++u) {
          if (z0 + zz < splits) {
            float er;
            two_sum(hi[u].x, v[zz][u].x, hi[u].x, er);
            lo[u].x += er;
            if constexpr (CPLX) {
              two_sum(hi[u].y, v[zz][u].y, hi[u].y, er);
              lo[u].y += er;
            }
          }
        }
    }
#pragma unroll
    for (int u = 0; u < UN; ++u) {
      const int64_t e = e0 + u * stride;
      if (e < pa) {
        DT a;
        if constexpr (CPLX)
          a = make_double2((double)hi[u].x + (double)lo[u].x, (double)hi[u].y + (double)lo[u].y);
        else
          a = (double)hi[u].x + (double)lo[u].x;
        if (p) a = axpy(eps, pp[u], a);
        if (e == corner) a = D<CPLX>::zero();
        out[e] = a;
        if (p) dot = add_cdot(dot, pp[u], a);
      }
    }
  }
  if (red) {
    double b = block_sum(dot);
    if (threadIdx.x == 0) red[bx] = b;
  }
}

// Few splits: two elements with four splits each in flight; many (small problems,
// bound by the latency of their partials): one element, sixteen splits; LEAN: one and
// eight (the fused kernel's five blocks per SM).  The order of the sums is the same.
template <bool CPLX, bool LEAN = false>
__device__ __forceinline__ void reduce_parts_body(int bx, int gx, const void* partv, int splits,
                                                  int64_t pa, int64_t corner, void* outv,
                                                  const void* pv, double eps, double* red,
                                                  const double* scal) {
  if (LEAN)
    reduce_parts_loop<CPLX, 8, 1>(bx, gx, partv, splits, pa, corner, outv, pv, eps, red, scal);
  else if (splits <= 12)
    reduce_parts_loop<CPLX, 4, kVecUnroll>(bx, gx, partv, splits, pa, corner, outv, pv, eps, red,
                                           scal);
  else
    reduce_parts_loop<CPLX, 16, 1>(bx, gx, partv, splits, pa, corner, outv, pv, eps, red, scal);
}

template <bool CPLX>
__global__ void __launch_bounds__(kVecThreads) reduce_parts_kernel(
    const void* __restrict__ partv, int splits, int64_t pa, int64_t corner, void* outv,
    const void* __restrict__ pv, double eps, double* red, const double* scal) {
  reduce_parts_body<CPLX>(blockIdx.x, gridDim.x, partv, splits, pa, corner, outv, pv, eps, red, scal);
}

// x = 0, r = p = F, rs = ||F||^2 (run after F was reduced into r)
template <bool CPLX>
__device__ __forceinline__ void cg_init_body(int bx, int gx, void* xv, void* rv, void* pv,
                                                              int64_t pa, double* red) {
  using DT = typename D<CPLX>::T;
  DT* x = reinterpret_cast<DT*>(xv);
  DT* r = reinterpret_cast<DT*>(rv);
  DT* p = reinterpret_cast<DT*>(pv);
  double nn = 0.0;
  const int64_t stride = (int64_t)gx * blockDim.x;
  for (int64_t e0 = bx * (int64_t)blockDim.x + threadIdx.x; e0 < pa;
       e0 += kVecUnroll * stride) {
    DT rr[kVecUnroll];
#pragma unroll
    for (int u = 0; u < kVecUnroll; ++u)
      if (e0 + u * stride < pa) rr[u] = r[e0 + u * stride];
#pragma unroll
    for (int u = 0; u < kVecUnroll; ++u) {
      const int64_t e = e0 + u * stride;
      if (e < pa) {
        x[e] = D<CPLX>::zero();
        p[e] = rr[u];
        nn = add_norm2(nn, rr[u]);
      }
    }
  }
  double b = block_sum(nn);
  if (threadIdx.x == 0) red[kVecBlocks + bx] = b;
}

template <bool CPLX>
__global__ void __launch_bounds__(kVecThreads) cg_init_kernel(void* xv, void* rv, void* pv,
                                                              int64_t pa, double* red) {
  cg_init_body<CPLX>(blockIdx.x, gridDim.x, xv, rv, pv, pa, red);
}

__device__ __forceinline__ void cg_init_scalars_body(int bx, int gx, const double* red, double* scal, double rtol, int nb) {
  double rs = sum_partials(red + kVecBlocks, nb);
  if (threadIdx.x == 0) {
    scal[SC_RS0] = rs;
    scal[SC_RS1] = rs;
    scal[SC_FNORM] = sqrt(rs);
    scal[SC_ITERS] = 0.0;
    scal[SC_DONE] = (rs == 0.0) ? 1.0 : 0.0;
    if (!isfinite(rs)) {
      scal[SC_NONFINITE] = 1.0;
      scal[SC_DONE] = 1.0;
    }
  }
}

__global__ void cg_init_scalars_kernel(const double* red, double* scal, double rtol, int nb) {
  cg_init_scalars_body(blockIdx.x, gridDim.x, red, scal, rtol, nb);
}

// alpha = rs / p^H A p; x += alpha p; r -= alpha A p; red2 = ||r||^2 partials
template <bool CPLX, int UN = kVecUnroll>
__device__ __forceinline__ void cg_step_x_body(int bx, int gx, void* xv, void* rv,
                                                                const void* pv, const void* apv,
                                                                int64_t pa, double* red,
                                                                double* scal, int it, int nb) {
  if (scal[SC_DONE] != 0.0) return;
  using DT = typename D<CPLX>::T;
  DT* x = reinterpret_cast<DT*>(xv);
  DT* r = reinterpret_cast<DT*>(rv);
  const DT* p = reinterpret_cast<const DT*>(pv);
  const DT* ap = reinterpret_cast<const DT*>(apv);
  const double alpha = sum_partials(
      red, nb, [&](double pap) { return scal[(it & 1) ? SC_RS1 : SC_RS0] / pap; });
  double nn = 0.0;
  const int64_t stride = (int64_t)gx * blockDim.x;
  for (int64_t e0 = bx * (int64_t)blockDim.x + threadIdx.x; e0 < pa;
       e0 += UN * stride) {
    DT pp[UN], xx[UN], aa[UN], rr[UN];
#pragma unroll
    for (int u = 0; u < UN; ++u) {
      const int64_t e = e0 + u * stride;
      if (e < pa) {
        pp[u] = p[e];
        xx[u] = x[e];
        aa[u] = ap[e];
        rr[u] = r[e];
      }
    }
#pragma unroll
    for (int u = 0; u < UN; ++u) {
      const int64_t e = e0 + u * stride;
      if (e < pa) {
        x[e] = axpy(alpha, pp[u], xx[u]);
        const DT q = axpy(-alpha, aa[u], rr[u]);
        r[e] = q;
        nn = add_norm2(nn, q);
      }
    }
  }
  double b = block_sum(nn);
  if (threadIdx.x == 0) red[kVecBlocks + bx] = b;
}

template <bool CPLX>
__global__ void __launch_bounds__(kVecThreads) cg_step_x_kernel(void* xv, void* rv,
                                                                const void* pv, const void* apv,
                                                                int64_t pa, double* red,
                                                                double* scal, int it, int nb) {
  cg_step_x_body<CPLX>(blockIdx.x, gridDim.x, xv, rv, pv, apv, pa, red, scal, it, nb);
}

// Element e of S p + eps p: its splits added as reduce_parts_loop adds them.
template <bool CPLX>
__device__ __forceinline__ void reduce_one(int64_t e, const void* partv, int splits, int64_t pa,
                                           int64_t corner, void* outv, const void* pv, double eps) {
  using DT = typename D<CPLX>::T;
  constexpr int KZ = 16;
  float2 hi = make_float2(0.f, 0.f), lo = make_float2(0.f, 0.f);
  for (int z0 = 0; z0 < splits; z0 += KZ) {
    float2 v[KZ];
#pragma unroll
    for (int z = 0; z < KZ; ++z) {
      v[z] = make_float2(0.f, 0.f);
      if (z0 + z < splits) {
        const int64_t o = (int64_t)(z0 + z) * pa + e;
        if constexpr (CPLX) v[z] = reinterpret_cast<const float2*>(partv)[o];
        else v[z].x = reinterpret_cast<const float*>(partv)[o];
      }
    }
#pragma unroll
    for (int z = 0; z < KZ; ++z)
      if (z0 + z < splits) {
        float er;
        two_sum(hi.x, v[z].x, hi.x, er);
        lo.x += er;
        if constexpr (CPLX) {
          two_sum(hi.y, v[z].y, hi.y, er);
          lo.y += er;
        }
      }
  }
  DT a;
  if constexpr (CPLX)
    a = make_double2((double)hi.x + (double)lo.x, (double)hi.y + (double)lo.y);
  else
    a = (double)hi.x + (double)lo.x;
  a = axpy(eps, reinterpret_cast<const DT*>(pv)[e], a);
  if (e == corner) a = D<CPLX>::zero();
  reinterpret_cast<DT*>(outv)[e] = a;
}

// Block bx's partial of Re p^H ap, in reduce_parts_loop's order.
template <bool CPLX>
__device__ __forceinline__ void dot_body(int bx, int gx, const void* pv, const void* apv,
                                         int64_t pa, double* red) {
  using DT = typename D<CPLX>::T;
  double dot = 0.0;
  for (int64_t e = bx * (int64_t)blockDim.x + threadIdx.x; e < pa; e += (int64_t)gx * blockDim.x)
    dot = add_cdot(dot, reinterpret_cast<const DT*>(pv)[e], reinterpret_cast<const DT*>(apv)[e]);
  const double b = block_sum(dot);
  if (threadIdx.x == 0) red[bx] = b;
}

// What the next forward contraction reads of element e of p.
template <bool CPLX>
__device__ __forceinline__ void store_p(const PlaneOut& po, int64_t e, typename D<CPLX>::T q) {
  if (po.planes) {
    const int j = (int)((uint32_t)e / (uint32_t)po.na), i = (int)(e - (int64_t)j * po.na);
    const int64_t pl = (int64_t)po.mt * 128 * po.na64;
    uint32_t hi, lo;
    split_bf16(re(q), hi, lo);
    const int64_t k0 = bplane_index(j, i, 0, CPLX, po.na64);
    po.planes[k0] = (uint16_t)hi;
    po.planes[pl + k0] = (uint16_t)lo;
    if constexpr (CPLX) {
      split_bf16(im(q), hi, lo);
      const int64_t k1 = bplane_index(j, i, 1, CPLX, po.na64);
      po.planes[k1] = (uint16_t)hi;
      po.planes[pl + k1] = (uint16_t)lo;
    }
  }
  if (po.xf) {
    if constexpr (CPLX)
      reinterpret_cast<float2*>(po.xf)[e] = make_float2((float)q.x, (float)q.y);
    else
      reinterpret_cast<float*>(po.xf)[e] = (float)q;
  }
}

// beta = rs_new / rs; p = r + beta p; convergence test on ||r|| <= rtol ||F||
template <bool CPLX, int UN = kVecUnroll>
__device__ __forceinline__ void cg_step_p_body(int bx, int gx, const void* rv, void* pv,
                                                                int64_t pa, const double* red,
                                                                double* scal, int it,
                                                                double rtol, int nb,
                                                                const PlaneOut& po = PlaneOut{}) {
  if (scal[SC_DONE] != 0.0) return;
  using DT = typename D<CPLX>::T;
  const DT* r = reinterpret_cast<const DT*>(rv);
  DT* p = reinterpret_cast<DT*>(pv);
  __shared__ double s_beta;
  __shared__ int s_stop;  // 1: converged, 2: not finite
  const double rs_new = sum_partials(red + kVecBlocks, nb, [&](double v) {
    s_beta = v / scal[(it & 1) ? SC_RS1 : SC_RS0];
    s_stop = !isfinite(v) ? 2 : sqrt(v) <= rtol * scal[SC_FNORM] ? 1 : 0;
    return v;
  });
  const bool conv = s_stop == 1, bad = s_stop == 2;
  if (!conv && !bad) {
    const double beta = s_beta;
    const int64_t stride = (int64_t)gx * blockDim.x;
    for (int64_t e0 = bx * (int64_t)blockDim.x + threadIdx.x; e0 < pa;
         e0 += UN * stride) {
      DT pp[UN], rr[UN];
#pragma unroll
      for (int u = 0; u < UN; ++u) {
        const int64_t e = e0 + u * stride;
        if (e < pa) {
          pp[u] = p[e];
          rr[u] = r[e];
        }
      }
#pragma unroll
      for (int u = 0; u < UN; ++u) {
        const int64_t e = e0 + u * stride;
        if (e < pa) {
          const DT q = axpy(beta, pp[u], rr[u]);
          p[e] = q;
          store_p<CPLX>(po, e, q);
        }
      }
    }
  }
  if (bx == 0 && threadIdx.x == 0) {
    scal[(it & 1) ? SC_RS0 : SC_RS1] = rs_new;
    scal[SC_ITERS] = (double)(it + 1);
    if (conv || bad) scal[SC_DONE] = 1.0;
    if (bad) scal[SC_NONFINITE] = 1.0;
  }
}

template <bool CPLX>
__global__ void __launch_bounds__(kVecThreads) cg_step_p_kernel(const void* rv, void* pv,
                                                                int64_t pa, const double* red,
                                                                double* scal, int it,
                                                                double rtol, int nb,
                                                                PlaneOut po) {
  cg_step_p_body<CPLX>(blockIdx.x, gridDim.x, rv, pv, pa, red, scal, it, rtol, nb, po);
}

// One grid barrier of a cooperative launch: arrival number `target` (counted over the
// launches of an SR step) opens it.  The wait is bounded; false: it gave up.
__device__ __forceinline__ bool grid_barrier(unsigned* ctr, unsigned target) {
  __shared__ int ok;
  __syncthreads();
  if (threadIdx.x == 0) {
    __threadfence();
    atomicAdd(ctr, 1u);
    unsigned v = 0;
    ok = 0;
    for (int it = 0; it < (1 << 22); ++it) {
      asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(ctr) : "memory");
      if ((int)(v - target) >= 0) {
        ok = 1;
        break;
      }
    }
    __threadfence();
  }
  __syncthreads();
  return ok != 0;
}

// The vector half of a CG iteration in one cooperative launch: the split reduction
// (S p + eps p and p^H A p), then alpha, x, r and ||r||^2, then beta, p and what the
// next forward reads of it, with two grid barriers where three launches had their
// gaps, ramps and drains (each 4-5 us whatever the size).  Same bodies, partial sums
// and reduction order as those launches (a block may take several of their blocks),
// which the batched and symmetric steps still use.  A small problem's few blocks
// would take the split reduction alone for most of the time (64 splits of a 40-site
// chain's 3321 elements on 4 SMs: 23 of 40 us), so it is spread over more blocks first
// (`spread`), one more barrier before the inner product.
struct CgFused {
  const void* part;
  int splits;
  int64_t pa, corner;
  void *x, *r, *p, *ap;
  double eps, rtol;
  double *red, *scal;
  int it, nb;  // nb: blocks of the partial sums (sr_vec_blocks)
  int spread;  // > 0: that many threads of each block reduce one element each
  PlaneOut po;
};
constexpr int kFusedPerSm = 5;  // resident blocks per SM (launch bounds)
template <bool CPLX>
__global__ void __launch_bounds__(kVecThreads, kFusedPerSm) cg_fused_kernel(CgFused A) {
  if (A.scal[SC_DONE] != 0.0) return;  // written by an earlier launch: the same in every block
  const int b0 = blockIdx.x, gb = gridDim.x, nb = A.nb;
  unsigned* ctr = reinterpret_cast<unsigned*>(A.scal + SC_BAR);
  unsigned arrived = (unsigned)(A.spread ? 3 : 2) * (unsigned)A.it * (unsigned)gb;
  bool ok = true;
  auto sync = [&]() { ok = grid_barrier(ctr, arrived += (unsigned)gb) && ok; };
  if (A.spread) {
    const int64_t e = (int64_t)b0 * A.spread + threadIdx.x;
    if ((int)threadIdx.x < A.spread && e < A.pa)
      reduce_one<CPLX>(e, A.part, A.splits, A.pa, A.corner, A.ap, A.p, A.eps);
    sync();
    for (int b = b0; b < nb; b += gb) dot_body<CPLX>(b, nb, A.p, A.ap, A.pa, A.red);
  } else {
    for (int b = b0; b < nb; b += gb)
      reduce_parts_body<CPLX, true>(b, nb, A.part, A.splits, A.pa, A.corner, A.ap, A.p, A.eps,
                                    A.red, nullptr);
  }
  sync();
  for (int b = b0; b < nb; b += gb)
    cg_step_x_body<CPLX, 1>(b, nb, A.x, A.r, A.p, A.ap, A.pa, A.red, A.scal, A.it, nb);
  sync();
  // block 0 ends with the scalars, so it takes its blocks last to first
  for (int b = b0 < nb ? b0 + (nb - 1 - b0) / gb * gb : -1; b >= 0; b -= gb)
    cg_step_p_body<CPLX, 1>(b, nb, A.r, A.p, A.pa, A.red, A.scal, A.it, A.rtol, nb, A.po);
  if (!ok && threadIdx.x == 0) {
    atomicOr(reinterpret_cast<int*>(A.scal + SC_ERR), 1);
    dev_status_set(1u << NK_ERR_TIMEOUT);
  }
}

// ------------------------------------------------------------------ CG of a small problem
// The whole CG of a small FP32 step in one cluster of eight CTAs.  Three launches an
// iteration spend nearly all their time on launches, ramps and a chain of dependent
// loads (10-site chain, 1008 samples, 121 parameters: 36 us an iteration); here the
// iterations stay in the cluster with two cluster barriers each, x and r in registers
// and p in shared memory, every CTA keeping all of them (19 us).  Samples are dealt
// to the CTAs in the forward kernel's tiles of 64 and the adjoint's elements in equal
// ranges; y, the centring partials and A p are passed through L2.  Every sum runs in
// the order of the three launches (forward_fp32_kernel, adjoint_fp32_kernel,
// cg_fused_kernel with one block).  FP64 adds and divisions that every warp needs are
// made by one and passed on: an SM does 1.6 per clock.
struct CgSmall {
  const int8_t* sigma;
  const void* T;
  const double* weights;
  int ns, n, m, splits, chunk, pa;
  void *x, *r, *y, *ap;
  double *mean_part, *scal;
  double eps, rtol;
  int n_cg;
};
constexpr int kCgCtas = 8;       // portable cluster size
constexpr int kCgPer = 4;        // elements per thread of the vector updates
constexpr int kCgMaxM = 63;      // one group of four columns per lane covers m + 1

// Where it is taken: problems that it has room for, and of those the ones whose busiest
// CTA has so little to do, in tiles of 64 samples (forward) and rounds of 256 products
// per sample of a split (adjoint), that it is done before three launches are; these take
// longer with more hidden units.  50 iterations here and in three launches, ms: real
// 10 x 10, 1200 samples 1.32 and 1.80, 20 x 20, 1200 samples 1.58 and 2.01, beyond the line
// 1500 samples 2.08 and 2.01; complex 14 x 14, 1500 samples 1.82 and 2.01, beyond 2000
// samples 2.12 and 2.05; 20 x 40, 600 samples 1.83 and 2.68, beyond 1200 samples 2.82 and
// 2.64.  (Complex problems of more than 1536 samples and 2^18 products win or lose within
// 6 % whatever the line.  Of 206 shapes measured, on the wrong side by more than that:
// real 8 x 8, 3000 samples, 7 %.)
static bool cg_small(int64_t ns, int m, int64_t pa, int cplx, int splits) {
  if (pa > kCgPer * kVecThreads || m > kCgMaxM || ns > 4096) return false;
  const int tiles = ceil_div(ceil_div((int)ns, 64), kCgCtas);
  const int rounds = ceil_div(ceil_div((int)pa, kCgCtas) * splits, kVecThreads);
  const int64_t adjoint = rounds * adjoint_chunk(ns, splits);
  const int64_t cols = pa / (m + 1) * ceil_div(m + 1, 16);  // of a tile's products, per lane
  if (cplx && ns > 1536 && ns * pa > 1 << 18) return false;
  return cplx ? tiles * (100 + 2 * cols) + adjoint <= 750 + 8 * m
              : tiles * 100 + adjoint <= 840 + 2 * m;
}

template <bool CPLX>
struct CgSmallSmem {
  using DT = typename D<CPLX>::T;
  using F = typename std::conditional<CPLX, float2, float>::type;
  DT p[kCgPer * kVecThreads];
  F xf[kCgPer * kVecThreads + kCgMaxM + 1];  // p as F32, rows a pitch apart
  DT part[64][17];              // a tile's row sums by lane
  DT y[64];
  DT sh8[8];
  DT mean;
  double sh[8], alpha, beta;
  int done;                     // 1: converged, 2: not finite
};

__device__ __forceinline__ double ld_l2(const double* p) { return __ldcg(p); }
__device__ __forceinline__ double2 ld_l2(const double2* p) { return __ldcg(p); }

__device__ __forceinline__ void cluster_sync_all() {
  asm volatile("barrier.cluster.arrive.release;" ::: "memory");
  asm volatile("barrier.cluster.wait.acquire;" ::: "memory");
}

template <bool CPLX>
__global__ void __cluster_dims__(kCgCtas, 1, 1) __launch_bounds__(kVecThreads)
    cg_small_kernel(CgSmall A) {
  using DT = typename D<CPLX>::T;
  using F = typename std::conditional<CPLX, float2, float>::type;
  if (A.scal[SC_DONE] != 0.0) return;  // written by an earlier launch: the same in every CTA
  extern __shared__ __align__(16) unsigned char smraw[];
  CgSmallSmem<CPLX>& S = *reinterpret_cast<CgSmallSmem<CPLX>*>(smraw);
  F* vs = reinterpret_cast<F*>(smraw + sizeof(CgSmallSmem<CPLX>));  // [ns]
  F* pz = vs + A.ns;                                                // [splits][ec]
  const int tid = threadIdx.x, lane = tid & 31, c = blockIdx.x;
  const int n = A.n, m = A.m, na = n + 1, ns = A.ns, pa = A.pa;
  const F* T = reinterpret_cast<const F*>(A.T);
  DT* y = reinterpret_cast<DT*>(A.y);
  DT* ap = reinterpret_cast<DT*>(A.ap);
  const int nvb = (ns + 63) / 64, vb0 = nvb * c / kCgCtas, vb1 = nvb * (c + 1) / kCgCtas;
  const int e0 = pa * c / kCgCtas, ec = pa * (c + 1) / kCgCtas - e0;
  const double invn = 1.0 / (double)ns;
  // pitch of xf: lanes read neighbouring rows, which fall into the same banks where the
  // pitch is a multiple of 16 (complex, 16 rows of 8 bytes: even); complex 15 x 30, 1500
  // samples 2.95 -> 2.16 ms
  const int xp = (na & (CPLX ? 1 : 15)) ? na : na + 1;
  int at[kCgPer];  // where the thread's elements lie in it
  DT x[kCgPer], r[kCgPer];
#pragma unroll
  for (int u = 0; u < kCgPer; ++u) {
    const int e = tid + u * kVecThreads;
    x[u] = r[u] = D<CPLX>::zero();
    at[u] = xp == na ? e : e + e / na;
    if (e < pa) {
      r[u] = reinterpret_cast<const DT*>(A.r)[e];
      S.p[e] = r[u];
      if constexpr (CPLX) S.xf[at[u]] = make_float2((float)r[u].x, (float)r[u].y);
      else S.xf[at[u]] = (float)r[u];
    }
  }
  double rs = A.scal[SC_RS0];
  const double fn = A.scal[SC_FNORM];
  int it = 0, done = 0;
  __syncthreads();
  while (it < A.n_cg && !done) {
    // forward: 64 samples at a time; lane x of 16 takes columns x + 16 q of four rows
    for (int vb = vb0; vb < vb1; ++vb) {
      const int xl = tid & 15, row0 = 4 * (tid >> 4);
      const int nq = (m + 16) / 16;  // column steps that any lane has
      F acc[4][4];
      const int8_t* sg[4];
      const F* X[4];
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        X[q] = S.xf + min(xl + 16 * q, m) * xp;
#pragma unroll
        for (int k = 0; k < 4; ++k) acc[q][k] = F{};
      }
      F tq[4][4];  // T', loaded ahead of the products
#pragma unroll
      for (int k = 0; k < 4; ++k)
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          if (q >= nq) break;
          const int j = xl + 16 * q;
          fg_one(tq[k][q]);
          if (j < m) tq[k][q] = __ldg(T + (int64_t)min(vb * 64 + row0 + k, ns - 1) * m + j);
        }
#pragma unroll
      for (int k = 0; k < 4; ++k) sg[k] = A.sigma + (int64_t)min(vb * 64 + row0 + k, ns - 1) * n;
#pragma unroll 4
      for (int i = 0; i < na; ++i) {
        float s4[4];
#pragma unroll
        for (int k = 0; k < 4; ++k) s4[k] = i < n ? (float)__ldg(sg[k] + i) : 1.f;
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          if (q >= nq) break;
          const F xv = X[q][i];
#pragma unroll
          for (int k = 0; k < 4; ++k) {
            if constexpr (CPLX) {
              acc[q][k].x = fmaf(s4[k], xv.x, acc[q][k].x);
              acc[q][k].y = fmaf(s4[k], xv.y, acc[q][k].y);
            } else {
              acc[q][k] = fmaf(s4[k], xv, acc[q][k]);
            }
          }
        }
      }
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        float pr = 0.f, pi = 0.f;
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          const int j = xl + 16 * q;
          if (j > m) continue;
          if constexpr (CPLX) {
            const float ar = acc[q][k].x, ai = acc[q][k].y;
            const float2 t = tq[k][q];
            pr += t.x * ar - t.y * ai;
            pi += t.x * ai + t.y * ar;
          } else {
            pr += tq[k][q] * acc[q][k];
          }
        }
        if constexpr (CPLX) S.part[row0 + k][xl] = make_double2((double)pr, (double)pi);
        else S.part[row0 + k][xl] = (double)pr;
      }
      __syncthreads();
      if (tid < 64) {
        // the 16 lanes of a row, halves first (lanes beyond m hold 0), then the tile's
        // part of the centring mean: four rows, pairs of those, the eight pairs in order
        const int s = vb * 64 + tid;
        DT v[16];
#pragma unroll
        for (int u = 0; u < 16; ++u) v[u] = S.part[tid][u];
#pragma unroll
        for (int off = 8; off >= 1; off >>= 1)
#pragma unroll
          for (int u = 0; u < off; ++u)
            if (u + off <= m) v[u] = vadd(v[u], v[u + off]);
        S.y[tid] = s < ns ? v[0] : D<CPLX>::zero();
        if (s < ns) y[s] = v[0];
        __syncwarp();
        double wr = 0.0, wi = 0.0;
        if (lane < 8) {
          const int q4 = (tid >> 5) * 32 + lane * 4;
#pragma unroll
          for (int k = 0; k < 4; ++k) {
            const int sk = vb * 64 + q4 + k;
            if (sk >= ns) break;
            const double w = A.weights ? __ldg(A.weights + sk) : invn;
            wr += w * re(S.y[q4 + k]);
            if (CPLX) wi += w * im(S.y[q4 + k]);
          }
        }
        wr += __shfl_xor_sync(0xffffffffu, wr, 1);
        if (CPLX) wi += __shfl_xor_sync(0xffffffffu, wi, 1);
        if (lane < 8 && !(lane & 1)) {
          DT& d = S.sh8[(tid >> 5) * 4 + lane / 2];
          if constexpr (CPLX) d = make_double2(wr, wi);
          else d = wr;
        }
      }
      __syncthreads();
      if (tid == 0) {
        double tr = 0.0, ti = 0.0;
#pragma unroll
        for (int u = 0; u < 8; ++u) {
          tr += re(S.sh8[u]);
          if (CPLX) ti += im(S.sh8[u]);
        }
        A.mean_part[vb] = tr;
        if (CPLX) A.mean_part[kVecBlocks + vb] = ti;
      }
    }
    cluster_sync_all();
    // v = w (y - <y>), every CTA for all samples
    // (one warp does each scalar's arithmetic: the FP64 pipe would make eight wait)
    if (tid < 32) {
      double mr = 0.0, mi = 0.0;
      for (int u = lane; u < nvb; u += 32) {
        mr += ld_l2(A.mean_part + u);
        if (CPLX) mi += ld_l2(A.mean_part + kVecBlocks + u);
      }
#pragma unroll
      for (int off = 16; off >= 1; off >>= 1) {
        mr += __shfl_xor_sync(0xffffffffu, mr, off);
        if (CPLX) mi += __shfl_xor_sync(0xffffffffu, mi, off);
      }
      if (lane == 0) {
        if constexpr (CPLX) S.mean = make_double2(mr, mi);
        else S.mean = mr;
      }
    }
    __syncthreads();
    {
      const double mr = re(S.mean), mi = im(S.mean);
      for (int s = tid; s < ns; s += kVecThreads) {
        const double w = A.weights ? __ldg(A.weights + s) : invn;
        const DT ys = ld_l2(y + s);
        store_v<CPLX>(vs, s, w * (re(ys) - mr), w * (im(ys) - mi));
      }
    }
    __syncthreads();
    // adjoint: one thread per element and split
    for (int w = tid; w < ec * A.splits; w += kVecThreads) {
      const int z = w / ec, e = e0 + w % ec, j = e / na, i = e % na;
      const int sb = z * A.chunk, se = min(ns, sb + A.chunk);
      F a = F{};
      const F* tp = T + min(j, m - 1);
      const int8_t* sp = A.sigma + min(i, n - 1);
#pragma unroll 8
      for (int s = sb; s < se; ++s) {
        F t = __ldg(tp + (int64_t)s * m);
        if (j == m) fg_one(t);
        const float sv = i < n ? (float)__ldg(sp + (int64_t)s * n) : 1.f;
        const F v = vs[s];
        if constexpr (CPLX) {
          const float2 zv = make_float2(t.x * v.x + t.y * v.y, t.x * v.y - t.y * v.x);
          a.x = fmaf(zv.x, sv, a.x);
          a.y = fmaf(zv.y, sv, a.y);
        } else {
          a = fmaf(__fmul_rn(t, v), sv, a);
        }
      }
      pz[w] = a;
    }
    __syncthreads();
    for (int w = tid; w < ec; w += kVecThreads) {
      float2 hi = make_float2(0.f, 0.f), lo = make_float2(0.f, 0.f);
      for (int z = 0; z < A.splits; ++z) {
        const F v = pz[z * ec + w];
        float er;
        if constexpr (CPLX) {
          two_sum(hi.x, v.x, hi.x, er);
          lo.x += er;
          two_sum(hi.y, v.y, hi.y, er);
          lo.y += er;
        } else {
          two_sum(hi.x, v, hi.x, er);
          lo.x += er;
        }
      }
      DT a;
      if constexpr (CPLX)
        a = make_double2((double)hi.x + (double)lo.x, (double)hi.y + (double)lo.y);
      else
        a = (double)hi.x + (double)lo.x;
      a = axpy(A.eps, S.p[e0 + w], a);
      if (e0 + w == pa - 1) a = D<CPLX>::zero();  // X'[m][n] is no parameter
      ap[e0 + w] = a;
    }
    cluster_sync_all();
    // alpha, x, r, beta and p, the same in every CTA
    DT q[kCgPer];
    double dot = 0.0;
#pragma unroll
    for (int u = 0; u < kCgPer; ++u) {
      const int e = tid + u * kVecThreads;
      if (e >= pa) break;
      q[u] = ld_l2(ap + e);
      dot = add_cdot(dot, S.p[e], q[u]);
    }
    const int nw = min(kVecThreads / 32, (pa + 31) / 32);  // warps with elements
    auto warp_part = [&](double v) {
      if (tid / 32 >= nw) return;
#pragma unroll
      for (int off = 16; off >= 1; off >>= 1) v += __shfl_xor_sync(0xffffffffu, v, off);
      if (lane == 0) S.sh[tid / 32] = v;
    };
    auto total = [&]() {
      double t = 0.0;
      for (int u = 0; u < nw; ++u) t += S.sh[u];
      return t;
    };
    warp_part(dot);
    __syncthreads();
    if (tid < 32) {
      const double alpha = rs / total();
      if (lane == 0) S.alpha = alpha;
    }
    __syncthreads();
    const double alpha = S.alpha;
    double nn = 0.0;
#pragma unroll
    for (int u = 0; u < kCgPer; ++u) {
      const int e = tid + u * kVecThreads;
      if (e >= pa) break;
      x[u] = axpy(alpha, S.p[e], x[u]);
      r[u] = axpy(-alpha, q[u], r[u]);
      nn = add_norm2(nn, r[u]);
    }
    warp_part(nn);
    __syncthreads();
    if (tid < 32) {
      const double rs_new = total(), beta = rs_new / rs;
      const bool bad = !isfinite(rs_new);
      if (lane == 0) {
        S.beta = beta;
        S.done = bad ? 2 : sqrt(rs_new) <= A.rtol * fn ? 1 : 0;
      }
      rs = rs_new;  // (in this warp)
    }
    __syncthreads();
    done = S.done;
    if (!done) {
      const double beta = S.beta;
#pragma unroll
      for (int u = 0; u < kCgPer; ++u) {
        const int e = tid + u * kVecThreads;
        if (e >= pa) break;
        const DT pn = axpy(beta, S.p[e], r[u]);
        S.p[e] = pn;
        if constexpr (CPLX) S.xf[at[u]] = make_float2((float)pn.x, (float)pn.y);
        else S.xf[at[u]] = (float)pn;
      }
    }
    ++it;
    __syncthreads();
  }
  if (c == 0) {
#pragma unroll
    for (int u = 0; u < kCgPer; ++u) {
      const int e = tid + u * kVecThreads;
      if (e < pa) reinterpret_cast<DT*>(A.x)[e] = x[u];
    }
    if (tid == 0) {
      A.scal[SC_RS0] = A.scal[SC_RS1] = rs;
      A.scal[SC_ITERS] = (double)it;
      if (done) A.scal[SC_DONE] = 1.0;
      if (done == 2) A.scal[SC_NONFINITE] = 1.0;
    }
  }
}

template <bool CPLX>
static nk_status launch_cg_small(const CgSmall& A, cudaStream_t st) {
  const size_t f = CPLX ? 8 : 4;
  const size_t smem = sizeof(CgSmallSmem<CPLX>) +
                      f * ((size_t)A.ns + (size_t)ceil_div(A.pa, kCgCtas) * A.splits);
  if (!allow_smem(cg_small_kernel<CPLX>, smem))
    return fail(NK_ERR_CUDA, "nk_sr_step: shared memory attribute");
  cg_small_kernel<CPLX><<<kCgCtas, kVecThreads, smem, st>>>(A);
  return check_launch("nk_sr_step(small cg)");
}

__device__ __forceinline__ void sr_write_info(const double* scal, double* info, double rtol);

// alpha <- alpha - lr delta (FP64 master), delta in the augmented layout; info.
template <bool CPLX>
__device__ __forceinline__ void sr_update_body(int bx, int gx, double* a, double* b, double* w, int n, int m,
                                 const void* __restrict__ xv, double lr, const double* scal,
                                 double* info, int n_iter_final, double rtol) {
  using DT = typename D<CPLX>::T;
  const DT* x = reinterpret_cast<const DT*>(xv);
  const int na = n + 1;
  const int64_t tot = (int64_t)(m + 1) * na;
  for (int64_t e = bx * (int64_t)blockDim.x + threadIdx.x; e < tot;
       e += (int64_t)gx * blockDim.x) {
    int j = (int)(e / na), i = (int)(e % na);
    double* dst;
    if (j < m && i < n) dst = w + (CPLX ? 2 : 1) * ((int64_t)j * n + i);
    else if (j < m) dst = b + (CPLX ? 2 : 1) * j;
    else if (i < n) dst = a + (CPLX ? 2 : 1) * i;
    else continue;
    if constexpr (CPLX) {
      dst[0] -= lr * x[e].x;
      dst[1] -= lr * x[e].y;
    } else {
      dst[0] -= lr * x[e];
    }
  }
  if (bx == 0 && threadIdx.x == 0) sr_write_info(scal, info, rtol);
}

// info {CG iterations, residual, ||F||, flags} from the CG scalars (one thread)
__device__ __forceinline__ void sr_write_info(const double* scal, double* info, double rtol) {
  {
    const double iters = scal[SC_ITERS];
    const double fn = scal[SC_FNORM];
    const double rs = scal[((int)iters & 1) ? SC_RS1 : SC_RS0];
    const double res = fn > 0.0 ? sqrt(rs) / fn : 0.0;
    info[NK_INFO_CG_ITERS] = iters;
    info[NK_INFO_CG_RESID] = res;
    info[NK_INFO_F_NORM] = fn;
    int flags = 0;
    if (res > rtol) flags |= 1 << NK_ERR_NOT_CONVERGED;
    if (scal[SC_NONFINITE] != 0.0 || !isfinite(res)) flags |= 1 << NK_ERR_NONFINITE;
    if (*reinterpret_cast<const int*>(scal + SC_ERR) != 0) flags |= 1 << NK_ERR_TIMEOUT;
    info[NK_INFO_FLAGS] = (double)flags;
  }
}

template <bool CPLX>
__global__ void sr_update_kernel(double* a, double* b, double* w, int n, int m,
                                 const void* __restrict__ xv, double lr, const double* scal,
                                 double* info, int n_iter_final, double rtol) {
  sr_update_body<CPLX>(blockIdx.x, gridDim.x, a, b, w, n, m, xv, lr, scal, info, n_iter_final, rtol);
}

// ------------------------------------------------------------------ symmetric RBM
// Tied parameters in the augmented layout [alpha + 1][n + 1]: (f, i < n) = Wt[f][i],
// (f, n) = bt[f], (alpha, 0) = at; the other entries of the last row stand for
// nothing and stay 0 in every CG vector (their fold lists are empty).

__device__ __forceinline__ double shfl_xor(double v, int o) {
  return __shfl_xor_sync(0xffffffffu, v, o);
}
__device__ __forceinline__ double2 shfl_xor(double2 v, int o) {
  return make_double2(__shfl_xor_sync(0xffffffffu, v.x, o), __shfl_xor_sync(0xffffffffu, v.y, o));
}

// P x: out[e] = x[tie[e]] over the untied augmented layout (0 where tie < 0)
template <bool CPLX>
__global__ void __launch_bounds__(kVecThreads) symm_expand_vec_kernel(
    const void* __restrict__ xv, const int* __restrict__ tie, int64_t pa, void* outv,
    const double* scal) {
  if (scal && scal[SC_DONE] != 0.0) return;
  using DT = typename D<CPLX>::T;
  const DT* x = reinterpret_cast<const DT*>(xv);
  DT* out = reinterpret_cast<DT*>(outv);
  for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < pa;
       e += (int64_t)gridDim.x * blockDim.x) {
    const int k = tie[e];
    out[e] = k >= 0 ? x[k] : D<CPLX>::zero();
  }
}

// P^T u (+ eps p): one warp per tied element sums its untied elements (lane l
// takes list entries l, l + 32, ..., then a fixed xor tree), so the result does
// not depend on scheduling; with p, per-block partials of Re p^H out -> red[bx].
template <bool CPLX>
__global__ void __launch_bounds__(kVecThreads) symm_fold_kernel(
    const void* __restrict__ uv, const int* __restrict__ off, const int* __restrict__ idx,
    int64_t pa_t, void* outv, const void* __restrict__ pv, double eps, double* red,
    const double* scal) {
  if (scal && scal[SC_DONE] != 0.0) return;
  using DT = typename D<CPLX>::T;
  const DT* u = reinterpret_cast<const DT*>(uv);
  const DT* p = reinterpret_cast<const DT*>(pv);
  DT* out = reinterpret_cast<DT*>(outv);
  const int lane = threadIdx.x & 31;
  const int64_t nw = ((int64_t)gridDim.x * blockDim.x) >> 5;
  double dot = 0.0;
  for (int64_t q = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5; q < pa_t; q += nw) {
    DT acc = D<CPLX>::zero();
    const int k1 = off[q + 1];
    for (int k = off[q] + lane; k < k1; k += 32) acc = vadd(acc, u[idx[k]]);
#pragma unroll
    for (int o = 16; o >= 1; o >>= 1) acc = vadd(acc, shfl_xor(acc, o));
    if (lane == 0) {
      if (p) {
        acc = axpy(eps, p[q], acc);
        dot = add_cdot(dot, p[q], acc);
      }
      out[q] = acc;
    }
  }
  if (red) {
    const double b = block_sum(dot);
    if (threadIdx.x == 0) red[blockIdx.x] = b;
  }
}

// theta_t <- theta_t - lr delta (tied layout); info
template <bool CPLX>
__global__ void symm_update_kernel(double* a, double* b, double* w, int n, int alpha,
                                   const void* __restrict__ xv, double lr,
                                   const double* scal, double* info, double rtol) {
  using DT = typename D<CPLX>::T;
  const DT* x = reinterpret_cast<const DT*>(xv);
  const int na = n + 1, c = CPLX ? 2 : 1;
  const int64_t tot = (int64_t)(alpha + 1) * na;
  for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < tot;
       e += (int64_t)gridDim.x * blockDim.x) {
    const int f = (int)(e / na), i = (int)(e % na);
    double* dst;
    if (f < alpha && i < n) dst = w + c * ((int64_t)f * n + i);
    else if (f < alpha) dst = b + c * f;
    else if (i == 0) dst = a;
    else continue;
    if constexpr (CPLX) {
      dst[0] -= lr * x[e].x;
      dst[1] -= lr * x[e].y;
    } else {
      dst[0] -= lr * x[e];
    }
  }
  if (blockIdx.x == 0 && threadIdx.x == 0) sr_write_info(scal, info, rtol);
}

// untied (a, b, W) from the tied parameters: a_i = at, b_(f,g) = bt_f,
// W[(f,g)][i] = Wt[f][perm[g][i]]
__global__ void symm_params_kernel(const double* __restrict__ ta, const double* __restrict__ tb,
                                   const double* __restrict__ tw, int n, int alpha, int ng,
                                   const int* __restrict__ perm, int cplx, double* a, double* b,
                                   double* w) {
  const int m = alpha * ng, c = cplx ? 2 : 1;
  const int64_t nw = (int64_t)m * n, tot = nw + m + n;
  for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < tot;
       e += (int64_t)gridDim.x * blockDim.x) {
    const double* src;
    double* dst;
    if (e < nw) {
      const int j = (int)(e / n), i = (int)(e % n);
      src = tw + c * ((int64_t)(j / ng) * n + perm[(int64_t)(j % ng) * n + i]);
      dst = w + c * e;
    } else if (e < nw + m) {
      const int j = (int)(e - nw);
      src = tb + c * (j / ng);
      dst = b + c * j;
    } else {
      src = ta;
      dst = a + c * (e - nw - m);
    }
    dst[0] = src[0];
    if (c == 2) dst[1] = src[1];
  }
}

// grad (a, b, W order) from the augmented adjoint result
template <bool CPLX>
__global__ void scatter_grad_kernel(const void* __restrict__ gv, int n, int m, double* grad) {
  using DT = typename D<CPLX>::T;
  const DT* g = reinterpret_cast<const DT*>(gv);
  const int na = n + 1;
  const int64_t tot = (int64_t)(m + 1) * na;
  for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < tot;
       e += (int64_t)gridDim.x * blockDim.x) {
    int j = (int)(e / na), i = (int)(e % na);
    int64_t k;
    if (j < m && i < n) k = (int64_t)n + m + (int64_t)j * n + i;
    else if (j < m) k = n + j;
    else if (i < n) k = i;
    else continue;
    if constexpr (CPLX) {
      grad[2 * k] = g[e].x;
      grad[2 * k + 1] = g[e].y;
    } else {
      grad[k] = g[e];
    }
  }
}

// ------------------------------------------------------------------ batched kernels
// The same kernels for every problem of an SR batch: blockIdx.y selects the
// problem (its SrDesc; complex and real problems share a launch and branch on
// its field), blockIdx.x runs over the problem's own grid (the one the
// single-problem launch uses), so each problem's reductions keep their order
// and a batched step computes exactly what nk_sr_step computes for it.

__global__ void __launch_bounds__(kVecThreads) stats_mean_batch(const SrDesc* __restrict__ D) {
  const SrDesc& d = D[blockIdx.y];
  if ((int)blockIdx.x >= d.nb_ns) return;
  if (d.cplx) stats_mean_body<true>(blockIdx.x, d.nb_ns, d.eloc, d.weights, d.ns, d.red);
  else stats_mean_body<false>(blockIdx.x, d.nb_ns, d.eloc, d.weights, d.ns, d.red);
}

__global__ void __launch_bounds__(kVecThreads) stats_dev_batch(const SrDesc* __restrict__ D) {
  const SrDesc& d = D[blockIdx.y];
  if ((int)blockIdx.x >= d.nb_ns) return;
  if (d.cplx)
    stats_dev_body<true>(blockIdx.x, d.nb_ns, d.eloc, d.weights, d.ns, d.n_chains, d.red, d.v,
                         d.nb_ns);
  else
    stats_dev_body<false>(blockIdx.x, d.nb_ns, d.eloc, d.weights, d.ns, d.n_chains, d.red, d.v,
                          d.nb_ns);
}

__global__ void stats_finish_batch(const SrDesc* __restrict__ D) {
  const SrDesc& d = D[blockIdx.y];
  stats_finish_body(d.weights, d.ns, d.n_chains, d.red, d.nb_ns, d.info, d.scal);
}

__global__ void flags_reset_batch(const SrDesc* __restrict__ D) {
  if (threadIdx.x == 0) {
    D[blockIdx.y].scal[SC_DONE] = 0.0;
    D[blockIdx.y].scal[SC_ERR] = 0.0;
  }
}

// in_cg = 0: F into r (no shift, no inner product); 1: S p + eps p into ap
__global__ void __launch_bounds__(kVecThreads) reduce_parts_batch(const SrDesc* __restrict__ D,
                                                                  int in_cg, double eps) {
  const SrDesc& d = D[blockIdx.y];
  if ((int)blockIdx.x >= d.nb_pa) return;
  char* out = in_cg ? d.ap : d.r;
  const void* p = in_cg ? d.p : nullptr;
  double* red = in_cg ? d.red : nullptr;
  const double* scal = in_cg ? d.scal : nullptr;
  const double e = in_cg ? eps : 0.0;
  if (d.cplx)
    reduce_parts_body<true>(blockIdx.x, d.nb_pa, d.part, d.splits, d.pa, d.corner, out, p, e,
                            red, scal);
  else
    reduce_parts_body<false>(blockIdx.x, d.nb_pa, d.part, d.splits, d.pa, d.corner, out, p, e,
                             red, scal);
}

__global__ void __launch_bounds__(kVecThreads) cg_init_batch(const SrDesc* __restrict__ D) {
  const SrDesc& d = D[blockIdx.y];
  if ((int)blockIdx.x >= d.nb_pa) return;
  if (d.cplx)
    cg_init_body<true>(blockIdx.x, d.nb_pa, d.x, d.r, d.p, d.pa, d.red);
  else
    cg_init_body<false>(blockIdx.x, d.nb_pa, d.x, d.r, d.p, d.pa, d.red);
}

__global__ void cg_init_scalars_batch(const SrDesc* __restrict__ D, double rtol) {
  const SrDesc& d = D[blockIdx.y];
  cg_init_scalars_body(0, 1, d.red, d.scal, rtol, d.nb_pa);
}

__global__ void __launch_bounds__(kVecThreads) center_partial_batch(const SrDesc* __restrict__ D) {
  const SrDesc& d = D[blockIdx.y];
  if ((int)blockIdx.x >= d.nb_ns || d.ctr_parts > 0) return;  // else the forward wrote them
  if (d.cplx)
    center_partial_body<true>(blockIdx.x, d.nb_ns, d.y, d.weights, d.ns, d.red, d.scal);
  else
    center_partial_body<false>(blockIdx.x, d.nb_ns, d.y, d.weights, d.ns, d.red, d.scal);
}

__global__ void __launch_bounds__(kVecThreads) center_apply_batch(const SrDesc* __restrict__ D) {
  const SrDesc& d = D[blockIdx.y];
  if ((int)blockIdx.x >= d.nb_ns) return;
  const int parts = d.ctr_parts > 0 ? d.ctr_parts : d.nb_ns;
  if (d.cplx)
    center_apply_body<true>(blockIdx.x, d.nb_ns, d.y, d.v, d.weights, d.ns, d.red, d.scal,
                            parts);
  else
    center_apply_body<false>(blockIdx.x, d.nb_ns, d.y, d.v, d.weights, d.ns, d.red, d.scal,
                             parts);
}

__global__ void __launch_bounds__(kVecThreads) cg_step_x_batch(const SrDesc* __restrict__ D,
                                                               int it) {
  const SrDesc& d = D[blockIdx.y];
  if ((int)blockIdx.x >= d.nb_pa) return;
  if (d.cplx)
    cg_step_x_body<true>(blockIdx.x, d.nb_pa, d.x, d.r, d.p, d.ap, d.pa, d.red, d.scal, it,
                       d.nb_pa);
  else
    cg_step_x_body<false>(blockIdx.x, d.nb_pa, d.x, d.r, d.p, d.ap, d.pa, d.red, d.scal, it,
                       d.nb_pa);
}

__global__ void __launch_bounds__(kVecThreads) cg_step_p_batch(const SrDesc* __restrict__ D,
                                                               int it, double rtol) {
  const SrDesc& d = D[blockIdx.y];
  if ((int)blockIdx.x >= d.nb_pa) return;
  PlaneOut po;
  po.planes = reinterpret_cast<uint16_t*>(d.xbf);
  po.na = d.n + 1;
  po.mt = d.mt1;
  po.na64 = d.na64;
  if (d.cplx)
    cg_step_p_body<true>(blockIdx.x, d.nb_pa, d.r, d.p, d.pa, d.red, d.scal, it, rtol, d.nb_pa,
                         po);
  else
    cg_step_p_body<false>(blockIdx.x, d.nb_pa, d.r, d.p, d.pa, d.red, d.scal, it, rtol, d.nb_pa,
                          po);
  if (d.fwd_nseg == 2) {
    // the next forward's two halves add onto zero (y of this iteration is consumed)
    double* y = reinterpret_cast<double*>(d.y);
    const int64_t len = d.ns * (d.cplx ? 2 : 1);
    for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < len;
         e += (int64_t)d.nb_pa * blockDim.x)
      y[e] = 0.0;
  }
}

__global__ void sr_update_batch(const SrDesc* __restrict__ D, double lr, int n_cg, double rtol) {
  const SrDesc& d = D[blockIdx.y];
  if ((int)blockIdx.x >= d.nb_pa) return;
  if (d.cplx)
    sr_update_body<true>(blockIdx.x, d.nb_pa, d.a, d.b, d.w, d.n, d.m, d.x, lr, d.scal, d.info,
                       n_cg, rtol);
  else
    sr_update_body<false>(blockIdx.x, d.nb_pa, d.a, d.b, d.w, d.n, d.m, d.x, lr, d.scal, d.info,
                       n_cg, rtol);
}

// ------------------------------------------------------------------ drivers

// A symmetric RBM's tables, tied parameters and tied CG vectors (nk_sr_step_symm).
struct SymmRun {
  const int *tie, *off, *idx, *perm;
  int64_t pa_t;
  int alpha, n_perm;
  double *a, *b, *w;
  char *x, *r, *p, *ap;
};

// sy = NULL: SR in the RBM's own parameters.  sy: SR in the tied parameters;
// the untied vectors x, r, p, ap of the scratch then hold expanded and
// not-yet-folded products only.
template <bool CPLX>
static nk_status sr_step_t(nk_rbm* r, const int8_t* sigma, const void* T, const double* eloc,
                           const double* weights, int64_t ns, int n_chains, double eps,
                           double lr, int n_cg, double rtol, int prec, char* sc,
                           double* info, cudaStream_t st, const SymmRun* sy = nullptr) {
  SrLayout L(r->n, r->m, CPLX, ns);
  double* scal = (double*)(sc + L.scal);
  double* red = (double*)(sc + L.red);
  const int n = r->n, m = r->m;
  const int64_t corner = (int64_t)m * L.na + n;
  const bool tc = prec == NK_PREC_BF16X2;
  // the CG runs on these vectors (the tied ones for a symmetric RBM)
  const int64_t pa_cg = sy ? sy->pa_t : L.pa;
  char* cx = sy ? sy->x : sc + L.x;
  char* cr = sy ? sy->r : sc + L.r;
  char* cp = sy ? sy->p : sc + L.p;
  char* cap = sy ? sy->ap : sc + L.ap;
  const int nbc = sr_vec_blocks(pa_cg);
  const int nbf = sy ? (int)std::min<int64_t>(kVecBlocks, (pa_cg + 7) / 8) : 0;
  int* err = reinterpret_cast<int*>(scal + SC_ERR);
  const int splits = sr_choose_splits(L, prec, r->sr_splits);
  AdjTcArgs aa{};
  FwdTcArgs fa{};
  if (tc) {
    aa.T = T;
    aa.ns = ns;
    aa.n = n;
    aa.m = m;
    aa.cplx = CPLX;
    aa.na64 = L.na64;
    aa.splits = splits;
    aa.part = sc + L.part;
    aa.err = err;
    fa.sigma = sigma;
    fa.ns = ns;
    fa.n = n;
    fa.m = m;
    fa.cplx = CPLX;
    fa.mode = 0;
    fa.mt = L.mt1;
    fa.na64 = L.na64;
    fa.rows = m + 1;
    fa.T = T;
    fa.y = sc + L.y;
    fa.skip = scal + SC_DONE;
    fa.err = err;
    fa.sig_rows = sc + L.sigr;
  }
  {
    const int nbs0 = sr_vec_blocks(ns);
    stats_mean_kernel<CPLX><<<nbs0, kVecThreads, 0, st>>>(eloc, weights, ns, red);
    stats_dev_kernel<CPLX><<<nbs0, kVecThreads, 0, st>>>(eloc, weights, ns, n_chains, red,
                                                        sc + L.v, nbs0);
    stats_finish_kernel<<<1, 32, 0, st>>>(weights, ns, n_chains, red, nbs0, info, scal);
  }
  if (nk_status e = check_launch("nk_sr_step(stats)")) return e;
  cudaMemsetAsync(scal + SC_DONE, 0, sizeof(double), st);
  cudaMemsetAsync(scal + SC_ERR, 0, 2 * sizeof(double), st);  // and SC_BAR
  // F = adjoint(w o (E - <E>)) -> r
  if (tc) {
    if (nk_status e = launch_sigma_t(sigma, ns, n, L.na64, sc + L.sigt, st)) return e;
    if (nk_status e = launch_sigma_rows(sigma, ns, n, L.na64, sc + L.sigr, st)) return e;
    aa.v = sc + L.v;
    aa.skip = nullptr;
    if (nk_status e = launch_adj_tc(aa, sc + L.sigt, st)) return e;
  } else {
    launch_adjoint_fp32<CPLX>(sigma, T, sc + L.v, ns, n, m, splits, sc + L.part, nullptr, st);
  }
  const int nbp = sr_vec_blocks(L.pa), nbs = sr_vec_blocks(ns);
  reduce_parts_kernel<CPLX><<<nbp, kVecThreads, 0, st>>>(sc + L.part, splits, L.pa, corner,
                                                         sc + L.r, nullptr, 0.0, nullptr,
                                                         nullptr);
  if (sy)
    symm_fold_kernel<CPLX><<<nbf, kVecThreads, 0, st>>>(sc + L.r, sy->off, sy->idx, pa_cg, cr,
                                                        nullptr, 0.0, nullptr, nullptr);
  cg_init_kernel<CPLX><<<nbc, kVecThreads, 0, st>>>(cx, cr, cp, pa_cg, red);
  cg_init_scalars_kernel<<<1, 32, 0, st>>>(red, scal, rtol, nbc);
  if (nk_status e = check_launch("nk_sr_step(force)")) return e;
  aa.v = sc + L.v;
  aa.skip = scal + SC_DONE;
  // The forward also writes the partial sums of the centring mean (one per CTA), when
  // they fit the partials buffer: no separate partial pass.
  const int64_t fp32_parts = tc ? 0 : forward_blocks(ns);
  const int ctr_parts = tc ? fwd_centring_parts(ns, L.mt1)
                           : (fp32_parts <= kVecBlocks ? (int)fp32_parts : 0);
  double* mean_part = ctr_parts ? red + 2 * kVecBlocks : nullptr;
  fa.mean_part = mean_part;
  fa.mean_stride = kVecBlocks;
  fa.weights = weights;
  fa.invn = 1.0 / (double)ns;
  // and where that is cheap the adjoint centres y itself while loading it
  const bool adj_ctr = ctr_parts && (tc ? adj_centres(m, CPLX) : adjoint_centres(ns, n, m, CPLX, splits));
  CentreArgs ca;
  if (adj_ctr) {
    aa.y = sc + L.y;
    aa.mean_part = red + 2 * kVecBlocks;
    aa.mean_stride = kVecBlocks;
    aa.invn = 1.0 / (double)ns;
    aa.mean_parts = ctr_parts;
    aa.weights = weights;
    ca.y = sc + L.y;
    ca.mean_part = mean_part;
    ca.parts = ctr_parts;
    ca.weights = weights;
    ca.invn = 1.0 / (double)ns;
  }
  // from the second CG iteration on, the p update writes the planes (or the F32 copy)
  // of p itself
  PlaneOut po;
  if (tc) {
    po.planes = (uint16_t*)(sc + L.xbf);
    po.na = L.na;
    po.mt = L.mt1;
    po.na64 = L.na64;
  } else {
    po.xf = sc + L.xf;
  }
  // the fused vector kernel's blocks have to be resident together
  int dev = 0, sms = 0;
  if (!sy && cudaGetDevice(&dev) == cudaSuccess)
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  int spread = 0, fused_grid = std::min(nbp, kFusedPerSm * sms);
  // Few blocks with little to reduce gain less from the fusion than the grid barriers take
  // (20 iterations, BF16 hi + lo, fused and in three launches: complex 100 x 100, 300
  // samples 888 us and 807, 100 x 400, 600 samples 1138 and 1079, but 16 x 64, 1000 samples
  // 650 and 691, 40 x 80, 1200 samples 746 and 860).
  if (tc && nbp < sms / 2 && splits <= 8 + nbp / 8) {
    fused_grid = 0;
  } else if (nbp < sms / 2 && splits > 4) {  // the smallest slices that stay under two per SM
    for (spread = 32; spread < 256 && ceil_div((int)L.pa, spread) > 2 * sms; spread *= 2) {}
    fused_grid = std::max(fused_grid, std::min(ceil_div((int)L.pa, spread), kFusedPerSm * sms));
    if (ceil_div((int)L.pa, spread) > fused_grid) spread = 0;
  }
  const bool small = !tc && !sy && cg_small(ns, m, L.pa, CPLX, splits);
  if (small && n_cg > 0) {
    const CgSmall A{sigma, T, weights, (int)ns, n, m, splits, (int)adjoint_chunk(ns, splits),
                    (int)L.pa, sc + L.x, sc + L.r, sc + L.y, sc + L.ap, red + 2 * kVecBlocks,
                    scal, eps, rtol, n_cg};
    if (nk_status e = launch_cg_small<CPLX>(A, st)) return e;
  }
  for (int it = 0; it < (small ? 0 : n_cg); ++it) {
    if (sy)  // the untied p = P p_t for the contractions
      symm_expand_vec_kernel<CPLX><<<nbp, kVecThreads, 0, st>>>(cp, sy->tie, L.pa, sc + L.p,
                                                                scal);
    if (tc) {
      if (it == 0 || sy) {
        if (nk_status e = launch_bplanes_from_f64(sc + L.p, m + 1, n + 1, L.na, CPLX, L.mt1,
                                                  L.na64, sc + L.xbf, scal + SC_DONE, st))
          return e;
      }
      if (nk_status e = launch_fwd_tc(fa, sc + L.xbf, st)) return e;
    } else {
      if (it == 0 || sy)
        to_f32_kernel<CPLX><<<nbp, kVecThreads, 0, st>>>(sc + L.p, sc + L.xf, L.pa, scal);
      launch_forward_fp32<CPLX>(sigma, ns, n, m, sc + L.xf, T, sc + L.y, scal, weights, mean_part,
                                st);
    }
    if (ctr_parts == 0)
      center_partial_kernel<CPLX><<<nbs, kVecThreads, 0, st>>>(sc + L.y, weights, ns, red, scal);
    if (!adj_ctr)
      center_apply_kernel<CPLX><<<nbs, kVecThreads, 0, st>>>(sc + L.y, sc + L.v, weights, ns,
                                                             red, scal, ctr_parts ? ctr_parts : nbs);
    if (tc) {
      if (nk_status e = launch_adj_tc(aa, sc + L.sigt, st)) return e;
    } else {
      launch_adjoint_fp32<CPLX>(sigma, T, sc + L.v, ns, n, m, splits, sc + L.part, scal, st, ca);
    }
    if (fused_grid > 0) {
      CgFused A{sc + L.part, splits, L.pa, corner, sc + L.x, sc + L.r, sc + L.p, sc + L.ap, eps,
                rtol,        red,    scal, it,     nbp,    spread, po};
      void* args[] = {&A};
      const cudaError_t e = cudaLaunchCooperativeKernel(
          cg_fused_kernel<CPLX>, dim3((unsigned)fused_grid), dim3(kVecThreads), args, 0, st);
      if (e == cudaSuccess) continue;
      if (e != cudaErrorCooperativeLaunchTooLarge && e != cudaErrorNotSupported)
        return fail(NK_ERR_CUDA, "nk_sr_step: cooperative launch failed: %s", cudaGetErrorString(e));
      // refused, as in a context with fewer SMs than the device: three launches from here
      // on, which make the same sums
      cudaGetLastError();
      fused_grid = 0;
    }
    if (sy) {  // S_t p_t + eps p_t = P^T (S P p_t) + eps p_t
      reduce_parts_kernel<CPLX><<<nbp, kVecThreads, 0, st>>>(
          sc + L.part, splits, L.pa, corner, sc + L.ap, nullptr, 0.0, nullptr, scal);
      symm_fold_kernel<CPLX><<<nbf, kVecThreads, 0, st>>>(sc + L.ap, sy->off, sy->idx, pa_cg,
                                                          cap, cp, eps, red, scal);
    } else {
      reduce_parts_kernel<CPLX><<<nbp, kVecThreads, 0, st>>>(
          sc + L.part, splits, L.pa, corner, sc + L.ap, sc + L.p, eps, red, scal);
    }
    cg_step_x_kernel<CPLX><<<nbc, kVecThreads, 0, st>>>(cx, cr, cp, cap, pa_cg, red, scal, it,
                                                        sy ? nbf : nbc);
    cg_step_p_kernel<CPLX><<<nbc, kVecThreads, 0, st>>>(cr, cp, pa_cg, red, scal, it, rtol, nbc,
                                                        sy ? PlaneOut{} : po);
    if (nk_status e = check_launch("nk_sr_step(cg)")) return e;
  }
  if (nk_status e = check_launch("nk_sr_step(cg)")) return e;
  if (sy) {
    symm_update_kernel<CPLX><<<nbc, kVecThreads, 0, st>>>(sy->a, sy->b, sy->w, n, sy->alpha, cx,
                                                          lr, scal, info, rtol);
    symm_params_kernel<<<nbp, kVecThreads, 0, st>>>(sy->a, sy->b, sy->w, n, sy->alpha,
                                                    sy->n_perm, sy->perm, CPLX, r->a, r->b, r->w);
  } else {
    sr_update_kernel<CPLX><<<nbp, kVecThreads, 0, st>>>(r->a, r->b, r->w, n, m, sc + L.x, lr,
                                                        scal, info, n_cg, rtol);
  }
  if (nk_status e = check_launch("nk_sr_step(update)")) return e;
  return launch_prepare(r, st);
}

nk_status run_sr_step(nk_rbm* r, const int8_t* sigma, const void* t, const double* eloc,
                      const double* weights, int64_t ns, int n_chains, double diag_shift,
                      double lr, int n_cg, double cg_rtol, int prec, void* scratch,
                      size_t scratch_bytes, double* info, cudaStream_t st) {
  size_t need = sr_scratch_bytes(r->n, r->m, r->is_complex, ns);
  if (scratch_bytes < need)
    return fail(NK_ERR_SHAPE, "nk_sr_step: scratch of %zu B, need %zu B", scratch_bytes, need);
  if (r->is_complex)
    return sr_step_t<true>(r, sigma, t, eloc, weights, ns, n_chains, diag_shift, lr, n_cg, cg_rtol,
                           prec, (char*)scratch, info, st);
  return sr_step_t<false>(r, sigma, t, eloc, weights, ns, n_chains, diag_shift, lr, n_cg, cg_rtol,
                          prec, (char*)scratch, info, st);
}

// ------------------------------------------------------------------ symmetric RBM (host)

SymmTables::SymmTables(int n_, int alpha_, int n_perm_) : n(n_), alpha(alpha_), n_perm(n_perm_) {
  const int64_t m = (int64_t)alpha * n_perm;
  pa = (m + 1) * (n + 1);
  pa_t = (int64_t)(alpha + 1) * (n + 1);
  size_t o = 0;
  auto take = [&](int64_t count) {
    size_t at = o;
    o += (size_t)round_up(count * (int64_t)sizeof(int32_t), 256);
    return at;
  };
  perm = take((int64_t)n_perm * n);
  tie = take(pa);
  off = take(pa_t + 1);
  idx = take(std::max<int64_t>(pa - 1, 1));
  total = o;
}

// tie: untied augmented element (j, i) -> tied element; the fold lists are the
// untied elements of each tied one in ascending order (a counting sort).
nk_status symm_build_tables(const int32_t* perm, int n, int alpha, int n_perm,
                            std::vector<int32_t>* out) {
  const SymmTables T(n, alpha, n_perm);
  std::vector<char> seen((size_t)n);
  for (int g = 0; g < n_perm; ++g) {
    std::fill(seen.begin(), seen.end(), 0);
    for (int i = 0; i < n; ++i) {
      const int32_t k = perm[(int64_t)g * n + i];
      if (k < 0 || k >= n || seen[k])
        return fail(NK_ERR_INVALID_ARG, "nk_symm_upload: row %d of perm is not a permutation", g);
      seen[k] = 1;
    }
  }
  out->assign(T.total / sizeof(int32_t), 0);
  int32_t* base = out->data();
  int32_t* P = base + T.perm / 4;
  int32_t* tie = base + T.tie / 4;
  int32_t* off = base + T.off / 4;
  int32_t* idx = base + T.idx / 4;
  std::copy(perm, perm + (int64_t)n_perm * n, P);
  const int na = n + 1, m = alpha * n_perm;
  for (int j = 0; j <= m; ++j)
    for (int i = 0; i <= n; ++i) {
      int64_t t;
      if (j < m && i < n) t = (int64_t)(j / n_perm) * na + perm[(int64_t)(j % n_perm) * n + i];
      else if (j < m) t = (int64_t)(j / n_perm) * na + n;
      else if (i < n) t = (int64_t)alpha * na;
      else t = -1;
      tie[(int64_t)j * na + i] = (int32_t)t;
    }
  std::vector<int64_t> cnt((size_t)T.pa_t + 1, 0);
  for (int64_t e = 0; e < T.pa; ++e)
    if (tie[e] >= 0) ++cnt[(size_t)tie[e] + 1];
  for (int64_t q = 0; q < T.pa_t; ++q) cnt[(size_t)q + 1] += cnt[(size_t)q];
  for (int64_t q = 0; q <= T.pa_t; ++q) off[q] = (int32_t)cnt[(size_t)q];
  for (int64_t e = 0; e < T.pa; ++e)
    if (tie[e] >= 0) idx[cnt[(size_t)tie[e]]++] = (int32_t)e;
  return NK_OK;
}

static size_t symm_vec_bytes(int n, int alpha, int cplx) {
  return (size_t)round_up((int64_t)(alpha + 1) * (n + 1) * (cplx ? 16 : 8), 256);
}

size_t sr_symm_scratch_bytes(int n, int alpha, int n_perm, int cplx, int64_t ns) {
  return sr_scratch_bytes(n, alpha * n_perm, cplx, ns) + 4 * symm_vec_bytes(n, alpha, cplx);
}

static SymmRun symm_run(const nk_rbm_symm* s, char* vec) {
  const SymmTables T(s->n, s->alpha, s->n_perm);
  const char* tb = (const char*)s->tables;
  SymmRun y;
  y.perm = (const int*)(tb + T.perm);
  y.tie = (const int*)(tb + T.tie);
  y.off = (const int*)(tb + T.off);
  y.idx = (const int*)(tb + T.idx);
  y.pa_t = T.pa_t;
  y.alpha = s->alpha;
  y.n_perm = s->n_perm;
  y.a = s->a;
  y.b = s->b;
  y.w = s->w;
  y.x = y.r = y.p = y.ap = nullptr;
  if (vec) {
    const size_t vb = symm_vec_bytes(s->n, s->alpha, s->is_complex);
    y.x = vec;
    y.r = vec + vb;
    y.p = vec + 2 * vb;
    y.ap = vec + 3 * vb;
  }
  return y;
}

nk_status run_symm_expand(const nk_rbm_symm* s, nk_rbm* r, cudaStream_t st) {
  const SymmRun y = symm_run(s, nullptr);
  const int64_t tot = (int64_t)r->m * r->n + r->m + r->n;
  const int blocks = (int)std::min<int64_t>(1024, std::max<int64_t>(1, (tot + 1023) / 1024));
  symm_params_kernel<<<blocks, kVecThreads, 0, st>>>(s->a, s->b, s->w, s->n, s->alpha, s->n_perm,
                                                     y.perm, s->is_complex, r->a, r->b, r->w);
  if (nk_status e = check_launch("nk_symm_expand")) return e;
  return launch_prepare(r, st);
}

nk_status run_sr_step_symm(nk_rbm_symm* s, nk_rbm* r, const int8_t* sigma, const void* t,
                           const double* eloc, const double* weights, int64_t ns,
                           int n_chains, double diag_shift, double lr, int n_cg,
                           double cg_rtol, int prec, void* scratch, size_t scratch_bytes,
                           double* info, cudaStream_t st) {
  const size_t base = sr_scratch_bytes(r->n, r->m, r->is_complex, ns);
  const size_t need = sr_symm_scratch_bytes(s->n, s->alpha, s->n_perm, s->is_complex, ns);
  if (scratch_bytes < need)
    return fail(NK_ERR_SHAPE, "nk_sr_step_symm: scratch of %zu B, need %zu B", scratch_bytes,
                need);
  const SymmRun y = symm_run(s, (char*)scratch + base);
  if (r->is_complex)
    return sr_step_t<true>(r, sigma, t, eloc, weights, ns, n_chains, diag_shift, lr, n_cg,
                           cg_rtol, prec, (char*)scratch, info, st, &y);
  return sr_step_t<false>(r, sigma, t, eloc, weights, ns, n_chains, diag_shift, lr, n_cg,
                          cg_rtol, prec, (char*)scratch, info, st, &y);
}

// ------------------------------------------------------------------ SR batches

// Split count of item i of a batch: the RBM's own setting, else a batch-wide
// default that spreads about two waves of adjoint CTAs over all problems.
static int batch_item_splits(const nk_sr_batch_item* items, int n_inst, int i, int prec) {
  const nk_rbm* r = items[i].rbm;
  SrLayout L(r->n, r->m, r->is_complex, items[i].ns);
  if (r->sr_splits > 0) return sr_choose_splits(L, prec, r->sr_splits);
  int64_t tiles = 0;
  for (int k = 0; k < n_inst; ++k) {
    const int hj = items[k].rbm->is_complex ? 64 : 128;
    tiles += (items[k].rbm->m + 1 + hj - 1) / hj;
  }
  // about four CTAs per SM over the whole batch: the instances' CTAs differ in
  // work (sites padded to 64 or 128, 1-7 hidden tiles), and finer pieces end the
  // launch with less idle time (64 uneven 1D instances: 34.5 -> 32.6 ms per
  // iteration against two per SM; eight per SM: 33.4)
  const int s = (int)std::max<int64_t>(1, (4 * 152) / std::max<int64_t>(tiles, 1));
  return sr_choose_splits(L, prec, s);
}

// Problems in descriptor order: complex ones first, then real ones (items order
// within each field).
static std::vector<int> batch_order(const nk_sr_batch_item* items, int n_inst) {
  std::vector<int> order;
  for (int pass = 0; pass < 2; ++pass)
    for (int i = 0; i < n_inst; ++i)
      if ((items[i].rbm->is_complex != 0) == (pass == 0)) order.push_back(i);
  return order;
}

nk_status sr_batch_check(const nk_sr_batch_item* items, int n_inst, int prec) {
  if (n_inst < 1 || !items) return fail(NK_ERR_INVALID_ARG, "SR batch: no items");
  if (prec != NK_PREC_BF16X2)
    return fail(NK_ERR_UNSUPPORTED, "SR batch: only the tensor-core precision NK_PREC_BF16X2");
  for (int i = 0; i < n_inst; ++i) {
    const nk_sr_batch_item& it = items[i];
    const nk_rbm* r = it.rbm;
    if (!r || !r->ws || !r->a || !r->b || !r->w)
      return fail(NK_ERR_INVALID_ARG, "SR batch: item %d has no RBM or workspace", i);
    if (it.ns < 1 || !it.sigma || !it.t || !it.eloc || !it.scratch || !it.info_out)
      return fail(NK_ERR_INVALID_ARG, "SR batch: item %d: NULL pointer or ns < 1", i);
    if (it.n_chains < 0 || (it.n_chains > 0 && it.ns % it.n_chains))
      return fail(NK_ERR_SHAPE, "SR batch: item %d: ns not a multiple of n_chains", i);
    if (((uintptr_t)it.scratch) & 255)
      return fail(NK_ERR_INVALID_ARG, "SR batch: item %d: scratch not 256-byte aligned", i);
    if (it.scratch_bytes < sr_scratch_bytes(r->n, r->m, r->is_complex, it.ns))
      return fail(NK_ERR_SHAPE, "SR batch: item %d: scratch too small", i);
    if (!tc_supported_shape(r->n, r->m))
      return fail(NK_ERR_UNSUPPORTED, "SR batch: item %d: n + 1 > 448", i);
  }
  return NK_OK;
}

size_t sr_batch_desc_bytes(int n_inst) { return (size_t)std::max(n_inst, 0) * sizeof(SrDesc); }

nk_status sr_batch_describe(const nk_sr_batch_item* items, int n_inst, int prec, void* host,
                            size_t bytes) {
  if (nk_status e = sr_batch_check(items, n_inst, prec)) return e;
  if (!host || bytes < sr_batch_desc_bytes(n_inst))
    return fail(NK_ERR_SHAPE, "SR batch: descriptor buffer of %zu B, need %zu B", bytes,
                sr_batch_desc_bytes(n_inst));
  const std::vector<int> order = batch_order(items, n_inst);
  SrDesc* out = reinterpret_cast<SrDesc*>(host);
  for (int z = 0; z < n_inst; ++z) {
    const nk_sr_batch_item& it = items[order[z]];
    nk_rbm* r = it.rbm;
    const int cplx = r->is_complex ? 1 : 0;
    SrLayout L(r->n, r->m, cplx, it.ns);
    WsLayout W(r->n, r->m, cplx);
    SrDesc d;
    memset(&d, 0, sizeof(d));
    char* sc = (char*)it.scratch;
    if (!tc_make_map(&d.fwd_map, sc + L.xbf, 2LL * L.mt1 * 128, L.na64, L.na64, 128))
      return NK_ERR_CUDA;
    if (!tc_make_map(&d.adj_map, sc + L.sigt, L.na64, L.ns8, L.ns8, L.na64 / 2))
      return NK_ERR_CUDA;
    if (!tc_make_map(&d.sig_map, sc + L.sigr, it.ns, L.na64, L.na64, 128)) return NK_ERR_CUDA;
    d.fwd_nseg = fwd_tc_nseg(it.ns, L.mt1);
    d.ctr_parts = fwd_centring_parts(it.ns, L.mt1);
    d.splits = batch_item_splits(items, n_inst, order[z], prec);
    d.nb_pa = sr_vec_blocks(L.pa);
    d.nb_ns = sr_vec_blocks(it.ns);
    d.cplx = cplx;
    d.n = r->n;
    d.m = r->m;
    d.n_chains = it.n_chains;
    d.na64 = L.na64;
    d.mt1 = L.mt1;
    d.mp = W.mp;
    d.wmt = W.mt;
    d.wna64 = W.na64;
    d.ns = it.ns;
    d.pa = L.pa;
    d.corner = (int64_t)r->m * L.na + r->n;
    d.ns8 = L.ns8;
    d.sigma = it.sigma;
    d.T = it.t;
    d.eloc = it.eloc;
    d.weights = it.weights;
    d.a = r->a;
    d.b = r->b;
    d.w = r->w;
    d.ws = (char*)r->ws;
    d.ws_a32 = W.a32;
    d.ws_b32 = W.b32;
    d.ws_wt = W.wt;
    d.ws_tab = W.tab;
    d.ws_xw = W.xw;
    d.ws_wbf = W.wbf;
    d.x = sc + L.x;
    d.r = sc + L.r;
    d.p = sc + L.p;
    d.ap = sc + L.ap;
    d.part = sc + L.part;
    d.y = sc + L.y;
    d.v = sc + L.v;
    d.sigt = sc + L.sigt;
    d.sigr = sc + L.sigr;
    d.xbf = sc + L.xbf;
    d.red = (double*)(sc + L.red);
    d.scal = (double*)(sc + L.scal);
    d.done = d.scal + SC_DONE;
    d.info = it.info_out;
    memcpy(&out[z], &d, sizeof(d));
  }
  return NK_OK;
}

// one sub-batch: problems [z0, z0 + G) of the descriptor order (up to kBatchMax)
static nk_status sr_batch_group(const nk_sr_batch_item* items, int n_inst,
                                const std::vector<int>& order, int z0, int G,
                                const SrDesc* D, double eps, double lr, int n_cg, double rtol,
                                int prec, cudaStream_t st) {
  const SrDesc* Dg = D + z0;
  FwdBatch fb{};
  AdjBatch ab{};
  int max_fwd = 1, max_adj = 1, max_sp = 1, max_na64 = 64;
  int64_t max_ns8 = 8, max_xp = 1, max_wp = 1, max_work = 1, max_minb = 1, max_rows = 1;
  for (int z = 0; z < G; ++z) {
    const nk_sr_batch_item& it = items[order[z0 + z]];
    const nk_rbm* r = it.rbm;
    const int cplx = r->is_complex ? 1 : 0;
    const int HJ = cplx ? 64 : 128;
    SrLayout L(r->n, r->m, cplx, it.ns);
    WsLayout W(r->n, r->m, cplx);
    char* sc = (char*)it.scratch;
    double* scal = (double*)(sc + L.scal);
    const int splits = batch_item_splits(items, n_inst, order[z0 + z], prec);
    FwdTcArgs& fa = fb.a[z];
    fa.sigma = it.sigma;
    fa.ns = it.ns;
    fa.n = r->n;
    fa.m = r->m;
    fa.cplx = cplx;
    fa.mode = 0;
    fa.mt = L.mt1;
    fa.na64 = L.na64;
    fa.rows = r->m + 1;
    fa.T = it.t;
    fa.y = sc + L.y;
    fa.skip = scal + SC_DONE;
    fa.err = reinterpret_cast<int*>(scal + SC_ERR);
    fa.nseg = fwd_tc_nseg(it.ns, L.mt1);
    if (fwd_centring_parts(it.ns, L.mt1)) {
      fa.mean_part = (double*)(sc + L.red) + 2 * kVecBlocks;
      fa.mean_stride = kVecBlocks;
      fa.invn = 1.0 / (double)it.ns;
      fa.weights = it.weights;
    }
    fb.map[z] = &Dg[z].fwd_map;
    fb.smap[z] = &Dg[z].sig_map;
    fb.tiles[z] = (int)((it.ns + 127) / 128);
    AdjTcArgs& aa = ab.a[z];
    aa.T = it.t;
    aa.v = sc + L.v;
    aa.ns = it.ns;
    aa.n = r->n;
    aa.m = r->m;
    aa.cplx = cplx;
    aa.na64 = L.na64;
    aa.splits = splits;
    aa.part = sc + L.part;
    aa.skip = nullptr;
    aa.err = reinterpret_cast<int*>(scal + SC_ERR);
    ab.map[z] = &Dg[z].adj_map;
    ab.chunk[z] = round_up(std::max<int64_t>((it.ns + splits - 1) / splits, 1), 64);
    ab.tiles[z] = (r->m + 1 + HJ - 1) / HJ;
    ab.splits[z] = splits;
    max_fwd = std::max(max_fwd, fb.tiles[z] * fa.nseg);
    max_rows = std::max<int64_t>(max_rows, it.ns * (L.na64 / 8));
    max_adj = std::max(max_adj, ab.tiles[z]);
    max_sp = std::max(max_sp, splits);
    max_na64 = std::max(max_na64, L.na64);
    max_ns8 = std::max<int64_t>(max_ns8, L.ns8);
    max_xp = std::max<int64_t>(max_xp, (int64_t)L.mt1 * 128 * L.na64);
    max_wp = std::max<int64_t>(max_wp, (int64_t)W.mt * 128 * W.na64);
    max_work = std::max<int64_t>(max_work, (int64_t)W.mp * (r->n + 1));
    max_minb = std::max<int64_t>(max_minb, (std::max(W.mp, r->n) + 255) / 256);
  }
  int max_nbp = 1, max_nbs = 1;
  for (int z = 0; z < G; ++z) {
    const nk_sr_batch_item& it = items[order[z0 + z]];
    SrLayout L(it.rbm->n, it.rbm->m, it.rbm->is_complex ? 1 : 0, it.ns);
    max_nbp = std::max(max_nbp, sr_vec_blocks(L.pa));
    max_nbs = std::max(max_nbs, sr_vec_blocks(it.ns));
  }
  const dim3 vg(max_nbp, G), vs(max_nbs, G), one(1, G);
  bool all_fused = true;  // every forward of the group writes its centring partials
  for (int z = 0; z < G; ++z) all_fused = all_fused && fb.a[z].mean_part != nullptr;
  stats_mean_batch<<<vs, kVecThreads, 0, st>>>(Dg);
  stats_dev_batch<<<vs, kVecThreads, 0, st>>>(Dg);
  stats_finish_batch<<<one, 32, 0, st>>>(Dg);
  flags_reset_batch<<<one, 32, 0, st>>>(Dg);
  if (nk_status e = check_launch("nk_sr_step_batch(stats)")) return e;
  if (nk_status e = launch_sigma_t_batch(Dg, G, max_ns8, max_na64, st)) return e;
  if (nk_status e = launch_sigma_rows_batch(Dg, G, max_rows, st)) return e;
  if (nk_status e = launch_adj_tc_batch(ab, G, max_adj, max_sp, max_na64, st)) return e;
  reduce_parts_batch<<<vg, kVecThreads, 0, st>>>(Dg, 0, 0.0);
  cg_init_batch<<<vg, kVecThreads, 0, st>>>(Dg);
  cg_init_scalars_batch<<<one, 32, 0, st>>>(Dg, rtol);
  if (nk_status e = check_launch("nk_sr_step_batch(force)")) return e;
  // the adjoints centre the forwards' outputs themselves when every problem of
  // the group qualifies (otherwise the centring launch runs for all of them)
  bool all_adj_ctr = all_fused;
  for (int z = 0; z < G; ++z) {
    const nk_rbm* r = items[order[z0 + z]].rbm;
    all_adj_ctr = all_adj_ctr && adj_centres(r->m, r->is_complex ? 1 : 0);
  }
  for (int z = 0; z < G; ++z) {
    ab.a[z].skip = fb.a[z].skip;
    if (all_adj_ctr) {
      const nk_sr_batch_item& it = items[order[z0 + z]];
      SrLayout L(it.rbm->n, it.rbm->m, it.rbm->is_complex ? 1 : 0, it.ns);
      ab.a[z].y = (char*)it.scratch + L.y;
      ab.a[z].mean_part = fb.a[z].mean_part;
      ab.a[z].mean_stride = kVecBlocks;
      ab.a[z].invn = 1.0 / (double)it.ns;
      ab.a[z].mean_parts = fwd_centring_parts(it.ns, L.mt1);
      ab.a[z].weights = it.weights;
    }
  }
  for (int it = 0; it < n_cg; ++it) {
    // from the second CG iteration on, cg_step_p_batch writes the planes of p itself
    if (it == 0) {
      if (nk_status e = launch_bplanes_p_batch(Dg, G, max_xp, st)) return e;
    }
    if (nk_status e = launch_fwd_tc_batch(fb, G, max_fwd, max_na64, st)) return e;
    if (!all_fused) center_partial_batch<<<vs, kVecThreads, 0, st>>>(Dg);
    if (!all_adj_ctr) center_apply_batch<<<vs, kVecThreads, 0, st>>>(Dg);
    if (nk_status e = launch_adj_tc_batch(ab, G, max_adj, max_sp, max_na64, st)) return e;
    reduce_parts_batch<<<vg, kVecThreads, 0, st>>>(Dg, 1, eps);
    cg_step_x_batch<<<vg, kVecThreads, 0, st>>>(Dg, it);
    cg_step_p_batch<<<vg, kVecThreads, 0, st>>>(Dg, it, rtol);
    if (nk_status e = check_launch("nk_sr_step_batch(cg)")) return e;
  }
  sr_update_batch<<<vg, kVecThreads, 0, st>>>(Dg, lr, n_cg, rtol);
  if (nk_status e = check_launch("nk_sr_step_batch(update)")) return e;
  if (nk_status e = launch_prepare_batch(Dg, G, max_work, max_minb, st)) return e;
  return launch_bplanes_rbm_batch(Dg, G, max_wp, st);
}

nk_status run_sr_step_batch(const nk_sr_batch_item* items, int n_inst, const void* desc_dev,
                            double eps, double lr, int n_cg, double rtol, int prec,
                            cudaStream_t st) {
  if (nk_status e = sr_batch_check(items, n_inst, prec)) return e;
  if (!desc_dev || (((uintptr_t)desc_dev) & 255))
    return fail(NK_ERR_INVALID_ARG, "nk_sr_step_batch: descriptors NULL or not 256-byte aligned");
  const std::vector<int> order = batch_order(items, n_inst);
  const SrDesc* D = reinterpret_cast<const SrDesc*>(desc_dev);
  for (int z = 0; z < n_inst; z += kBatchMax) {
    const int G = std::min(kBatchMax, n_inst - z);
    if (nk_status e = sr_batch_group(items, n_inst, order, z, G, D, eps, lr, n_cg, rtol, prec, st))
      return e;
  }
  return NK_OK;
}

// ------------------------------------------------------------------ autotuner

template <bool CPLX>
static nk_status time_adjoint(const nk_rbm* r, const int8_t* sigma, const void* T, int64_t ns,
                              int prec, char* sc, const SrLayout& L, int splits,
                              cudaStream_t st, float* ms) {
  const int64_t corner = (int64_t)r->m * L.na + r->n;
  cudaEvent_t e0, e1;
  if (cudaEventCreate(&e0) != cudaSuccess || cudaEventCreate(&e1) != cudaSuccess)
    return fail(NK_ERR_CUDA, "nk_sr_tune: cannot create events");
  AdjTcArgs aa{};
  aa.T = T;
  aa.v = sc + L.v;
  aa.ns = ns;
  aa.n = r->n;
  aa.m = r->m;
  aa.cplx = CPLX;
  aa.na64 = L.na64;
  aa.splits = splits;
  aa.part = sc + L.part;
  nk_status e = NK_OK;
  float best = 1e30f;
  for (int rep = 0; rep < 4 && e == NK_OK; ++rep) {
    cudaEventRecord(e0, st);
    if (prec == NK_PREC_BF16X2)
      e = launch_adj_tc(aa, sc + L.sigt, st);
    else
      launch_adjoint_fp32<CPLX>(sigma, T, sc + L.v, ns, r->n, r->m, splits, sc + L.part, nullptr,
                                st);
    reduce_parts_kernel<CPLX><<<sr_vec_blocks(L.pa), kVecThreads, 0, st>>>(
        sc + L.part, splits, L.pa, corner, sc + L.ap, nullptr, 0.0, nullptr, nullptr);
    cudaEventRecord(e1, st);
    if (e == NK_OK) e = check_launch("nk_sr_tune");
    if (cudaEventSynchronize(e1) != cudaSuccess) e = fail(NK_ERR_CUDA, "nk_sr_tune: sync");
    float t = 0.f;
    cudaEventElapsedTime(&t, e0, e1);
    if (rep > 0) best = std::min(best, t);  // first repetition is a warm-up
  }
  cudaEventDestroy(e0);
  cudaEventDestroy(e1);
  *ms = best;
  return e;
}

nk_status run_sr_tune(nk_rbm* r, const int8_t* sigma, const void* t, int64_t ns, int prec,
                      void* scratch, size_t scratch_bytes, cudaStream_t st) {
  SrLayout L(r->n, r->m, r->is_complex, ns);
  if (scratch_bytes < L.total)
    return fail(NK_ERR_SHAPE, "nk_sr_tune: scratch of %zu B, need %zu B", scratch_bytes, L.total);
  char* sc = (char*)scratch;
  // any finite v: only the timing matters
  if (cudaMemsetAsync(sc + L.v, 0, (size_t)ns * (r->is_complex ? 16 : 8), st) != cudaSuccess)
    return fail(NK_ERR_CUDA, "nk_sr_tune: memset");
  if (prec == NK_PREC_BF16X2) {
    if (nk_status e = launch_sigma_t(sigma, ns, r->n, L.na64, sc + L.sigt, st)) return e;
  }
  const int h = prec == NK_PREC_BF16X2 ? L.splits_tc : L.splits_fp32;
  // candidates: the heuristic, half of it, and the split counts that fill
  // one to four whole waves of adjoint CTAs (one per SM)
  const int hj = tc_hidden_per_tile(r->is_complex);
  const int tiles = prec == NK_PREC_BF16X2 ? (r->m + 1 + hj - 1) / hj
                                           : ceil_div(L.na, 64) * ceil_div(L.ma, 64);
  int cand[6] = {h, h / 2};
  for (int k = 1; k <= 4; ++k) cand[1 + k] = (k * 152) / tiles;
  int best_s = sr_choose_splits(L, prec, h);
  float best_t = 1e30f;
  int tried[6];
  int n_tried = 0;
  for (int k = 0; k < 6; ++k) {
    const int sp = sr_choose_splits(L, prec, std::max(1, cand[k]));
    bool seen = false;
    for (int u = 0; u < n_tried; ++u) seen = seen || tried[u] == sp;
    if (seen) continue;
    tried[n_tried++] = sp;
    float ms = 0.f;
    nk_status e = r->is_complex
                      ? time_adjoint<true>(r, sigma, t, ns, prec, sc, L, sp, st, &ms)
                      : time_adjoint<false>(r, sigma, t, ns, prec, sc, L, sp, st, &ms);
    if (e) return e;
    if (ms < best_t) {
      best_t = ms;
      best_s = sp;
    }
  }
  r->sr_splits = best_s;
  return NK_OK;
}

// ------------------------------------------------------------------ K8 backward
// grad_k = sum_s conj(O_sk) g_s (analytic RBM log-derivatives, Sec. 2.2.5) over
// chunks of at most kBackChunk samples: per chunk, T = tanh(theta) is
// recomputed from sigma (the theta contraction of ln psi with a tanh epilogue
// and no ln cosh), the adjoint contraction writes its split-K partials, the
// partials are reduced over splits (fixed order) and the chunk's sum is added
// to an FP64 accumulator in chunk order.  Scratch holds one chunk's T and the
// adjoint's buffers for one chunk: it does not grow with ns beyond kBackChunk.

constexpr int64_t kBackChunk = 16384;

static int64_t backward_chunk(int64_t ns) {
  return std::min<int64_t>(std::max<int64_t>(ns, 1), kBackChunk);
}

size_t backward_scratch_bytes(int n, int m, int cplx, int64_t ns) {
  const int64_t c = backward_chunk(ns);
  SrLayout L(n, m, cplx, c);
  const size_t f = cplx ? 8 : 4;
  return L.total + (size_t)round_up(c * m * f, 256) +
         (size_t)round_up(L.pa * (cplx ? 16 : 8), 256);
}

template <bool CPLX>
__global__ void copy_g_kernel(const double* g, void* v, int64_t ns) {
  for (int64_t s = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; s < ns;
       s += (int64_t)gridDim.x * blockDim.x) {
    store_v<CPLX>(v, s, g[2 * s], CPLX ? g[2 * s + 1] : 0.0);
  }
}

// acc = x (first chunk) or acc + x
template <bool CPLX>
__global__ void accumulate_kernel(void* accv, const void* xv, int64_t pa, int first) {
  using DT = typename D<CPLX>::T;
  DT* acc = reinterpret_cast<DT*>(accv);
  const DT* x = reinterpret_cast<const DT*>(xv);
  for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < pa;
       e += (int64_t)gridDim.x * blockDim.x) {
    if (first) {
      acc[e] = x[e];
    } else if constexpr (CPLX) {
      acc[e] = make_double2(acc[e].x + x[e].x, acc[e].y + x[e].y);
    } else {
      acc[e] += x[e];
    }
  }
}

template <bool CPLX>
static nk_status backward_t(const nk_rbm* r, const int8_t* sigma, int64_t ns, const double* g,
                            double* grad, int prec, char* sc, cudaStream_t st) {
  const int64_t chunk = backward_chunk(ns);
  SrLayout L(r->n, r->m, CPLX, chunk);
  const size_t f = CPLX ? 8 : 4;
  char* T = sc + L.total;
  char* acc = T + round_up(chunk * r->m * f, 256);
  const bool tc = prec == NK_PREC_BF16X2;
  const int splits = sr_choose_splits(L, prec, r->sr_splits);
  const int64_t corner = (int64_t)r->m * L.na + r->n;
  const int64_t nchunks = (ns + chunk - 1) / chunk;
  for (int64_t k = 0; k < nchunks; ++k) {
    const int64_t c0 = k * chunk, cn = std::min<int64_t>(chunk, ns - c0);
    const int8_t* sg = sigma + c0 * r->n;
    const int sp = (int)std::max<int64_t>(1, std::min<int64_t>(splits, (cn + 63) / 64));
    nk_status e = tc ? launch_logpsi_bf16(r, sg, cn, nullptr, nullptr, st, T)
                     : launch_logpsi_fp32(r, sg, cn, nullptr, nullptr, st, T);
    if (e) return e;
    const int64_t blocks = std::max<int64_t>(1, std::min<int64_t>((cn + 255) / 256, 1024));
    copy_g_kernel<CPLX><<<(unsigned)blocks, 256, 0, st>>>(g + 2 * c0, sc + L.v, cn);
    if (tc) {
      if ((e = launch_sigma_t(sg, cn, r->n, L.na64, sc + L.sigt, st))) return e;
      AdjTcArgs aa{};
      aa.T = T;
      aa.v = sc + L.v;
      aa.ns = cn;
      aa.n = r->n;
      aa.m = r->m;
      aa.cplx = CPLX;
      aa.na64 = L.na64;
      aa.splits = sp;
      aa.part = sc + L.part;
      if ((e = launch_adj_tc(aa, sc + L.sigt, st))) return e;
    } else {
      launch_adjoint_fp32<CPLX>(sg, T, sc + L.v, cn, r->n, r->m, sp, sc + L.part, nullptr, st);
    }
    reduce_parts_kernel<CPLX><<<sr_vec_blocks(L.pa), kVecThreads, 0, st>>>(
        sc + L.part, sp, L.pa, corner, sc + L.x, nullptr, 0.0, nullptr, nullptr);
    if (nchunks > 1)
      accumulate_kernel<CPLX><<<sr_vec_blocks(L.pa), kVecThreads, 0, st>>>(acc, sc + L.x, L.pa,
                                                                           k == 0 ? 1 : 0);
  }
  scatter_grad_kernel<CPLX><<<sr_vec_blocks(L.pa), kVecThreads, 0, st>>>(
      nchunks > 1 ? acc : sc + L.x, r->n, r->m, grad);
  return check_launch("nk_rbm_logpsi_backward");
}

nk_status run_backward(const nk_rbm* r, const int8_t* sigma, int64_t ns, const double* g,
                       double* grad, int prec, void* scratch, size_t scratch_bytes,
                       cudaStream_t st) {
  size_t need = backward_scratch_bytes(r->n, r->m, r->is_complex, ns);
  if (scratch_bytes < need)
    return fail(NK_ERR_SHAPE, "nk_rbm_logpsi_backward: scratch of %zu B, need %zu B",
                scratch_bytes, need);
  return r->is_complex ? backward_t<true>(r, sigma, ns, g, grad, prec, (char*)scratch, st)
                       : backward_t<false>(r, sigma, ns, g, grad, prec, (char*)scratch, st);
}

NK_STATUS_COLLECTOR(collect_status_sr)

}  // namespace nk
