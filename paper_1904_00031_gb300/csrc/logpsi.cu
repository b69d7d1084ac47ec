// K1 (FP32 path): ln psi(sigma) = a . sigma + sum_j ln cosh(theta_j),
// theta = W sigma + b (Sec. 2.2.2: RbmSpin; an RBM is a one-layer FFNN with
// ln cosh activation).  theta is computed as the augmented contraction
// [W | b] [sigma; 1] on the CUDA cores (16-site chunks summed in FP32 and
// carried with TwoSum: theta to about one FP32 rounding), ln cosh is fused into
// the epilogue and summed per sample in FP64; a . sigma is added in FP64 from
// the master a.
// Without a ln psi output the epilogue only stores theta and / or tanh(theta)
// (the local energies need theta; the backward recomputes tanh(theta) per
// chunk of samples).
#include "common.cuh"
#include "fgemm.cuh"
#include "internal.h"

namespace nk {

constexpr int kLpTR = 4;            // rows per thread: 64 samples per CTA
constexpr int kLpBS = 16 * kLpTR;

template <bool CPLX>
struct LogpsiArgs {
  using F = typename std::conditional<CPLX, float2, float>::type;
  const int8_t* sigma;
  int64_t ns;
  int n, m;
  const F* xw;        // [m][n + 1] W | b
  const double* a;    // master a (F64)
  double* logpsi;     // c128 [ns], or null: theta / tanh(theta) only, no ln cosh
  F* theta_out;       // [ns][m] or null
  F* t_out;           // [ns][m] tanh(theta) or null
  int segs;           // CTAs per sample tile, each with its share of the hidden tiles
};

// s + e += x exactly (Knuth's TwoSum in FP32, two values at a time)
__device__ __forceinline__ void two_sum2(float2& s, float2& e, float2 x) {
  const float2 m1 = make_float2(-1.f, -1.f);
  const float2 t = __fadd2_rn(s, x);
  const float2 bp = fg_fma(s, m1, t);
  const float2 u = fg_fma(fg_fma(bp, m1, t), m1, s);
  e = __fadd2_rn(e, __fadd2_rn(u, fg_fma(bp, m1, x)));
  s = t;
}

// CTAs per sample tile of a call of `tiles`: theta and tanh(theta) are independent by
// hidden tile, which are dealt out while CTAs are fewer than two per SM (complex 100 x
// 400, 300 samples: 125 us with one, 23 here; 50 x 100, 8192 samples 26.8 and 19.8).
static int logpsi_segs(const double* logpsi, int m, int64_t tiles) {
  return logpsi ? 1 : (int)std::max<int64_t>(1, std::min<int64_t>(ceil_div(m, 64), 2 * 152 / tiles));
}

// One CTA: 64 samples, all hidden units (or the segment's) in tiles of 64.
// Every 16-site chunk is summed in a fresh accumulator and carried with TwoSum, so
// that theta is accurate to about one FP32 rounding instead of growing with the
// number of sites; the units of a row are folded four at a time (x + 16 q of a tile)
// in FP32, then in FP64.  At 10x10 real (16,383 samples, m = 400) theta
// takes 79 us (scalar 4 x 4 blocks: 118; 128-unit tiles, whose sums did not fit the
// registers: 118).
// (SEGS = false: one CTA per sample tile; as a run-time count it cost complex calls 3 %.)
template <bool CPLX, bool SEGS>
__device__ __forceinline__ void logpsi_fp32_body(const LogpsiArgs<CPLX>& A, int bx) {
  using F = typename LogpsiArgs<CPLX>::F;
  using L = Tile<CPLX ? kMulRealA : kMulReal, kLpTR, true, 16, 64>;
  __shared__ __align__(16) unsigned char smem[L::STAGE_BYTES];
  const int segs = SEGS ? A.segs : 1;
  const int64_t s0 = (int64_t)(bx / segs) * kLpBS;
  const int n = A.n, m = A.m, K = n + 1;
  const int jt = (m + L::BC - 1) / L::BC, seg = bx % segs;  // hidden tiles, this CTA's share
  const int jt0 = jt * seg / segs, jt1 = jt * (seg + 1) / segs;
  __shared__ double2 psum[kLpTR][kFThreads];  // each thread's own sums, out of registers
#pragma unroll
  for (int p = 0; p < kLpTR; ++p) psum[p][threadIdx.x] = make_double2(0.0, 0.0);
  Operand<int8_t, false, L::BR, L::NA, false, false, true, false, 16> oa;
  Operand<F, false, L::BC, L::NB, false, false, false, true, 16> ob;
  oa.init(A.sigma, n, s0, A.ns, 0, K);
  ob.init(A.xw, K, jt0 * L::BC, m, 0, K);
  L acc;
  float2 sx[L::TP][L::TC], ex[L::TP][L::TC];
  float2 sy[CPLX ? L::TP : 1][L::TC], ey[CPLX ? L::TP : 1][L::TC];
  auto clear = [&]() {
    const float2 z = make_float2(0.f, 0.f);
#pragma unroll
    for (int p = 0; p < L::TP; ++p)
#pragma unroll
      for (int q = 0; q < L::TC; ++q) {
        sx[p][q] = ex[p][q] = z;
        if constexpr (CPLX) sy[p][q] = ey[p][q] = z;
      }
  };
  clear();
  acc.zero();
  acc.bounds(A.ns - s0, m);
  const int nk = (K + 15) / 16;  // chunks per tile of hidden units
  int kc = 0, j0 = jt0 * L::BC;
  acc.template run<1>(smem, nk * (jt1 - jt0), oa, ob, [&](int) {
#pragma unroll
    for (int p = 0; p < L::TP; ++p)
#pragma unroll
      for (int q = 0; q < L::TC; ++q) {
        two_sum2(sx[p][q], ex[p][q], acc.x[p][q]);
        if constexpr (CPLX) two_sum2(sy[p][q], ey[p][q], acc.y[p][q]);
      }
    acc.zero();
    if (++kc < nk) return;
#pragma unroll
    for (int r = 0; r < kLpTR; ++r) {
      const int64_t s = s0 + L::lr() + r;
      if (s >= A.ns) continue;
#pragma unroll
      for (int g = 0; g < L::TC / 4; ++g) {
        float lr = 0.f, li = 0.f;
#pragma unroll
        for (int qq = 0; qq < 4; ++qq) {
          const int q = 4 * g + qq, j = j0 + L::col(q);
          if (j >= m) continue;
          const float2 x2 = __fadd2_rn(sx[r / 2][q], ex[r / 2][q]);
          const float x = (r & 1) ? x2.y : x2.x;
          if constexpr (CPLX) {
            const float2 y2 = __fadd2_rn(sy[r / 2][q], ey[r / 2][q]);
            const float y = (r & 1) ? y2.y : y2.x;
            if (A.logpsi) {
              cf l = lncosh_c(cf{x, y});
              lr += l.x;
              li += l.y;
            }
            if (A.theta_out) A.theta_out[s * m + j] = make_float2(x, y);
            if (A.t_out) {
              cf t = tanh_c(cf{x, y});
              A.t_out[s * m + j] = make_float2(t.x, t.y);
            }
          } else {
            if (A.logpsi) lr += lncosh_f(x);
            if (A.theta_out) A.theta_out[s * m + j] = x;
            if (A.t_out) A.t_out[s * m + j] = tanh_f(x);
          }
        }
        if (A.logpsi) {
          psum[r][threadIdx.x].x += (double)lr;
          psum[r][threadIdx.x].y += (double)li;
        }
      }
    }
    clear();
    kc = 0;
    j0 += L::BC;
  });
  if (!A.logpsi) return;
  // a . sigma of the row's sites x, x + 16, ..., then the sum over the 16 lanes
  const int x = threadIdx.x & 15;
#pragma unroll
  for (int r = 0; r < kLpTR; ++r) {
    const int64_t s = s0 + L::lr() + r;
    double2 part = psum[r][threadIdx.x];
    if (s < A.ns) {
      const int8_t* sg = A.sigma + s * n;
      for (int i = x; i < n; i += 16) {
        const double si = (double)sg[i];
        part.x += (CPLX ? A.a[2 * i] : A.a[i]) * si;
        if (CPLX) part.y += A.a[2 * i + 1] * si;
      }
    }
#pragma unroll
    for (int off = 8; off >= 1; off >>= 1) {
      part.x += __shfl_xor_sync(0xffffffffu, part.x, off);
      part.y += __shfl_xor_sync(0xffffffffu, part.y, off);
    }
    if (x == 0 && s < A.ns) {
      A.logpsi[2 * s] = part.x;
      A.logpsi[2 * s + 1] = part.y;
    }
  }
}

template <bool CPLX, bool SEGS>
__global__ void __launch_bounds__(kFThreads, 2) logpsi_fp32_kernel(LogpsiArgs<CPLX> A) {
  logpsi_fp32_body<CPLX, SEGS>(A, blockIdx.x);
}

// Up to kLogpsiBatch problems of one field in one launch: CTA b runs sample
// tile b - start[k] of problem k, as that problem's own launch would.
constexpr int kLogpsiBatch = 64;
template <bool CPLX>
struct LogpsiFp32Batch {
  int n;
  int start[kLogpsiBatch + 1];
  LogpsiArgs<CPLX> j[kLogpsiBatch];
};

template <bool CPLX, bool SEGS>
__global__ void __launch_bounds__(kFThreads, 2)
    logpsi_fp32_batch(const __grid_constant__ LogpsiFp32Batch<CPLX> B) {
  int k = 0;
  while (k + 1 < B.n && (int)blockIdx.x >= B.start[k + 1]) ++k;
  logpsi_fp32_body<CPLX, SEGS>(B.j[k], (int)blockIdx.x - B.start[k]);
}

template <bool CPLX>
static LogpsiArgs<CPLX> logpsi_args(const nk_rbm* r, const int8_t* sigma, int64_t ns,
                                    double* logpsi, void* theta_out, void* t_out, int segs) {
  using F = typename LogpsiArgs<CPLX>::F;
  WsLayout L(r->n, r->m, r->is_complex);
  return LogpsiArgs<CPLX>{sigma, ns, r->n, r->m, (const F*)((const char*)r->ws + L.xw), r->a,
                          logpsi, (F*)theta_out, (F*)t_out, segs};
}

// the problems of one field, at most kLogpsiBatch to a launch
template <bool CPLX>
static nk_status logpsi_fp32_field(const nk_logpsi_item* items, const int* idx, int n,
                                   cudaStream_t st) {
  int64_t tiles = 0;
  for (int u = 0; u < n; ++u)
    if ((items[idx[u]].rbm->is_complex != 0) == CPLX)
      tiles += (items[idx[u]].ns + kLpBS - 1) / kLpBS;
  for (int u0 = 0; u0 < n;) {
    LogpsiFp32Batch<CPLX> B;
    B.n = 0;
    B.start[0] = 0;
    bool split = false;
    int u = u0;
    for (; u < n && B.n < kLogpsiBatch; ++u) {
      const nk_logpsi_item& it = items[idx[u]];
      if ((it.rbm->is_complex != 0) != CPLX) continue;
      const int64_t t = (it.ns + kLpBS - 1) / kLpBS;
      const int segs = logpsi_segs(it.logpsi_out, it.rbm->m, tiles);
      split = split || segs > 1;
      B.j[B.n] = logpsi_args<CPLX>(it.rbm, it.sigma, it.ns, it.logpsi_out, it.theta_out, nullptr, segs);
      B.start[B.n + 1] = B.start[B.n] + (int)(t * segs);
      ++B.n;
    }
    u0 = u;
    if (B.n == 0) continue;
    auto kern = split ? logpsi_fp32_batch<CPLX, true> : logpsi_fp32_batch<CPLX, false>;
    kern<<<B.start[B.n], kFThreads, 0, st>>>(B);
    if (nk_status e = check_launch("nk_batch_logpsi")) return e;
  }
  return NK_OK;
}

nk_status launch_logpsi_fp32_fused(const nk_logpsi_item* items, const int* idx, int n,
                                   cudaStream_t st) {
  if (nk_status e = logpsi_fp32_field<false>(items, idx, n, st)) return e;
  return logpsi_fp32_field<true>(items, idx, n, st);
}

nk_status launch_logpsi_fp32(const nk_rbm* r, const int8_t* sigma, int64_t ns, double* logpsi,
                             void* theta_out, cudaStream_t st, void* t_out) {
  const int64_t tiles = (ns + kLpBS - 1) / kLpBS;
  const int segs = logpsi_segs(logpsi, r->m, tiles);
  const unsigned blocks = (unsigned)(tiles * segs);
  if (r->is_complex) {
    auto kern = segs > 1 ? logpsi_fp32_kernel<true, true> : logpsi_fp32_kernel<true, false>;
    kern<<<blocks, kFThreads, 0, st>>>(logpsi_args<true>(r, sigma, ns, logpsi, theta_out, t_out, segs));
  } else {
    auto kern = segs > 1 ? logpsi_fp32_kernel<false, true> : logpsi_fp32_kernel<false, false>;
    kern<<<blocks, kFThreads, 0, st>>>(logpsi_args<false>(r, sigma, ns, logpsi, theta_out, t_out, segs));
  }
  return check_launch("nk_rbm_logpsi");
}

}  // namespace nk
