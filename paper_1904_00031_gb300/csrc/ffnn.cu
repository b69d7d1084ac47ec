// Multi-layer feed-forward network with ln cosh activations (Sec. 2.2.2: FFNN
// machines of dense layers y = W x + b and Lncosh activations with a sum
// output; the one-layer network is the RBM without visible bias):
//   x_0 = sigma,  h_l = W_l x_(l-1) + b_l,  x_l = ln cosh(h_l),  ln psi = sum_j x_(L, j),
// and its backward grad_k = sum_s conj(O_sk) g_s (the convention of the RBM
// backward) by the holomorphic chain rule:
//   e_L = conj(tanh h_L) g,  e_(l-1) = conj(tanh h_(l-1)) (e_l conj(W_l)),
//   grad W_l = e_l^T conj(x_(l-1)),  grad b_l = sum_s e_l.
// Every contraction runs on the CUDA cores in FP32 (128- or 64-row output tiles,
// packed pair instructions) on an FP32 copy of the master parameters made once per
// call; ln psi and the gradients are summed in FP64 (the weight gradients over
// sample splits in a fixed order).  The backward recomputes the forward into its
// scratch, so it needs nothing from an earlier call.
#include "common.cuh"
#include "fgemm.cuh"
#include "internal.h"

namespace nk {

namespace {

constexpr int kFSplitStep = 16;  // granularity of the weight gradients' sample splits
constexpr int kFMaxLayers = 8;

template <bool CPLX>
struct FT;
template <>
struct FT<true> {
  using F = float2;
  static __device__ __forceinline__ float2 zero() { return make_float2(0.f, 0.f); }
};
template <>
struct FT<false> {
  using F = float;
  static __device__ __forceinline__ float zero() { return 0.f; }
};

__device__ __forceinline__ float2 cconj(float2 a) { return make_float2(a.x, -a.y); }
__device__ __forceinline__ float cconj(float a) { return a; }
__device__ __forceinline__ float2 cmul(float2 a, float2 b) {
  return make_float2(fmaf(a.x, b.x, -a.y * b.y), fmaf(a.x, b.y, a.y * b.x));
}
__device__ __forceinline__ float cmul(float a, float b) { return a * b; }

template <bool CPLX>
__device__ __forceinline__ typename FT<CPLX>::F lncosh_t(typename FT<CPLX>::F h) {
  if constexpr (CPLX) {
    cf l = lncosh_c(cf{h.x, h.y});
    return make_float2(l.x, l.y);
  } else {
    return lncosh_f(h);
  }
}

template <bool CPLX>
__device__ __forceinline__ typename FT<CPLX>::F tanh_t(typename FT<CPLX>::F h) {
  if constexpr (CPLX) {
    cf t = tanh_c(cf{h.x, h.y});
    return make_float2(t.x, t.y);
  } else {
    return tanh_f(h);
  }
}

// The tiles of 16 TR rows.  Real ones of 64 rows have 64 columns (4 x 4 elements per
// thread) in chunks of 16, two operand sets ahead: they run where CTAs are few, and a
// CTA that has its SM to itself takes twice as long for twice the columns.
template <int MUL, int TR>
struct FTileOf {
  using T = Tile<MUL, TR>;
};
template <>
struct FTileOf<kMulReal, 4> {
  using T = Tile<kMulReal, 4, false, 16, 64>;
};
template <int MUL, int TR>
using FTile = typename FTileOf<MUL, TR>::T;

// C[r][c] = sum_{k in [kb, ke)} A(r, k) B(c, k) for one tile (fgemm.cuh); epi(r, c,
// acc) receives every element of the tile that lies inside R x C.
// Measured at [400, 1600, 400] complex, 16,384 samples, forward + backward: 18.2 ms
// with scalar operands staged per 64 x 64 tile, 13.0 with packed instructions on
// operands staged ready-made (192 bytes per 64 instructions: shared-memory bound,
// FMA pipe 57 %), 9.6 as here (6.7 at the measured FMA rate).
template <int MUL, int TR>
struct GemmSmem {
  using L = FTile<MUL, TR>;
  static constexpr int PT = L::CPLX ? L::BC + 8 : L::BC + 16;  // row pitch of the result tile
  static constexpr size_t bytes() {
    const size_t tile = (size_t)L::BR * PT * (L::CPLX ? 8 : 4);
    return L::STAGE_BYTES > tile ? L::STAGE_BYTES : tile;
  }
};

template <int MUL, int TR, class OA, class OB, class Epi>
__device__ __forceinline__ void gemm_tile(int64_t R, int64_t C, int64_t kb, int64_t ke,
                                          int64_t r0, int64_t c0, OA& oa, OB& ob,
                                          const Epi& epi) {
  using L = FTile<MUL, TR>;
  constexpr bool CPLX = L::CPLX;
  constexpr int PT = GemmSmem<MUL, TR>::PT;
  extern __shared__ __align__(16) unsigned char smraw[];
  L acc;
  acc.zero();
  acc.bounds(R - r0, C - c0);
  acc.template run<L::kFK == 16 ? 2 : 1>(smraw, (int)((ke - kb + L::kFK - 1) / L::kFK), oa, ob, [](int) {});
  // The tile goes through shared memory so that the epilogue is a rolled loop (its
  // transcendentals, inlined once per element of the register tile, would not fit
  // the instruction cache) over whole row segments.
  using F = typename FT<CPLX>::F;
  F* tile = reinterpret_cast<F*>(smraw);
#pragma unroll
  for (int p = 0; p < L::TP; ++p)
#pragma unroll
    for (int q = 0; q < L::TC; ++q) {
      F* d = tile + L::row(p) * PT + L::col(q);
      if constexpr (CPLX) {
        d[0] = make_float2(acc.x[p][q].x, acc.y[p][q].x);
        d[PT] = make_float2(acc.x[p][q].y, acc.y[p][q].y);
      } else {
        d[0] = acc.x[p][q].x;
        d[PT] = acc.x[p][q].y;
      }
    }
  __syncthreads();
  const int c = threadIdx.x % L::BC;
  if (c0 + c < C) {
#pragma unroll 1
    for (int r = threadIdx.x / L::BC; r < L::BR && r0 + r < R; r += kFThreads / L::BC)
      epi(r0 + r, c0 + c, tile[r * PT + c]);
  }
}

// The FP32 copy of the flat FP64 parameters (scalars) that the contractions read:
// converted once per call, because the conversions share the slow FP64 pipe (one
// per staged element would cost as much as the products).
__global__ void ffnn_params_kernel(const double* __restrict__ p, int64_t cnt, float* out) {
  for (int64_t x = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; x < cnt;
       x += (int64_t)gridDim.x * blockDim.x)
    out[x] = (float)p[x];
}

// ---------------------------------------------------------------- forward

// h_l = x_(l-1) W_l^T + b_l for a tile of samples x outputs.  Layer 1 reads
// sigma (int8).  Stores h_l and x_l = ln cosh(h_l) (either may be null), or,
// given an upstream vector g, only e_l = conj(tanh h_l) g (the backward's top).
template <bool CPLX, bool FIRST, int TR>
__global__ void __launch_bounds__(kFThreads, TR == 8 ? 2 : 3) ffnn_fwd_kernel(const int8_t* __restrict__ sigma,
                                                                const void* __restrict__ xin,
                                                                int64_t ns, int win, int wout,
                                                                const float* __restrict__ Wv,
                                                                const float* __restrict__ bv,
                                                                void* hout, void* xout,
                                                                const double* __restrict__ g,
                                                                void* eout) {
  using F = typename FT<CPLX>::F;
  constexpr int MUL = CPLX ? (FIRST ? kMulRealA : kMulFull) : kMulReal;
  const F* X = reinterpret_cast<const F*>(xin);
  const F* Wm = reinterpret_cast<const F*>(Wv);
  const F* bm = reinterpret_cast<const F*>(bv);
  F* H = reinterpret_cast<F*>(hout);
  F* Y = reinterpret_cast<F*>(xout);
  F* E = reinterpret_cast<F*>(eout);
  auto epi = [&](int64_t s, int64_t j, F acc) {
    const F b = bm[j];
    F h;
    if constexpr (CPLX) h = make_float2(acc.x + b.x, acc.y + b.y); else h = acc + b;
    if (E) {
      const F t = cconj(tanh_t<CPLX>(h));
      if constexpr (CPLX)
        E[s * wout + j] = cmul(t, make_float2((float)g[2 * s], (float)g[2 * s + 1]));
      else
        E[s * wout + j] = t * (float)g[2 * s];
      return;
    }
    if (H) H[s * wout + j] = h;
    Y[s * wout + j] = lncosh_t<CPLX>(h);
  };
  using L = FTile<MUL, TR>;
  const int64_t r0 = (int64_t)blockIdx.y * L::BR, c0 = (int64_t)blockIdx.x * L::BC;
  Operand<F, false, L::BC, L::NB, false, false, false, false, L::kFK> ob;
  ob.init(Wm, win, c0, wout, 0, win);
  if constexpr (FIRST) {
    Operand<int8_t, false, L::BR, L::NA, false, false, false, false, L::kFK> oa;
    oa.init(sigma, win, r0, ns, 0, win);
    gemm_tile<MUL, TR>(ns, wout, 0, win, r0, c0, oa, ob, epi);
  } else {
    Operand<F, false, L::BR, L::NA, false, false, false, false, L::kFK> oa;
    oa.init(X, win, r0, ns, 0, win);
    gemm_tile<MUL, TR>(ns, wout, 0, win, r0, c0, oa, ob, epi);
  }
}

// ln psi_s = sum_j x_(L, s, j), FP64, one warp per sample (fixed order)
template <bool CPLX>
__global__ void ffnn_rowsum_kernel(const void* __restrict__ xl, int64_t ns, int w,
                                   double* __restrict__ logpsi) {
  using F = typename FT<CPLX>::F;
  const F* X = reinterpret_cast<const F*>(xl);
  const int lane = threadIdx.x & 31;
  const int64_t s = (int64_t)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
  if (s >= ns) return;
  double r = 0.0, i = 0.0;
  for (int j = lane; j < w; j += 32) {
    const F v = X[s * w + j];
    if constexpr (CPLX) {
      r += (double)v.x;
      i += (double)v.y;
    } else {
      r += (double)v;
    }
  }
#pragma unroll
  for (int off = 16; off >= 1; off >>= 1) {
    r += __shfl_xor_sync(0xffffffffu, r, off);
    i += __shfl_xor_sync(0xffffffffu, i, off);
  }
  if (lane == 0) {
    logpsi[2 * s] = r;
    logpsi[2 * s + 1] = i;
  }
}

// ---------------------------------------------------------------- backward

// e_(l-1)[s][i] = conj(tanh h_(l-1)[s][i]) sum_j e_l[s][j] conj(W_l[j][i])
template <bool CPLX, int TR>
__global__ void __launch_bounds__(kFThreads, TR == 8 ? 2 : 3) ffnn_bwd_kernel(const void* __restrict__ ein,
                                                                const void* __restrict__ hprev,
                                                                int64_t ns, int wl, int wprev,
                                                                const float* __restrict__ Wv,
                                                                void* eout) {
  using F = typename FT<CPLX>::F;
  const F* E = reinterpret_cast<const F*>(ein);
  const F* H = reinterpret_cast<const F*>(hprev);
  const F* Wm = reinterpret_cast<const F*>(Wv);
  F* Eo = reinterpret_cast<F*>(eout);
  auto epi = [&](int64_t s, int64_t i, F acc) {
    Eo[s * wprev + i] = cmul(cconj(tanh_t<CPLX>(H[s * wprev + i])), acc);
  };
  constexpr int MUL = CPLX ? kMulFull : kMulReal;
  using L = FTile<MUL, TR>;
  const int64_t r0 = (int64_t)blockIdx.y * L::BR, c0 = (int64_t)blockIdx.x * L::BC;
  Operand<F, false, L::BR, L::NA, false, false, false, false, L::kFK> oa;
  Operand<F, true, L::BC, L::NB, true, false, false, false, L::kFK> ob;
  oa.init(E, wl, r0, ns, 0, wl);
  ob.init(Wm, wprev, c0, wprev, 0, wl);
  gemm_tile<MUL, TR>(ns, wprev, 0, wl, r0, c0, oa, ob, epi);
}

// Where this layer's gradient (W then b, flat) holds element (j, i); i = wprev: b_j.
__device__ __forceinline__ int64_t grad_index(int64_t j, int64_t i, int wl, int wprev) {
  return i < wprev ? j * wprev + i : (int64_t)wl * wprev + j;
}

// partial[z][j][i] = sum_{s in split z} e_l[s][j] conj(x'_(l-1)[s][i]),
// x' = [x | 1] (i = wprev is the bias column); layer 1 reads sigma.  Given grad (one
// split), the gradient itself, as the reduction would write it: small calls are bound by
// their launches.
template <bool CPLX, bool FIRST, int TR>
__global__ void __launch_bounds__(kFThreads, TR == 8 ? 2 : 3) ffnn_wgrad_kernel(const void* __restrict__ ein,
                                                                  const int8_t* __restrict__ sigma,
                                                                  const void* __restrict__ xprev,
                                                                  int64_t ns, int wl, int wprev,
                                                                  int64_t chunk, void* partv,
                                                                  double* grad) {
  using F = typename FT<CPLX>::F;
  constexpr int MUL = CPLX ? (FIRST ? kMulRealB : kMulFull) : kMulReal;
  const F* E = reinterpret_cast<const F*>(ein);
  const F* X = reinterpret_cast<const F*>(xprev);
  F* part = reinterpret_cast<F*>(partv) + (int64_t)blockIdx.z * wl * (wprev + 1);
  auto epi = [&](int64_t j, int64_t i, F acc) {
    if (!grad) {
      part[j * (wprev + 1) + i] = acc;
      return;
    }
    const int64_t k = grad_index(j, i, wl, wprev);
    if constexpr (CPLX) {
      grad[2 * k] = 0.0 + (double)acc.x;
      grad[2 * k + 1] = 0.0 + (double)acc.y;
    } else {
      grad[k] = 0.0 + (double)acc;
    }
  };
  const int64_t kb = (int64_t)blockIdx.z * chunk, ke = std::min<int64_t>(ns, kb + chunk);
  using L = FTile<MUL, TR>;
  const int64_t r0 = (int64_t)blockIdx.y * L::BR, c0 = (int64_t)blockIdx.x * L::BC;
  Operand<F, true, L::BR, L::NA, false, false, false, false, L::kFK> oa;
  oa.init(E, wl, r0, wl, kb, ke);
  if constexpr (FIRST) {
    Operand<int8_t, true, L::BC, L::NB, false, true, false, false, L::kFK> ob;
    ob.init(sigma, wprev, c0, wprev + 1, kb, ke);
    gemm_tile<MUL, TR>(wl, wprev + 1, kb, ke, r0, c0, oa, ob, epi);
  } else {
    Operand<F, true, L::BC, L::NB, true, true, false, false, L::kFK> ob;
    ob.init(X, wprev, c0, wprev + 1, kb, ke);
    gemm_tile<MUL, TR>(wl, wprev + 1, kb, ke, r0, c0, oa, ob, epi);
  }
}

// grad (this layer's W then b, flat, FP64) = fixed-order sum over the splits
template <bool CPLX>
__global__ void ffnn_wreduce_kernel(const void* __restrict__ partv, int splits, int wl, int wprev,
                                    double* __restrict__ grad) {
  using F = typename FT<CPLX>::F;
  const F* part = reinterpret_cast<const F*>(partv);
  const int64_t per = (int64_t)wl * (wprev + 1);
  for (int64_t x = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; x < per;
       x += (int64_t)gridDim.x * blockDim.x) {
    double r = 0.0, im = 0.0;
    for (int z = 0; z < splits; ++z) {
      const F v = part[z * per + x];
      if constexpr (CPLX) {
        r += (double)v.x;
        im += (double)v.y;
      } else {
        r += (double)v;
      }
    }
    const int64_t j = x / (wprev + 1), i = x % (wprev + 1);
    const int64_t k = grad_index(j, i, wl, wprev);
    if constexpr (CPLX) {
      grad[2 * k] = r;
      grad[2 * k + 1] = im;
    } else {
      grad[k] = r;
    }
  }
}

struct FfnnLayout {
  int L, cplx;
  int w[kFMaxLayers + 1];
  int64_t ns;
  int splits;
  size_t h[kFMaxLayers], x[kFMaxLayers], e0, e1, part, p32, total;
  int64_t n_params;
  int64_t off[kFMaxLayers];  // flat parameter offset of each layer (in parameters)
  int64_t chunk;
  FfnnLayout(const nk_ffnn* f, int64_t ns_) {
    L = f->n_layers;
    cplx = f->is_complex ? 1 : 0;
    ns = std::max<int64_t>(ns_, 1);
    for (int l = 0; l <= L; ++l) w[l] = f->widths[l];
    const size_t fs = cplx ? 8 : 4;
    auto up = [](size_t b) { return (b + 255) / 256 * 256; };
    size_t o = 0;
    int wmax = 0;
    int64_t pmax = 0, po = 0;
    for (int l = 1; l <= L; ++l) {
      h[l - 1] = o;
      o += up((size_t)ns * w[l] * fs);
      x[l - 1] = o;
      o += up((size_t)ns * w[l] * fs);
      wmax = std::max(wmax, w[l]);
      pmax = std::max<int64_t>(pmax, (int64_t)w[l] * (w[l - 1] + 1));
      off[l - 1] = po;
      po += (int64_t)w[l] * (w[l - 1] + 1);
    }
    splits = (int)std::min<int64_t>(16, std::max<int64_t>(1, ns / 1024));
    chunk = ((ns + splits - 1) / splits + kFSplitStep - 1) / kFSplitStep * kFSplitStep;
    e0 = o;
    o += up((size_t)ns * wmax * fs);
    e1 = o;
    o += up((size_t)ns * wmax * fs);
    part = o;
    o += up((size_t)splits * pmax * fs);
    n_params = po;
    p32 = o;
    o += up((size_t)po * fs);
    total = o;
  }
};

// Rows per thread of a contraction: 8 (128 rows) where its tiles fill every SM's two CTAs
// and do not pad the rows much more than 64-row tiles would, else 4.  Real, forward +
// backward: [400, 1600, 400], 16,384 samples 4.45 ms, 64 x 128 tiles everywhere 4.95; on
// 64 x 64 tiles [400, 800, 800, 400], 500 samples 355 us, 64 x 128 792.  Complex with the
// sample operand real (a first layer's forward): [400, 800], 16,384 samples 585 us, 64
// rows 691.  The other complex contractions keep 64 rows, three CTAs to an SM, as far as a
// grid's y goes: [400, 400, 400, 400], 6000 samples, backward 1526 us, 128 rows where they
// fill 1764; [400, 800], 16,384 samples, backward 1074 and 1218.
template <int MUL>
int tile_rows(int64_t rows, int64_t cols, int z) {
  constexpr int BC = FTile<MUL, 8>::BC;
  const int64_t t8 = (rows + 127) / 128, t4 = (rows + 63) / 64, ct = (cols + BC - 1) / BC;
  if (MUL == kMulFull || MUL == kMulRealB) return t4 > 65535 ? 8 : 4;
  return t8 * ct * z >= 2 * 152 && 8 * t8 * 128 <= 9 * t4 * 64 ? 8 : 4;
}

// Launches kern8 or kern4 (the two tiles of one contraction) over rows x cols x z.
template <int MUL, class K8, class K4, class... Args>
nk_status gemm_launch(K8 kern8, K4 kern4, int64_t rows, int64_t cols, int z, cudaStream_t st,
                      Args... args) {
  using L8 = FTile<MUL, 8>;
  using L4 = FTile<MUL, 4>;
  auto go = [&](auto kern, int br, int bc, size_t smem) -> nk_status {
    const dim3 grid((unsigned)((cols + bc - 1) / bc), (unsigned)((rows + br - 1) / br), (unsigned)z);
    if (smem > 48 * 1024 && cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                                 (int)smem) != cudaSuccess)
      return fail(NK_ERR_CUDA, "nk_ffnn: shared memory attribute");
    kern<<<grid, kFThreads, smem, st>>>(args...);
    return NK_OK;
  };
  return tile_rows<MUL>(rows, cols, z) == 8
             ? go(kern8, L8::BR, L8::BC, GemmSmem<MUL, 8>::bytes())
             : go(kern4, L4::BR, L4::BC, GemmSmem<MUL, 4>::bytes());
}

// The forward through all layers.  keep_h: h_l is stored for the backward, and
// the last layer stores e_L = conj(tanh h_L) g into etop instead of x_L.
template <bool CPLX>
nk_status forward_t(const nk_ffnn* f, const FfnnLayout& Lo, const int8_t* sigma, int64_t ns,
                    double* logpsi, char* sc, cudaStream_t st, const double* g = nullptr,
                    char* etop = nullptr) {
  const int64_t fs = CPLX ? 2 : 1;  // scalars per parameter
  float* p32 = reinterpret_cast<float*>(sc + Lo.p32);
  const int64_t cnt = fs * Lo.n_params;
  ffnn_params_kernel<<<(unsigned)std::min<int64_t>(152 * 8, (cnt + 255) / 256), 256, 0, st>>>(
      f->params, cnt, p32);
  for (int l = 1; l <= Lo.L; ++l) {
    const float* Wm = p32 + fs * Lo.off[l - 1];
    const float* bm = Wm + fs * (int64_t)Lo.w[l] * Lo.w[l - 1];
    const bool top = g && l == Lo.L;
    void* h = g && !top ? sc + Lo.h[l - 1] : nullptr;
    void* x = top ? nullptr : sc + Lo.x[l - 1];
    const double* gl = top ? g : nullptr;
    void* el = top ? etop : nullptr;
    nk_status e;
    if (l == 1)
      e = gemm_launch<CPLX ? kMulRealA : kMulReal>(
          ffnn_fwd_kernel<CPLX, true, 8>, ffnn_fwd_kernel<CPLX, true, 4>, ns, Lo.w[1], 1, st, sigma,
          (const void*)nullptr, ns, Lo.w[0], Lo.w[1], Wm, bm, h, x, gl, el);
    else
      e = gemm_launch<CPLX ? kMulFull : kMulReal>(
          ffnn_fwd_kernel<CPLX, false, 8>, ffnn_fwd_kernel<CPLX, false, 4>, ns, Lo.w[l], 1, st,
          sigma, (const void*)(sc + Lo.x[l - 2]), ns, Lo.w[l - 1], Lo.w[l], Wm, bm, h, x, gl, el);
    if (e) return e;
  }
  if (logpsi)
    ffnn_rowsum_kernel<CPLX><<<(unsigned)((ns + 7) / 8), 256, 0, st>>>(sc + Lo.x[Lo.L - 1], ns,
                                                                      Lo.w[Lo.L], logpsi);
  return check_launch("nk_ffnn forward");
}

template <bool CPLX>
nk_status backward_t(const nk_ffnn* f, const FfnnLayout& Lo, const int8_t* sigma, int64_t ns,
                     const double* g, double* grad, char* sc, cudaStream_t st) {
  char* ecur = sc + Lo.e0;
  char* enext = sc + Lo.e1;
  if (nk_status e = forward_t<CPLX>(f, Lo, sigma, ns, nullptr, sc, st, g, ecur)) return e;
  const int64_t fs = CPLX ? 2 : 1;
  const float* p32 = reinterpret_cast<const float*>(sc + Lo.p32);
  for (int l = Lo.L; l >= 1; --l) {
    const float* Wm = p32 + fs * Lo.off[l - 1];
    const int wl = Lo.w[l], wp = Lo.w[l - 1];
    double* gl = grad + fs * Lo.off[l - 1];
    double* direct = Lo.splits == 1 ? gl : nullptr;
    nk_status e;
    if (l == 1)
      e = gemm_launch<CPLX ? kMulRealB : kMulReal>(
          ffnn_wgrad_kernel<CPLX, true, 8>, ffnn_wgrad_kernel<CPLX, true, 4>, wl, wp + 1, Lo.splits,
          st, (const void*)ecur, sigma, (const void*)nullptr, ns, wl, wp, Lo.chunk,
          (void*)(sc + Lo.part), direct);
    else
      e = gemm_launch<CPLX ? kMulFull : kMulReal>(
          ffnn_wgrad_kernel<CPLX, false, 8>, ffnn_wgrad_kernel<CPLX, false, 4>, wl, wp + 1,
          Lo.splits, st, (const void*)ecur, sigma, (const void*)(sc + Lo.x[l - 2]), ns, wl, wp,
          Lo.chunk, (void*)(sc + Lo.part), direct);
    if (e) return e;
    const int64_t per = (int64_t)wl * (wp + 1);
    if (!direct)
      ffnn_wreduce_kernel<CPLX><<<(unsigned)std::min<int64_t>(1024, (per + 255) / 256), 256, 0, st>>>(
          sc + Lo.part, Lo.splits, wl, wp, gl);
    if (l > 1) {
      e = gemm_launch<CPLX ? kMulFull : kMulReal>(
          ffnn_bwd_kernel<CPLX, 8>, ffnn_bwd_kernel<CPLX, 4>, ns, wp, 1, st, (const void*)ecur,
          (const void*)(sc + Lo.h[l - 2]), ns, wl, wp, Wm, (void*)enext);
      if (e) return e;
      std::swap(ecur, enext);
    }
  }
  return check_launch("nk_ffnn backward");
}

}  // namespace

nk_status check_ffnn(const nk_ffnn* f, const char* who) {
  if (!f || !f->widths || !f->params) return fail(NK_ERR_INVALID_ARG, "%s: NULL network", who);
  if (f->n_layers < 1 || f->n_layers > kFMaxLayers)
    return fail(NK_ERR_SHAPE, "%s: n_layers = %d outside [1, %d]", who, f->n_layers, kFMaxLayers);
  for (int l = 0; l <= f->n_layers; ++l)
    if (f->widths[l] < 1 || f->widths[l] > (1 << 20))
      return fail(NK_ERR_SHAPE, "%s: width %d of layer %d", who, f->widths[l], l);
  return NK_OK;
}

size_t ffnn_scratch_bytes(const nk_ffnn* f, int64_t ns) { return FfnnLayout(f, ns).total; }

nk_status run_ffnn_logpsi(const nk_ffnn* f, const int8_t* sigma, int64_t ns, double* logpsi,
                          void* scratch, size_t bytes, cudaStream_t st) {
  FfnnLayout Lo(f, ns);
  if (bytes < Lo.total)
    return fail(NK_ERR_SHAPE, "nk_ffnn_logpsi: scratch of %zu B, need %zu B", bytes, Lo.total);
  return f->is_complex ? forward_t<true>(f, Lo, sigma, ns, logpsi, (char*)scratch, st)
                       : forward_t<false>(f, Lo, sigma, ns, logpsi, (char*)scratch, st);
}

nk_status run_ffnn_backward(const nk_ffnn* f, const int8_t* sigma, int64_t ns, const double* g,
                            double* grad, void* scratch, size_t bytes, cudaStream_t st) {
  FfnnLayout Lo(f, ns);
  if (bytes < Lo.total)
    return fail(NK_ERR_SHAPE, "nk_ffnn_backward: scratch of %zu B, need %zu B", bytes, Lo.total);
  return f->is_complex ? backward_t<true>(f, Lo, sigma, ns, g, grad, (char*)scratch, st)
                       : backward_t<false>(f, Lo, sigma, ns, g, grad, (char*)scratch, st);
}

}  // namespace nk
