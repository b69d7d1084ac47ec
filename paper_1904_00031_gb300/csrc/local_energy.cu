// K3: local energies E_loc(sigma) = sum_sigma' <sigma|H|sigma'> psi(sigma')/psi(sigma)
// (Eq. 5, Sec. 2.2.5) for a Hamiltonian of 1-local and 2-local terms, and K4:
// the factored log-derivatives T = tanh(theta) (Sec. 2.2.5: O_b = tanh theta,
// O_W = tanh theta (x) sigma, O_a = sigma).
//
// Every move's psi ratio is exp(visible) * prod_j (cosh c_j - t_j sinh c_j)
// (c = 2 s_i W_i (+ 2 s_k W_k), t = tanh theta) from the cosh/sinh(2W) tables,
// with each running product kept as mantissa * 2^e; matrix elements, visible
// factors and the sums over moves are FP64.
#include "common.cuh"
#include "internal.h"
#include "opdev.h"
#include "ratio.cuh"
#include "tc.cuh"
#include "status.cuh"
#include "umma.cuh"

#include <stddef.h>
#include <string.h>

#include <memory>
#include <type_traits>

namespace nk {

struct ElocArgs {
  int n, m, mp, n_moves;
  int64_t ns;
  const int8_t* sigma;
  const void* theta;   // [ns][m] F
  const char* op;      // compiled operator
  const double* a;     // master a
  const double2* fac;  // [nm_pad][4] mel x exp(visible) per move and spin pattern (built per call)
  const void* tab;     // [n][mp] T2
  double* eloc;        // c128 [ns]
  void* t_out;         // [ns][m] F or null
  int nseg;            // 1, or 2: each configuration tile is split over two CTAs
                       // taking half of the move tiles each, whose sums are added
                       // into eloc (zeroed first) atomically
  int seg_fast;        // 1: the grid is (nseg, tiles), so the two halves of a
                       // configuration tile run back to back and share its theta /
                       // T rows in L2; 0: (tiles, nseg)
};

__device__ __forceinline__ int idx_of(int8_t s) { return s > 0 ? 0 : 1; }

// Tiled form (complex RBMs on operators without the site-quad layout): a CTA owns 64
// configurations and walks the move list in tiles of 64 moves; every thread advances a
// 4 x 4 block of running products
// prod_j (cosh c_j - s_i t_j sinh c_j / s_i) held in registers, so each staged
// value is reused by 16 threads and the kernel is bound by the FP32 pipe.  The
// (cosh c, sinh c / s_i) columns of all moves are built once per call in the
// caller's scratch as a [m][moves] table (a two-spin move has cosh c =
// A_i A_k +/- B_i B_k, sinh c / s_i = B_i A_k +/- A_i B_k from the site tables;
// the sign is fixed per move by the alignment split at compilation); 16 x 64
// tiles of it arrive by 2-D TMA into a double buffer, one chunk ahead, while
// the t = tanh(theta) tile of the next chunk is loaded into registers.
constexpr int kEBS = 64;   // configurations per CTA
constexpr int kEBM = 64;   // moves per tile
constexpr int kEBK = 16;   // hidden units per chunk
constexpr int kETS = kEBS + 1;  // padded row of the t tile (conflict-free transposed stores)

// (cosh c_j, sinh c_j / s_i) of move mv: the two-spin form from the site tables
template <bool CPLX>
__device__ __forceinline__ typename RatioTypes<CPLX>::T2 move_column(const OpMove& M,
                                                                     const void* tabv, int mp,
                                                                     int j) {
  using T2 = typename RatioTypes<CPLX>::T2;
  const T2* tab = reinterpret_cast<const T2*>(tabv);
  const T2 ai = tab[(int64_t)M.i * mp + j];
  if (!M.two) return ai;
  const T2 ak = tab[(int64_t)M.k * mp + j];
  const float al = (float)M.align;
  if constexpr (CPLX) {
    cf Ai{ai.x, ai.y}, Bi{ai.z, ai.w}, Ak{ak.x, ak.y}, Bk{ak.z, ak.w};
    cf c = Ai * Ak + al * (Bi * Bk);
    cf d = Bi * Ak + al * (Ai * Bk);
    return make_float4(c.x, c.y, d.x, d.y);
  } else {
    return make_float2(fmaf(al * ai.y, ak.y, ai.x * ak.x), fmaf(al * ai.x, ak.y, ai.y * ak.x));
  }
}

// Real RBMs: table[j][mv] = (cosh c_j, sinh c_j / s_i) of move mv.
// Complex RBMs: row j holds, per tile of 64 moves, 32 slots for move pairs
// (a, b = a + 16) with a = (s mod 16) + 32 (s div 16): first the C plane,
// slot s = (Re C_a, Re C_b, Im C_a, Im C_b), then the D plane (same for
// D = sinh c / s_i), so that one 16-byte load gives a thread the operands of
// two moves as packed FP32 pairs.
// Complex RBMs on a site-quad operator: row j holds (C, D) of the moves in order
// (eloc_wide_body).
// Element x of the table (complex: of mp * ntile * 32 slot pairs; real: of mp * nm_pad)
template <bool CPLX>
__device__ __forceinline__ void move_table_elem(int64_t x, const OpMove* __restrict__ mvs,
                                                const void* __restrict__ tabv, int mp, int nm,
                                                int nm_pad, bool quad, void* outv) {
  if constexpr (CPLX) {
    float4* out = reinterpret_cast<float4*>(outv);
    const int ntile = nm_pad / kEBM;
    const int slot = (int)(x & 31);
    const int64_t jt = x >> 5;
    const int j = (int)(jt / ntile), mt = (int)(jt % ntile);
    const int a = mt * kEBM + (slot & 15) + 32 * (slot >> 4), b = a + 16;
    const float4 za = make_float4(0.f, 0.f, 0.f, 0.f);
    const float4 va = a < nm ? move_column<true>(mvs[a], tabv, mp, j) : za;
    const float4 vb = b < nm ? move_column<true>(mvs[b], tabv, mp, j) : za;
    float4* row = out + ((int64_t)j * ntile + mt) * 64;
    if (quad) {
      row[a - mt * kEBM] = va;
      row[b - mt * kEBM] = vb;
      return;
    }
    row[slot] = make_float4(va.x, vb.x, va.y, vb.y);
    row[32 + slot] = make_float4(va.z, vb.z, va.w, vb.w);
  } else {
    float2* out = reinterpret_cast<float2*>(outv);
    const int j = (int)(x / nm_pad), mv = (int)(x % nm_pad);
    out[x] = mv < nm ? move_column<false>(mvs[mv], tabv, mp, j) : make_float2(0.f, 0.f);
  }
}

__host__ __device__ inline int64_t move_table_elems(int cplx, int mp, int nm_pad) {
  return cplx ? (int64_t)mp * (nm_pad / kEBM) * 32 : (int64_t)mp * nm_pad;
}

// Byte offset of the factor table in the scratch: after the move table of
// mp x nm_pad entries (T2: 16 bytes complex, 8 real).
__host__ __device__ inline int64_t move_factor_offset(int cplx, int mp, int nm_pad) {
  return ((int64_t)mp * nm_pad * (cplx ? 16 : 8) + 255) / 256 * 256;
}

// Element y = 4 mv + x of the factor table: mel(x) exp(-2 s_i a_i (- 2 s_k a_k)) of
// move mv for the spin pattern x = 2 idx(s_i) + idx(s_k) (zero for a padding move
// or a zero matrix element), in FP64: the per-move constant of every ratio.
template <bool CPLX>
__device__ __forceinline__ void move_factor_elem(int64_t y, const OpMove* __restrict__ mvs,
                                                 const double* __restrict__ a, int nm,
                                                 double2* out) {
  const int mv = (int)(y >> 2), x = (int)(y & 3);
  double cr = 0.0, ci = 0.0;
  if (mv < nm) {
    const double mr = mvs[mv].mel[x][0], mi = mvs[mv].mel[x][1];
    if (mr != 0.0 || mi != 0.0) {
      const double si = (x >> 1) ? -1.0 : 1.0, sk = (x & 1) ? -1.0 : 1.0;
      const int i = mvs[mv].i, k = mvs[mv].k;
      double vr, vi;
      if (CPLX) {
        vr = -2.0 * si * a[2 * i];
        vi = -2.0 * si * a[2 * i + 1];
        if (mvs[mv].two) {
          vr += -2.0 * sk * a[2 * k];
          vi += -2.0 * sk * a[2 * k + 1];
        }
      } else {
        vr = -2.0 * si * a[i];
        vi = 0.0;
        if (mvs[mv].two) vr += -2.0 * sk * a[k];
      }
      const double ev = exp(vr), fr = ev * cos(vi), fi = ev * sin(vi);
      cr = mr * fr - mi * fi;
      ci = mr * fi + mi * fr;
    }
  }
  out[y] = make_double2(cr, ci);
}

// Element x of a call's tables: the move table, then the factor table.
template <bool CPLX>
__device__ __forceinline__ void move_job_elem(int64_t x, const OpMove* __restrict__ mvs,
                                              const void* __restrict__ tabv,
                                              const double* __restrict__ a, int mp, int nm,
                                              int nm_pad, bool quad, void* outv) {
  const int64_t te = move_table_elems(CPLX, mp, nm_pad);
  if (x < te) {
    move_table_elem<CPLX>(x, mvs, tabv, mp, nm, nm_pad, quad, outv);
  } else {
    double2* fac = reinterpret_cast<double2*>(reinterpret_cast<char*>(outv) +
                                              move_factor_offset(CPLX, mp, nm_pad));
    move_factor_elem<CPLX>(x - te, mvs, a, nm, fac);
  }
}

__host__ __device__ inline int64_t move_job_elems(int cplx, int mp, int nm_pad) {
  return move_table_elems(cplx, mp, nm_pad) + (int64_t)nm_pad * 4;
}

template <bool CPLX>
__global__ void move_tables_kernel(const char* __restrict__ op, const void* __restrict__ tabv,
                                   const double* __restrict__ a, int mp, int nm, int nm_pad,
                                   void* outv) {
  const OpDevHeader* H = reinterpret_cast<const OpDevHeader*>(op);
  const OpMove* mvs = reinterpret_cast<const OpMove*>(op + H->off_moves);
  const int64_t total = move_job_elems(CPLX, mp, nm_pad);
  for (int64_t x = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; x < total;
       x += (int64_t)gridDim.x * blockDim.x)
    move_job_elem<CPLX>(x, mvs, tabv, a, mp, nm, nm_pad, (H->flags & kOpQuadMoves) != 0, outv);
}

// The move tables of many problems in one launch (job k owns elements
// [start[k], start[k + 1]) of the concatenated range; real and complex jobs mix).
constexpr int kMoveJobs = 64;
struct MoveTableJob {
  int cplx, mp, nm, nm_pad;
  const char* op;
  const void* tab;
  const double* a;
  void* out;
};
struct MoveTableBatch {
  int n;
  int64_t start[kMoveJobs + 1];
  MoveTableJob j[kMoveJobs];
};

__global__ void move_tables_batch_kernel(const __grid_constant__ MoveTableBatch B) {
  const int64_t total = B.start[B.n];
  for (int64_t x = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; x < total;
       x += (int64_t)gridDim.x * blockDim.x) {
    int lo = 0, hi = B.n - 1;
    while (lo < hi) {
      const int mid = (lo + hi + 1) >> 1;
      if (B.start[mid] <= x) lo = mid; else hi = mid - 1;
    }
    const MoveTableJob& J = B.j[lo];
    const OpDevHeader* H = reinterpret_cast<const OpDevHeader*>(J.op);
    const OpMove* mvs = reinterpret_cast<const OpMove*>(J.op + H->off_moves);
    if (J.cplx)
      move_job_elem<true>(x - B.start[lo], mvs, J.tab, J.a, J.mp, J.nm, J.nm_pad,
                          (H->flags & kOpQuadMoves) != 0, J.out);
    else
      move_job_elem<false>(x - B.start[lo], mvs, J.tab, J.a, J.mp, J.nm, J.nm_pad, false, J.out);
  }
}

// Packed FP32 pair arithmetic (two independent lanes per instruction).
__device__ __forceinline__ float2 f2fma(float2 a, float2 b, float2 c) { return __ffma2_rn(a, b, c); }
__device__ __forceinline__ float2 f2mul(float2 a, float2 b) { return __fmul2_rn(a, b); }

// Two running products (the lanes of a packed pair, complex: Re in x, Im in y)
// renormalised with one shared power of two, the exponent of the largest of
// their four parts: each is kept as mantissa * 2^e with the pair's e.  The
// smaller product keeps its full FP32 precision unless it is below 2^-126 of
// the larger, where its local-energy term is negligible against the larger one.
// Exponents count up to 126 only: 2^-127 is no normal number, and of an infinity any
// positive power of two leaves what it is.
__device__ __forceinline__ void renorm_pair(float2& x, float2& y, int& e) {
  const float mx = fmaxf(fmaxf(fabsf(x.x), fabsf(x.y)), fmaxf(fabsf(y.x), fabsf(y.y)));
  int ex = min((__float_as_int(mx) >> 23) & 0xff, 253) - 127;
  if (mx == 0.f) ex = 0;
  const float sc = __int_as_float((127 - ex) << 23);
  x = f2mul(x, make_float2(sc, sc));
  y = f2mul(y, make_float2(sc, sc));
  e += ex;
}

// p 2^e, as ldexp gives it (one multiplication where 2^e is a normal number)
__device__ __forceinline__ double scale_exp(float p, int e) {
  if (e > -1000 && e < 1000) return (double)p * __longlong_as_double((long long)(1023 + e) << 52);
  return ldexp((double)p, e);
}

__device__ __forceinline__ void local_energy_body(const CUtensorMap* mtab, const ElocArgs& A,
                                                  const int tile_idx, const int seg) {
  using F = float2;
  using T2 = float4;
  extern __shared__ __align__(128) unsigned char smraw[];
  using TS = float4;  // t tile entry: (Re t, Re t, Im t, Im t), two packed pairs
  T2* mvt = reinterpret_cast<T2*>(smraw);                                    // [2][BK][BM]
  TS* tS = reinterpret_cast<TS*>(smraw + 2 * kEBK * kEBM * sizeof(T2));      // [2][BK][BS+1]
  int* mvi = reinterpret_cast<int*>(reinterpret_cast<char*>(tS) +
                                    round_up(2 * kEBK * kETS * sizeof(TS), 16));
  int* mvk = mvi + kEBM;
  int* mvtwo = mvk + kEBM;
  double2* cvs = reinterpret_cast<double2*>(mvtwo + kEBM);                   // [BM][4]
  double2* eacc = cvs + 4 * kEBM;  // [4][256] per-thread partial E_loc (kept out of registers)
  uint64_t* mbar = reinterpret_cast<uint64_t*>(eacc + 4 * 256);              // [2]

  const int tid = threadIdx.x, ts = tid >> 4, tm = tid & 15;
  const int64_t s0 = (int64_t)tile_idx * kEBS;
  const int n = A.n, m = A.m, mp = A.mp;
  const OpDevHeader* H = reinterpret_cast<const OpDevHeader*>(A.op);
  const OpDSite* ds = reinterpret_cast<const OpDSite*>(A.op + H->off_dsite);
  const OpDBond* db = reinterpret_cast<const OpDBond*>(A.op + H->off_dbond);
  const OpMove* mvs = reinterpret_cast<const OpMove*>(A.op + H->off_moves);
  const F* th = reinterpret_cast<const F*>(A.theta);
  F* tout = reinterpret_cast<F*>(A.t_out);
  const int nm = A.n_moves;
  if (H->flags & kOpQuadMoves) return;  // eloc_wide_body's
  const int ntile = (nm + kEBM - 1) / kEBM, nchunk = mp / kEBK;
  const int tile_begin = ntile * seg / A.nseg, tile_end = ntile * (seg + 1) / A.nseg;
  const int it_begin = tile_begin * nchunk, it_end = tile_end * nchunk;
  const uint32_t tile_bytes = kEBK * kEBM * sizeof(T2);

  if (tid == 0) {
    mbar_init(&mbar[0], 1);
    mbar_init(&mbar[1], 1);
    mbar_fence_init();
  }

  // diagonal part: the 16 threads of a configuration split the terms
  double er[4], ei[4];
#pragma unroll
  for (int p = 0; p < 4; ++p) {
    er[p] = ei[p] = 0.0;
    const int64_t s = s0 + ts * 4 + p;
    if (s < A.ns && seg == 0) {  // the diagonal belongs to the first segment
      const int8_t* sg = A.sigma + s * n;
      for (int u = tm; u < H->n_dsite; u += 16) {
        int x = idx_of(sg[ds[u].i]);
        er[p] += ds[u].d[x][0];
        ei[p] += ds[u].d[x][1];
      }
      for (int u = tm; u < H->n_dbond; u += 16) {
        int x = 2 * idx_of(sg[db[u].i]) + idx_of(sg[db[u].k]);
        er[p] += db[u].d[x][0];
        ei[p] += db[u].d[x][1];
      }
    }
    eacc[p * 256 + tid] = make_double2(er[p], ei[p]);
  }

  // Hidden-unit chunk of iteration it: each move tile walks the chunks in the
  // direction opposite to the previous one, so its first chunks are the ones the
  // CTA read last (still in L2) -- fewer DRAM re-reads of the t rows.
  auto chunk_of = [&](int it) {
    const int r = it % nchunk;
    return ((it / nchunk - tile_begin) & 1) ? nchunk - 1 - r : r;
  };
  // t tile of a chunk: thread covers (ss, kk) = (e >> 4, e & 15), e = tid + 256 u
  F tv[4];
  auto load_t = [&](int it) {
    const int kc = chunk_of(it), mt = it / nchunk;
    const bool reuse = tout && mt > tile_begin;  // t was written by this CTA at its first tile
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const int e = tid + u * 256, ss = e >> 4, kk = e & 15;
      const int64_t s = s0 + ss;
      const int j = kc * kEBK + kk;
      tv[u] = make_float2(0.f, 0.f);
      if (s < A.ns && j < m) tv[u] = reuse ? tout[s * m + j] : th[s * m + j];
    }
  };
  auto store_t = [&](int it, int buf) {
    const int kc = chunk_of(it), mt = it / nchunk;
    const bool reuse = tout && mt > tile_begin;
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const int e = tid + u * 256, ss = e >> 4, kk = e & 15;
      const int64_t s = s0 + ss;
      const int j = kc * kEBK + kk;
      F v = tv[u];
      if (!reuse && s < A.ns && j < m) {
        cf c = tanh_c(cf{v.x, v.y});
        v = make_float2(c.x, c.y);
        if (tout) tout[s * m + j] = v;
      }
      tS[(buf * kEBK + kk) * kETS + ss] = make_float4(v.x, v.x, v.y, v.y);
    }
  };

  __syncthreads();
  if (it_end > it_begin) {
    if (tid == 0) {
      mbar_arrive_expect_tx(&mbar[0], tile_bytes);
      tma_load_2d(mvt, mtab, tile_begin * kEBM * 4, 0, &mbar[0]);
    }
    load_t(it_begin);
    store_t(it_begin, 0);
  }

  // running products packed over the move pairs (q = 2 qp, 2 qp + 1): Px/Py[p][qp] =
  // (Re, Im) parts, shared exponent Pe[p][qp]
  float2 Px[4][2], Py[4][2];
  int Pe[4][2];
  float2 ns2[4][2];     // -sigma_i packed over the move pairs
  bool bad = false;     // a bounded wait for a move-table chunk gave up
  __shared__ volatile int s_bad;
  if (tid == 0) s_bad = 0;
  __syncthreads();
  int it_stop = it_end; // first chunk not processed
  for (int it = it_begin; it < it_end; ++it) {
    const int b = (it - it_begin) & 1, kc = it % nchunk, mt = it / nchunk, mt0 = mt * kEBM;
    __syncthreads();  // chunk it-1 fully consumed; t tile of chunk it stored
    if (s_bad) {      // a wait timed out: all threads stop together
      it_stop = it;
      break;
    }
    if (kc == 0) {
      // new tile of moves: metadata and mel * exp(visible) per sign pattern
      if (tid < kEBM) {
        const int mv = mt0 + tid;
        mvi[tid] = mv < nm ? mvs[mv].i : 0;
        mvk[tid] = mv < nm ? mvs[mv].k : 0;
        mvtwo[tid] = mv < nm ? mvs[mv].two : -1;  // -1: padding move
      }
      // the tile's mel x exp(visible) factors, built once per call by the
      // move-table launch (tile mt0 .. mt0 + 63 lies inside the padded table)
      cvs[tid] = A.fac[(int64_t)mt0 * 4 + tid];
      __syncthreads();
#pragma unroll
      for (int p = 0; p < 4; ++p) {
        const int64_t s = s0 + ts * 4 + p;
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          const float sv = (s < A.ns) ? (float)A.sigma[s * n + mvi[tm + 16 * q]] : 1.f;
          if (q & 1) ns2[p][q >> 1].y = -sv; else ns2[p][q >> 1].x = -sv;
        }
#pragma unroll
        for (int qp = 0; qp < 2; ++qp) {
          Px[p][qp] = make_float2(1.f, 1.f);
          Py[p][qp] = make_float2(0.f, 0.f);
          Pe[p][qp] = 0;
        }
      }
    }
    if (tid == 0 && it + 1 < it_end) {
      const int it1 = it + 1;
      mbar_arrive_expect_tx(&mbar[b ^ 1], tile_bytes);
      tma_load_2d(mvt + (size_t)(b ^ 1) * kEBK * kEBM, mtab,
                      (it1 / nchunk) * kEBM * 4, chunk_of(it1) * kEBK, &mbar[b ^ 1]);
    }
    if (it + 1 < it_end) load_t(it + 1);
    if (!mbar_wait_bounded(&mbar[b], (uint32_t)(((it - it_begin) >> 1) & 1))) {
      bad = true;
      s_bad = 1;
    }
    const T2* mv_b = mvt + (size_t)b * kEBK * kEBM;
    const TS* t_b = tS + (size_t)b * kEBK * kETS;
    // r = C - s t D for two moves at once: with ns = -s,
    // Re r = Re C + ns (Re t Re D - Im t Im D), Im r = Im C + ns (Re t Im D + Im t Re D),
    // then P *= r.
    const float4* mvc = reinterpret_cast<const float4*>(mv_b);
#pragma unroll
    for (int kk = 0; kk < kEBK; ++kk) {
      float4 t4[4], c4[2], d4[2];
#pragma unroll
      for (int p = 0; p < 4; ++p) t4[p] = t_b[kk * kETS + ts * 4 + p];
#pragma unroll
      for (int qp = 0; qp < 2; ++qp) {
        c4[qp] = mvc[kk * kEBM + tm + 16 * qp];
        d4[qp] = mvc[kk * kEBM + 32 + tm + 16 * qp];
      }
#pragma unroll
      for (int p = 0; p < 4; ++p) {
        const float2 tx = make_float2(t4[p].x, t4[p].y), ty = make_float2(t4[p].z, t4[p].w);
        const float2 nty = make_float2(-t4[p].z, -t4[p].w);
#pragma unroll
        for (int qp = 0; qp < 2; ++qp) {
          const float2 cx = make_float2(c4[qp].x, c4[qp].y), cy = make_float2(c4[qp].z, c4[qp].w);
          const float2 dx = make_float2(d4[qp].x, d4[qp].y), dy = make_float2(d4[qp].z, d4[qp].w);
          const float2 tdx = f2fma(tx, dx, f2mul(nty, dy));
          const float2 tdy = f2fma(tx, dy, f2mul(ty, dx));
          const float2 rx = f2fma(ns2[p][qp], tdx, cx);
          const float2 ry = f2fma(ns2[p][qp], tdy, cy);
          const float2 px = Px[p][qp], py = Py[p][qp];
          Px[p][qp] = f2fma(make_float2(-py.x, -py.y), ry, f2mul(px, rx));
          Py[p][qp] = f2fma(py, rx, f2mul(px, ry));
        }
      }
      if (kk == kEBK - 1) {  // once per chunk of 16 hidden units
#pragma unroll
        for (int p = 0; p < 4; ++p)
#pragma unroll
          for (int qp = 0; qp < 2; ++qp) renorm_pair(Px[p][qp], Py[p][qp], Pe[p][qp]);
      }
    }
    if (it + 1 < it_end) store_t(it + 1, b ^ 1);
    if (kc == nchunk - 1) {
      // fold the tile's ratios into the local energies (FP64)
#pragma unroll
      for (int p = 0; p < 4; ++p) {
        const int64_t s = s0 + ts * 4 + p;
        if (s >= A.ns) continue;
        double2 acc = eacc[p * 256 + tid];
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          const int mm = tm + 16 * q;
          if (mvtwo[mm] < 0) continue;
          const int x = 2 * idx_of(A.sigma[s * n + mvi[mm]]) + idx_of(A.sigma[s * n + mvk[mm]]);
          const double2 cv = cvs[mm * 4 + x];
          if (cv.x == 0.0 && cv.y == 0.0) continue;
          double pr, pi;
          const float2 px = Px[p][q >> 1], py = Py[p][q >> 1];
          pr = scale_exp((q & 1) ? px.y : px.x, Pe[p][q >> 1]);
          pi = scale_exp((q & 1) ? py.y : py.x, Pe[p][q >> 1]);
          acc.x += cv.x * pr - cv.y * pi;
          acc.y += cv.x * pi + cv.y * pr;
        }
        eacc[p * 256 + tid] = acc;
      }
    }
  }
  __syncthreads();
  bad = s_bad != 0;
  if (bad) {
    if (tid == 0) {
      // let the chunk copies still in flight (the one waited for and the next)
      // land before the CTA exits
      for (int c = it_stop - 1; c <= it_stop && c < it_end; ++c)
        if (c >= it_begin)
          mbar_wait_bounded(&mbar[(c - it_begin) & 1], (uint32_t)(((c - it_begin) >> 1) & 1),
                            1u << 20);
      dev_status_set(1u << NK_ERR_TIMEOUT);
    }
  }
  // the 16 threads of a configuration are lanes tid ^ 1, 2, 4, 8 of one warp
#pragma unroll
  for (int p = 0; p < 4; ++p) {
    er[p] = bad ? __longlong_as_double(0x7ff8000000000000ll) : eacc[p * 256 + tid].x;
    ei[p] = bad ? __longlong_as_double(0x7ff8000000000000ll) : eacc[p * 256 + tid].y;
#pragma unroll
    for (int off = 8; off >= 1; off >>= 1) {
      er[p] += __shfl_xor_sync(0xffffffffu, er[p], off);
      ei[p] += __shfl_xor_sync(0xffffffffu, ei[p], off);
    }
    const int64_t s = s0 + ts * 4 + p;
    if (tm == 0 && s < A.ns) {
      if (A.nseg == 1) {
        A.eloc[2 * s] = er[p];
        A.eloc[2 * s + 1] = ei[p];
      } else {
        // two addends onto an exact zero: 0 + x + y = 0 + y + x in IEEE
        // arithmetic, so the result does not depend on the order
        atomicAdd(&A.eloc[2 * s], er[p]);
        atomicAdd(&A.eloc[2 * s + 1], ei[p]);
      }
    }
  }
  // with no moves at all, t = tanh(theta) is still written
  if (nm == 0 && tout && seg == 0) {
    for (int e = tid; e < kEBS * m; e += blockDim.x) {
      const int64_t s = s0 + e / m;
      const int j = e % m;
      if (s >= A.ns) continue;
      const F x = th[s * m + j];
      const cf c = tanh_c(cf{x.x, x.y});
      tout[s * m + j] = make_float2(c.x, c.y);
    }
  }
}

__global__ void __launch_bounds__(256, 2) local_energy_tiled(const __grid_constant__ CUtensorMap mtab,
                                                          ElocArgs A) {
  local_energy_body(&mtab, A, A.seg_fast ? blockIdx.y : blockIdx.x,
                          A.seg_fast ? blockIdx.x : blockIdx.y);
}

// ------------------------------------------------------------------ wide form
// Real RBMs, and complex RBMs on operators in the site-quad layout (a thread's four
// moves share their first spin): a CTA takes 128 configurations x 64 moves, each thread
// 8 configurations x 4 moves, packed over pairs of configurations.  What bounds the
// 4 x 4 form is not the FMA pipe but shared memory: complex, 128 operand bytes per
// thread and hidden unit for 72 packed instructions (an SM returns 128 bytes per clock,
// so 128 cycles against the FMA pipe's 144).  Here it is 128 bytes for 136: t as it
// lies (planes of real and imaginary parts, a pair of configurations is one operand),
// the move's (C, D) put in both lanes by register moves; real: 64 bytes for 48.
// 20x20 J1-J2, 65,536 samples: 62.9 -> 52.6 ms; 10x10 Ising, 16,383 samples, with
// theta: 373 -> 315 us.  The order of the instructions within a unit does not matter (five tried,
// 53.4 - 53.5 ms), scalar multiply-adds with a negated operand cost more (55.9).
// Complex operators without quads would need a sign per configuration and move, which
// does not fit the registers: the 4 x 4 form (local_energy_body) keeps them.
//
// The (configuration tile, move tile) units are dealt to the CTAs as contiguous ranges
// of equal length; a range is at least one configuration tile long (or exactly half of
// one), so at most two CTAs share a tile and their sums meet in eloc as two addends
// onto zero, whatever the order.
//
// Fewer tiles than CTA slots: a tile's move tiles are dealt to a cluster of up to eight
// CTAs, whose sums the first adds up in rank order, and tiles are of 64 configurations
// (4 x 4 per thread) where that is faster still (wide_plan).
template <bool CPLX, int NP>            // NP pairs of configurations per thread
struct WideSmem {
  using T2 = typename RatioTypes<CPLX>::T2;
  static constexpr int BS = 32 * NP;    // configurations per tile
  static constexpr int TS = BS + 4;     // pitch of a t plane row (one hidden unit)
  T2 tab[2][kEBK][kEBM];                // (C, D) of the chunk's units and the tile's moves
  float t[2][CPLX ? 2 : 1][kEBK][TS];   // [stage][re, im]
  double2 cvs[4 * kEBM];                // mel x exp(visible)
  double2 eacc[BS];                     // E_loc of the configurations so far
  int mvi[kEBM], mvk[kEBM];
  uint64_t mbar[2];
  int bad;
  // exponents of a pair's running products: E0 + (E1 << 16) in the first plane, or, for
  // more units than 16 bits can count (wide_exps), a plane each.  A tile starts at 127 per
  // renormalisation to come, which takes off its renorm_scale's field.
  int pe[2][4 * NP][256];
};

// Whether exponents may need more than 16 bits: a renormalisation (16 units, real: 8)
// adds at most 127 in magnitude.
__host__ __device__ inline bool wide_exps(int mp, bool cplx) {
  return mp / (cplx ? kEBK : kEBK / 2) > 255;
}

template <bool CPLX, int NP>
static size_t wide_smem(int mp) {
  return sizeof(WideSmem<CPLX, NP>) -
         (wide_exps(mp, CPLX) ? 0 : sizeof(WideSmem<CPLX, NP>::pe) / 2);
}

__device__ __forceinline__ void cluster_barrier() {
  asm volatile("barrier.cluster.arrive.release;" ::: "memory");
  asm volatile("barrier.cluster.wait.acquire;" ::: "memory");
}

// *p of the cluster's CTA `rank`
__device__ __forceinline__ double2 ld_cluster(const double2* p, int rank) {
  uint32_t a;
  double2 v;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(a) : "r"(smem_addr(p)), "r"(rank));
  asm volatile("ld.shared::cluster.v2.f64 {%0, %1}, [%2];" : "=d"(v.x), "=d"(v.y) : "r"(a) : "memory");
  return v;
}

__device__ __forceinline__ void cp_async4(void* dst, const void* src) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(smem_addr(dst)), "l"(src) : "memory");
}

// Bits of the power of two that a renormalisation multiplies v by: 2^(127 - E), E the
// biased exponent, but never below 2^-126 (renorm_pair has the reason).  127 - E comes
// from the complemented field, so that the limit costs no instruction (one more per
// product took 2.5 % of a real call's time).
__device__ __forceinline__ uint32_t renorm_scale(float v) {
  return (uint32_t)__viaddmax_s32((int)(~__float_as_uint(v) & 0x7f800000u), -(1 << 23), 1 << 23);
}

// Sum over the 16 lanes of a configuration (nothing to do where it is zero in the
// whole warp, as the imaginary parts of a real problem are).
__device__ __forceinline__ void sum16(double& v) {
  if (!__any_sync(0xffffffffu, v != 0.0)) return;
#pragma unroll
  for (int off = 8; off >= 1; off >>= 1) v += __shfl_xor_sync(0xffffffffu, v, off);
}

// CTA bx of the gx that share the call's units; CLUSTER: of the `parts` that make up
// the cluster of a configuration tile.
template <bool CPLX, int NP, bool CLUSTER>
__device__ __forceinline__ void eloc_wide_body(const CUtensorMap* mtab, const ElocArgs& A, int bx,
                                               int gx, int parts) {
  constexpr int kQBS = WideSmem<CPLX, NP>::BS;
  using F = typename RatioTypes<CPLX>::F;
  const OpDevHeader* H = reinterpret_cast<const OpDevHeader*>(A.op);
  if (CPLX && !(H->flags & kOpQuadMoves)) return;  // local_energy_body's
  extern __shared__ __align__(128) unsigned char smraw[];
  using Smem = WideSmem<CPLX, NP>;
  Smem& S = *reinterpret_cast<Smem*>(smraw);
  const OpDSite* ds = reinterpret_cast<const OpDSite*>(A.op + H->off_dsite);
  const OpDBond* db = reinterpret_cast<const OpDBond*>(A.op + H->off_dbond);
  const OpMove* mvs = reinterpret_cast<const OpMove*>(A.op + H->off_moves);
  const F* th = reinterpret_cast<const F*>(A.theta);
  F* tout = reinterpret_cast<F*>(A.t_out);
  const int tid = threadIdx.x, ts = tid >> 4, tm = tid & 15;
  const int n = A.n, m = A.m, nchunk = A.mp / kEBK, nm = A.n_moves;
  const int ntile = nm > 0 ? (nm + kEBM - 1) / kEBM : 1;  // no moves: one empty tile
  const int half = A.nseg == 2 ? ntile / 2 : ntile;
  const int64_t tiles = (A.ns + kQBS - 1) / kQBS, units = tiles * ntile;
  const int64_t u_begin = CLUSTER ? (int64_t)(bx / parts) * ntile + ntile * (bx % parts) / parts
                                  : units * bx / gx;
  const int64_t u_end = CLUSTER ? (int64_t)(bx / parts) * ntile + ntile * (bx % parts + 1) / parts
                                : units * (bx + 1) / gx;
  const bool big = wide_exps(A.mp, CPLX);
  const uint32_t tab_bytes = sizeof(S.tab[0]);
  if (tid == 0) {
    mbar_init(&S.mbar[0], 1);
    mbar_init(&S.mbar[1], 1);
    mbar_fence_init();
    S.bad = 0;
  }
  __syncthreads();
  uint32_t fills = 0;  // table chunks waited for so far (stage and phase of the next)
  bool bad = false;

  int64_t u0 = u_begin;
  while (u0 < u_end && !bad) {
    // one configuration tile's share: move tiles [mt_begin, mt_end)
    const int64_t tile = u0 / ntile;
    const int mt_begin = (int)(u0 - tile * ntile);
    const int mt_end = (int)std::min<int64_t>(ntile, mt_begin + (u_end - u0));
    u0 += mt_end - mt_begin;
    const int64_t s0 = tile * kQBS;
    const bool whole = mt_end - mt_begin == ntile;
    __syncthreads();  // the last tile's readers of eacc are done
    // diagonal part: the threads of a configuration (and the CTAs of a cluster) split the
    // terms, FP64 adds being what this part costs; the configurations
    // are staged in the tiles' memory (not in use yet) where they fit, so that a warp
    // reads one term and 32 configurations at a time
    {
      const int c = tid & (kQBS - 1), h = tid / kQBS;
      const int64_t s = std::min<int64_t>(s0 + c, A.ns - 1);
      const int pitch = (int)round_up(n, 128) + 4;  // neighbouring configurations one bank apart
      const bool staged = (size_t)pitch * kQBS <= offsetof(Smem, cvs);
      const int8_t* sg = A.sigma + s * n;
      double er = 0.0, ei = 0.0;
      if (CLUSTER || mt_begin == 0) {
        if (staged) {
          int8_t* st = reinterpret_cast<int8_t*>(smraw);
          const int64_t lim = (A.ns - s0) * n;
          for (int x = tid; x < kQBS * n; x += 256)
            st[x / n * pitch + x % n] = x < lim ? A.sigma[s0 * n + x] : 1;
          __syncthreads();
          sg = st + c * pitch;
        }
        constexpr int TPC = 256 / kQBS;  // threads per configuration
        auto terms = [&](int first, int step, double& er, double& ei) {
#pragma unroll 4
          for (int u = first; u < H->n_dsite; u += step) {
            const double* d = ds[u].d[idx_of(sg[ds[u].i])];
            er += d[0];
            if (d[1] != 0.0) ei += d[1];
          }
#pragma unroll 4
          for (int u = first; u < H->n_dbond; u += step) {
            const double* d = db[u].d[2 * idx_of(sg[db[u].i]) + idx_of(sg[db[u].k])];
            er += d[0];
            if (d[1] != 0.0) ei += d[1];
          }
        };
        if (CLUSTER) {
          terms(h + TPC * (bx % parts), TPC * parts, er, ei);
        } else {
          // four partial sums, (0 + 2) + (1 + 3) whatever the tile: a call's sums do not
          // depend on whether it runs in a batch
          terms(h, 4, er, ei);
          if (TPC == 2) {
            double er2 = 0.0, ei2 = 0.0;
            terms(h + 2, 4, er2, ei2);
            er += er2;
            ei += ei2;
          }
        }
        S.cvs[tid] = make_double2(er, ei);  // (not in use yet)
        __syncthreads();
        if (h == 0) {
          double2 b = S.cvs[kQBS + c];
          if (TPC == 4) {
            er += S.cvs[2 % TPC * kQBS + c].x;
            ei += S.cvs[2 % TPC * kQBS + c].y;
            b.x += S.cvs[3 % TPC * kQBS + c].x;
            b.y += S.cvs[3 % TPC * kQBS + c].y;
          }
          er += b.x;
          ei += b.y;
        }
      }
      if (h == 0) S.eacc[c] = make_double2(er, ei);
      // the staged configurations are read before the tiles' copies may land on them
      asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
      __syncthreads();
    }
    const int it_begin = mt_begin * nchunk, it_end = nm > 0 ? mt_end * nchunk : it_begin;
    // each move tile walks the chunks in the direction opposite to the previous one, so
    // its first chunks are the ones read last (still in L2); the directions are those
    // of the two halves a call may be split into, so that the products' order is fixed
    auto chunk_of = [&](int it) {
      const int r = it % nchunk, mt = it / nchunk;
      return ((mt >= half ? mt - half : mt) & 1) ? nchunk - 1 - r : r;
    };
    // t of a chunk: thread (c, kk) = (tid / 16 + 16 u, tid % 16) copies its elements
    // asynchronously, from t_out after the CTA's first move tile of these configurations.
    // Before (or without t_out) theta is copied, and the thread turns its own elements
    // into tanh(theta) where they lie, after the chunk's products.
    auto from_t = [&](int it) { return tout && it / nchunk > mt_begin; };
    auto copy_t = [&](int it, int b) {
      const int kk = tid & 15, j = chunk_of(it) * kEBK + kk;
      const F* base = from_t(it) ? tout : th;
#pragma unroll
      for (int u = 0; u < 2 * NP; ++u) {
        const int c = ts + 16 * u;
        const int64_t s = s0 + c;
        if (s < A.ns && j < m) {
          const float* src = reinterpret_cast<const float*>(base + s * m + j);
          cp_async4(&S.t[b][0][kk][c], src);
          if constexpr (CPLX) cp_async4(&S.t[b][1][kk][c], src + 1);
        } else {
          S.t[b][0][kk][c] = 0.f;
          if constexpr (CPLX) S.t[b][1][kk][c] = 0.f;
        }
      }
      asm volatile("cp.async.commit_group;" ::: "memory");
    };
    auto tanh_t = [&](int it, int b) {
      const int kk = tid & 15, j = chunk_of(it) * kEBK + kk;
#pragma unroll (CPLX ? 2 : 4)
      for (int u = 0; u < 2 * NP; ++u) {
        const int c = ts + 16 * u;
        const int64_t s = s0 + c;
        if (s >= A.ns || j >= m) continue;
        if constexpr (CPLX) {
          const cf y = tanh_c(cf{S.t[b][0][kk][c], S.t[b][1][kk][c]});
          S.t[b][0][kk][c] = y.x;
          S.t[b][1][kk][c] = y.y;
          if (tout) tout[s * m + j] = make_float2(y.x, y.y);
        } else {
          const float y = tanh_f(S.t[b][0][kk][c]);
          S.t[b][0][kk][c] = y;
          if (tout) tout[s * m + j] = y;
        }
      }
    };
    auto land_t = [&](int it, int b) {
      asm volatile("cp.async.wait_all;" ::: "memory");
      if (!from_t(it)) tanh_t(it, b);
    };
    auto load_tab = [&](int it, int b) {  // one thread
      mbar_arrive_expect_tx(&S.mbar[b], tab_bytes);
      tma_load_2d(S.tab[b], mtab, (it / nchunk) * kEBM * (CPLX ? 4 : 2), chunk_of(it) * kEBK,
                  &S.mbar[b]);
    };
    if (it_begin < it_end) {
      if (tid == 0) load_tab(it_begin, (int)(fills & 1));
      copy_t(it_begin, (int)(fills & 1));
      land_t(it_begin, (int)(fills & 1));
    } else if (tout) {  // no moves at all: t = tanh(theta) is still written
      for (int e = tid; e < kQBS * m; e += 256) {
        const int64_t o = (s0 + e / m) * m + e % m;
        if (s0 + e / m >= A.ns) continue;
        if constexpr (CPLX) {
          const cf y = tanh_c(cf{th[o].x, th[o].y});
          tout[o] = make_float2(y.x, y.y);
        } else {
          tout[o] = tanh_f(th[o]);
        }
      }
    }

    float2 Px[NP][4], Py[CPLX ? NP : 1][4];  // [configuration pair][move]
    float2 ns2[NP][CPLX ? 1 : 4];            // -s_i of the pair's configurations (and move)
    for (int it = it_begin; it < it_end; ++it, ++fills) {
      const int b = (int)(fills & 1), kc = it % nchunk, mt0 = it / nchunk * kEBM;
      __syncthreads();  // chunk it - 1 fully consumed; t of chunk it stored
      if (S.bad) {      // a wait timed out: all threads stop together
        bad = true;
        break;
      }
      if (kc == 0) {
        if (tid < kEBM) {
          S.mvi[tid] = mt0 + tid < nm ? mvs[mt0 + tid].i : 0;
          S.mvk[tid] = mt0 + tid < nm ? mvs[mt0 + tid].k : 0;
        }
        S.cvs[tid] = A.fac[(int64_t)mt0 * 4 + tid];  // zero for a padding move
        __syncthreads();
#pragma unroll
        for (int p = 0; p < NP; ++p) {
          const int64_t s = s0 + ts * (2 * NP) + 2 * p;
#pragma unroll
          for (int q = 0; q < (CPLX ? 1 : 4); ++q) {
            const int i = S.mvi[tm + 16 * q];
            ns2[p][q].x = s < A.ns ? -(float)A.sigma[s * n + i] : -1.f;
            ns2[p][q].y = s + 1 < A.ns ? -(float)A.sigma[(s + 1) * n + i] : -1.f;
          }
#pragma unroll
          for (int q = 0; q < 4; ++q) {
            Px[p][q] = make_float2(1.f, 1.f);
            if constexpr (CPLX) Py[p][q] = make_float2(0.f, 0.f);
            const int e = 127 * (CPLX ? 1 : 2) * nchunk;
            S.pe[0][p * 4 + q][tid] = big ? e : e * 65537;
            if (big) S.pe[1][p * 4 + q][tid] = e;
          }
        }
      }
      const bool more = it + 1 < it_end;
      if (more) {
        if (tid == 0) load_tab(it + 1, b ^ 1);
        copy_t(it + 1, b ^ 1);
      }
      if (!mbar_wait_bounded(&S.mbar[b], (fills >> 1) & 1)) S.bad = 1;
      auto renorm = [&]() {  // every product by its own power of two
#pragma unroll
        for (int p = 0; p < NP; ++p)
#pragma unroll
          for (int q = 0; q < 4; ++q) {
            uint32_t b0, b1;
            if constexpr (CPLX) {
              b0 = renorm_scale(fmaxf(fabsf(Px[p][q].x), fabsf(Py[p][q].x)));
              b1 = renorm_scale(fmaxf(fabsf(Px[p][q].y), fabsf(Py[p][q].y)));
            } else {
              b0 = renorm_scale(Px[p][q].x);
              b1 = renorm_scale(Px[p][q].y);
            }
            const float2 sc = make_float2(__uint_as_float(b0), __uint_as_float(b1));
            Px[p][q] = f2mul(Px[p][q], sc);
            if constexpr (CPLX) Py[p][q] = f2mul(Py[p][q], sc);
            if (big) {
              S.pe[0][p * 4 + q][tid] -= (int)(b0 >> 23);
              S.pe[1][p * 4 + q][tid] -= (int)(b1 >> 23);
            } else {
              S.pe[0][p * 4 + q][tid] -= (int)((b0 >> 23) + (b1 >> 7));
            }
          }
      };
      // r = C - s t D for two configurations at once: with nu = -s t,
      // Re r = nu_x D_x + (-nu_y D_y + C_x), Im r = nu_x D_y + (nu_y D_x + C_y); P *= r
#pragma unroll
      for (int kk = 0; kk < kEBK; ++kk) {
        float2 tx[NP], ty[CPLX ? NP : 1];
#pragma unroll
        for (int h = 0; h < NP / 2; ++h) {
          const float4 x = *reinterpret_cast<const float4*>(&S.t[b][0][kk][ts * (2 * NP) + 4 * h]);
          tx[2 * h] = make_float2(x.x, x.y);
          tx[2 * h + 1] = make_float2(x.z, x.w);
          if constexpr (CPLX) {
            const float4 y = *reinterpret_cast<const float4*>(&S.t[b][1][kk][ts * (2 * NP) + 4 * h]);
            tx[2 * h] = f2mul(ns2[2 * h][0], tx[2 * h]);
            tx[2 * h + 1] = f2mul(ns2[2 * h + 1][0], tx[2 * h + 1]);
            ty[2 * h] = f2mul(ns2[2 * h][0], make_float2(y.x, y.y));
            ty[2 * h + 1] = f2mul(ns2[2 * h + 1][0], make_float2(y.z, y.w));
          }
        }
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          const auto v = S.tab[b][kk][tm + 16 * q];
          if constexpr (CPLX) {
            const float2 cx = make_float2(v.x, v.x), cy = make_float2(v.y, v.y);
            const float2 dx = make_float2(v.z, v.z), dy = make_float2(v.w, v.w);
            const float2 ndy = make_float2(-v.w, -v.w);
#pragma unroll
            for (int p = 0; p < NP; ++p) {
              const float2 rx = f2fma(tx[p], dx, f2fma(ty[p], ndy, cx));
              const float2 ry = f2fma(tx[p], dy, f2fma(ty[p], dx, cy));
              const float2 px = Px[p][q], py = Py[p][q];
              Px[p][q] = f2fma(make_float2(-py.x, -py.y), ry, f2mul(px, rx));
              Py[p][q] = f2fma(py, rx, f2mul(px, ry));
            }
          } else {
            const float2 c2 = make_float2(v.x, v.x), d2 = make_float2(v.y, v.y);
#pragma unroll
            for (int p = 0; p < NP; ++p)
              Px[p][q] = f2mul(Px[p][q], f2fma(f2mul(ns2[p][q], tx[p]), d2, c2));
          }
        }
        if (!CPLX && kk == 7) renorm();
      }
      renorm();  // once per chunk of 16 hidden units (real: of 8)
      if (more) land_t(it + 1, b ^ 1);
      if (kc == nchunk - 1) {
        // fold the tile's ratios into the local energies (FP64); the 16 threads of a
        // configuration are lanes tid ^ 1, 2, 4, 8 of one warp
#pragma unroll
        for (int c = 0; c < 2 * NP; ++c) {
          const int64_t s = s0 + ts * (2 * NP) + c;
          double ar = 0.0, ai = 0.0;
          if (s < A.ns) {
#pragma unroll
            for (int q = 0; q < 4; ++q) {
              const int mm = tm + 16 * q;
              const int x = 2 * idx_of(A.sigma[s * n + S.mvi[mm]]) + idx_of(A.sigma[s * n + S.mvk[mm]]);
              const double2 cv = S.cvs[mm * 4 + x];
              if (cv.x == 0.0 && cv.y == 0.0) continue;
              const int e01 = S.pe[0][(c / 2) * 4 + q][tid], e0 = big ? e01 : (int16_t)(e01 & 0xffff);
              const int e = !(c & 1) ? e0 : big ? S.pe[1][(c / 2) * 4 + q][tid] : (e01 - e0) >> 16;
              const float2 px = Px[c / 2][q];
              const double pr = scale_exp((c & 1) ? px.y : px.x, e);
              if constexpr (CPLX) {
                const float2 py = Py[c / 2][q];
                const double pi = scale_exp((c & 1) ? py.y : py.x, e);
                ar += cv.x * pr - cv.y * pi;
                ai += cv.x * pi + cv.y * pr;
              } else {
                ar += cv.x * pr;
                if (cv.y != 0.0) ai += cv.y * pr;
              }
            }
          }
          sum16(ar);
          sum16(ai);
          if (tm == 0) {
            S.eacc[ts * (2 * NP) + c].x += ar;
            S.eacc[ts * (2 * NP) + c].y += ai;
          }
        }
      }
    }
    __syncthreads();
    bad = bad || S.bad != 0;
    if (bad && tid == 0) {
      // the table copies still in flight (the one waited for and the next) land before
      // the CTA exits
      for (uint32_t f = fills > 0 ? fills - 1 : 0; f <= fills + 1; ++f)
        mbar_wait_bounded(&S.mbar[f & 1], (f >> 1) & 1, 1u << 20);
      dev_status_set(1u << NK_ERR_TIMEOUT);
    }
    if (tid < kQBS && s0 + tid < A.ns) {
      const double nan = __longlong_as_double(0x7ff8000000000000ll);
      const double er = bad ? nan : S.eacc[tid].x, ei = bad ? nan : S.eacc[tid].y;
      double* e = A.eloc + 2 * (s0 + tid);
      if (CLUSTER) {
        S.eacc[tid] = make_double2(er, ei);
      } else if (whole) {
        e[0] = er;
        e[1] = ei;
      } else {
        atomicAdd(e, er);
        atomicAdd(e + 1, ei);
      }
    }
  }
  if (CLUSTER) {
    cluster_barrier();
    const int64_t s = (int64_t)(bx / parts) * kQBS + tid;
    if (bx % parts == 0 && tid < kQBS && s < A.ns) {
      double2 e = S.eacc[tid];
      for (int k = 1; k < parts; ++k) {
        const double2 v = ld_cluster(&S.eacc[tid], k);
        e.x += v.x;
        e.y += v.y;
      }
      A.eloc[2 * s] = e.x;
      A.eloc[2 * s + 1] = e.y;
    }
    cluster_barrier();  // the sums are read before their CTAs exit
    return;
  }
  // after a timeout the rest of the CTA's range is marked too
  if (bad)
    for (; u0 < u_end; u0 = (u0 / ntile + 1) * ntile)
      if (tid < kQBS && u0 / ntile * kQBS + tid < A.ns)
        atomicAdd(A.eloc + 2 * (u0 / ntile * kQBS + tid), __longlong_as_double(0x7ff8000000000000ll));
}

template <bool CPLX, int NP, bool CLUSTER>
__global__ void __launch_bounds__(256, 2) local_energy_wide(const __grid_constant__ CUtensorMap mtab,
                                                            ElocArgs A, int parts) {
  eloc_wide_body<CPLX, NP, CLUSTER>(&mtab, A, blockIdx.x, gridDim.x, parts);
}

// Clusters of `parts` CTAs of a wide kernel that run at once (less than the SMs would
// give, where a GPC's do not divide by the cluster); 0 where none do.
template <class K>
static int64_t wide_slots(K kern, size_t smem, int parts) {
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3((unsigned)parts);
  cfg.blockDim = dim3(256);
  cfg.dynamicSmemBytes = smem;
  cudaLaunchAttribute at{};
  at.id = cudaLaunchAttributeClusterDimension;
  at.val.clusterDim.x = (unsigned)parts;
  at.val.clusterDim.y = at.val.clusterDim.z = 1;
  cfg.attrs = &at;
  cfg.numAttrs = 1;
  int n = 0;
  if (!allow_smem(kern, smem) ||
      cudaOccupancyMaxActiveClusters(&n, kern, &cfg) != cudaSuccess) {
    cudaGetLastError();
    return 0;
  }
  return n;
}

// Shared memory that keeps a CTA alone on its SM: a cluster is otherwise put on as few
// SMs as hold it, whatever else is idle.
constexpr size_t kAloneSmem = 116 * 1024;

template <bool CPLX, int NP>
static int64_t wide_clusters(int parts, bool alone) {
  struct Table {
    int64_t n[2][9];
    Table() {  // asked of the driver once
      const size_t smem = wide_smem<CPLX, NP>(32);
      for (int p = 2; p <= 8; ++p) {
        n[0][p] = wide_slots(local_energy_wide<CPLX, NP, true>, smem, p);
        n[1][p] = wide_slots(local_energy_wide<CPLX, NP, true>, std::max(smem, kAloneSmem), p);
      }
    }
  };
  static const Table t;
  return t.n[alone][parts];
}

// How the wide form runs: configurations per tile (32 np), CTAs per tile (a cluster),
// CTAs.  With 304 tiles or more, ranges of units dealt to two CTAs per SM.  Below, the
// cheapest by this measure: rounds of CTAs times move tiles a CTA takes, times what two
// CTAs on an SM cost over one alone (20x20, one move tile: complex 0.71 and 1.28 ms, real
// 0.38 and 0.53), times what 64 configurations cost over 128.  theta + local energies,
// 4 x 4 blocks of 64 configurations in halves -> here: 20x20 J1-J2, 300 samples 5.58 ->
// 1.64 ms, 1500 samples 5.63 -> 2.00, 6000 samples 9.84 -> 6.60; 20x20 Ising, 1500 samples 1.87 -> 1.00; 64-site
// Ising chain, 1500 samples 72 -> 61 us.
struct WidePlan {
  int np, parts;
  int64_t grid;
  bool ranges, alone;
};
static WidePlan wide_plan(int64_t ns, int n_moves, bool cplx) {
  const int64_t slots = 2 * 152;
  const int ntile = std::max(1, (n_moves + kEBM - 1) / kEBM);
  if ((ns + 127) / 128 >= slots) return {4, 1, slots, true, false};
  WidePlan best{};
  double least = 0.0;
  for (int np = 4; np >= 2; np -= 2)
    for (int parts = 1; parts <= std::min(8, ntile); ++parts)
      for (int alone = 1; alone >= 0; --alone) {
        const int64_t tiles = std::max<int64_t>(1, (ns + 32 * np - 1) / (32 * np));
        int64_t at_once = alone ? slots / 2 : slots;
        if (parts > 1)
          at_once = cplx ? (np == 4 ? wide_clusters<true, 4>(parts, alone)
                                    : wide_clusters<true, 2>(parts, alone))
                         : (np == 4 ? wide_clusters<false, 4>(parts, alone)
                                    : wide_clusters<false, 2>(parts, alone));
        if (at_once < 1 || (alone && tiles > at_once)) continue;
        const double cost = (double)((tiles + at_once - 1) / at_once) *
                            ((ntile + parts - 1) / parts) * (np == 4 ? 1.0 : cplx ? 0.6 : 0.75) *
                            (alone ? 1.0 : cplx ? 1.8 : 1.4);
        if (best.np == 0 || cost < 0.97 * least) {
          best = {np, parts, tiles * parts, false, alone != 0};
          least = cost;
        }
      }
  return best;
}

// Up to kElocBatch problems of one field in one launch: CTA b runs CTA
// b - start[k] of problem k, numbered as its own launch with the segment as
// the fast index (the two halves of a configuration tile back to back).
constexpr int kElocBatch = 64;
struct ElocBatch {
  int n;
  int start[kElocBatch + 1];
  ElocArgs a[kElocBatch];
  CUtensorMap map[kElocBatch];
};

__global__ void __launch_bounds__(256, 2) local_energy_batch(const __grid_constant__ ElocBatch B) {
  int k = 0;
  while (k + 1 < B.n && (int)blockIdx.x >= B.start[k + 1]) ++k;
  const int b = (int)blockIdx.x - B.start[k];
  const ElocArgs& A = B.a[k];
  local_energy_body(&B.map[k], A, b / A.nseg, b % A.nseg);
}

// (CLUSTER: every problem's tiles are shared by `parts` CTAs, so that the problems start
// at whole clusters)
template <bool CPLX, int NP, bool CLUSTER>
__global__ void __launch_bounds__(256, 2)
    local_energy_wide_batch(const __grid_constant__ ElocBatch B, int parts) {
  int k = 0;
  while (k + 1 < B.n && (int)blockIdx.x >= B.start[k + 1]) ++k;
  eloc_wide_body<CPLX, NP, CLUSTER>(&B.map[k], B.a[k], (int)blockIdx.x - B.start[k],
                                    B.start[k + 1] - B.start[k], parts);
}

size_t local_energy_scratch_bytes(int m, int cplx, int n_moves) {
  const int64_t nm_pad = round_up(std::max(n_moves, 1), kEBM);
  // the move table, then the factor table (one double2 per move and spin pattern)
  return (size_t)(move_factor_offset(cplx, padded_m(m), (int)nm_pad) + nm_pad * 4 * 16);
}

// Two CTAs per SM: when the last wave of CTAs would be far from full, the move tiles of a
// configuration tile are split into two halves (twice the CTAs) to even out the waves.
int local_energy_segs(int n_moves, int64_t ns) {
  const int64_t blocks = (ns + kEBS - 1) / kEBS;
  auto wave_eff = [&](int64_t b) {
    const int64_t slots = 2 * 152;
    return (double)b / (double)(((b + slots - 1) / slots) * slots);
  };
  return (n_moves > kEBM && wave_eff(2 * blocks) > wave_eff(blocks)) ? 2 : 1;
}

// Everything one local-energy call needs, before anything is enqueued.
struct ElocPlan {
  ElocArgs A;
  CUtensorMap map;
  bool cplx;
  size_t smem;
  int64_t blocks;  // configuration tiles of 64 (local_energy_body)
  bool wide;       // the wide form may run: real, or whole move tiles of a complex operator
                   // that may be in the site-quad layout (only the device knows)
  WidePlan wp;
  MoveTableJob job;
  int64_t tab_elems;
};

static nk_status plan_local_energy(const nk_rbm* r, const void* op_dev, int n_moves,
                                   const int8_t* sigma, const void* theta, int64_t ns,
                                   double* eloc, void* t_out, void* scratch, size_t scratch_bytes,
                                   ElocPlan* P) {
  WsLayout L(r->n, r->m, r->is_complex);
  const bool cplx = r->is_complex != 0;
  const size_t need = local_energy_scratch_bytes(r->m, cplx, n_moves);
  if (n_moves > 0 && (!scratch || scratch_bytes < need))
    return fail(NK_ERR_SHAPE, "nk_local_energy: scratch of %zu B, need %zu B", scratch_bytes, need);
  ElocArgs& A = P->A;
  A.n = r->n;
  A.m = r->m;
  A.mp = L.mp;
  A.ns = ns;
  A.n_moves = n_moves;
  A.sigma = sigma;
  A.theta = theta;
  A.op = (const char*)op_dev;
  A.a = r->a;
  A.tab = (const char*)r->ws + L.tab;
  A.eloc = eloc;
  A.t_out = t_out;
  P->cplx = cplx;
  const int nm_pad = (int)round_up(std::max(n_moves, 1), kEBM);
  memset(&P->map, 0, sizeof(P->map));
  P->job = MoveTableJob{cplx ? 1 : 0, L.mp, n_moves, nm_pad, A.op, A.tab, r->a, scratch};
  P->tab_elems = n_moves > 0 ? move_job_elems(cplx, L.mp, nm_pad) : 0;
  A.fac = n_moves > 0 ? reinterpret_cast<const double2*>(
                            (const char*)scratch + move_factor_offset(cplx, L.mp, nm_pad))
                      : nullptr;
  if (n_moves > 0) {
    const int fl = cplx ? 4 : 2;  // floats per table entry
    if (!make_map_f32(&P->map, scratch, L.mp, (int64_t)nm_pad * fl, (int64_t)nm_pad * fl * 4,
                      kEBM * fl, kEBK))
      return NK_ERR_CUDA;
  }
  P->smem = 2 * kEBK * kEBM * 16 + round_up(2 * kEBK * kETS * 16, 16) + 3 * kEBM * 4 +
            kEBM * 4 * 16 + 4 * 256 * 16 + 16;  // of local_energy_body
  P->blocks = (ns + kEBS - 1) / kEBS;
  A.nseg = local_energy_segs(n_moves, ns);
  if (r->eloc_segs > 0) A.nseg = (r->eloc_segs >= 2 && n_moves > kEBM) ? 2 : 1;  // tuned or set
  A.seg_fast = A.nseg == 2 && P->blocks <= 65535 ? 1 : 0;
  P->wide = !cplx || (n_moves > 0 && n_moves % kEBM == 0);
  if (P->wide) P->wp = wide_plan(ns, n_moves, cplx);
  return NK_OK;
}

// Whether CTAs of one form or the other add their sums up in eloc, which starts at zero.
static bool adds_up(const ElocPlan& P) {
  return (P.cplx && P.A.nseg == 2) || (P.wide && P.wp.ranges);
}

nk_status launch_local_energy(const nk_rbm* r, const void* op_dev, int n_moves,
                              const int8_t* sigma, const void* theta, int64_t ns, double* eloc,
                              void* t_out, void* scratch, size_t scratch_bytes, cudaStream_t st) {
  ElocPlan P;
  if (nk_status e = plan_local_energy(r, op_dev, n_moves, sigma, theta, ns, eloc, t_out, scratch,
                                      scratch_bytes, &P))
    return e;
  const ElocArgs& A = P.A;
  if (P.tab_elems > 0) {
    const int64_t blocks = std::max<int64_t>(1, std::min<int64_t>((P.tab_elems + 255) / 256, 152 * 8));
    if (P.cplx)
      move_tables_kernel<true><<<(unsigned)blocks, 256, 0, st>>>(A.op, A.tab, A.a, A.mp, n_moves,
                                                                 P.job.nm_pad, scratch);
    else
      move_tables_kernel<false><<<(unsigned)blocks, 256, 0, st>>>(A.op, A.tab, A.a, A.mp,
                                                                  n_moves, P.job.nm_pad, scratch);
    if (nk_status e = check_launch("nk_local_energy(move tables)")) return e;
  }
  const WidePlan& wp = P.wp;
  if (adds_up(P) && cudaMemsetAsync(eloc, 0, (size_t)ns * 2 * sizeof(double), st) != cudaSuccess)
    return fail(NK_ERR_CUDA, "nk_local_energy: cudaMemsetAsync failed");
  auto go_wide = [&](auto kern, size_t smem) -> nk_status {
    if (wp.alone && wp.parts > 1) smem = std::max(smem, kAloneSmem);
    if (!allow_smem(kern, smem)) return fail(NK_ERR_CUDA, "nk_local_energy: shared memory attribute");
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3((unsigned)wp.grid);
    cfg.blockDim = dim3(256);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cudaLaunchAttribute at{};
    at.id = cudaLaunchAttributeClusterDimension;
    at.val.clusterDim.x = (unsigned)wp.parts;
    at.val.clusterDim.y = at.val.clusterDim.z = 1;
    cfg.attrs = &at;
    cfg.numAttrs = wp.parts > 1 ? 1 : 0;
    if (cudaLaunchKernelEx(&cfg, kern, P.map, A, wp.parts) != cudaSuccess)
      return fail(NK_ERR_CUDA, "nk_local_energy: launch failed");
    return NK_OK;
  };
  if (P.wide) {
    // complex: only the device knows the operator's layout, and the kernel that it is
    // not for returns
    // one CTA per tile: ranges of whole tiles
    auto pick = [&](auto r4, auto r2, auto c4, auto c2) {
      const size_t s4 = P.cplx ? wide_smem<true, 4>(A.mp) : wide_smem<false, 4>(A.mp);
      const size_t s2 = P.cplx ? wide_smem<true, 2>(A.mp) : wide_smem<false, 2>(A.mp);
      if (wp.parts > 1) return wp.np == 4 ? go_wide(c4, s4) : go_wide(c2, s2);
      return wp.np == 4 ? go_wide(r4, s4) : go_wide(r2, s2);
    };
    const nk_status e =
        P.cplx ? pick(local_energy_wide<true, 4, false>, local_energy_wide<true, 2, false>,
                      local_energy_wide<true, 4, true>, local_energy_wide<true, 2, true>)
               : pick(local_energy_wide<false, 4, false>, local_energy_wide<false, 2, false>,
                      local_energy_wide<false, 4, true>, local_energy_wide<false, 2, true>);
    if (e || !P.cplx) return e;
  }
  if (!allow_smem(local_energy_tiled, P.smem))
    return fail(NK_ERR_CUDA, "nk_local_energy: shared memory attribute");
  local_energy_tiled<<<A.seg_fast ? dim3((unsigned)A.nseg, (unsigned)P.blocks)
                                  : dim3((unsigned)P.blocks, (unsigned)A.nseg),
                       256, P.smem, st>>>(P.map, A);
  return check_launch("nk_local_energy");
}

// Problems that a launch of the batch takes, started one after another.
static void batch_add(ElocBatch* B, const ElocPlan& P, int64_t ctas) {
  B->a[B->n] = P.A;
  B->map[B->n] = P.map;
  B->start[B->n + 1] = B->start[B->n] + (int)ctas;
  ++B->n;
}

// The wide form of a batch's problems, one launch per field, tile and cluster size (at
// most kElocBatch problems each).  A problem keeps the cluster size and ranges of its own
// call, which fix the order of its sums; where one CTA takes a whole tile the sums do not
// depend on the tile, and 64 configurations are taken where 128 leave SMs idle.
static nk_status launch_wide_batch(const std::vector<ElocPlan>& plans, cudaStream_t st) {
  const int n = (int)plans.size();
  int64_t c64[2] = {0, 0};  // tiles of 64 of the problems that are free to choose
  auto free_np = [&](const ElocPlan& P) { return P.wp.parts == 1 && !P.wp.ranges; };
  for (const ElocPlan& P : plans)
    if (P.wide && free_np(P)) c64[P.cplx] += (P.A.ns + 63) / 64;
  auto np_of = [&](const ElocPlan& P) {
    return free_np(P) ? (c64[P.cplx] <= 2 * 152 ? 2 : 4) : P.wp.np;
  };
  std::vector<bool> done((size_t)n, false);
  std::unique_ptr<ElocBatch> B(new ElocBatch);  // 15 KB: kept off the stack
  for (int u = 0; u < n; ++u) {
    if (done[u] || !plans[u].wide) continue;
    const bool cplx = plans[u].cplx;
    const int np = np_of(plans[u]);
    int parts = plans[u].wp.parts;
    size_t smem = 0;
    B->n = 0;
    B->start[0] = 0;
    for (int v = u; v < n && B->n < kElocBatch; ++v) {
      const ElocPlan& P = plans[v];
      if (done[v] || !P.wide || P.cplx != cplx || np_of(P) != np || P.wp.parts != parts) continue;
      done[v] = true;
      batch_add(B.get(), P, free_np(P) ? (P.A.ns + 32 * np - 1) / (32 * np) : P.wp.grid);
      smem = std::max(smem, cplx ? (np == 4 ? wide_smem<true, 4>(P.A.mp) : wide_smem<true, 2>(P.A.mp))
                                 : (np == 4 ? wide_smem<false, 4>(P.A.mp) : wide_smem<false, 2>(P.A.mp)));
    }
    const int64_t ctas = B->start[B->n];
    auto go = [&](auto kern, int64_t alone) -> nk_status {
      // few clusters: one CTA per SM (kAloneSmem)
      if (ctas / parts <= alone) smem = std::max(smem, kAloneSmem);
      if (!allow_smem(kern, smem))
        return fail(NK_ERR_CUDA, "nk_batch_local_energy: shared memory attribute");
      cudaLaunchConfig_t cfg{};
      cfg.gridDim = dim3((unsigned)ctas);
      cfg.blockDim = dim3(256);
      cfg.dynamicSmemBytes = smem;
      cfg.stream = st;
      cudaLaunchAttribute at{};
      at.id = cudaLaunchAttributeClusterDimension;
      at.val.clusterDim.x = (unsigned)parts;
      at.val.clusterDim.y = at.val.clusterDim.z = 1;
      cfg.attrs = &at;
      cfg.numAttrs = parts > 1 ? 1 : 0;
      void* args[] = {B.get(), &parts};
      if (cudaLaunchKernelExC(&cfg, (const void*)kern, args) != cudaSuccess)
        return fail(NK_ERR_CUDA, "nk_batch_local_energy: launch failed");
      return NK_OK;
    };
    auto pick = [&](auto r4, auto r2, auto c4, auto c2, int64_t alone) {
      if (parts > 1) return np == 4 ? go(c4, alone) : go(c2, alone);
      return np == 4 ? go(r4, 0) : go(r2, 0);
    };
    const nk_status e =
        cplx ? pick(local_energy_wide_batch<true, 4, false>, local_energy_wide_batch<true, 2, false>,
                    local_energy_wide_batch<true, 4, true>, local_energy_wide_batch<true, 2, true>,
                    parts > 1 ? (np == 4 ? wide_clusters<true, 4>(parts, true)
                                         : wide_clusters<true, 2>(parts, true)) : 0)
             : pick(local_energy_wide_batch<false, 4, false>, local_energy_wide_batch<false, 2, false>,
                    local_energy_wide_batch<false, 4, true>, local_energy_wide_batch<false, 2, true>,
                    parts > 1 ? (np == 4 ? wide_clusters<false, 4>(parts, true)
                                         : wide_clusters<false, 2>(parts, true)) : 0);
    if (e) return e;
  }
  return NK_OK;
}

// Fused local energies of many problems: one move-table launch for all of them, then
// one launch of the 4 x 4 form for the complex ones and of the wide form per field, tile
// and cluster size; of whole move tiles in complex problems, as in single calls, the form
// that the operator's layout is not for returns at once.  (Problems of several move tiles
// launched one after another: 48 of 72-site Ising, 256 samples each, 2140 us, here 119;
// 48 of 64-site Heisenberg, 1024 samples each, 2535, here 201.)
// Every problem runs its own launch's arithmetic and move-tile split, so the results are
// those of separate calls.
nk_status launch_local_energy_fused(const nk_eloc_item* items, const int* idx, int n,
                                    cudaStream_t st) {
  std::vector<ElocPlan> plans((size_t)n);
  for (int u = 0; u < n; ++u) {
    const nk_eloc_item& it = items[idx[u]];
    if (nk_status e = plan_local_energy(it.rbm, it.op_dev, it.n_moves, it.sigma, it.theta, it.ns,
                                        it.eloc_out, it.t_out, it.scratch, it.scratch_bytes,
                                        &plans[u]))
      return e;
  }
  for (int u0 = 0; u0 < n; u0 += kMoveJobs) {
    MoveTableBatch TB;
    TB.n = 0;
    TB.start[0] = 0;
    for (int u = u0; u < std::min(n, u0 + kMoveJobs); ++u) {
      if (plans[u].tab_elems == 0) continue;
      TB.j[TB.n] = plans[u].job;
      TB.start[TB.n + 1] = TB.start[TB.n] + plans[u].tab_elems;
      ++TB.n;
    }
    if (TB.n > 0) {
      const int64_t blocks =
          std::max<int64_t>(1, std::min<int64_t>((TB.start[TB.n] + 255) / 256, 152 * 8));
      move_tables_batch_kernel<<<(unsigned)blocks, 256, 0, st>>>(TB);
      if (nk_status e = check_launch("nk_batch_local_energy(move tables)")) return e;
    }
  }
  for (const ElocPlan& P : plans)
    if (adds_up(P) &&
        cudaMemsetAsync(P.A.eloc, 0, (size_t)P.A.ns * 2 * sizeof(double), st) != cudaSuccess)
      return fail(NK_ERR_CUDA, "nk_batch_local_energy: cudaMemsetAsync failed");
  if (nk_status e = launch_wide_batch(plans, st)) return e;
  std::unique_ptr<ElocBatch> B(new ElocBatch);
  for (int u = 0; u < n;) {
    size_t smem = 0;
    B->n = 0;
    B->start[0] = 0;
    for (; u < n && B->n < kElocBatch; ++u) {
      if (!plans[u].cplx) continue;
      batch_add(B.get(), plans[u], plans[u].blocks * plans[u].A.nseg);
      smem = std::max(smem, plans[u].smem);
    }
    if (B->n == 0) continue;
    if (!allow_smem(local_energy_batch, smem))
      return fail(NK_ERR_CUDA, "nk_batch_local_energy: shared memory attribute");
    local_energy_batch<<<(unsigned)B->start[B->n], 256, smem, st>>>(*B);
    if (nk_status e = check_launch("nk_batch_local_energy")) return e;
  }
  return NK_OK;
}

// ------------------------------------------------------------------ K4 logderiv

template <bool CPLX>
__global__ void logderiv_kernel(int n, int m, int64_t ns, const int8_t* __restrict__ sigma,
                                const void* __restrict__ theta, int layout, void* out) {
  using F = typename RatioTypes<CPLX>::F;
  const F* th = reinterpret_cast<const F*>(theta);
  F* o = reinterpret_cast<F*>(out);
  const int64_t P = (int64_t)n + m + (int64_t)n * m;
  const int64_t total = layout == NK_LAYOUT_DENSE ? ns * P : ns * m;
  for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < total;
       e += (int64_t)gridDim.x * blockDim.x) {
    F v;
    if (layout != NK_LAYOUT_DENSE) {
      F x = th[e];
      if constexpr (CPLX) {
        cf tt = tanh_c(cf{x.x, x.y});
        v = make_float2(tt.x, tt.y);
      } else {
        v = tanh_f(x);
      }
    } else {
      int64_t s = e / P, k = e % P;
      if (k < n) {
        float sv = (float)sigma[s * n + k];
        if constexpr (CPLX) v = make_float2(sv, 0.f); else v = sv;
      } else {
        int64_t kk = k - n;
        int j = (int)(kk < m ? kk : (kk - m) / n);
        float mult = kk < m ? 1.f : (float)sigma[s * n + (kk - m) % n];
        F x = th[s * m + j];
        if constexpr (CPLX) {
          cf tt = tanh_c(cf{x.x, x.y});
          v = make_float2(mult * tt.x, mult * tt.y);
        } else {
          v = mult * tanh_f(x);
        }
      }
    }
    o[e] = v;
  }
}

nk_status launch_logderiv(const nk_rbm* r, const int8_t* sigma, const void* theta, int64_t ns,
                          int layout, void* o_out, cudaStream_t st) {
  int64_t P = (int64_t)r->n + r->m + (int64_t)r->n * r->m;
  int64_t total = layout == NK_LAYOUT_DENSE ? ns * P : ns * r->m;
  int64_t blocks = std::min<int64_t>((total + 255) / 256, 152 * 16);
  if (blocks < 1) blocks = 1;
  if (r->is_complex)
    logderiv_kernel<true><<<(unsigned)blocks, 256, 0, st>>>(r->n, r->m, ns, sigma, theta, layout,
                                                           o_out);
  else
    logderiv_kernel<false><<<(unsigned)blocks, 256, 0, st>>>(r->n, r->m, ns, sigma, theta, layout,
                                                            o_out);
  return check_launch("nk_logderiv");
}

NK_STATUS_COLLECTOR(collect_status_local_energy)

}  // namespace nk
