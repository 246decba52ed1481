// Norm bound of Sec. 3.4 (Theorem 2, Algorithm 2 steps 1-2) and the scaled
// cast X_0 = X / lam~ (Algorithm 2 step 3).
//
// Lanczos on A = X^2 (Parlett, The Symmetric Eigenvalue Problem, Ch. 13):
// 20 steps, A q = X (X q), Lanczos vectors and all recurrences in FP64: the
// three-term recurrence, then full re-orthogonalisation (one classical
// Gram-Schmidt pass), then the
// largest Ritz pair (sigma, q) of the tridiagonal T_m and
//     lam~ = sqrt(sigma + ||X (X q) - sigma q||_2),
// raised to max(lam~, ||X||_F / sqrt(n), max_i |X_ii|) (both lower bounds of
// ||X||_2; they only matter when the start vector misses the top eigenvector).
//
// The mat-vec reads only the upper triangle of the FP32 input, once per
// product (an HBM-bound pass of n^2/2 words), in 128 x 128 tiles: each tile
// adds its rows' dot products (X(i,j) v_j, i <= j) and its columns' dot
// products (X(i,j) v_i, i < j) into per-tile partial sums, reduced afterwards
// in a fixed order (deterministic).  GB300's FP64 pipe is narrow, so the
// element level runs in FP32: each thread forms 8-term FP32 FMA sums, which
// are combined exactly into double-float (FP32 pair) partial sums with the
// TwoSum error-free transformation (Knuth; Ogita, Rump & Oishi, "Accurate sum
// and dot product", SIAM J. Sci. Comput. 2005), converted to FP64 per vector
// element.  A mat-vec is thus accurate to a few FP32 roundings of the 8-term
// runs (~1e-7 relative); the recurrences and the re-orthogonalisation are FP64,
// the dot products and norms that feed them double-float (FP32 pairs, ~48
// bits), all in a fixed order.
#include <cuda_bf16.h>
#include <cuda_fp16.h>

#include <algorithm>
#include <cmath>
#include <map>
#include <mutex>
#include <tuple>
#include <type_traits>

#include "epilogue.cuh"
#include "internal.h"
#include "normbound.cuh"
#include "ptx.cuh"
#include "tridiag.cuh"

namespace psd {

namespace {

// Host-side fault injection (psd_debug_set): a factor applied to lam~ (1.0:
// none; a factor below 1 drives the chain past the composite's basin and
// exercises the overshoot report) and the limit of the grid barriers' waits
// (0: every barrier that is not already complete gives up at once and the
// bound returns PSD_ERR_TIMEOUT; the cluster form, whose barriers are the
// hardware's, takes up the limit 0 only).  Read by the kernels at run time, so
// captured graphs see the current values.
__device__ double g_debug_bound_scale = 1.0;
__device__ unsigned long long g_debug_barrier_limit_ns = kWaitLimitNs;

// ------------------------------------------------------------------ phases
//
// Every phase of the norm bound is a device function over virtual blocks of
// kNT = 256 threads.  It runs either as the body of its own kernel (one CTA
// per virtual block: the multi-launch path, kNormBoundLaunches per bound) or inside
// one persistent cooperative kernel whose CTAs take virtual blocks
// blockIdx.x, blockIdx.x + gridDim.x, ... between grid-wide barriers.  Both
// execute the same arithmetic in the same order and give the same bits.
// Vectors an earlier phase wrote are read with ld.global.cg (through L2): in
// the persistent kernel they change while it runs, which the non-coherent
// read-only path must not be used for.
static_assert(kVecThreads == kNT, "vector phases: one element per thread of a 256-thread block");

// Shared memory of one CTA, reused by the phases (each virtual block ends
// with a barrier before the next one writes it again).
struct NBShared {
  union {
    struct {
      float2 red[2][8][kRedStride];  // two buffers: consecutive tiles of a run alternate
      double fro[8];
    } mv;
    float2 part[8][32];
    struct {
      float2 s[32];
    } orth;
    struct {
      double y[kMaxSteps];
      float a[kMaxSteps], b[kMaxSteps];
    } tri;
  } u;
  double bs[8];  // block_sum64 (apart from u: a phase may still read u.orth.h when a warp enters it)
  double scalar[2];
};

// Everything the phases read: sizes, the argument block, state and buffers.
struct NBCtx {
  int n, nb, ntiles, nv, npart;
  int64_t npad;
  const DevArgs* args;
  DevState* st;
  double *Qv, *w, *q, *zsave;
  float2* Qf;            // Lanczos vectors as double-float pairs (for the dot products), kMaxSteps x npad
  float* vh;             // mat-vec input (the vector rounded to FP32)
  float2 *P1, *P2;
  float2* dots;          // per chunk: 32 double-float partials (dot products, slot 31 ||w'||^2)
  double* norms;         // per 256-element block: FP64 partial of ||q_0||^2
  float2* norms2;        // per chunk: double-float partial of a squared norm (same storage as norms)
  double* tile_fro;
  float4* pack;          // room for the packed tiles, or null
};

// Block-wide FP64 sum of one value per thread (kNT threads), fixed order;
// every thread receives the sum.
__device__ __forceinline__ double block_sum64(double v, double* sh) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  const int w = threadIdx.x >> 5;
  if ((threadIdx.x & 31) == 0) sh[w] = v;
  __syncthreads();
  double s = 0.0;
  for (int k = 0; k < kNT / 32; ++k) s += sh[k];
  __syncthreads();
  return s;
}

// Fixed-order warp sum of cnt FP64 values (lane-strided, then a butterfly).
// Each lane's values are loaded 8 at a time before they are added (in order):
// the sums are L2-latency chains otherwise.
__device__ __forceinline__ double warp_sum_array(const double* a, int cnt, int stride) {
  const int lane = threadIdx.x & 31;
  double s = 0.0;
  for (int c0 = 0; c0 < cnt; c0 += 8 * 32) {
    double t[8];
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      const int c = c0 + 32 * i + lane;
      t[i] = c < cnt ? __ldcg(a + static_cast<int64_t>(c) * stride) : 0.0;
    }
#pragma unroll
    for (int i = 0; i < 8; ++i)
      if (c0 + 32 * i + lane < cnt) s += t[i];
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
  return s;
}

// The thread's 8-element slices of v: rows (vi) and columns (vj); zeros past n.
// vh holds npad (a multiple of 256) floats and the slices start at multiples of 8.
__device__ __forceinline__ void tile_load_v(int n, const TileGeom& g, const float* vh, float (&vi)[8],
                                            float (&vj)[8]) {
  const float4 a0 = __ldcg(reinterpret_cast<const float4*>(vh + g.ib));
  const float4 a1 = __ldcg(reinterpret_cast<const float4*>(vh + g.ib) + 1);
  const float4 b0 = __ldcg(reinterpret_cast<const float4*>(vh + g.jb));
  const float4 b1 = __ldcg(reinterpret_cast<const float4*>(vh + g.jb) + 1);
  const float a[8] = {a0.x, a0.y, a0.z, a0.w, a1.x, a1.y, a1.z, a1.w};
  const float b[8] = {b0.x, b0.y, b0.z, b0.w, b1.x, b1.y, b1.z, b1.w};
#pragma unroll
  for (int k = 0; k < 8; ++k) {
    vi[k] = g.ib + k < n ? a[k] : 0.f;
    vj[k] = g.jb + k < n ? b[k] : 0.f;
  }
}

// Tile `t` = (bi, bj)'s results in global memory: row partials P1[bj][rows],
// column partials P2[bi][columns], ||X||_F^2 share, max |X_ii|.
struct GlobalSink {
  const NBCtx& c;
  const TileGeom& g;
  int tile;
  __device__ __forceinline__ void row(int i, float2 v) const { c.P1[static_cast<int64_t>(g.bj) * c.npad + i] = v; }
  __device__ __forceinline__ void col(int j, float2 v) const { c.P2[static_cast<int64_t>(g.bi) * c.npad + j] = v; }
  __device__ __forceinline__ void diag(unsigned m) const { atomicMax(&c.st->maxdiag_bits, m); }
  __device__ __forceinline__ void fro(double f) const { c.tile_fro[tile] = f; }
};

// Tile t of a product over X (t in [0, ntiles)), one tile per call.
template <bool STATS>
__device__ __forceinline__ void ph_symv(const NBCtx& c, const float* X, int64_t ld, int t, NBShared& sh) {
  const TileGeom g = tile_geom(t);
  float vi[8], vj[8], x[8][8], rsum[8], csum[8], fro;
  unsigned mdiag;
  tile_load_v(c.n, g, c.vh, vi, vj);
  tile_load_x(X, ld, c.n, g, x);
  tile_fma_reg<STATS>(c.n, g, vi, vj, x, rsum, csum, fro, mdiag);
  tile_reduce<STATS>(c.n, g, rsum, csum, fro, mdiag, sh.u.mv.red[0], sh.u.mv.fro, GlobalSink{c, g, t}, true);
}

// Tiles r = first, first + stride, ... < ntiles of a product (in the
// opposite order of the tile list if `rev`), each loaded while the previous
// one is reduced: the same arithmetic per tile as ph_symv.  The caller ends
// the run with a CTA barrier (the grid barrier after the phase).
// pack: the first product (STATS) also stores the tiles there, each thread's 16
// float4 at [tile][q][thread], and the later ones read them from there; null:
// all products read X.
template <bool STATS>
__device__ __forceinline__ void ph_symv_run(const NBCtx& c, const float* X, int64_t ld, float4* pack, int first,
                                            int stride, bool rev, NBShared& sh) {
  if (first >= c.ntiles) return;
  auto tile_at = [&](int r) { return rev ? c.ntiles - 1 - r : r; };
  float vi[8], vj[8], x[8][8];
  int r = first;
  int buf = 0;
  TileGeom g = tile_geom(tile_at(r));
  auto load_x = [&](int tile, const TileGeom& tg) {
    float4* p = pack ? pack + static_cast<int64_t>(tile) * (16 * kNT) + threadIdx.x : nullptr;
    if (STATS || !pack) {
      tile_load_x(X, ld, c.n, tg, x);
      if (STATS && pack) {
#pragma unroll
        for (int k = 0; k < 8; ++k) {
          p[kNT * (2 * k)] = make_float4(x[k][0], x[k][1], x[k][2], x[k][3]);
          p[kNT * (2 * k + 1)] = make_float4(x[k][4], x[k][5], x[k][6], x[k][7]);
        }
      }
    } else {
#pragma unroll
      for (int k = 0; k < 8; ++k) {
        const float4 a = __ldcg(p + kNT * (2 * k)), b = __ldcg(p + kNT * (2 * k + 1));
        x[k][0] = a.x; x[k][1] = a.y; x[k][2] = a.z; x[k][3] = a.w;
        x[k][4] = b.x; x[k][5] = b.y; x[k][6] = b.z; x[k][7] = b.w;
      }
    }
  };
  tile_load_v(c.n, g, c.vh, vi, vj);
  load_x(tile_at(r), g);
  while (true) {
    float rsum[8], csum[8], fro;
    unsigned mdiag;
    tile_fma_reg<STATS>(c.n, g, vi, vj, x, rsum, csum, fro, mdiag);
    const int rn = r + stride;
    const TileGeom gn = tile_geom(tile_at(rn < c.ntiles ? rn : r));
    if (rn < c.ntiles) {  // in flight during the reduction
      tile_load_v(c.n, gn, c.vh, vi, vj);
      load_x(tile_at(rn), gn);
    }
    tile_reduce<STATS>(c.n, g, rsum, csum, fro, mdiag, sh.u.mv.red[buf], sh.u.mv.fro, GlobalSink{c, g, tile_at(r)},
                       false);
    if (rn >= c.ntiles) break;
    r = rn;
    g = gn;
    buf ^= 1;
  }
}

// The product over a CTA's resident tiles: tile b0 in registers (x, geometry
// g), tile b0 + stride (if any; g1) in shared memory, each thread's own 16 float4
// of it at xs[256 q + thread] (read and written by that thread only).
template <bool STATS>
__device__ __forceinline__ void ph_symv_resident(const NBCtx& c, int b0, int stride, const TileGeom& g,
                                                 const TileGeom& g1, const float (&x)[8][8], const float4* xs,
                                                 NBShared& sh) {
  if (b0 >= c.ntiles) return;
  float vi[8], vj[8], rsum[8], csum[8], fro;
  unsigned mdiag;
  tile_load_v(c.n, g, c.vh, vi, vj);
  tile_fma_reg<STATS>(c.n, g, vi, vj, x, rsum, csum, fro, mdiag);
  const int t1 = b0 + stride;
  if (t1 < c.ntiles) tile_load_v(c.n, g1, c.vh, vi, vj);
  tile_reduce<STATS>(c.n, g, rsum, csum, fro, mdiag, sh.u.mv.red[0], sh.u.mv.fro, GlobalSink{c, g, b0}, false);
  if (t1 >= c.ntiles) return;
  auto col = [&](int k, float (&o)[8]) {
    const float4 a = xs[kNT * (2 * k) + threadIdx.x], b = xs[kNT * (2 * k + 1) + threadIdx.x];
    o[0] = a.x; o[1] = a.y; o[2] = a.z; o[3] = a.w;
    o[4] = b.x; o[5] = b.y; o[6] = b.z; o[7] = b.w;
  };
  tile_fma<STATS>(c.n, g1, vi, vj, col, rsum, csum, fro, mdiag);
  tile_reduce<STATS>(c.n, g1, rsum, csum, fro, mdiag, sh.u.mv.red[1], sh.u.mv.fro, GlobalSink{c, g1, t1}, false);
}

// State reset and the start vector q_0 (unit SplitMix64 vector, before scaling).
__device__ __forceinline__ void ph_init(const NBCtx& c, int vb, NBShared& sh) {
  const int e = vb * kNT + threadIdx.x;
  double v = 0.0;
  if (e < c.n) v = lanczos_start(e);
  const double s = block_sum64(v * v, sh.bs);
  if (threadIdx.x == 0) c.norms[vb] = s;
  if (e < c.n) c.Qv[e] = v;  // unnormalised; ph_norm0 scales it
  if (vb == 0 && threadIdx.x == 0) {
    DevState* st = c.st;
    st->m = 0;
    st->done = 0;
    st->status = 0;
    st->maxdiag_bits = 0;
    st->absmax_bits = 0;
    st->sigma = st->resid = st->lambda = st->fro = st->maxdiag = st->inv_lambda = 0.0;
  }
}

// Broadcast of a value computed by warp 0 (slot k of the CTA's scalars).
__device__ __forceinline__ double bcast(double v, NBShared& sh, int k) {
  if (threadIdx.x == 0) sh.scalar[k] = v;
  __syncthreads();
  const double r = sh.scalar[k];
  __syncthreads();
  return r;
}

// Element e of Lanczos vector k: FP64, double-float pair and mat-vec input.
__device__ __forceinline__ void put_lanczos(const NBCtx& c, int k, int e, double q) {
  const float2 p = d_to_f2(q);
  c.Qv[static_cast<int64_t>(k) * c.npad + e] = q;
  c.Qf[static_cast<int64_t>(k) * c.npad + e] = p;
  c.vh[e] = p.x;
}

// q_0 /= ||v||, split.
__device__ __forceinline__ void ph_norm0(const NBCtx& c, int vb, NBShared& sh) {
  double s = 0.0;
  if (threadIdx.x < 32) s = warp_sum_array(c.norms, c.nv, 1);
  if (threadIdx.x == 0) s = 1.0 / sqrt(s);  // FP64 scalar work in one thread
  const double inv = bcast(s, sh, 0);
  const int e = vb * kNT + threadIdx.x;
  if (e < c.n) {
    put_lanczos(c, 0, e, __ldcg(c.Qv + e) * inv);
  }
}

// ||X||_F from the per-tile sums of the first product (one warp, fixed order).
__device__ __forceinline__ void ph_fro(const NBCtx& c) {
  const double f = warp_sum_array(c.tile_fro, c.ntiles, 1);
  if (threadIdx.x == 0) c.st->fro = sqrt(f);
}

// The chunk-reducing phases take two chunks per CTA at once, one per half
// of the CTA (warps 0-3 and 4-7): a chunk pair index cp covers chunks 2 cp and
// 2 cp + 1.  With one chunk per CTA, orders just above 32 x the CTA count
// (n = 10,000: 313 chunks, 304 CTAs) left a few CTAs a second chunk and the
// whole phase waiting for them.
__device__ __forceinline__ int chunk_of_half(int cp) { return 2 * cp + static_cast<int>(threadIdx.x >> 7); }
__device__ __forceinline__ bool half_lead_warp() { return (threadIdx.x & 127) < 32; }

// y_e = sum_{bj >= b(e)} P1[bj][e] + sum_{bi <= b(e)} P2[bi][e] for the 32
// elements e of chunk `ch`, by the 4 warps of this thread's half of the CTA:
// warp h (0-3 in the half) adds the blocks congruent to h mod 4 in
// double-float, then the half's first warp combines the 4 warp sums in a fixed
// order.  Returns y_e (a normalised pair) in that warp; other warps return 0.  Both halves
// call it together (CTA barriers).
__device__ __forceinline__ F2 reduce_partials(const NBCtx& c, int ch, NBShared& sh) {
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, hw = w & 3;
  const int e = ch * 32 + lane;
  F2 a{0.f, 0.f}, d{0.f, 0.f};
  if (e < c.n) {
    // P1 of bj = b + hw, + 4, ... then P2 of bi = hw, + 4, ... <= b: about (nb + 1) / 4
    // entries, ten loads in flight (a loop unrolled over a few entries waits for
    // the loads of its remainder one by one): the bound at n = 2000 417 -> 389 us,
    // 4096 578 -> 546, 10000 2042 -> 1981, and unchanged where one cluster runs it
    const int b = e / kSymvTile;
    const int c1 = (c.nb - b - hw + 3) / 4, c2 = (b - hw + 4) / 4, cnt = c1 + c2;
    for (int i0 = 0; i0 < cnt; i0 += 10) {
      float2 p[10];
#pragma unroll
      for (int k = 0; k < 10; ++k) {
        const int i = i0 + k;
        const float2* at = i < c1 ? c.P1 + static_cast<int64_t>(b + hw + 4 * i) * c.npad
                                  : c.P2 + static_cast<int64_t>(hw + 4 * (i - c1)) * c.npad;
        p[k] = i < cnt ? __ldcg(at + e) : make_float2(0.f, 0.f);
      }
#pragma unroll
      for (int k = 0; k < 10; ++k) {
        if (i0 + k < c1)
          a = f2_add(a, F2{p[k].x, p[k].y});
        else if (i0 + k < cnt)
          d = f2_add(d, F2{p[k].x, p[k].y});
      }
    }
  }
  const F2 t = f2_add(a, d);
  sh.u.part[w][lane] = make_float2(t.h, t.l);
  __syncthreads();
  F2 y{0.f, 0.f};
  if (hw == 0) {
    F2 acc{sh.u.part[w][lane].x, sh.u.part[w][lane].y};
#pragma unroll
    for (int q = 1; q < 4; ++q) acc = f2_add(acc, F2{sh.u.part[w + q][lane].x, sh.u.part[w + q][lane].y});
    y = f2_norm(acc);
  }
  __syncthreads();
  return y;
}

// u = X v (first product of X (X v)): the second product's input, the chunk's
// share of ||u||^2 (= alpha_j, q_j being a unit vector), and u itself if asked
// for.  Chunk pair cp.
__device__ __forceinline__ void ph_reduce_split(const NBCtx& c, int cp, double* u, NBShared& sh) {
  const int ch = chunk_of_half(cp);
  const F2 y = reduce_partials(c, ch, sh);
  if (!half_lead_warp() || ch >= c.npart) return;
  const int e = ch * 32 + (threadIdx.x & 31);
  if (e < c.n) {
    if (u) u[e] = f2_to_d(y);
    c.vh[e] = y.h;
  }
  const F2 t = warp_sum_f2(f2_mul(y, y));  // y is 0 past n
  if ((threadIdx.x & 31) == 0) c.norms2[ch] = make_float2(t.h, t.l);
}

// ---- Lanczos step j after the second product: w = X u, the three-term
// recurrence, one full Gram-Schmidt pass and q_{j+1}.
//
// alpha_j = q_j . X u = ||u||^2 is known from the first product, so the
// recurrence w' = w - alpha_j q_j - beta_{j-1} q_{j-1} is applied as soon as w
// is reduced.  In exact arithmetic w' is orthogonal to every Lanczos vector; in
// this one its components along them are at the mat-vec's rounding level, and a
// single Gram-Schmidt pass over all of them takes those out down to the FP64
// rounding of w' (two passes are only needed where the first cancels most of
// the vector).  The pass's coefficient along q_j is added to alpha_j.  Two
// passes on w itself took a phase and a grid barrier more per step.
//
// Element work is done per chunk of 32 elements by one warp (lane =
// element): the vectors and their updates in FP64, the dot products (q_k . w'
// and ||w'||^2) and their sums over the chunks as double-float pairs (FP32 hi +
// lo, about 48 bits), because this GPU issues FP64 at a small fraction of its
// FP32 rate.  Every CTA adds the chunks' partials itself, in the same order.

// w' = w - alpha_j q_j - beta_{j-1} q_{j-1}; the chunk's shares of q_k . w'
// (k <= j) and ||w'||^2 (slot 31) into dots.  Chunk pair cp.
__device__ __forceinline__ void ph_reduce_dots(const NBCtx& c, int cp, int j, NBShared& sh) {
  const int ch = chunk_of_half(cp);
  const int lane = threadIdx.x & 31;
  const int e = ch * 32 + lane;
  const bool lead = half_lead_warp() && ch < c.npart;
  // alpha_j by a warp of the other half of the CTA's work; loads before the partial sums'
  if (threadIdx.x >= 32 && threadIdx.x < 64) {
    const double a = warp_sum_chunks(c.norms2, c.npart, LoadCg());
    if (lane == 0) sh.scalar[0] = a;
  }
  float2 qf[kMaxSteps];
  double beta = 0.0, qj = 0.0, qp = 0.0;
#pragma unroll
  for (int k = 0; k < kMaxSteps; ++k)
    qf[k] = (lead && k <= j && e < c.n) ? __ldcg(c.Qf + static_cast<int64_t>(k) * c.npad + e) : make_float2(0.f, 0.f);
  if (lead && e < c.n) qj = __ldcg(c.Qv + static_cast<int64_t>(j) * c.npad + e);
  if (lead && j > 0) {
    beta = __ldcg(&c.st->beta[j - 1]);
    if (e < c.n) qp = __ldcg(c.Qv + static_cast<int64_t>(j - 1) * c.npad + e);
  }
  const F2 y = reduce_partials(c, ch, sh);  // its barriers publish sh.scalar[0]
  const double alpha = sh.scalar[0];
  if (cp == 0 && threadIdx.x == 0) c.st->alpha[j] = alpha;
  if (!lead) return;
  const double w = lanczos_recur(f2_to_d(y), alpha, qj, beta, qp);
  if (e < c.n) c.w[e] = w;
  c.dots[static_cast<int64_t>(lane) * c.npart + ch] =
      chunk_dots(f2_of(e < c.n ? w : 0.0), j, [&](int k) { return F2{qf[k].x, qf[k].y}; });
}

// The Gram-Schmidt pass and the next Lanczos vector.  Every CTA sums the
// chunks' dots h and ||w'||^2; w'' = w' - Q h is orthogonal to Q and (Q
// orthonormal) ||w''||^2 = ||w'||^2 - ||h||^2, so beta_j = ||w''|| needs no
// further reduction (h is at the mat-vec's rounding level: no cancellation
// until w' itself is down there).  Stops on breakdown (beta_j <= 1e-12
// ||X||_F^2) or after the last step; otherwise q_{j+1} = w'' / beta_j per chunk.
// The chunks' warps form w'' (four independent chains: an FP64 operation's
// latency is 64 cycles) while the last warp forms beta_j.  Returns `stop` (the
// same in every CTA).
__device__ __forceinline__ bool ph_orth_next(const NBCtx& c, int cta, int ncta, int j, NBShared& sh) {
  const int lane = threadIdx.x & 31, wp = threadIdx.x >> 5;
  constexpr int kW = kNT / 32;
  const int ch0 = cta + ncta * wp;  // most CTAs have one chunk, on warp 0
  const double fro = __ldcg(&c.st->fro);
  chunk_sums(c.dots, c.npart, c.npart, j, sh.u.orth.s, LoadCg());
  __syncthreads();
  if (wp == kW - 1) beta_of_sums(sh.u.orth.s, j, sh.scalar);
  const double h = ch0 < c.npart && lane <= j ? f2_to_d(F2{sh.u.orth.s[lane].x, sh.u.orth.s[lane].y}) : 0.0;
  auto next = [&](int ch) {  // w'' of the lane's element
    const int e = ch * 32 + lane;
    double qk[kMaxSteps];
#pragma unroll
    for (int k = 0; k < kMaxSteps; ++k)
      qk[k] = (k <= j && e < c.n) ? __ldcg(c.Qv + static_cast<int64_t>(k) * c.npad + e) : 0.0;
    return lanczos_orth(e < c.n ? __ldcg(c.w + e) : 0.0, h, qk, j);
  };
  const double w0 = ch0 < c.npart ? next(ch0) : 0.0;
  __syncthreads();
  const double beta = sh.scalar[0];
  const bool stop = !(beta > kBreakdown * (fro * fro)) || j == kMaxSteps - 1;  // also true for NaN
  if (cta == 0 && threadIdx.x == 0) {
    c.st->alpha[j] = __ldcg(&c.st->alpha[j]) + f2_to_d(F2{sh.u.orth.s[j].x, sh.u.orth.s[j].y});
    c.st->beta[j] = beta;
    c.st->m = j + 1;
    if (stop) c.st->done = j + 1;
  }
  if (!stop) {
    const double inv = sh.scalar[1];
    auto put = [&](int ch, double w) {
      const int e = ch * 32 + lane;
      if (e >= c.n) return;
      put_lanczos(c, j + 1, e, w * inv);
    };
    if (ch0 < c.npart) put(ch0, w0);
    for (int ch = ch0 + ncta * kW; ch < c.npart; ch += ncta * kW) put(ch, next(ch));
  }
  __syncthreads();
  return stop;
}

// Largest eigenpair of the Lanczos tridiagonal (tridiag.cuh): sigma and the
// Ritz vector's coordinates y in the Lanczos basis.  One warp.
__device__ __forceinline__ void ph_tridiag(const NBCtx& c, NBShared& sh) {
  DevState* st = c.st;
  // alpha, beta and m were written by thread 0 of this CTA (persistent kernel)
  // or by earlier kernels: plain loads
  const int m = *reinterpret_cast<volatile int*>(&st->m);
  const double sigma = tridiag_top_eig(st->alpha, st->beta, m, sh.u.tri.y, sh.u.tri.a, sh.u.tri.b);
  if (threadIdx.x == 0) {
    st->sigma = sigma;
    for (int k = 0; k < kMaxSteps; ++k) st->y[k] = sh.u.tri.y[k];
  }
}

// q = sum_k y_k q_k per chunk (one warp), partial ||q||^2 into norms[ch] (double-float).
__device__ __forceinline__ void ph_ritz(const NBCtx& c, int cta, int ncta, NBShared& sh) {
  (void)sh;
  const int m = __ldcg(&c.st->m);
  const int lane = threadIdx.x & 31, wp = threadIdx.x >> 5;
  for (int ch = cta + ncta * wp; ch < c.npart; ch += ncta * (kNT / 32)) {
    const int e = ch * 32 + lane;
    double s = 0.0;
    if (e < c.n) {
      double qk[kMaxSteps], yk[kMaxSteps];
#pragma unroll
      for (int k = 0; k < kMaxSteps; ++k) {
        qk[k] = k < m ? __ldcg(c.Qv + static_cast<int64_t>(k) * c.npad + e) : 0.0;
        yk[k] = k < m ? __ldcg(&c.st->y[k]) : 0.0;
      }
      s = lanczos_ritz(yk, qk, m);
      c.q[e] = s;
    }
    const F2 t = warp_sum_f2(f2_of(s * s));
    if (lane == 0) c.norms2[ch] = make_float2(t.h, t.l);
  }
}

// 1 / sqrt of the sum of the chunks' double-float partials norms2[0 .. npart)
// (fixed order; 0 for a zero sum); every thread of the CTA receives it.
__device__ __forceinline__ double inv_norm_of_sum(const NBCtx& c, NBShared& sh) {
  if (threadIdx.x < 32) {
    const double s2 = warp_sum_chunks(c.norms2, c.npart, LoadCg());
    if (threadIdx.x == 0) sh.scalar[0] = s2 > 0.0 ? 1.0 / sqrt(s2) : 0.0;
  }
  __syncthreads();
  const double r = sh.scalar[0];
  __syncthreads();
  return r;
}

// q /= ||q|| (inv = 1 / ||q||), split for the residual products.
__device__ __forceinline__ void ph_ritz_norm(const NBCtx& c, int vb, double inv) {
  const int e = vb * kNT + threadIdx.x;
  if (e < c.n) {
    const double v = __ldcg(c.q + e) * inv;
    c.q[e] = v;
    c.vh[e] = __double2float_rn(v);
  }
}

// r = X (X q) - sigma q, partial ||r||^2 of the chunk into norms2[ch].
__device__ __forceinline__ void ph_resid(const NBCtx& c, int cp, NBShared& sh) {
  const int ch = chunk_of_half(cp);
  const F2 y = reduce_partials(c, ch, sh);
  if (!half_lead_warp() || ch >= c.npart) return;
  const int lane = threadIdx.x & 31;
  const int e = ch * 32 + lane;
  double r = 0.0;
  if (e < c.n) r = fma(-__ldcg(&c.st->sigma), __ldcg(c.q + e), f2_to_d(y));
  const F2 t = warp_sum_f2(f2_of(r * r));
  if (lane == 0) c.norms2[ch] = make_float2(t.h, t.l);
}

// lam~ = max(sqrt(sigma + r), ||X||_F / sqrt n, max |X_ii|) times `scale` (1.0
// unless a test injects a bound that is too small) into the state and the
// report.  One thread; r2 = r^2.
__device__ void record_bound(DevState* st, psd_info_t* info, int n, double r2, double fro, double md, double sigma,
                             int m, double scale) {
  const double r = sqrt(r2);
  const double fro2 = fro * fro;
  double lam = sqrt(fmax(sigma + r, 0.0));
  lam = fmax(lam, fro / sqrt(static_cast<double>(n)));
  lam = fmax(lam, md);
  lam *= scale;
  st->resid = r;
  st->maxdiag = md;
  const bool finite = isfinite(fro2) && isfinite(lam) && isfinite(sigma);
  if (!finite) {
    atomicCAS(&st->status, 0, PSD_ERR_NONFINITE);
    lam = 0.0;
  }
  st->lambda = lam;
  st->inv_lambda = lam > 0.0 ? 1.0 / lam : 0.0;
  if (info) {
    info->lambda_bound = lam;
    info->lanczos_sigma = sigma;
    info->lanczos_resid = r;
    info->fro_X = fro;
    info->max_diag = md;
    info->lanczos_steps = m;
    info->status = __ldcg(&st->status);
    info->compl_resid = __longlong_as_double(0x7ff8000000000000ll);  // set by a projection's last step
  }
}

// The bound from the residual's partials.  One warp.
__device__ __forceinline__ void ph_final(const NBCtx& c) {
  const double r2 = warp_sum_chunks(c.norms2, c.npart, LoadCg());
  if (threadIdx.x != 0) return;
  DevState* st = c.st;
  record_bound(st, c.args->info, c.n, r2, __ldcg(&st->fro),
               static_cast<double>(__uint_as_float(__ldcg(&st->maxdiag_bits))), __ldcg(&st->sigma), __ldcg(&st->m),
               g_debug_bound_scale);
}

// ------------------------------------------------- multi-launch kernels
// One CTA per virtual block; `skip` kernels of Lanczos step j >= 1 return at
// once after a breakdown (the state's `done`).
__global__ void __launch_bounds__(kNT) nb_init_kernel(NBCtx c) {
  __shared__ NBShared sh;
  ph_init(c, blockIdx.x, sh);
}
__global__ void __launch_bounds__(kNT) nb_norm0_kernel(NBCtx c) {
  __shared__ NBShared sh;
  ph_norm0(c, blockIdx.x, sh);
}
// `reverse` deals the tiles to the CTAs in the opposite order: consecutive
// products over the same X alternate direction, so each starts on the tiles
// the previous one read last, which are still in L2.  The tile -> partial slot
// mapping does not depend on the order: results are identical.
template <bool STATS>
__global__ void __launch_bounds__(kNT, 2) nb_symv_kernel(NBCtx c, int skip, int reverse) {
  if (skip && c.st->done) return;
  __shared__ NBShared sh;
  const int t = reverse ? c.ntiles - 1 - static_cast<int>(blockIdx.x) : static_cast<int>(blockIdx.x);
  ph_symv<STATS>(c, c.args->X, c.args->ld, t, sh);
}
__global__ void nb_fro_kernel(NBCtx c) { ph_fro(c); }
__global__ void __launch_bounds__(kNT) nb_reduce_split_kernel(NBCtx c, double* u, int skip) {
  if (skip && c.st->done) return;
  __shared__ NBShared sh;
  ph_reduce_split(c, blockIdx.x, u, sh);
}
__global__ void __launch_bounds__(kNT) nb_reduce_dots_kernel(NBCtx c, int j) {
  if (c.st->done) return;
  __shared__ NBShared sh;
  ph_reduce_dots(c, blockIdx.x, j, sh);
}
__global__ void __launch_bounds__(kNT) nb_orth_kernel(NBCtx c, int j) {
  // `done` is j + 1 once step j stopped: set by this very launch in the last step,
  // while CTAs of it may still be starting -- they must not take it for an earlier
  // step's, some warps before and some after it is set
  const int done = c.st->done;
  if (done != 0 && done <= j) return;
  __shared__ NBShared sh;
  ph_orth_next(c, blockIdx.x, gridDim.x, j, sh);
}
__global__ void nb_tridiag_kernel(NBCtx c) {
  __shared__ NBShared sh;
  ph_tridiag(c, sh);
}
__global__ void __launch_bounds__(kNT) nb_ritz_kernel(NBCtx c) {
  __shared__ NBShared sh;
  ph_ritz(c, blockIdx.x, gridDim.x, sh);
}
__global__ void __launch_bounds__(kNT) nb_ritz_norm_kernel(NBCtx c) {
  __shared__ NBShared sh;
  ph_ritz_norm(c, blockIdx.x, inv_norm_of_sum(c, sh));
}
__global__ void __launch_bounds__(kNT) nb_resid_kernel(NBCtx c) {
  __shared__ NBShared sh;
  ph_resid(c, blockIdx.x, sh);
}
__global__ void nb_final_kernel(NBCtx c) { ph_final(c); }

// ----------------------------------------------------- persistent kernel
__device__ __forceinline__ unsigned long long ld_acquire_u64(const unsigned long long* p) {
  unsigned long long v;
  asm volatile("ld.acquire.gpu.global.u64 %0, [%1];" : "=l"(v) : "l"(p) : "memory");
  return v;
}
__device__ __forceinline__ void red_release_add_u32(unsigned* p, unsigned v) {
  asm volatile("red.release.gpu.global.add.u32 [%0], %1;" ::"l"(p), "r"(v) : "memory");
}

// Grid-wide barrier of a cooperative launch: every CTA adds 1 to sync[0]
// (zeroed before the launch) with release semantics, which the CTA barrier in
// front extends to all its threads' writes; the k-th barrier is passed when it
// reaches k * gridDim.x.  A poll is one 64-bit acquire load of the count and
// the abort word sync[1] next to it; the clock is read on every 32nd poll only.
// The wait is bounded: after the limit the CTA raises PSD_ERR_TIMEOUT and
// sync[1], and every CTA that sees sync[1] leaves the kernel at its next
// barrier.  Thread 0 keeps the count of barriers.
struct GridBarrier {
  unsigned* sync;  // 8-byte aligned
  unsigned long long limit;
  unsigned epoch;
  __device__ __forceinline__ bool wait(int* status, volatile int* ok_sh) {
    __syncthreads();
    if (threadIdx.x == 0) {
      ++epoch;
      const unsigned target = epoch * gridDim.x;
      red_release_add_u32(sync, 1u);
      int ok = 1;
      unsigned long long t0 = 0;
      for (unsigned poll = 0;; ++poll) {
        const unsigned long long v = ld_acquire_u64(reinterpret_cast<const unsigned long long*>(sync));
        if (static_cast<unsigned>(v) >= target) break;
        if (static_cast<unsigned>(v >> 32) != 0u) {
          // another CTA gave up; record it too: the first phase resets the
          // status word in CTA 0, which may run after that CTA's record, and
          // every CTA (CTA 0 included) leaves through a barrier after its own
          // first phase
          atomicCAS(status, 0, PSD_ERR_TIMEOUT);
          ok = 0;
          break;
        }
        if ((poll & 31u) == 0u) {
          const unsigned long long now = globaltimer_ns();
          if (poll == 0u) t0 = now;
          if (now - t0 >= limit) {  // >=: a zero limit gives up on the first poll
            atomicExch(sync + 1, 1u);
            atomicCAS(status, 0, PSD_ERR_TIMEOUT);
            ok = 0;
            break;
          }
        }
      }
      *ok_sh = ok;
    }
    __syncthreads();
    return *ok_sh != 0;
  }
};

// The whole bound in one launch: the phases of the multi-launch path in the
// same order, separated by grid barriers instead of kernel boundaries (108 of
// them, each a few microseconds shorter than a kernel boundary, and no
// launch of a small FP64 vector kernel waits on an empty GPU).
//
// RESIDENT: at most two tiles per CTA, loaded once -- the first into registers,
// the second into shared memory (64 KB, dynamic; not allocated when no CTA has
// two) -- so X is read from global memory once instead of 42 times.
template <bool RESIDENT>
__global__ void __launch_bounds__(kNT, 2) nb_persistent_kernel(NBCtx c, unsigned* sync) {
  extern __shared__ float4 xs[];
  __shared__ NBShared sh;
  __shared__ volatile int ok_sh;
  GridBarrier gb{sync, g_debug_barrier_limit_ns, 0u};
  int* status = &c.st->status;
  const int G = gridDim.x, b0 = blockIdx.x;
  const int npair = (c.npart + 1) / 2;  // chunk pairs of the reducing phases
  const float* X = c.args->X;
  const int64_t ld = c.args->ld;
  // rows that 16-byte loads cannot take: 41 of the 42 products read a packed copy
  float4* pack = (ld & 3) != 0 || (reinterpret_cast<uintptr_t>(X) & 15) != 0 ? c.pack : nullptr;
  float x[8][8];
  const TileGeom g0 = tile_geom(b0 < c.ntiles ? b0 : 0), g1 = tile_geom(b0 + G < c.ntiles ? b0 + G : 0);
  if (RESIDENT) {
    if (b0 + G < c.ntiles) {
      tile_load_x(X, ld, c.n, g1, x);
#pragma unroll
      for (int k = 0; k < 8; ++k) {
        xs[kNT * (2 * k) + threadIdx.x] = make_float4(x[k][0], x[k][1], x[k][2], x[k][3]);
        xs[kNT * (2 * k + 1) + threadIdx.x] = make_float4(x[k][4], x[k][5], x[k][6], x[k][7]);
      }
    }
    if (b0 < c.ntiles) tile_load_x(X, ld, c.n, g0, x);
  }
  int pass = 0;
  auto product = [&](auto stats) {
    constexpr bool kStats = decltype(stats)::value;
    if constexpr (RESIDENT)
      ph_symv_resident<kStats>(c, b0, G, g0, g1, x, xs, sh);
    else
      ph_symv_run<kStats>(c, X, ld, pack, b0, G, (pass++ & 1) != 0, sh);
  };
#define NB_SYNC()                           \
  do {                                      \
    if (!gb.wait(status, &ok_sh)) return;   \
  } while (0)
  for (int vb = b0; vb < c.nv; vb += G) ph_init(c, vb, sh);
  NB_SYNC();
  for (int vb = b0; vb < c.nv; vb += G) ph_norm0(c, vb, sh);
  NB_SYNC();
  for (int j = 0; j < kMaxSteps; ++j) {
    if (j == 0)
      product(std::true_type{});
    else
      product(std::false_type{});
    NB_SYNC();
    if (j == 0 && b0 == 0 && threadIdx.x < 32) ph_fro(c);
    double* u = c.zsave ? c.zsave + j * c.npad : nullptr;
    for (int cp = b0; cp < npair; cp += G) ph_reduce_split(c, cp, u, sh);
    NB_SYNC();
    product(std::false_type{});
    NB_SYNC();
    for (int cp = b0; cp < npair; cp += G) ph_reduce_dots(c, cp, j, sh);
    NB_SYNC();
    if (ph_orth_next(c, b0, G, j, sh)) break;  // the same decision in every CTA
    NB_SYNC();
  }
  __syncthreads();  // thread 0's record of the last step, for warp 0
  if (b0 == 0 && threadIdx.x < 32) ph_tridiag(c, sh);
  NB_SYNC();
  ph_ritz(c, b0, G, sh);
  NB_SYNC();
  {
    const double inv = inv_norm_of_sum(c, sh);
    for (int vb = b0; vb < c.nv; vb += G) ph_ritz_norm(c, vb, inv);
  }
  NB_SYNC();
  product(std::false_type{});
  NB_SYNC();
  for (int cp = b0; cp < npair; cp += G) ph_reduce_split(c, cp, nullptr, sh);
  NB_SYNC();
  product(std::false_type{});
  NB_SYNC();
  for (int cp = b0; cp < npair; cp += G) ph_resid(c, cp, sh);
  NB_SYNC();
  if (b0 == 0 && threadIdx.x < 32) ph_final(c);
#undef NB_SYNC
}

#include "normbound_cluster.cuh"

// Four consecutive elements (positions pos .. pos+3 of a row) of the output
// matrix in the chain's storage: 16-bit, or an FP16 hi/lo pair of v * scale.
__device__ __forceinline__ void put16(uint16_t* H, const uint16_t (&u)[4], int valid) {
  if (valid == 4) {
    *reinterpret_cast<uint2*>(H) =
        make_uint2(u[0] | (static_cast<uint32_t>(u[1]) << 16), u[2] | (static_cast<uint32_t>(u[3]) << 16));
  } else {
    for (int k = 0; k < valid; ++k) H[k] = u[k];
  }
}

template <int DT>
__device__ __forceinline__ void store4(void* M, void* M_lo, int64_t pos, const float (&v)[4], int valid,
                                       float scale) {
  uint16_t u[4];
  if (DT == DT_F16X2) {
    uint16_t l[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      split_h2_sat(v[k] * scale, u[k], l[k]);
    }
    put16(static_cast<uint16_t*>(M_lo) + pos, l, valid);
  } else {
#pragma unroll
    for (int k = 0; k < 4; ++k)
      u[k] = DT == DT_BF16 ? __bfloat16_as_ushort(__float2bfloat16_rn(v[k])) : __half_as_ushort(__float2half_rn(v[k]));
  }
  put16(static_cast<uint16_t*>(M) + pos, u, valid);
}

// X_0 = RN(X * (1/lam~)) into a full symmetric matrix (16-bit, or a scaled FP16
// hi/lo pair), from the upper triangle of X, in 64 x 64 tiles through shared memory.
// Thread (tx, ty): rows i0 + 4 tx .. +3 (one 16-byte load), columns
// j0 + ty + 16 c, c = 0..3.  Both output positions are written with
// row-contiguous vector stores.
template <int DT>
__global__ void __launch_bounds__(256) scale_cast_kernel(const DevArgs* __restrict__ args, int n,
                                                         const DevState* __restrict__ st, void* __restrict__ M,
                                                         void* __restrict__ M_lo,
                                                         int64_t ldm, float scale) {
  __shared__ float s[64][65];
  int bi, bj;
  tile_of(blockIdx.x, bi, bj);
  const int i0 = bi * 64, j0 = bj * 64;
  const float* __restrict__ X = args->X;
  const int64_t ld = args->ld;
  const float inv = static_cast<float>(st->inv_lambda);
  const int tx = threadIdx.x & 15, ty = threadIdx.x >> 4;
  const bool diag = bi == bj;
  const bool vec = ((ld & 3) == 0) && ((reinterpret_cast<uintptr_t>(X) & 15) == 0);
  const int ib = i0 + 4 * tx;
#pragma unroll
  for (int c = 0; c < 4; ++c) {
    const int jj = ty + 16 * c, j = j0 + jj;
    float x[4] = {0.f, 0.f, 0.f, 0.f};
    if (j < n) {
      const float* col = X + static_cast<int64_t>(j) * ld + ib;
      if (vec && ib + 3 < n) {
        const float4 q = __ldg(reinterpret_cast<const float4*>(col));
        x[0] = q.x; x[1] = q.y; x[2] = q.z; x[3] = q.w;
      } else {
#pragma unroll
        for (int k = 0; k < 4; ++k)
          if (ib + k < n) x[k] = __ldg(col + k);
      }
    }
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      const int ii = 4 * tx + k;
      s[ii][jj] = (!diag || ii <= jj) ? x[k] * inv : 0.f;
    }
  }
  __syncthreads();
  if (diag) {
#pragma unroll
    for (int c = 0; c < 4; ++c) {
      const int jj = ty + 16 * c;
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        const int ii = 4 * tx + k;
        if (ii > jj) s[ii][jj] = s[jj][ii];
      }
    }
    __syncthreads();
  }
  const int valid_i = min(4, n - ib);
#pragma unroll
  for (int c = 0; c < 4; ++c) {
    const int jj = ty + 16 * c, j = j0 + jj;
    // position (i + j ldm): memory row j, elements i0 + 4 tx .. +3
    if (j < n && valid_i > 0) {
      const float v[4] = {s[4 * tx][jj], s[4 * tx + 1][jj], s[4 * tx + 2][jj], s[4 * tx + 3][jj]};
      store4<DT>(M, M_lo, static_cast<int64_t>(j) * ldm + ib, v, valid_i, scale);
    }
    // mirrored position (j + i ldm): memory row i = i0 + jj, elements j0 + 4 tx .. +3
    const int i = i0 + jj, jc = j0 + 4 * tx;
    const int valid_j = min(4, n - jc);
    if (!diag && i < n && valid_j > 0) {
      const float v[4] = {s[jj][4 * tx], s[jj][4 * tx + 1], s[jj][4 * tx + 2], s[jj][4 * tx + 3]};
      store4<DT>(M, M_lo, static_cast<int64_t>(i) * ldm + jc, v, valid_j, scale);
    }
  }
}

// Caller pointers of one replay: the argument block, and (single projection)
// the caller-facing fields of the one block record.
__global__ void set_args_kernel(DevArgs* d, DevArgs h, BlockRec* blk) {
  *d = h;
  if (blk) {
    blk->X = h.X;
    blk->ld = h.ld;
    blk->out = h.out;
    blk->ld_out = h.ld_out;
  }
}

__global__ void set_block_kernel(BlockRec* dst, BlockRec v) { *dst = v; }

// Status word and overshoot of the last stage into the report, and the
// complementarity residual from the final product's per-warp shares (256
// threads: strided sums, warp trees, then the 8 warp sums in order).
__global__ void __launch_bounds__(kComplSumThreads)
    finalize_kernel(const DevArgs* args, DevState* st, const double* cres, int ncompl) {
  __shared__ double wsum[kComplSumThreads / 32];
  psd_info_t* info = args->info;
  const double v = compl_cta_sum<kComplSumThreads>(cres, cres ? ncompl : 0, wsum);
  if (threadIdx.x != 0) return;
  finalize_report(st, info);
  if (info) {
    const double f2 = st->fro * st->fro;
    info->compl_resid = !cres ? __longlong_as_double(0x7ff8000000000000ll) : (f2 > 0.0 ? v / f2 : 0.0);
  }
}

}  // namespace

cudaError_t set_norm_bound_debug(int knob, double value) {
  if (knob == 1) return cudaMemcpyToSymbol(g_debug_bound_scale, &value, sizeof(double));
  if (knob == 2) {
    const unsigned long long ns = static_cast<unsigned long long>(value);
    return cudaMemcpyToSymbol(g_debug_barrier_limit_ns, &ns, sizeof(ns));
  }
  return cudaErrorInvalidValue;
}

size_t lanczos_bytes(int64_t n) {
  const int64_t npad = (n + 255) / 256 * 256;
  const int64_t nb = (n + kSymvTile - 1) / kSymvTile;
  const int64_t ntiles = nb * (nb + 1) / 2;
  const int64_t nctas = (n + kVecThreads - 1) / kVecThreads;
  const int64_t npart = (n + 31) / 32;
  size_t b = 0;
  auto add = [&](size_t bytes) { b += (bytes + 255) / 256 * 256; };
  add(sizeof(double) * (kMaxSteps + 1) * npad);  // Qv
  add(sizeof(float2) * kMaxSteps * npad);        // Qf
  add(sizeof(double) * npad * 2);                // w, q
  add(sizeof(float) * npad);                     // vh
  add(sizeof(float2) * nb * npad * 2);           // P1, P2
  add(sizeof(float2) * npart * 32);              // dots
  add(sizeof(double) * std::max(npart, nctas));  // norms
  add(sizeof(double) * ntiles);                  // tile_fro
  add(sizeof(unsigned) * 2);                     // grid barrier of the persistent kernel
  return b;
}

void lanczos_carve(LanczosBufs& L, int64_t n, uint8_t* base) {
  L.zsave = nullptr;
  L.pack = nullptr;
  L.n = n;
  L.npad = (n + 255) / 256 * 256;
  L.nb = static_cast<int>((n + kSymvTile - 1) / kSymvTile);
  L.ntiles = L.nb * (L.nb + 1) / 2;
  L.nvec_ctas = static_cast<int>((n + kVecThreads - 1) / kVecThreads);
  L.npart = static_cast<int>((n + 31) / 32);
  size_t off = 0;
  auto take = [&](size_t bytes) {
    uint8_t* p = base + off;
    off += (bytes + 255) / 256 * 256;
    return p;
  };
  L.Qv = reinterpret_cast<double*>(take(sizeof(double) * (kMaxSteps + 1) * L.npad));
  L.Qf = reinterpret_cast<float2*>(take(sizeof(float2) * kMaxSteps * L.npad));
  double* v2 = reinterpret_cast<double*>(take(sizeof(double) * L.npad * 2));
  L.w = v2;
  L.q = v2 + L.npad;
  L.vh = reinterpret_cast<float*>(take(sizeof(float) * L.npad));
  float2* P = reinterpret_cast<float2*>(take(sizeof(float2) * L.nb * L.npad * 2));
  L.P1 = P;
  L.P2 = P + static_cast<int64_t>(L.nb) * L.npad;
  L.dots = reinterpret_cast<float2*>(take(sizeof(float2) * L.npart * 32));
  L.norms = reinterpret_cast<double*>(take(sizeof(double) * std::max(L.npart, L.nvec_ctas)));
  L.tile_fro = reinterpret_cast<double*>(take(sizeof(double) * L.ntiles));
  L.sync = reinterpret_cast<unsigned*>(take(sizeof(unsigned) * 2));
}

namespace {

NBCtx make_ctx(const LanczosBufs& L, const DevArgs* args, DevState* st) {
  NBCtx c{};
  c.n = static_cast<int>(L.n);
  c.nb = L.nb;
  c.ntiles = L.ntiles;
  c.nv = L.nvec_ctas;
  c.npart = L.npart;
  c.npad = L.npad;
  c.args = args;
  c.st = st;
  c.Qv = L.Qv;
  c.w = L.w;
  c.q = L.q;
  c.zsave = L.zsave;
  c.vh = L.vh;
  c.Qf = L.Qf;
  c.P1 = L.P1;
  c.P2 = L.P2;
  c.dots = L.dots;
  c.norms = L.norms;
  c.norms2 = reinterpret_cast<float2*>(L.norms);
  c.tile_fro = L.tile_fro;
  c.pack = reinterpret_cast<float4*>(L.pack);
  return c;
}

constexpr int kTileSmem = static_cast<int>(sizeof(float)) * kSymvTile * kSymvTile;  // one resident tile

// Form and grid of the persistent kernel.  A cooperative launch needs every CTA
// resident: up to 2 per SM (128 registers; 64 KB + 17 KB of shared memory
// each), no more than the largest phase has virtual blocks.  RESIDENT when two
// tiles per CTA hold the whole triangle (304 CTAs: 608 tiles, n <= 4352).
// grid 0: the device cannot run it.
struct PersistentForm {
  int grid = 0;
  bool resident = false;
  int smem = 0;
};
PersistentForm persistent_form(const NBCtx& c) {
  // occupancies by device, looked up once (callers on several threads and streams)
  struct Occ {
    int sms = 0, stream = 0, one = 0, two = 0;
  };
  static std::mutex mu;
  static std::map<int, Occ> known;
  PersistentForm f;
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess) return f;
  Occ o;
  {
    std::lock_guard<std::mutex> lk(mu);
    auto it = known.find(dev);
    if (it != known.end()) {
      o = it->second;
    } else {
      if (cudaDeviceGetAttribute(&o.sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess ||
          cudaFuncSetAttribute(nb_persistent_kernel<true>, cudaFuncAttributeMaxDynamicSharedMemorySize, kTileSmem) !=
              cudaSuccess ||
          cudaOccupancyMaxActiveBlocksPerMultiprocessor(&o.stream, nb_persistent_kernel<false>, kNT, 0) !=
              cudaSuccess ||
          cudaOccupancyMaxActiveBlocksPerMultiprocessor(&o.one, nb_persistent_kernel<true>, kNT, 0) != cudaSuccess ||
          cudaOccupancyMaxActiveBlocksPerMultiprocessor(&o.two, nb_persistent_kernel<true>, kNT, kTileSmem) !=
              cudaSuccess)
        return f;
      known[dev] = o;
    }
  }
  const int work = std::max(std::max(std::max(c.ntiles, c.npart), c.nv), 1);
  if (c.ntiles <= o.one * o.sms) {
    f = PersistentForm{std::min(o.one * o.sms, work), true, 0};
  } else if (c.ntiles <= 2 * o.two * o.sms) {
    f = PersistentForm{std::min(o.two * o.sms, work), true, kTileSmem};
  } else {
    f = PersistentForm{std::min(o.stream * o.sms, work), false, 0};
  }
  return f;
}

// Whether the current device runs clusters of `csize` CTAs with `smem` bytes
// each (looked up once per device and shape).
bool cluster_fits(int csize, int smem) {
  static std::mutex mu;
  static std::map<std::tuple<int, int, int>, bool> known;
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess) return false;
  std::lock_guard<std::mutex> lk(mu);
  const auto key = std::make_tuple(dev, csize, smem);
  auto it = known.find(key);
  if (it != known.end()) return it->second;
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3(csize);
  cfg.blockDim = dim3(kNT);
  cfg.dynamicSmemBytes = smem;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = csize;
  attr[0].val.clusterDim.y = attr[0].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  int num = 0;
  const bool ok =
      cudaFuncSetAttribute(nb_cluster_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, 232448) ==
          cudaSuccess &&
      cudaFuncSetAttribute(nb_cluster_kernel, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) ==
          cudaSuccess &&
      cudaOccupancyMaxActiveClusters(&num, nb_cluster_kernel, &cfg) == cudaSuccess && num > 0;
  cudaGetLastError();
  known[key] = ok;
  return ok;
}

// The shape of a launch for a matrix of nb tile rows.
ClusterJob cluster_job(int nb, int& smem) {
  ClusterJob jb{};
  cluster_shape(nb * (nb + 1) / 2, jb.csize, jb.extra);
  jb.nbmax = nb;
  jb.own = (4 * nb + jb.csize - 1) / jb.csize;
  smem = cluster_carve(nullptr, nullptr, jb.extra, jb.own, nb);
  return jb;
}

cudaError_t launch_cluster(const ClusterJob& jb, int smem, cudaStream_t s) {
  cudaError_t e;  // the attributes on every call: a device reset drops them
  if ((e = cudaFuncSetAttribute(nb_cluster_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, 232448)) !=
      cudaSuccess)
    return e;
  if ((e = cudaFuncSetAttribute(nb_cluster_kernel, cudaFuncAttributeNonPortableClusterSizeAllowed, 1)) !=
      cudaSuccess)
    return e;
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3(jb.csize);
  cfg.blockDim = dim3(kNT);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = jb.csize;
  attr[0].val.clusterDim.y = attr[0].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, nb_cluster_kernel, jb);
}

}  // namespace

cudaError_t enqueue_norm_bound(const LanczosBufs& L, const DevArgs* args, DevState* st, cudaStream_t s,
                               bool persistent) {
  const NBCtx c = make_ctx(L, args, st);
  if (persistent && c.nb <= kClusterMaxNb) {
    int smem = 0;
    ClusterJob jb = cluster_job(c.nb, smem);
    if (cluster_fits(jb.csize, smem)) {
      jb.args = args;
      jb.n = c.n;
      jb.st = st;
      jb.Qv = c.Qv;
      jb.zsave = c.zsave;
      jb.npad = c.npad;
      return launch_cluster(jb, smem, s);
    }
  }
  if (persistent) {
    const PersistentForm f = persistent_form(c);
    if (f.grid > 0) {
      cudaError_t e = cudaMemsetAsync(L.sync, 0, 2 * sizeof(unsigned), s);
      if (e != cudaSuccess) return e;
      cudaLaunchConfig_t cfg{};
      cfg.gridDim = dim3(f.grid);
      cfg.blockDim = dim3(kNT);
      if (f.smem > 0) {  // on every call: a device reset drops it
        e = cudaFuncSetAttribute(nb_persistent_kernel<true>, cudaFuncAttributeMaxDynamicSharedMemorySize, f.smem);
        if (e != cudaSuccess) return e;
      }
      cfg.dynamicSmemBytes = f.smem;
      cfg.stream = s;
      cudaLaunchAttribute attr[1];
      attr[0].id = cudaLaunchAttributeCooperative;
      attr[0].val.cooperative = 1;
      cfg.attrs = attr;
      cfg.numAttrs = 1;
      return f.resident ? cudaLaunchKernelEx(&cfg, nb_persistent_kernel<true>, c, L.sync)
                        : cudaLaunchKernelEx(&cfg, nb_persistent_kernel<false>, c, L.sync);
    }
  }
  const int vb = c.nv, rb = c.npart, pb = (c.npart + 1) / 2;  // pb: chunk pairs
  nb_init_kernel<<<vb, kNT, 0, s>>>(c);
  nb_norm0_kernel<<<vb, kNT, 0, s>>>(c);
  int pass = 0;  // products over X so far: odd ones traverse the tiles backwards
  for (int j = 0; j < kMaxSteps; ++j) {
    if (j == 0) {
      nb_symv_kernel<true><<<c.ntiles, kNT, 0, s>>>(c, 0, pass++ & 1);
      nb_fro_kernel<<<1, 32, 0, s>>>(c);
    } else {
      nb_symv_kernel<false><<<c.ntiles, kNT, 0, s>>>(c, 1, pass++ & 1);
    }
    double* u = L.zsave ? L.zsave + j * L.npad : nullptr;
    nb_reduce_split_kernel<<<pb, kNT, 0, s>>>(c, u, 1);
    nb_symv_kernel<false><<<c.ntiles, kNT, 0, s>>>(c, 1, pass++ & 1);
    nb_reduce_dots_kernel<<<pb, kNT, 0, s>>>(c, j);
    nb_orth_kernel<<<rb, kNT, 0, s>>>(c, j);
  }
  nb_tridiag_kernel<<<1, 32, 0, s>>>(c);
  nb_ritz_kernel<<<rb, kNT, 0, s>>>(c);
  nb_ritz_norm_kernel<<<vb, kNT, 0, s>>>(c);
  // (after a breakdown the remaining steps' products do no work, so these two
  // may not continue the alternation; results do not depend on the direction)
  nb_symv_kernel<false><<<c.ntiles, kNT, 0, s>>>(c, 0, pass++ & 1);
  nb_reduce_split_kernel<<<pb, kNT, 0, s>>>(c, nullptr, 0);
  nb_symv_kernel<false><<<c.ntiles, kNT, 0, s>>>(c, 0, pass++ & 1);
  nb_resid_kernel<<<pb, kNT, 0, s>>>(c);
  nb_final_kernel<<<1, 32, 0, s>>>(c);
  return cudaGetLastError();
}


cudaError_t enqueue_scale_cast(int dtype, const DevArgs* args, const DevState* st, int64_t n, void* M,
                               void* M_lo, int64_t ldm, cudaStream_t s, float scale) {
  const int nb = static_cast<int>((n + 63) / 64);
  const int tiles = nb * (nb + 1) / 2;
  const int blk = 256;
  const int ni = static_cast<int>(n);
  switch (dtype) {
    case DT_F16: scale_cast_kernel<DT_F16><<<tiles, blk, 0, s>>>(args, ni, st, M, M_lo, ldm, scale); break;
    case DT_BF16: scale_cast_kernel<DT_BF16><<<tiles, blk, 0, s>>>(args, ni, st, M, M_lo, ldm, scale); break;
    case DT_F16X2: scale_cast_kernel<DT_F16X2><<<tiles, blk, 0, s>>>(args, ni, st, M, M_lo, ldm, scale); break;
    default: return cudaErrorInvalidValue;
  }
  return cudaGetLastError();
}

cudaError_t enqueue_set_args(DevArgs* d_args, const DevArgs& h, cudaStream_t s, BlockRec* blk) {
  set_args_kernel<<<1, 1, 0, s>>>(d_args, h, blk);
  return cudaGetLastError();
}

cudaError_t enqueue_set_block(BlockRec* d_blk, const BlockRec& v, cudaStream_t s) {
  set_block_kernel<<<1, 1, 0, s>>>(d_blk, v);
  return cudaGetLastError();
}

cudaError_t enqueue_finalize(const DevArgs* args, DevState* st, cudaStream_t s, const double* cres, int ncompl) {
  finalize_kernel<<<1, kComplSumThreads, 0, s>>>(args, st, cres, ncompl);
  return cudaGetLastError();
}

}  // namespace psd
