// Device pieces of the norm bound shared by its forms: the persistent and the
// multi-launch form (normbound.cu) and the cluster form (normbound_cluster.cu).
// All forms run the same arithmetic in the same order and give the same bits.
#pragma once

#include <cuda_runtime.h>

#include <cstdint>

#include "internal.h"

namespace psd {
namespace {

constexpr int kNT = 256;  // threads of a CTA (of each tile group)
constexpr uint64_t kSeed = 0x243F6A8885A308D3ull;  // Lanczos start vector seed
constexpr uint64_t kGolden = 0x9E3779B97F4A7C15ull;

// ------------------------------------------------------- double-float helpers
struct F2 {
  float h, l;
};
__device__ __forceinline__ void two_sum(float a, float b, float& s, float& e) {
  s = __fadd_rn(a, b);
  const float z = __fsub_rn(s, a);
  e = __fadd_rn(__fsub_rn(a, __fsub_rn(s, z)), __fsub_rn(b, z));
}
__device__ __forceinline__ F2 f2_add(F2 a, F2 b) {
  float s, e;
  two_sum(a.h, b.h, s, e);
  return F2{s, __fadd_rn(__fadd_rn(a.l, b.l), e)};
}
__device__ __forceinline__ double f2_to_d(F2 a) { return static_cast<double>(a.h) + static_cast<double>(a.l); }
__device__ __forceinline__ F2 shfl_xor_f2(F2 a, int m) {
  return F2{__shfl_xor_sync(0xffffffffu, a.h, m), __shfl_xor_sync(0xffffffffu, a.l, m)};
}

// Normalised pair: h = RN(h + l).
__device__ __forceinline__ F2 f2_norm(F2 a) {
  const float s = __fadd_rn(a.h, a.l);
  return F2{s, __fsub_rn(a.l, __fsub_rn(s, a.h))};
}
// Product of two normalised pairs (Dekker's, with fma; error ~2^-47 relative).
__device__ __forceinline__ F2 f2_mul(F2 a, F2 b) {
  const float p = __fmul_rn(a.h, b.h);
  float e = fmaf(a.h, b.h, -p);
  e = fmaf(a.h, b.l, e);
  e = fmaf(a.l, b.h, e);
  return F2{p, e};
}

// --------------------------------------------------------------- SplitMix64
__device__ __forceinline__ uint64_t splitmix64(uint64_t seed, uint64_t i) {
  uint64_t z = seed + (i + 1) * kGolden;
  z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
  z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
  return z ^ (z >> 31);
}

// The FP32 estimate (FP64 runs at a small fraction of the FP32 rate on this GPU,
// and every thread of a tile's CTA evaluates this) is corrected exactly by the
// integer loops.
__device__ __forceinline__ void tile_of(int t, int& bi, int& bj) {
  int j = static_cast<int>((sqrtf(8.f * static_cast<float>(t) + 1.f) - 1.f) * 0.5f);
  while ((j + 1) * (j + 2) / 2 <= t) ++j;
  while (j * (j + 1) / 2 > t) --j;
  bj = j;
  bi = t - j * (j + 1) / 2;
}

// Recursive-halving sum of 32 double-float values over a warp; on return lane l
// holds the warp total of value l.  The dot products of a chunk are formed and
// added in FP32 pairs (~48 bits, what their partial sums are stored in): the
// same sums in FP64 cost ~4,000 cycles per chunk on this GPU's FP64 unit.
__device__ __forceinline__ F2 warp_multi_sum(F2 (&v)[32], int lane) {
#pragma unroll
  for (int half = 16, m = 16; half >= 1; half >>= 1, m >>= 1) {
    const bool upper = (lane & m) != 0;
#pragma unroll
    for (int i = 0; i < half; ++i) {
      const F2 send = upper ? v[i] : v[i + half];
      const F2 keep = upper ? v[i + half] : v[i];
      v[i] = f2_add(keep, shfl_xor_f2(send, m));
    }
  }
  return v[0];
}

// One tile of y = X v over the upper triangle (see file comment), in three
// pieces so that the persistent kernel can load the next tile while it
// reduces the current one.  Thread (tr, tc) = (lane & 15, 2 warp + lane / 16)
// owns rows i0 + 8 tr .. +7 and columns j0 + 8 tc .. +7: each column's 128
// rows are read by a half-warp as 512 contiguous bytes.  DIAG tiles mask to
// i <= j (rows) and i < j (columns).  STATS adds the tile's share of
// ||X||_F^2 and max |X_ii|.
struct TileGeom {
  int bi, bj, ib, jb;
  bool diag;    // the tile lies on the diagonal
  bool ondiag;  // the thread's block does
};
__device__ __forceinline__ TileGeom tile_geom_at(int bi, int bj) {
  TileGeom g;
  g.bi = bi;
  g.bj = bj;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  g.ib = g.bi * kSymvTile + 8 * (lane & 15);
  g.jb = g.bj * kSymvTile + 8 * (2 * warp + (lane >> 4));
  g.diag = g.bi == g.bj;
  g.ondiag = g.ib == g.jb;
  return g;
}
__device__ __forceinline__ TileGeom tile_geom(int t) {
  int bi, bj;
  tile_of(t, bi, bj);
  return tile_geom_at(bi, bj);
}

// The thread's 64 elements: 16 independent 16-byte loads of X in flight; zeros
// below the diagonal of a diagonal tile (those entries of X are not read for use).
__device__ __forceinline__ void tile_load_x(const float* __restrict__ X, int64_t ld, int n, const TileGeom& g,
                                            float (&x)[8][8]) {
  const bool full = (g.ib + 7 < n) && (g.jb + 7 < n);
  const bool vec = full && ((ld & 3) == 0) && ((reinterpret_cast<uintptr_t>(X) & 15) == 0);
#pragma unroll
  for (int c = 0; c < 8; ++c) {
    const float* col = X + static_cast<int64_t>(g.jb + c) * ld + g.ib;
    if (vec) {
      const float4 a4 = __ldg(reinterpret_cast<const float4*>(col));
      const float4 b4 = __ldg(reinterpret_cast<const float4*>(col + 4));
      x[c][0] = a4.x; x[c][1] = a4.y; x[c][2] = a4.z; x[c][3] = a4.w;
      x[c][4] = b4.x; x[c][5] = b4.y; x[c][6] = b4.z; x[c][7] = b4.w;
    } else {
#pragma unroll
      for (int k = 0; k < 8; ++k) x[c][k] = (g.jb + c < n && g.ib + k < n) ? __ldg(col + k) : 0.f;
    }
  }
  if (g.diag) {
#pragma unroll
    for (int c = 0; c < 8; ++c)
#pragma unroll
      for (int k = 0; k < 8; ++k)
        if (g.ib + k > g.jb + c) x[c][k] = 0.f;
  }
}

// Per-thread row and column dot products of the 8 x 8 block (8-term FP32 FMA runs).
// `col(c, x)` gives column c of the block (zeros below the diagonal).  Row sums
// take i <= j, column sums i < j: only a block on the diagonal has elements
// (c == k) that the two treat differently.
template <bool STATS, class Col>
__device__ __forceinline__ void tile_fma(int n, const TileGeom& g, const float (&vi)[8], const float (&vj)[8],
                                         const Col& col, float (&rsum)[8], float (&csum)[8], float& fro,
                                         unsigned& mdiag) {
  fro = 0.f;
  mdiag = 0;
#pragma unroll
  for (int k = 0; k < 8; ++k) rsum[k] = 0.f;
#pragma unroll
  for (int c = 0; c < 8; ++c) {
    float x[8];
    col(c, x);
    csum[c] = 0.f;
#pragma unroll
    for (int k = 0; k < 8; ++k) {
      const float xr = x[k], xc = (k == c && g.ondiag) ? 0.f : x[k];
      if (STATS && k == c && g.ondiag && g.ib + k < n) mdiag = max(mdiag, __float_as_uint(fabsf(x[k])));
      rsum[k] = fmaf(xr, vj[c], rsum[k]);
      csum[c] = fmaf(xc, vi[k], csum[c]);
      if (STATS) fro = fmaf(xr, xc + xr, fro);  // x^2 on the diagonal, 2 x^2 above it
    }
  }
}

// tile_fma of a tile held in registers.
template <bool STATS>
__device__ __forceinline__ void tile_fma_reg(int n, const TileGeom& g, const float (&vi)[8], const float (&vj)[8],
                                             const float (&x)[8][8], float (&rsum)[8], float (&csum)[8], float& fro,
                                             unsigned& mdiag) {
  auto col = [&](int c, float (&o)[8]) {
#pragma unroll
    for (int k = 0; k < 8; ++k) o[k] = x[c][k];
  };
  tile_fma<STATS>(n, g, vi, vj, col, rsum, csum, fro, mdiag);
}

// The warps' row sums lie at red[warp][17 k + tr] for row 8 tr + k: the stores (a
// half-warp along tr) and the reads (a warp along k and tr) spread over the banks.
constexpr int kRedStride = 8 * 17;

// Combines the threads' sums in a fixed order (double-float) into the tile's
// row partials (sink.row(i, v): row i's dot product with this tile) and column
// partials (sink.col(j, v)), through the row buffer `red`; with STATS the tile's
// share of ||X||_F^2 goes to sink.fro (one thread) and each warp's max |X_ii|
// to sink.diag.  Ends with a CTA barrier unless `sync_after` is false: a run
// of tiles alternates the two buffers instead, since a tile two ahead writes a
// buffer only after every thread has passed the barrier of the tile between
// (and so finished reading it); the run is followed by a CTA barrier.
template <bool STATS, class Sink>
__device__ __forceinline__ void tile_reduce(int n, const TileGeom& g, const float (&rsum)[8], const float (&csum)[8],
                                            float fro, unsigned mdiag, float2 (*red)[kRedStride], double* fro_sh,
                                            const Sink& sink, bool sync_after) {
  const int i0 = g.bi * kSymvTile;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int tr = lane & 15;
  // rows: the two column groups of a warp (exact TwoSum), then the 8 warps
  F2 rs[8], cs[8];
#pragma unroll
  for (int k = 0; k < 8; ++k) {
    const float o = __shfl_xor_sync(0xffffffffu, rsum[k], 16);
    float h, e;
    if (lane < 16) two_sum(rsum[k], o, h, e); else two_sum(o, rsum[k], h, e);
    rs[k] = F2{h, e};
    cs[k] = F2{csum[k], 0.f};
  }
  if (lane < 16) {
#pragma unroll
    for (int k = 0; k < 8; ++k) red[warp][17 * k + tr] = make_float2(rs[k].h, rs[k].l);
  }
  // columns: recursive halving over the 16 row groups of a half-warp
#pragma unroll
  for (int half = 4, m = 8; half >= 1; half >>= 1, m >>= 1) {
    const bool upper = (tr & m) != 0;
#pragma unroll
    for (int i = 0; i < half; ++i) {
      const F2 send = upper ? cs[i] : cs[i + half];
      const F2 keep = upper ? cs[i + half] : cs[i];
      cs[i] = f2_add(keep, shfl_xor_f2(send, m));
    }
  }
  {
    const F2 o = shfl_xor_f2(cs[0], 1);
    cs[0] = (tr & 1) ? f2_add(o, cs[0]) : f2_add(cs[0], o);
    const int j = g.jb + (tr >> 1);
    if ((tr & 1) == 0 && j < n) sink.col(j, make_float2(cs[0].h, cs[0].l));
  }
  __syncthreads();
  if (threadIdx.x < kSymvTile) {
    const int r = threadIdx.x;
    const int at = 17 * (r & 7) + (r >> 3);
    F2 p[8];
#pragma unroll
    for (int w = 0; w < 8; ++w) p[w] = F2{red[w][at].x, red[w][at].y};
#pragma unroll
    for (int h = 1; h < 8; h *= 2)
#pragma unroll
      for (int w = 0; w < 8; w += 2 * h) p[w] = f2_add(p[w], p[w + h]);
    const F2 a = p[0];
    if (i0 + r < n) sink.row(i0 + r, make_float2(a.h, a.l));
  }
  if (STATS) {
    double f = static_cast<double>(fro);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) f += __shfl_xor_sync(0xffffffffu, f, o);
    if (lane == 0) fro_sh[warp] = f;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) mdiag = max(mdiag, __shfl_xor_sync(0xffffffffu, mdiag, o));
    if (lane == 0 && mdiag) sink.diag(mdiag);
    __syncthreads();
    if (threadIdx.x == 0) {
      double sum = 0.0;
      for (int w = 0; w < 8; ++w) sum += fro_sh[w];
      sink.fro(sum);
    }
  }
  if (sync_after) __syncthreads();
}

__device__ __forceinline__ float2 d_to_f2(double v) {
  const float h = __double2float_rn(v);
  return make_float2(h, __double2float_rn(v - static_cast<double>(h)));
}

// Warp sum of one double-float value per lane (fixed order; every lane).
__device__ __forceinline__ F2 warp_sum_f2(F2 t) {
  const int lane = threadIdx.x & 31;
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    const F2 other = shfl_xor_f2(t, o);
    t = (lane & o) ? f2_add(other, t) : f2_add(t, other);
  }
  return t;
}
__device__ __forceinline__ F2 f2_of(double v) {
  const float2 p = d_to_f2(v);
  return F2{p.x, p.y};
}

// Loads of the double-float partials: through L2 (vectors other CTAs wrote), or plain (shared memory).
struct LoadCg {
  __device__ __forceinline__ float2 operator()(const float2* p) const { return __ldcg(p); }
};
struct LoadPlain {
  __device__ __forceinline__ float2 operator()(const float2* p) const { return *p; }
};

// Sum of nch double-float partials by one warp (lanes stride over them, 8 loads
// in flight, then a butterfly; fixed order), as FP64 in every lane.
template <class Load>
__device__ __forceinline__ double warp_sum_chunks(const float2* part, int nch, const Load& load) {
  const int lane = threadIdx.x & 31;
  F2 acc{0.f, 0.f};
  for (int c0 = 0; c0 < nch; c0 += 8 * 32) {
    float2 t[8];
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      const int ch = c0 + 32 * i + lane;
      t[i] = ch < nch ? load(part + ch) : make_float2(0.f, 0.f);
    }
#pragma unroll
    for (int i = 0; i < 8; ++i) acc = f2_add(acc, F2{t[i].x, t[i].y});
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    const F2 other = shfl_xor_f2(acc, o);
    acc = (lane & o) ? f2_add(other, acc) : f2_add(acc, other);
  }
  return f2_to_d(acc);
}

// S[k] = sum over the chunks of part[k * stride + ch] (slot-major: a warp's 32
// lanes read 256 contiguous bytes) for the slots k <= j and 31, double-float in a
// fixed order (lanes stride over the chunks, then a butterfly), into shared
// memory.  Warp w takes the slots w, w + 8, w + 16, w + 24 together: four
// independent chains of loads and adds.
template <class Load>
__device__ __forceinline__ void chunk_sums(const float2* part, int nch, int stride, int j, float2* S, const Load& load) {
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  F2 acc[4];
  bool use[4];
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const int k = w + 8 * i;
    use[i] = k <= j || k == 31;
    acc[i] = F2{0.f, 0.f};
  }
  for (int c0 = 0; c0 < nch; c0 += 2 * 32) {
    float2 t[4][2];
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
      for (int q = 0; q < 2; ++q) {
        const int ch = c0 + 32 * q + lane;
        t[i][q] = use[i] && ch < nch ? load(part + static_cast<int64_t>(w + 8 * i) * stride + ch) : make_float2(0.f, 0.f);
      }
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
      for (int q = 0; q < 2; ++q) acc[i] = f2_add(acc[i], F2{t[i][q].x, t[i][q].y});
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1)
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const F2 other = shfl_xor_f2(acc[i], o);
      acc[i] = (lane & o) ? f2_add(other, acc[i]) : f2_add(acc[i], other);
    }
  if (lane == 0) {
#pragma unroll
    for (int i = 0; i < 4; ++i)
      if (use[i]) S[w + 8 * i] = make_float2(acc[i].h, acc[i].l);
  }
}

// beta_j = sqrt(b2) and its reciprocal (one rsqrt in place of a square root and a division).
__device__ __forceinline__ void lanczos_beta(double b2, double& beta, double& inv) {
  inv = rsqrt(b2);
  beta = b2 > 0.0 ? b2 * inv : (b2 <= 0.0 ? 0.0 : b2);  // NaN stays NaN
}
// beta_j and 1 / beta_j from the summed dots S (one warp; lane 0 writes): beta^2 =
// ||w'||^2 - ||h||^2, the difference in double-float.
__device__ __forceinline__ void beta_of_sums(const float2* S, int j, double* out) {
  const int lane = threadIdx.x & 31;
  F2 q{0.f, 0.f};
  if (lane <= j) {
    const F2 s = f2_norm(F2{S[lane].x, S[lane].y});
    q = f2_mul(s, s);
  }
  q = warp_sum_f2(q);
  if (lane == 0) {
    const F2 d = f2_add(F2{S[31].x, S[31].y}, F2{-q.h, -q.l});
    double b, inv;
    lanczos_beta(f2_to_d(d), b, inv);
    out[0] = b;
    out[1] = inv;
  }
}

// The dot products of a chunk's element w' (lane = element) with the Lanczos
// vectors q_k, k <= j (q[k]: double-float), and ||w'||^2 in slot 31: lane l returns
// slot l's sum over the chunk.
template <class LoadQ>
__device__ __forceinline__ float2 chunk_dots(F2 w, int j, const LoadQ& q) {
  F2 v[32];
#pragma unroll
  for (int k = 0; k < 32; ++k) {
    v[k] = F2{0.f, 0.f};
    if (k < kMaxSteps && k <= j) v[k] = f2_mul(q(k), w);
  }
  v[31] = f2_mul(w, w);
  const F2 s = warp_multi_sum(v, threadIdx.x & 31);
  return make_float2(s.h, s.l);
}

// Vector elements of a Lanczos step (one lane = one element).
// w' = w - alpha q_j - beta q_{j-1}.
__device__ __forceinline__ double lanczos_recur(double w, double alpha, double qj, double beta, double qp) {
  return fma(-beta, qp, fma(-alpha, qj, w));
}
// w'' = w' - sum_{k <= j} h_k q_k in four independent chains (an FP64
// operation's latency is 64 cycles).  h: h_k in lane k (one conversion to FP64
// per warp; done by the warps that sum the slots it was 32 of them, on a unit
// that issues one every ~19 cycles).
__device__ __forceinline__ double lanczos_orth(double w, double h, const double (&qk)[kMaxSteps], int j) {
  double a[4] = {0.0, 0.0, 0.0, 0.0};
#pragma unroll
  for (int k = 0; k < kMaxSteps; ++k)
    if (k <= j) a[k & 3] = fma(__shfl_sync(0xffffffffu, h, k), qk[k], a[k & 3]);
  return w - ((a[0] + a[1]) + (a[2] + a[3]));
}
// sum_k y_k q_k, k < m.
__device__ __forceinline__ double lanczos_ritz(const double (&yk)[kMaxSteps], const double (&qk)[kMaxSteps], int m) {
  double s = 0.0;
#pragma unroll
  for (int k = 0; k < kMaxSteps; ++k)
    if (k < m) s = fma(yk[k], qk[k], s);
  return s;
}
// Element `i` of the start vector, before scaling to unit length.
__device__ __forceinline__ double lanczos_start(int i) {
  const uint64_t z = splitmix64(kSeed, static_cast<uint64_t>(i));
  return 2.0 * (static_cast<double>(z >> 11) * 0x1.0p-53) - 1.0;
}

}  // namespace
}  // namespace psd
