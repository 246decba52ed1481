// Norm bound of a small matrix by one thread-block cluster (included by
// normbound.cu inside its namespace).
//
// Up to order kClusterMaxOrder the whole bound of a matrix runs on one cluster
// of C <= 16 CTAs: the tiles of X stay on chip for all 42 products (a CTA's
// first tile in registers, up to two more in shared memory), every vector lives
// in shared memory, and the phases are separated by hardware cluster barriers.
// What bounds it is the latency of the phases, so all communication is remote
// shared-memory stores into the place where the next phase reads: a tile's
// partial sums go to the CTA that owns their chunk of 32 elements (chunk ch:
// rank ch % C), and what every CTA needs (the mat-vec input, the chunks'
// partial dot products) is stored to all of them.  The arithmetic and its order
// are those of the other forms (normbound.cuh): the same bits for any C.
//
// psd_norm_bound against the persistent grid kernel on the same phases: n = 256
// 278 against 436 us, 701 368 against 449, 1000 424 against 460 (then 208, 284 and
// 333 us with double-float dot products).  The order ends where 16 CTAs of three
// tiles do.

constexpr int kClusterMaxNb = 9;   // 45 tiles on 16 CTAs of 3
constexpr int kClusterMaxSize = 16;
constexpr int kClusterMaxExtra = 2;  // tiles in shared memory per CTA
constexpr int kClusterMaxOrder = kClusterMaxNb * kSymvTile;

struct ClusterJob {
  const DevArgs* args;
  int n;
  DevState* st;
  double *Qv, *zsave;       // zsave set: Lanczos vectors and X q_j are also kept in global memory (row length npad)
  int64_t npad;
  int csize, extra;         // CTAs, tiles in shared memory per CTA
  int own, nbmax;           // chunks per CTA and tile rows that the shared memory is laid out for
};

__host__ __device__ constexpr int cluster_round16(int b) { return (b + 15) / 16 * 16; }

// Shared memory of a CTA, carved in this order.
struct ClusterSmem {
  float4* xs;        // extra x 64 KB
  float2 (*red)[8][kRedStride];  // 2 buffers
  double* Q;         // own x kMaxSteps x 32
  float2* Qf;        // the same as double-float pairs
  double* w;         // own x 32
  double* fro;       // per tile (every CTA has all of them)
  double *alpha, *beta, *y;
  float2* hs;        // the summed dots as pairs
  int2* geo;         // (bi, bj) of the CTA's tiles
  double* norms;     // per 256-element block (start vector)
  double* bs;        // block_sum64
  double* scalar;    // 4
  float2* part;      // own x (nbmax + 1) x 32 partial sums of the own chunks
  float2* dots;      // 32 slots x dstride
  float2* norms2;    // per chunk
  float2* stg;       // 8 x 32
  float* vh;         // mat-vec input, nbmax x 128
  float *a32, *b32;
  unsigned* mdiag;
  int dstride;
};
__host__ __device__ inline int cluster_carve(ClusterSmem* s, uint8_t* base, int extra, int own, int nbmax) {
  int off = 0;
  auto take = [&](int bytes) {
    const int o = off;
    off += cluster_round16(bytes);
    return base + o;
  };
  const int nch = 4 * nbmax, ntl = nbmax * (nbmax + 1) / 2, ds = nch | 1;
  ClusterSmem t;
  t.xs = reinterpret_cast<float4*>(take(extra * 4 * kSymvTile * kSymvTile));
  t.red = reinterpret_cast<float2(*)[8][kRedStride]>(take(2 * 8 * kRedStride * 8));
  t.Q = reinterpret_cast<double*>(take(own * kMaxSteps * 32 * 8));
  t.Qf = reinterpret_cast<float2*>(take(own * kMaxSteps * 32 * 8));
  t.w = reinterpret_cast<double*>(take(own * 32 * 8));
  t.fro = reinterpret_cast<double*>(take(ntl * 8));
  t.hs = reinterpret_cast<float2*>(take(32 * 8));
  t.geo = reinterpret_cast<int2*>(take((kClusterMaxExtra + 1) * 8));
  t.alpha = reinterpret_cast<double*>(take(kMaxSteps * 8));
  t.beta = reinterpret_cast<double*>(take(kMaxSteps * 8));
  t.y = reinterpret_cast<double*>(take(kMaxSteps * 8));
  t.norms = reinterpret_cast<double*>(take((nbmax + 1) / 2 * 8));
  t.bs = reinterpret_cast<double*>(take(8 * 8));
  t.scalar = reinterpret_cast<double*>(take(4 * 8));
  t.part = reinterpret_cast<float2*>(take(own * (nbmax + 1) * 32 * 8));
  t.dots = reinterpret_cast<float2*>(take(32 * ds * 8));
  t.norms2 = reinterpret_cast<float2*>(take(nch * 8));
  t.stg = reinterpret_cast<float2*>(take(8 * 32 * 8));
  t.vh = reinterpret_cast<float*>(take(nbmax * kSymvTile * 4));
  t.a32 = reinterpret_cast<float*>(take(kMaxSteps * 4));
  t.b32 = reinterpret_cast<float*>(take(kMaxSteps * 4));
  t.mdiag = reinterpret_cast<unsigned*>(take(4));
  t.dstride = ds;
  if (s) *s = t;
  return off;
}

// Stores to the same place (shared address `a` of this CTA) in CTA `rank` of the cluster.
__device__ __forceinline__ void st_remote(uint32_t a, uint32_t rank, float v) {
  asm volatile("st.shared::cluster.f32 [%0], %1;" ::"r"(mapa_shared(a, rank)), "f"(v) : "memory");
}
__device__ __forceinline__ void st_remote(uint32_t a, uint32_t rank, float2 v) {
  asm volatile("st.shared::cluster.v2.f32 [%0], {%1, %2};" ::"r"(mapa_shared(a, rank)), "f"(v.x), "f"(v.y) : "memory");
}
__device__ __forceinline__ void st_remote(uint32_t a, uint32_t rank, double v) {
  asm volatile("st.shared::cluster.f64 [%0], %1;" ::"r"(mapa_shared(a, rank)), "d"(v) : "memory");
}
__device__ __forceinline__ unsigned ld_remote(const unsigned* p, uint32_t rank) {
  unsigned v;
  asm volatile("ld.shared::cluster.u32 %0, [%1];" : "=r"(v) : "r"(mapa_shared(smem_u32(p), rank)) : "memory");
  return v;
}

// Tile (bi, bj)'s partial sums to the owners of their chunks: slot bi holds
// column partials (bi <= the chunk's tile row b), slot bj + 1 row partials (bj >= b).
struct ClusterSink {
  const ClusterSmem& s;
  const TileGeom& g;
  int tile, csize, clog, nbmax;  // csize = 2^clog
  __device__ __forceinline__ void put(int i, int slot, float2 v) const {
    const int ch = i >> 5;
    st_remote(smem_u32(s.part + ((ch >> clog) * (nbmax + 1) + slot) * 32 + (i & 31)), ch & (csize - 1), v);
  }
  __device__ __forceinline__ void row(int i, float2 v) const { put(i, g.bj + 1, v); }
  __device__ __forceinline__ void col(int j, float2 v) const { put(j, g.bi, v); }
  __device__ __forceinline__ void diag(unsigned m) const { atomicMax(s.mdiag, m); }
  __device__ __forceinline__ void fro(double f) const {
    for (int r = 0; r < csize; ++r) st_remote(smem_u32(s.fro + tile), r, f);
  }
};

// The matrix-vector product over the CTA's tiles rank, rank + C, ...: the first
// in registers, the rest in shared memory (each thread's own 16 float4).
template <bool STATS>
__device__ __forceinline__ void cl_product(const ClusterSmem& s, int n, int ntiles, int rank, int csize, int nbmax,
                                           const float (&x)[8][8]) {
  int buf = 0;
  for (int t = rank, i = 0; t < ntiles; t += csize, ++i, buf ^= 1) {
    const TileGeom g = tile_geom_at(s.geo[i].x, s.geo[i].y);
    float vi[8], vj[8], rsum[8], csum[8], fro;
    unsigned mdiag;
#pragma unroll
    for (int k = 0; k < 8; k += 4) {
      const float4 a = *reinterpret_cast<const float4*>(s.vh + g.ib + k);
      const float4 b = *reinterpret_cast<const float4*>(s.vh + g.jb + k);
      vi[k] = a.x; vi[k + 1] = a.y; vi[k + 2] = a.z; vi[k + 3] = a.w;
      vj[k] = b.x; vj[k + 1] = b.y; vj[k + 2] = b.z; vj[k + 3] = b.w;
    }
    if (i == 0) {
      tile_fma_reg<STATS>(n, g, vi, vj, x, rsum, csum, fro, mdiag);
    } else {
      const float4* xt = s.xs + (i - 1) * 16 * kNT;
      auto col = [&](int k, float (&o)[8]) {
        const float4 a = xt[kNT * (2 * k) + threadIdx.x], b = xt[kNT * (2 * k + 1) + threadIdx.x];
        o[0] = a.x; o[1] = a.y; o[2] = a.z; o[3] = a.w;
        o[4] = b.x; o[5] = b.y; o[6] = b.z; o[7] = b.w;
      };
      tile_fma<STATS>(n, g, vi, vj, col, rsum, csum, fro, mdiag);
    }
    tile_reduce<STATS>(n, g, rsum, csum, fro, mdiag, s.red[buf], s.bs, ClusterSink{s, g, t, csize, 31 - __clz(csize), nbmax}, false);
  }
}

// y of own chunk `o` (global chunk o C + rank) by the four warps of this half
// of the CTA, in reduce_partials' order; the half's first warp receives it.
// Both halves call it together (CTA barriers).
__device__ __forceinline__ F2 cl_reduce(const ClusterSmem& s, int n, int nb, int o, int nown, int e, int nbmax) {
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, hw = w & 3;
  F2 a{0.f, 0.f}, d{0.f, 0.f};
  if (o < nown && e < n) {
    const int b = e / kSymvTile;
    const float2* p = s.part + o * (nbmax + 1) * 32 + lane;
    for (int bj = b + hw; bj < nb; bj += 4) a = f2_add(a, F2{p[(bj + 1) * 32].x, p[(bj + 1) * 32].y});
    for (int bi = hw; bi <= b; bi += 4) d = f2_add(d, F2{p[bi * 32].x, p[bi * 32].y});
  }
  const F2 t = f2_add(a, d);
  s.stg[w * 32 + lane] = make_float2(t.h, t.l);
  __syncthreads();
  F2 y{0.f, 0.f};
  if (hw == 0) {
    F2 acc{s.stg[w * 32 + lane].x, s.stg[w * 32 + lane].y};
#pragma unroll
    for (int q = 1; q < 4; ++q) acc = f2_add(acc, F2{s.stg[(w + q) * 32 + lane].x, s.stg[(w + q) * 32 + lane].y});
    y = f2_norm(acc);
  }
  __syncthreads();
  return y;
}

__global__ void __launch_bounds__(kNT, 2) nb_cluster_kernel(const ClusterJob jb) {
  extern __shared__ __align__(16) uint8_t cl_raw[];
  const int C = jb.csize, rank = static_cast<int>(cluster_ctarank());
  const int n = jb.n;
  const float* X = jb.args->X;
  const int64_t ld = jb.args->ld;
  DevState* st = jb.st;
  ClusterSmem s;
  cluster_carve(&s, cl_raw, jb.extra, jb.own, jb.nbmax);
  const int nbmax = jb.nbmax;
  const int nb = (n + kSymvTile - 1) / kSymvTile, ntiles = nb * (nb + 1) / 2;
  const int nch = (n + 31) / 32, nv = (n + kNT - 1) / kNT;
  const int nown = nch > rank ? (nch - 1 - rank) / C + 1 : 0;  // own chunks rank, rank + C, ...
  const int nit = (nown + 1) / 2;                              // two at a time, one per half of the CTA
  const int tid = threadIdx.x, lane = tid & 31, wp = tid >> 5, half = tid >> 7;
  const bool lead = half_lead_warp();
  auto elem_of = [&](int o) { return (o * C + rank) * 32 + lane; };

  auto put_q = [&](int o, int k, double q) {
    s.Q[(o * kMaxSteps + k) * 32 + lane] = q;
    s.Qf[(o * kMaxSteps + k) * 32 + lane] = d_to_f2(q);
  };

  // tiles: the extra ones into shared memory, the first into registers
  float x[8][8];
  for (int t = rank + C, i = 0; t < ntiles; t += C, ++i) {
    const TileGeom g = tile_geom(t);
    if (tid == 0) s.geo[i + 1] = make_int2(g.bi, g.bj);
    tile_load_x(X, ld, n, g, x);
    float4* xt = s.xs + i * 16 * kNT;
#pragma unroll
    for (int k = 0; k < 8; ++k) {
      xt[kNT * (2 * k) + tid] = make_float4(x[k][0], x[k][1], x[k][2], x[k][3]);
      xt[kNT * (2 * k + 1) + tid] = make_float4(x[k][4], x[k][5], x[k][6], x[k][7]);
    }
  }
  if (rank < ntiles) {
    const TileGeom g = tile_geom(rank);
    if (tid == 0) s.geo[0] = make_int2(g.bi, g.bj);
    tile_load_x(X, ld, n, g, x);
  }

  // start vector: every CTA forms all of it (no communication)
  for (int vb = 0; vb < nv; ++vb) {
    const int e = vb * kNT + tid;
    const double v = e < n ? lanczos_start(e) : 0.0;
    const double sum = block_sum64(v * v, s.bs);
    if (tid == 0) s.norms[vb] = sum;
  }
  if (tid == 0) *s.mdiag = 0u;
  __syncthreads();
  if (tid < 32) {
    double t = lane < nv ? s.norms[lane] : 0.0;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
    if (lane == 0) s.scalar[0] = 1.0 / sqrt(t);
  }
  __syncthreads();
  {
    const double inv = s.scalar[0];
    for (int e = tid; e < nb * kSymvTile; e += kNT)
      s.vh[e] = e < n ? __double2float_rn(lanczos_start(e) * inv) : 0.f;
    for (int o = wp; o < nown; o += kNT / 32) {
      const int e = elem_of(o);
      const double q = e < n ? lanczos_start(e) * inv : 0.0;
      put_q(o, 0, q);
      if (jb.zsave && e < n) jb.Qv[e] = q;
    }
  }
  cluster_sync_all();  // every CTA of the cluster runs before any remote store
  // The cluster's barriers are the hardware's and have no limit of their own.  A wait
  // limit of 0 (psd_debug_set) gives up here, where the other forms' first barrier
  // does: one CTA alone (one chunk of 32 elements) has nobody to wait for.
  if (g_debug_barrier_limit_ns == 0ull && nch > 1) {  // the same in every CTA
    if (rank == 0 && tid == 0) {
      st->m = st->done = 0;
      st->maxdiag_bits = st->absmax_bits = 0;
      st->sigma = st->resid = st->lambda = st->fro = st->maxdiag = st->inv_lambda = 0.0;
      st->status = PSD_ERR_TIMEOUT;
    }
    return;
  }

  // an element of the mat-vec input (0 past n) to every CTA
  auto put_vh = [&](int e, float h) {
    const uint32_t a = smem_u32(s.vh + e);
    if (e >= n) h = 0.f;
#pragma unroll 4
    for (int r = 0; r < C; ++r) st_remote(a, r, h);
  };
  // a double-float partial of chunk ch to every CTA
  auto put_norm2 = [&](int ch, const F2& t) {
    if (lane < C) st_remote(smem_u32(s.norms2 + ch), lane, make_float2(t.h, t.l));
  };
  // u = X v: split for the second product, the chunks' shares of ||u||^2
  auto reduce_split = [&](double* u) {
    for (int it = 0; it < nit; ++it) {
      const int o = 2 * it + half, e = elem_of(o);
      const F2 y = cl_reduce(s, n, nb, o, nown, e, nbmax);
      if (lead && o < nown) {
        put_vh(e, y.h);
        if (u && e < n) u[e] = f2_to_d(y);
        put_norm2(o * C + rank, warp_sum_f2(f2_mul(y, y)));
      }
    }
  };

  double fro = 0.0;
  int m = 0;
  for (int j = 0; j < kMaxSteps; ++j) {
    if (j == 0)
      cl_product<true>(s, n, ntiles, rank, C, nbmax, x);
    else
      cl_product<false>(s, n, ntiles, rank, C, nbmax, x);
    cluster_sync_all();
    if (j == 0) {  // ||X||_F from the tiles' sums (each warp alike)
      double t = 0.0;
      for (int k = lane; k < ntiles; k += 32) t += s.fro[k];
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
      fro = sqrt(t);
    }
    reduce_split(jb.zsave ? jb.zsave + j * jb.npad : nullptr);
    cluster_sync_all();
    cl_product<false>(s, n, ntiles, rank, C, nbmax, x);
    cluster_sync_all();
    // w = X u, w' and its dots (ph_reduce_dots); alpha_j by a warp that only helps to reduce
    if (wp == 1) {
      const double a = warp_sum_chunks(s.norms2, nch, LoadPlain());
      if (lane == 0) s.scalar[3] = a;
    }
    if (nit == 0) __syncthreads();
    for (int it = 0; it < nit; ++it) {
      const int o = 2 * it + half, e = elem_of(o);
      const F2 y = cl_reduce(s, n, nb, o, nown, e, nbmax);
      if (!(lead && o < nown)) continue;
      const double alpha = s.scalar[3];  // published by cl_reduce's barriers
      const double* Qo = s.Q + o * kMaxSteps * 32 + lane;
      const float2* Qfo = s.Qf + o * kMaxSteps * 32 + lane;
      const double w = lanczos_recur(f2_to_d(y), alpha, Qo[j * 32], j > 0 ? s.beta[j - 1] : 0.0,
                                     j > 0 ? Qo[(j - 1) * 32] : 0.0);
      s.w[o * 32 + lane] = w;
      const float2 d = chunk_dots(f2_of(e < n ? w : 0.0), j, [&](int k) { return F2{Qfo[k * 32].x, Qfo[k * 32].y}; });
      const uint32_t a = smem_u32(s.dots + lane * s.dstride + o * C + rank);
#pragma unroll 4
      for (int r = 0; r < C; ++r) st_remote(a, r, d);
    }
    cluster_sync_all();
    // Gram-Schmidt pass and q_{j+1} (ph_orth_next)
    chunk_sums(s.dots, nch, s.dstride, j, s.hs, LoadPlain());
    __syncthreads();
    if (wp == 7) {
      beta_of_sums(s.hs, j, s.scalar);
    } else if (wp == 6) {
      const double alpha = s.scalar[3];
      if (lane == 0) s.alpha[j] = alpha + f2_to_d(F2{s.hs[j].x, s.hs[j].y});
    }
    const double h = wp < nown && lane <= j ? f2_to_d(F2{s.hs[lane].x, s.hs[lane].y}) : 0.0;
    double wo[2] = {0.0, 0.0};  // own chunks wp, wp + 8 (at most 16 chunks a CTA)
    auto next = [&](int o) {
      double qk[kMaxSteps];
#pragma unroll
      for (int k = 0; k < kMaxSteps; ++k) qk[k] = k <= j ? s.Q[(o * kMaxSteps + k) * 32 + lane] : 0.0;
      return lanczos_orth(s.w[o * 32 + lane], h, qk, j);
    };
    if (wp < nown) wo[0] = next(wp);
    if (wp + 8 < nown) wo[1] = next(wp + 8);
    __syncthreads();
    const double bt = s.scalar[0], inv = s.scalar[1];
    const bool stop = !(bt > kBreakdown * (fro * fro)) || j == kMaxSteps - 1;  // also true for NaN
    if (tid == 0) s.beta[j] = bt;
    m = j + 1;
    if (stop) break;  // the same decision in every CTA
#pragma unroll
    for (int i = 0; i < 2; ++i) {
      const int o = wp + 8 * i;
      if (o < nown) {
        const int e = elem_of(o);
        const double q = wo[i] * inv;
        put_q(o, j + 1, q);
        if (jb.zsave && e < n) jb.Qv[static_cast<int64_t>(j + 1) * jb.npad + e] = q;
        put_vh(e, __double2float_rn(q));
      }
    }
    cluster_sync_all();
  }
  __syncthreads();
  // largest Ritz pair (every CTA alike), the Ritz vector and its residual
  if (wp == 0) {
    const double sigma = tridiag_top_eig(s.alpha, s.beta, m, s.y, s.a32, s.b32);
    if (lane == 0) s.scalar[2] = sigma;
  }
  __syncthreads();
  const double sigma = s.scalar[2];
  double ro[2] = {0.0, 0.0};
#pragma unroll
  for (int i = 0; i < 2; ++i) {
    const int o = wp + 8 * i;
    if (o < nown) {
      const int e = elem_of(o);
      double qk[kMaxSteps], yk[kMaxSteps];
#pragma unroll
      for (int k = 0; k < kMaxSteps; ++k) {
        qk[k] = k < m ? s.Q[(o * kMaxSteps + k) * 32 + lane] : 0.0;
        yk[k] = k < m ? s.y[k] : 0.0;
      }
      ro[i] = e < n ? lanczos_ritz(yk, qk, m) : 0.0;
      put_norm2(o * C + rank, warp_sum_f2(f2_of(ro[i] * ro[i])));
    }
  }
  cluster_sync_all();
  {
    const double s2 = warp_sum_chunks(s.norms2, nch, LoadPlain());
    const double inv = s2 > 0.0 ? 1.0 / sqrt(s2) : 0.0;
#pragma unroll
    for (int i = 0; i < 2; ++i) {
      const int o = wp + 8 * i;
      if (o < nown) {
        const double q = ro[i] * inv;
        s.w[o * 32 + lane] = q;
        put_vh(elem_of(o), __double2float_rn(q));
      }
    }
  }
  cluster_sync_all();
  cl_product<false>(s, n, ntiles, rank, C, nbmax, x);
  cluster_sync_all();
  reduce_split(nullptr);
  cluster_sync_all();
  cl_product<false>(s, n, ntiles, rank, C, nbmax, x);
  cluster_sync_all();
  for (int it = 0; it < nit; ++it) {
    const int o = 2 * it + half, e = elem_of(o);
    const F2 y = cl_reduce(s, n, nb, o, nown, e, nbmax);
    if (!(lead && o < nown)) continue;
    const double r = e < n ? fma(-sigma, s.w[o * 32 + lane], f2_to_d(y)) : 0.0;
    put_norm2(o * C + rank, warp_sum_f2(f2_of(r * r)));
  }
  cluster_sync_all();
  if (rank == 0 && wp == 0) {
    const double r2 = warp_sum_chunks(s.norms2, nch, LoadPlain());
    unsigned md = lane < C ? ld_remote(s.mdiag, lane) : 0u;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) md = max(md, __shfl_xor_sync(0xffffffffu, md, o));
    if (lane < kMaxSteps) {
      st->alpha[lane] = lane < m ? s.alpha[lane] : 0.0;
      st->beta[lane] = lane < m ? s.beta[lane] : 0.0;
      st->y[lane] = s.y[lane];
    }
    if (lane == 0) {
      st->sigma = sigma;
      st->fro = fro;
      st->m = m;
      st->done = m;
      st->status = 0;
      st->maxdiag_bits = md;
      st->absmax_bits = 0;
      record_bound(st, jb.args->info, n, r2, fro, static_cast<double>(__uint_as_float(md)), sigma, m,
                   g_debug_bound_scale);
    }
  }
  cluster_sync_all();  // no CTA exits while another reads its shared memory
}

// CTAs for `ntiles` tiles (one tile per CTA as far as 16 CTAs go), and tiles
// per CTA beyond the first.
inline void cluster_shape(int ntiles, int& csize, int& extra) {
  csize = 1;
  while (csize < kClusterMaxSize && csize < ntiles) csize *= 2;
  extra = (ntiles + csize - 1) / csize - 1;
}
