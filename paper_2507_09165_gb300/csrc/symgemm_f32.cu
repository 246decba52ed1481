// Symmetric product of the FP32 path: operands as scaled FP16 hi/lo pairs, three
// FP16 tensor-core products per K-step, promoted FP32 accumulation in registers.
//
// A matrix M of the FP32 chain is stored as hi = RN16(2^s M), lo = RN16(2^s M -
// hi): about 22 significant bits.  The power of two 2^s lifts the lo parts of
// the iterates' entries (~1/sqrt(n)) out of FP16's subnormals, which otherwise
// cap an unscaled pair at an absolute 2^-25 (chain.h F32Range).  The products
// run on SM pairs (tcgen05.mma.cta_group::2, M = 256) as in symgemm.cu and
// symgemm_x3.cu, at the FP16 rate: twice that of the TF32 split.
//
// The tensor cores add into FP32 accumulators without rounding to nearest, so
// over a whole product the error would grow like n.  K is therefore
// accumulated in chunks of kChunkK elements: the MMA warp alternates two
// 256-column tensor-memory buffers, and the 8 epilogue warps add each finished
// chunk to running FP32 sums (round to nearest, chunks in order) that they keep
// in registers, 128 per thread.  The sums used to live in tensor memory next to
// the only chunk buffer, and the tensor cores waited for every fold.
// What bounds it: the tensor cores (n = 10,000: 1.72 ms alone, 1,789 TFLOP/s, 0.94
// of the measured 16-bit rate; TF32 pairs on one SM took 4.0 ms); at small orders the
// K loop of a single round of tiles and the launch itself (n = 256: ~9 us a product).
#include <cuda_fp16.h>

#include <algorithm>
#include <mutex>

#include "epilogue.cuh"
#include "internal.h"
#include "ptx.cuh"

namespace psd {

namespace {

constexpr int kBM = 128;
constexpr int kBN = 256;
constexpr int kEW = 8;                    // epilogue warps: two per 32-lane quarter
// Warps 0-3: producer, MMA issue, two idle; warps 4-11: epilogue.  384 threads
// x 168 registers = 64,512 at launch, dealt as 128 x 40 + 256 x 232 = 64,512.
constexpr int kThreadsF = 128 + 32 * kEW;
constexpr int kRegsIo = 40, kRegsEpi = 232;
static_assert(128 * kRegsIo + 256 * kRegsEpi <= kThreadsF * 168, "register shares within the launch's registers");
// 3 stages of 64 KB: 128 rows of A_hi, A_lo, B_hi, B_lo (B: this CTA's half),
// 64 K elements (128-byte rows, 128-byte swizzle).  6 stages of 64-byte rows in
// the same space measured 4-8% slower (n = 3001: 4.07 against 3.76 ms).
constexpr int kRowBytesF = kRowBytesF32;
constexpr int kKElems = kRowBytesF / 2;
constexpr int kOpBytes = kBM * kRowBytesF;  // 16 KB
constexpr int kStageBytesF = 4 * kOpBytes;
constexpr int kStagesF = 3;
constexpr int kChunkK = 128;
constexpr int kChunkBlocks = kChunkK / kKElems;
constexpr int kEpiBytesF = 32 * kStgWords * 4;  // per warp: 32 x 32 words (stage outputs) or 32 x 33 (final)
constexpr int kTmemCols = 512;
__host__ __device__ constexpr int smem_bytes_f32() {
  return 1024 + kStagesF * kStageBytesF + kEW * kEpiBytesF + 8 * (2 * kStagesF + 5) + 16;
}
static_assert(smem_bytes_f32() <= 232448, "shared memory per CTA");
// A wait that has given up leaves copies of this CTA in flight, which signal
// the leader's barrier: they are given this long to land before the CTA exits.
constexpr unsigned long long kDrainNs = 200000ull;

__device__ __forceinline__ __half2 as_h2(uint32_t w) { return *reinterpret_cast<const __half2*>(&w); }
__device__ __forceinline__ float2 unpack_h2(uint32_t w) { return __half22float2(*reinterpret_cast<const __half2*>(&w)); }

// 8 consecutive pair elements (w[e] = hi | lo << 16) to memory, clipped at `valid`.
__device__ __forceinline__ void store_pair8(uint16_t* dh, uint16_t* dl, const uint32_t (&w)[8], int valid) {
  uint32_t h[4], l[4];
#pragma unroll
  for (int e = 0; e < 4; ++e) {
    h[e] = __byte_perm(w[2 * e], w[2 * e + 1], 0x5410);
    l[e] = __byte_perm(w[2 * e], w[2 * e + 1], 0x7632);
  }
  if (valid >= 8) {
    *reinterpret_cast<uint4*>(dh) = make_uint4(h[0], h[1], h[2], h[3]);
    *reinterpret_cast<uint4*>(dl) = make_uint4(l[0], l[1], l[2], l[3]);
  } else {
    for (int e = 0; e < valid; ++e) {
      dh[e] = static_cast<uint16_t>(w[e]);
      dl[e] = static_cast<uint16_t>(w[e] >> 16);
    }
  }
}

// A warp's staging square: 32 rows of 32 words, the 16-byte group g of row t at
// g ^ (t & 7).  Word stores down a column of rows, 16-byte stores and loads along
// a row per lane, and 16-byte loads of 64-byte segments (4 lanes a row) are all
// free of bank conflicts.
__device__ __forceinline__ int sq_word(int t, int e) { return 32 * t + ((((e >> 2) ^ (t & 7)) << 2) | (e & 3)); }
__device__ __forceinline__ uint4* sq_group(uint32_t* S, int t, int g) {
  return reinterpret_cast<uint4*>(S + 32 * t) + (g ^ (t & 7));
}
// Row t of the square: the 8 words from 8 seg on.
__device__ __forceinline__ void sq_load8(uint32_t* S, int t, int seg, uint32_t (&w)[8]) {
  const uint4 a = *sq_group(S, t, 2 * seg), b = *sq_group(S, t, 2 * seg + 1);
  w[0] = a.x; w[1] = a.y; w[2] = a.z; w[3] = a.w;
  w[4] = b.x; w[5] = b.y; w[6] = b.z; w[7] = b.w;
}

// Moves the sums of a warp's later chunks one chunk down (a loop over chunks
// with the sums in fixed registers: unrolled code for four chunks spills).
__device__ __forceinline__ void next_chunk(float (&sum)[4][32]) {
#pragma unroll
  for (int i = 0; i < 3; ++i)
#pragma unroll
    for (int j = 0; j < 32; ++j) sum[i][j] = sum[i + 1][j];
}

__device__ __forceinline__ void prefetch_l2(const void* p) {
  asm volatile("prefetch.global.L2 [%0];" ::"l"(p));
}

struct EpiOut {
  uint16_t *hi, *lo;         // the block's output pair
  const uint16_t *yh, *yl;   // EPI_POLY: the block's Y pair
  float cacc, cy, cdiag;     // stored value = cacc * acc + cy * (y_hi + y_lo) (+ cdiag on the diagonal)
  float unscale;             // stored value -> value (the report's largest)
};

// One 32 x 32 chunk: lane l holds row r0 + l, v[j] the FP32 sum at column c0 + j.
// Global memory is read (Y) and written in segments of 64 bytes by 4 lanes
// (whole sectors), 8 rows an instruction; between that shape and a row per
// lane everything goes through the staging square as hi | lo words.  The square
// holds the chunk transposed for the mirrored rows (c, r) and then as it is for
// (r, c); a diagonal chunk is symmetrised from its upper part and written once.
// With scalar conversions and staged words read one by one a chunk took
// 5000-7500 cycles and the tensor cores waited at the end of every tile; with a
// row per lane in global memory (16-byte pieces of sectors) n = 3001 was 10% slower.
template <int EPI>
__device__ __forceinline__ void epilogue_pair(const EpiOut& eo, int n, int64_t ldc, int64_t ldy, int r0, int c0,
                                              const float* v, uint32_t* S, int lane, bool track,
                                              unsigned& amax_bits) {
  const int r = r0 + lane;
  const bool diag = r0 == c0;
  const int seg = lane & 3, sr = lane >> 2;  // segment and row (+ 8 k) of the global accesses
  const int nc = n - c0;                     // columns below the order, for the range check
  __half2 big = __float2half2_rn(0.f);
  uint32_t w[32];                            // the lane's row: hi | lo << 16
  if (EPI == EPI_POLY) {
    uint4 yh[4], yl[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      yh[k] = yl[k] = make_uint4(0u, 0u, 0u, 0u);
      const int rr = r0 + sr + 8 * k, c = c0 + 8 * seg;
      // rows hold round_up(n, 64) elements: a 16-byte load that starts below n stays inside (what lies past n is not used)
      if (rr < n && c < n) {
        yh[k] = __ldg(reinterpret_cast<const uint4*>(eo.yh + static_cast<int64_t>(rr) * ldy + c));
        yl[k] = __ldg(reinterpret_cast<const uint4*>(eo.yl + static_cast<int64_t>(rr) * ldy + c));
      }
    }
    __syncwarp();  // the previous chunk's reads of S are done
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      const uint32_t h[4] = {yh[k].x, yh[k].y, yh[k].z, yh[k].w}, l[4] = {yl[k].x, yl[k].y, yl[k].z, yl[k].w};
#pragma unroll
      for (int g = 0; g < 2; ++g)
        *sq_group(S, sr + 8 * k, 2 * seg + g) =
            make_uint4(__byte_perm(h[2 * g], l[2 * g], 0x5410), __byte_perm(h[2 * g], l[2 * g], 0x7632),
                       __byte_perm(h[2 * g + 1], l[2 * g + 1], 0x5410), __byte_perm(h[2 * g + 1], l[2 * g + 1], 0x7632));
    }
    __syncwarp();
#pragma unroll
    for (int g = 0; g < 8; ++g) {
      const uint4 a = *sq_group(S, lane, g);
      w[4 * g] = a.x; w[4 * g + 1] = a.y; w[4 * g + 2] = a.z; w[4 * g + 3] = a.w;
    }
  }
#pragma unroll
  for (int q = 0; q < 16; ++q) {
    float a = eo.cacc * v[2 * q], b = eo.cacc * v[2 * q + 1];
    if (EPI == EPI_POLY) {
      const float2 ya = unpack_h2(w[2 * q]), yb = unpack_h2(w[2 * q + 1]);  // (hi, lo)
      a = fmaf(eo.cacc, v[2 * q], eo.cy * (ya.x + ya.y));
      b = fmaf(eo.cacc, v[2 * q + 1], eo.cy * (yb.x + yb.y));
      if (diag && 2 * q == lane) a += eo.cdiag;
      if (diag && 2 * q + 1 == lane) b += eo.cdiag;
    }
    const uint32_t hi = pack_h2_sat(a, b);
    if (2 * q < nc) big = __hmax2(big, __habs2(as_h2(2 * q + 1 < nc ? hi : hi & 0xFFFFu)));
    const float2 h = unpack_h2(hi);
    const uint32_t lo = pack_h2_sat(a - h.x, b - h.y);
    w[2 * q] = __byte_perm(hi, lo, 0x5410);
    w[2 * q + 1] = __byte_perm(hi, lo, 0x7632);
  }
  // a value beyond FP16 is stored as +-65504 (+ up to as much in lo): the iterates stay
  // finite, and whatever the stage the report gives the size that did not fit
  const float2 bg = __half22float2(big);
  if (r < n && (track || fmaxf(bg.x, bg.y) == 65504.f)) {
#pragma unroll
    for (int j = 0; j < 32; ++j) {
      const float2 t = unpack_h2(w[j]);
      float m = fabsf(t.x + t.y);
      if (EPI != EPI_POLY && fabsf(eo.cacc * v[j]) > 65504.f) m = fabsf(eo.cacc * v[j]);
      if (c0 + j < n && (track || m >= 65504.f)) amax_bits = max(amax_bits, __float_as_uint(m * eo.unscale));
    }
  }
  __syncwarp();
#pragma unroll
  for (int j = 0; j < 32; ++j) S[sq_word(j, lane)] = w[j];  // row j = column c0 + j
  __syncwarp();
  if (!diag) {
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      const int jj = sr + 8 * k, c = c0 + jj, e0 = r0 + 8 * seg;
      uint32_t u[8];
      sq_load8(S, jj, seg, u);
      const int64_t at = static_cast<int64_t>(c) * ldc + e0;
      if (c < n && e0 < n) store_pair8(eo.hi + at, eo.lo + at, u, n - e0);
    }
  } else {
#pragma unroll
    for (int j = 0; j < 32; ++j) {
      const uint32_t up = S[sq_word(lane, j)];  // element (j, lane) of the upper part
      if (j < lane) w[j] = up;
    }
  }
  __syncwarp();
#pragma unroll
  for (int g = 0; g < 8; ++g) *sq_group(S, lane, g) = make_uint4(w[4 * g], w[4 * g + 1], w[4 * g + 2], w[4 * g + 3]);
  __syncwarp();
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    const int tt = sr + 8 * k, rr = r0 + tt, e0 = c0 + 8 * seg;
    uint32_t u[8];
    sq_load8(S, tt, seg, u);
    const int64_t at = static_cast<int64_t>(rr) * ldc + e0;
    if (rr < n && e0 < n) store_pair8(eo.hi + at, eo.lo + at, u, n - e0);
  }
}

template <int EPI>
__global__ void __launch_bounds__(kThreadsF, 1)
    symgemm_f32_kernel(const __grid_constant__ CUtensorMap tmAh, const __grid_constant__ CUtensorMap tmAl,
                       const __grid_constant__ CUtensorMap tmBh, const __grid_constant__ CUtensorMap tmBl,
                       const GemmParams p) {
  tmem_pair_enter();
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) &
                                             ~static_cast<uintptr_t>(1023));
  uint8_t* stages = smem;
  uint8_t* epi = smem + kStagesF * kStageBytesF;
  uint64_t* bars = reinterpret_cast<uint64_t*>(epi + kEW * kEpiBytesF);
  // bars: full[S] | empty[S] | tfull[2] | tempty[2] | drain
  uint32_t* tmem_holder = reinterpret_cast<uint32_t*>(bars + 2 * kStagesF + 5);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_holder + 1);

  const int warp = threadIdx.x >> 5;
  const int lane = threadIdx.x & 31;
  const uint32_t rank = cluster_ctarank();
  const bool leader = rank == 0;
  const int cl = static_cast<int>(blockIdx.x >> 1), ncl = static_cast<int>(gridDim.x >> 1);
  auto full_bar = [&](int s) { return smem_u32(bars + s); };
  auto empty_bar = [&](int s) { return smem_u32(bars + kStagesF + s); };
  auto tfull_bar = [&](int a) { return smem_u32(bars + 2 * kStagesF + a); };
  auto tempty_bar = [&](int a) { return smem_u32(bars + 2 * kStagesF + 2 + a); };
  const uint32_t drain_bar = smem_u32(bars + 2 * kStagesF + 4);

  if (threadIdx.x == 0) {
    for (int s = 0; s < kStagesF; ++s) {
      mbar_init(full_bar(s), 1);
      mbar_init(empty_bar(s), 1);
    }
    for (int a = 0; a < 2; ++a) {
      mbar_init(tfull_bar(a), 1);
      mbar_init(tempty_bar(a), 2 * kEW);  // the leader's: the epilogue warps of both CTAs
    }
    mbar_init(drain_bar, 1);
    *abort_flag = 0;
    fence_mbar_init();
    tma_prefetch_desc(&tmAh);
    tma_prefetch_desc(&tmAl);
    tma_prefetch_desc(&tmBh);
    tma_prefetch_desc(&tmBl);
  }
  const uint32_t tmem_base = tmem_pair_setup(tmem_holder, kTmemCols);

  if (warp < 4) {
    reg_dec<kRegsIo>();
    if (warp == 0) {
      if (lane == 0) {
        uint32_t s = 0, ph = 0;
        bool ok = true, issued = false;
        const uint32_t stage_tx = 4 * (kOpBytes + p.b_rows() * kRowBytesF);
        for (TileStream ts(p, cl, ncl); ok && ts.valid(); ts.advance()) {
          ts.prefetch();
          const TileMeta& m = ts.cur();
          const int4 tc = m.tc;
          const int kbn = (m.n + kKElems - 1) / kKElems;
          // this CTA's 128 rows of A and its N/2 rows of B
          const int ya = static_cast<int>(m.off + tc.x + 128 * static_cast<int>(rank));
          const int yb = static_cast<int>(m.off + m.db + tc.y + (tc.w >> 1) * static_cast<int>(rank));
          for (int kb = 0; kb < kbn; ++kb) {
            if (!wait_bounded(empty_bar(s), ph ^ 1u, abort_flag)) {
              ok = false;
              break;
            }
            if (leader) mbar_arrive_expect_tx(full_bar(s), stage_tx);  // both CTAs' copies
            const uint32_t dst = smem_u32(stages + s * kStageBytesF);
            const uint32_t fb = mapa_shared(full_bar(s), 0);
            tma_load_2d_pair(dst, &tmAh, kb * kKElems, ya, fb);
            tma_load_2d_pair(dst + kOpBytes, &tmAl, kb * kKElems, ya, fb);
            tma_load_2d_pair(dst + 2 * kOpBytes, &tmBh, kb * kKElems, yb, fb);
            tma_load_2d_pair(dst + 3 * kOpBytes, &tmBl, kb * kKElems, yb, fb);
            issued = true;
            if (++s == kStagesF) {
              s = 0;
              ph ^= 1u;
            }
          }
        }
        // the ring's last commits have arrived: none is on its way to a CTA that has left
        for (int q = 0; ok && q < kStagesF; ++q) {
          ok = wait_bounded(empty_bar(s), ph ^ 1u, abort_flag);
          if (++s == kStagesF) {
            s = 0;
            ph ^= 1u;
          }
        }
        if (!ok && issued) {
          const unsigned long long t0 = globaltimer_ns();
          while (globaltimer_ns() - t0 < kDrainNs) {
          }
        }
      }
    } else if (warp == 1) {
      if (leader) {  // issues for both CTAs
        uint32_t s = 0, ph = 0, acc = 0, acc_ph = 0;
        bool ok = true;
        for (TileStream ts(p, cl, ncl); ok && ts.valid(); ts.advance()) {
          ts.prefetch();
          const int4 tc = ts.cur().tc;
          const int kbn = (ts.cur().n + kKElems - 1) / kKElems;
          const uint32_t idesc = p.idesc | (static_cast<uint32_t>(tc.w >> 3) << 17);  // M = 256, N = tile width
          for (int kc = 0; ok && kc < kbn; kc += kChunkBlocks) {
            if (!wait_bounded(tempty_bar(acc), acc_ph ^ 1u, abort_flag)) {
              ok = false;
              break;
            }
            tc_fence_after();
            const uint32_t d_tmem = tmem_base + acc * kBN;
            const int kend = min(kbn, kc + kChunkBlocks);
            for (int kb = kc; kb < kend; ++kb) {
              if (!wait_bounded(full_bar(s), ph, abort_flag)) {
                ok = false;
                break;
              }
              tc_fence_after();
              if (lane == 0) {
                const uint32_t ah = smem_u32(stages + s * kStageBytesF);
                const uint32_t al = ah + kOpBytes, bh = ah + 2 * kOpBytes, bl = ah + 3 * kOpBytes;
  #pragma unroll
                for (int k = 0; k < kRowBytesF / 32; ++k) {
                  const uint32_t off = 32 * k;
                  const uint32_t more = ((kb - kc) | k) == 0 ? 0u : 1u;
                  mma_f16_pair(d_tmem, sw128_kmajor_desc(ah + off), sw128_kmajor_desc(bl + off), idesc, more);
                  mma_f16_pair(d_tmem, sw128_kmajor_desc(al + off), sw128_kmajor_desc(bh + off), idesc, 1u);
                  mma_f16_pair(d_tmem, sw128_kmajor_desc(ah + off), sw128_kmajor_desc(bh + off), idesc, 1u);
                }
                mma_commit_pair(empty_bar(s), 3);  // frees the stage in both CTAs
              }
              __syncwarp();
              if (++s == kStagesF) {
                s = 0;
                ph ^= 1u;
              }
            }
            if (!ok) break;
            if (lane == 0) mma_commit_pair(tfull_bar(acc), 3);
            __syncwarp();
            acc ^= 1u;
            if (acc == 0) acc_ph ^= 1u;
          }
        }
        if (!ok && lane == 0) {
          mma_commit_pair(drain_bar, 1);  // the MMAs already issued, before tensor memory is released
          const unsigned long long t0 = globaltimer_ns();
          while (!mbar_try_wait(drain_bar, 0) && globaltimer_ns() - t0 < kWaitLimitNs) {
          }
        }
        __syncwarp();
      }
    }
  } else {
    reg_inc<kRegsEpi>();
    const int ew = warp & 3;   // tensor-memory lane quarter
    const int ewi = warp - 4;  // epilogue warp 0 .. 7
    const int half = ewi >> 2; // this warp's chunks of the quarter: half, half + 2, ... (32 columns each)
    uint8_t* wbuf = epi + ewi * kEpiBytesF;
    uint32_t acc = 0, acc_ph = 0;
    unsigned amax_bits = 0;
    int amax_block = -1;
    const bool track_launch = p.ep.absmax_blocks != 0 || p.ep.absmax != nullptr;
    auto flush_amax = [&](int blk) {
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) amax_bits = max(amax_bits, __shfl_xor_sync(0xffffffffu, amax_bits, o));
      if (lane == 0 && amax_bits) {
        unsigned* dst = p.ep.absmax ? p.ep.absmax : &p.blocks[blk].st->absmax_bits;
        atomicMax(dst, amax_bits);
      }
      amax_bits = 0;
    };
    const uint32_t tempty_leader[2] = {mapa_shared(tempty_bar(0), 0), mapa_shared(tempty_bar(1), 0)};
    for (int t = cl; t < p.num_tiles; t += ncl) {
      const int4 tc = p.tiles[t];
      const BlockRec& br = p.blocks[tc.z];
      const int n = br.n;
      if (EPI != EPI_FINAL && amax_block != tc.z) {
        if (amax_block >= 0) flush_amax(amax_block);
        amax_block = tc.z;
      }
      const int r0 = tc.x + 128 * static_cast<int>(rank) + 32 * ew;
      // chunks of this warp's 32 rows that lie on or above the diagonal and inside n
      const int ch_begin = max(0, (r0 - tc.y) >> 5);
      const int ch_end = r0 < n ? min((tc.w + 31) >> 5, (n - tc.y + 31) >> 5) : ch_begin;
      const uint32_t lanes = static_cast<uint32_t>(32 * ew) << 16;
      const int kbn = (n + kKElems - 1) / kKElems;
      if (EPI == EPI_POLY && r0 + lane < n) {  // this tile's Y towards L2 while the products run
        const int64_t at = (br.off + br.dy + r0 + lane) * p.ep.ldy + tc.y;
        for (int ch = max(half, ch_begin + ((ch_begin ^ half) & 1)); ch < ch_end; ch += 2) {
          prefetch_l2(static_cast<const uint16_t*>(p.ep.Y) + at + 32 * ch);
          prefetch_l2(static_cast<const uint16_t*>(p.ep.Y_lo) + at + 32 * ch);
        }
      }
      float sum[4][32] = {};
      bool ok = true;
      for (int kc = 0; kc < kbn; kc += kChunkBlocks) {
        if (!wait_bounded(tfull_bar(acc), acc_ph, abort_flag)) {
          ok = false;
          break;
        }
        tc_fence_after();
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          const int ch = half + 2 * i;
          if (ch >= ch_begin && ch < ch_end) {  // the same for the whole warp
            uint32_t v[32];
            tmem_ld32(tmem_base + lanes + acc * kBN + 32 * ch, v);
#pragma unroll
            for (int j = 0; j < 32; ++j) sum[i][j] += __uint_as_float(v[j]);
          }
        }
        tc_fence_before();
        __syncwarp();
        if (lane == 0) {
          if (leader)
            mbar_arrive(tempty_bar(acc));
          else
            mbar_arrive_remote(tempty_leader[acc]);
        }
        acc ^= 1u;
        if (acc == 0) acc_ph ^= 1u;
      }
      if (!ok) break;
      if constexpr (EPI == EPI_FINAL) {
        const float lam = static_cast<float>(br.st->lambda) * p.ep.in_scale;  // a power of two: exact
        ComplAcc cacc;
        ComplAcc* cap = p.ep.cres ? &cacc : nullptr;
#pragma unroll 1
        for (int ch = half; ch < kBN / 32; ch += 2) {
          if (ch >= ch_begin && ch < ch_end) {
            uint32_t v[32];
#pragma unroll
            for (int j = 0; j < 32; ++j) v[j] = __float_as_uint(sum[0][j]);
            epilogue_chunk_final(br, r0, tc.y + 32 * ch, v, wbuf, lane, lam, cap);
          }
          next_chunk(sum);
        }
        if (cap) {
          const double cs = compl_warp_sum(cacc);
          if (lane == 0) p.ep.cres[2 * kEW * static_cast<int64_t>(t) + kEW * static_cast<int>(rank) + ewi] = cs;
        }
      } else {
        const int64_t row = br.off + br.dc, yrow = br.off + br.dy;
        EpiOut eo;
        eo.hi = static_cast<uint16_t*>(p.ep.C) + row * p.ep.ldc;
        eo.lo = static_cast<uint16_t*>(p.ep.C_lo) + row * p.ep.ldc;
        eo.yh = EPI == EPI_POLY ? static_cast<const uint16_t*>(p.ep.Y) + yrow * p.ep.ldy : nullptr;
        eo.yl = EPI == EPI_POLY ? static_cast<const uint16_t*>(p.ep.Y_lo) + yrow * p.ep.ldy : nullptr;
        const float factor = EPI == EPI_POLY ? p.ep.c : EPI == EPI_SCALE ? p.ep.s : 1.f;
        eo.cacc = factor * (p.ep.in_scale * p.ep.out_scale);  // scales: powers of two, exact
        eo.cy = p.ep.b * (p.ep.y_scale * p.ep.out_scale);
        eo.cdiag = p.ep.a * p.ep.out_scale;
        eo.unscale = 1.f / p.ep.out_scale;
#pragma unroll 1
        for (int ch = half; ch < kBN / 32; ch += 2) {
          if (ch >= ch_begin && ch < ch_end)
            epilogue_pair<EPI>(eo, n, p.ep.ldc, p.ep.ldy, r0, tc.y + 32 * ch, sum[0],
                               reinterpret_cast<uint32_t*>(wbuf), lane, track_launch, amax_bits);
          next_chunk(sum);
        }
      }
      __syncwarp();
    }
    if (EPI != EPI_FINAL && amax_block >= 0) flush_amax(amax_block);
  }

  // every operand read, remote arrival and copy of the pair is complete
  // before either CTA releases tensor memory or exits
  tmem_pair_teardown(tmem_base, kTmemCols);
  if (threadIdx.x == 0 && *abort_flag) raise_status(p.ep.status, PSD_ERR_TIMEOUT);
}

using KernelF32 = void (*)(const CUtensorMap, const CUtensorMap, const CUtensorMap, const CUtensorMap,
                           const GemmParams);

}  // namespace

cudaError_t launch_symgemm_f32(int epi, const CUtensorMap* tm, const GemmParams& p, int grid, cudaStream_t stream) {
  if (p.num_tiles == 0) return cudaSuccess;
  static const KernelF32 kernels[4] = {symgemm_f32_kernel<EPI_COPY>, symgemm_f32_kernel<EPI_POLY>,
                                       symgemm_f32_kernel<EPI_SCALE>, symgemm_f32_kernel<EPI_FINAL>};
  if (epi < EPI_COPY || epi > EPI_FINAL) return cudaErrorInvalidValue;
  static std::mutex attr_mu;  // launches come from several callers' threads
  static bool attr_set[4] = {};
  {
    std::lock_guard<std::mutex> lk(attr_mu);
    if (!attr_set[epi]) {
      cudaError_t e =
          cudaFuncSetAttribute(kernels[epi], cudaFuncAttributeMaxDynamicSharedMemorySize, smem_bytes_f32());
      if (e != cudaSuccess) return e;
      attr_set[epi] = true;
    }
  }
  GemmParams q = p;
  q.idesc = make_idesc(0u, 2 * kBM, 0);  // FP16 operands, M = 256; N comes from each tile
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3(2 * std::max(1, std::min(grid / 2, p.num_tiles)));
  cfg.blockDim = dim3(kThreadsF);
  cfg.dynamicSmemBytes = smem_bytes_f32();
  cfg.stream = stream;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = 2;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, kernels[epi], tm[0], tm[1], tm[2], tm[3], q);
}

}  // namespace psd
