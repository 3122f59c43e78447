// mmd.cu -- corpus similarity by maximum mean discrepancy (Sec. 5 of the
// paper, the MMD equation): MMD(X, Y) = 1/(n n) sum over i, j of
// [2 d(x_i, y_j) - d(x_i, x_j) - d(y_i, y_j)], with d an l1 distance between
// embeddings of the sounds. The library's embedding is its log-mel feature
// vector (345 frames x 128 bands = 44160 bf16 values for a 4 s voice).
//
// Two kernels:
//  * l1_distance_kernel: the pooled pairwise distance matrix of m embeddings,
//    d[i][j] = sum_k |e_i[k] - e_j[k]|, through
//      sum_k |a - b| = 2 sum_k max(a, b) - sum_k a - sum_k b.
//    A maximum of two bf16 values is a bf16 value, so one packed instruction
//    takes two exact maxima, and the sums over k are products with a vector of
//    ones on the tensor cores (mma.sync: the maxima are made in registers,
//    where the operand of tcgen05.mma cannot lie). See the kernel.
//  * mmd_trials_kernel: one CTA per trial; a trial labels each pooled sound
//    0 (in X), 1 (in Y) or neither. Each warp walks rows of the distance
//    matrix that belong to X or Y and sums them by the column's label (FP32
//    within a row, FP64 across rows); the block adds its warps' sums in warp
//    order (deterministic) and forms
//    2 S_xy / (n_x n_y) - S_xx / n_x^2 - S_yy / n_y^2.

#include <cooperative_groups.h>
#include <cuda_bf16.h>

#include <algorithm>
#include <array>
#include <climits>
#include <cstdint>
#include <map>
#include <mutex>

#include "internal.h"

namespace synth {

namespace cg = cooperative_groups;

namespace {

// ---- pairwise l1 distances ---------------------------------------------------
// What bounds it: instruction issue. 256 element pairs cost four packed maxima
// and one m16n8k16 product, which holds a scheduler for eight slots (measured:
// a loop of nothing else reaches 81 pairs a clock and SM), twelve slots
// against sixteen for a subtraction and an addition of an absolute value per
// pair, the form that this replaces. Rows taken term by term beside the
// products did not overlap with them (a quarter of them: 10% slower).
// 3072 sounds x 44160 values: 14.93 ms before, 12.82 ms; 1024 sounds: 8.58
// -> 1.61 ms and 256: 8.29 -> 0.24 ms, where 128 x 128 tiles left SMs
// without work.
//
// Work: a CTA of 16 warps takes a 64 x 64 tile of the upper triangle (the
// mirror is written by the same CTA); a warp takes 8 rows x 32 columns. The 16
// rows of a product are 16 pairs: row g (g < 8) pairs one row i with column
// 8 jj + g, row g + 8 with column 8 (jj + 1) + g, and a lane's four values of
// k lie together in the embedding (the order of k does not matter to a sum),
// so that one 16-byte shared-memory load feeds two products. Chunks of 128
// values arrive by cp.async through three stages.
//
// Precision: with M the sum of maxima over 64 values, started from zero, and
// S_i, S_j the two rows' own sums over them formed by the same products, the
// running FP32 sum takes M - (S_i + S_j) / 2, half the distance over those
// values. It thus grows like the distance, not like the values, has 690
// additions at 44160 values instead of 44160, and is exactly 0 for equal rows. What
// the products lose is relative to the rows' sums of absolute values, N = N_i + N_j:
// at most 28 2^-24 N, so 28 2^-24 N / d of d. A sum of |a - b| term by term in FP32
// loses at most dim 2^-24 of d. So a pair goes through the maxima where
// N / d <= dim / 128, at most kCloseRatio (a bound of 4.3e-4 of d then, from dim =
// 32768 on; 1.3e-5 at 1024), and is computed again term by term beyond, as where a
// value is not finite. The line is where the errors of unrelated, shifted and heavy-
// tailed rows meet those of the term-by-term sum in order: root mean square against
// 64 bits, heavy-tailed rows, maxima / in order: 1024 values, N / d = 8.6: 9.3e-8 /
// 1.4e-7, 16: 1.3e-7 / 1.1e-7; 2816, 16: 1.3e-7 / 2.4e-7, 32: 2.0e-7 / 1.8e-7; 44160,
// 1.1: 1.0e-7 / 3.1e-6, 231: 6.4e-7 / 1.0e-6. Below kTermsDim values the maxima would
// pay for few pairs, and every tile is computed term by term: 3000 sounds of 512
// values 206 us (maxima and then terms for most tiles 380), of 128 values 65 (74).
constexpr int kDT = 64;            // distance tile (rows and columns)
constexpr int kDK = 128;           // embedding values per stage
constexpr int kDStages = 3;
constexpr int kDThreads = 512;
constexpr int kMaxCluster = 8;
constexpr float kCloseRatio = 256.f, kDimPerRatio = 128.f;
constexpr int kTermsDim = 1024;
constexpr int kListed = 512;       // close pairs of a tile computed one by one; more: the whole tile

struct L1Smem {
  uint4 stage[kDStages][2 * kDT][kDK / 8];  // rows of the tile, then its columns; 16-byte chunks
                                            // swizzled (l1_chunk)
  float h[2][2][2 * kDT];                   // of two stages, half the sum over each 64 values, per row
  float norm[2 * kDT];                      // sum of |e| over all values, per row
  int n_close;
  uint16_t close[kListed];
};

// Chunk c of a row: neighbouring rows lie 4 chunks apart and 8 consecutive
// rows in 8 different chunk columns, so that the 16-byte loads of 8 lanes (two
// rows of four chunks, or eight rows of one) cover all 32 banks.
__device__ __forceinline__ int l1_chunk(int row, int c) {
  return c ^ (((row & 1) << 2) | ((row >> 1) & 3));
}

__device__ __forceinline__ uint32_t max_bf16x2(uint32_t a, uint32_t b) {
  uint32_t r;
  asm("max.bf16x2 %0, %1, %2;" : "=r"(r) : "r"(a), "r"(b));
  return r;
}

// d += (the 16 x 16 bf16 values a) x ones: every column of d is the row's sum
__device__ __forceinline__ void add_rows(float (&d)[4], uint32_t a0, uint32_t a1, uint32_t a2,
                                         uint32_t a3, bool first) {
  const uint32_t ones = 0x3f803f80u;
  if (first) {
    asm("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%8}, "
        "{%9,%9,%9,%9};"
        : "=f"(d[0]), "=f"(d[1]), "=f"(d[2]), "=f"(d[3])
        : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(ones), "f"(0.f));
  } else {
    asm("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%8}, "
        "{%0,%1,%2,%3};"
        : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
        : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(ones));
  }
}

__device__ __forceinline__ float bf16_lo(uint32_t w) { return __uint_as_float(w << 16); }
__device__ __forceinline__ float bf16_hi(uint32_t w) { return __uint_as_float(w & 0xffff0000u); }

// acc += |a - b| over the 8 values of a 16-byte chunk, in order
__device__ __forceinline__ float add_abs_diff8(float acc, const uint4& a, const uint4& b) {
  const uint32_t wa[4] = {a.x, a.y, a.z, a.w}, wb[4] = {b.x, b.y, b.z, b.w};
#pragma unroll
  for (int u = 0; u < 4; ++u) {
    acc += fabsf(bf16_lo(wa[u]) - bf16_lo(wb[u]));
    acc += fabsf(bf16_hi(wa[u]) - bf16_hi(wb[u]));
  }
  return acc;
}

// Stage c of the tile at rows r0, columns c0: 2 x 64 rows of 128 values, zeros
// past the end of the rows and of dim.
__device__ __forceinline__ void l1_load(L1Smem& s, int slot, int c, const __nv_bfloat16* emb,
                                        int64_t ld, int m, int dim, int r0, int c0) {
  constexpr int kPer = 2 * kDT * (kDK / 8) / kDThreads;
#pragma unroll
  for (int l = 0; l < kPer; ++l) {
    const int e = threadIdx.x + l * kDThreads;
    const int row = e / (kDK / 8), ch = e % (kDK / 8);
    const int g = row < kDT ? r0 + row : c0 + row - kDT;
    const int k = c * kDK + ch * 8;
    const int bytes = g < m ? 2 * min(max(dim - k, 0), 8) : 0;
    const __nv_bfloat16* src = bytes > 0 ? emb + (int64_t)g * ld + k : emb;
    const uint32_t dst =
        (uint32_t)__cvta_generic_to_shared(&s.stage[slot][row][l1_chunk(row, ch)]);
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst), "l"(src), "r"(bytes)
                 : "memory");
  }
}
__device__ __forceinline__ void l1_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
__device__ __forceinline__ void l1_wait() { asm volatile("cp.async.wait_group 1;" ::: "memory"); }
__device__ __forceinline__ void l1_wait_all() { asm volatile("cp.async.wait_all;" ::: "memory"); }

// The tile's distances term by term. Two groups of 256 threads take half of the
// values each (every other 16-byte chunk); thread t of a group has rows
// t / 16 + 16 {0..3} and columns t % 16 + 16 {0..3}. The halves are then added, and
// the tile and its mirror written row by row.
__device__ __noinline__ void l1_tile_by_terms(L1Smem& s, const __nv_bfloat16* emb, int64_t ld,
                                              int m, int dim, int r0, int c0, float* dist) {
  const int n_chunks = (dim + kDK - 1) / kDK;
  const int group = threadIdx.x >> 8, ti = (threadIdx.x >> 4) & 15, tj = threadIdx.x & 15;
  float acc[4][4] = {};
  __syncthreads();
  l1_load(s, 0, 0, emb, ld, m, dim, r0, c0);
  l1_commit();
  if (n_chunks > 1) l1_load(s, 1, 1, emb, ld, m, dim, r0, c0);
  l1_commit();
  for (int c = 0; c < n_chunks; ++c) {
    l1_wait();
    __syncthreads();
    if (c + 2 < n_chunks) l1_load(s, (c + 2) % kDStages, c + 2, emb, ld, m, dim, r0, c0);
    l1_commit();
    const auto& st = s.stage[c % kDStages];
#pragma unroll 1
    for (int ch = group; ch < kDK / 8; ch += 2) {
      uint4 b[4];
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        const int row = kDT + tj + 16 * q;
        b[q] = st[row][l1_chunk(row, ch)];
      }
#pragma unroll
      for (int p = 0; p < 4; ++p) {
        const int row = ti + 16 * p;
        const uint4 a = st[row][l1_chunk(row, ch)];
#pragma unroll
        for (int q = 0; q < 4; ++q) acc[p][q] = add_abs_diff8(acc[p][q], a, b[q]);
      }
    }
  }
  l1_wait_all();
  __syncthreads();
  using Part = float[kDT][kDT + 1];
  static_assert(2 * sizeof(Part) <= sizeof(s.stage), "the halves fit the stages");
  Part* part = reinterpret_cast<Part*>(&s.stage[0][0][0]);
#pragma unroll
  for (int p = 0; p < 4; ++p)
#pragma unroll
    for (int q = 0; q < 4; ++q) part[group][ti + 16 * p][tj + 16 * q] = acc[p][q];
  __syncthreads();
  for (int e = threadIdx.x; e < kDT * kDT; e += kDThreads) {
    const int i = e / kDT, j = e % kDT;
    const float d = part[0][i][j] + part[1][i][j];
    part[0][i][j] = d;
    if (r0 + i < m && c0 + j < m) dist[(int64_t)(r0 + i) * m + c0 + j] = d;
  }
  __syncthreads();
  for (int e = threadIdx.x; e < kDT * kDT; e += kDThreads) {
    const int j = e / kDT, i = e % kDT;
    if (r0 + i < m && c0 + j < m) dist[(int64_t)(c0 + j) * m + r0 + i] = part[0][i][j];
  }
}

// A cluster of CTAs (1 to 8) shares a tile: each takes a part of the chunks,
// and the first adds their sums in rank order.
__global__ void __launch_bounds__(kDThreads, 1)
    l1_distance_kernel(const __nv_bfloat16* __restrict__ emb, int64_t ld, int m, int dim,
                       float* __restrict__ dist, float close_ratio) {
  extern __shared__ __align__(16) unsigned char l1_smem[];
  L1Smem& s = *reinterpret_cast<L1Smem*>(l1_smem);
  const cg::cluster_group cluster = cg::this_cluster();
  const int rank = (int)cluster.block_rank(), ranks = (int)cluster.num_blocks();
  // tile t of the upper triangle, row by row from the bottom: the last r + 1
  // tile rows hold (r + 1)(r + 2) / 2 tiles
  const int nb = (m + kDT - 1) / kDT;
  const int t = nb * (nb + 1) / 2 - 1 - (int)(blockIdx.x / ranks);
  int r = (int)((sqrtf(8.f * (float)t + 1.f) - 1.f) * 0.5f);
  while (r * (r + 1) / 2 > t) --r;
  while ((r + 1) * (r + 2) / 2 <= t) ++r;
  const int bi = nb - 1 - r, bj = nb - 1 - (t - r * (r + 1) / 2);
  const int r0 = bi * kDT, c0 = bj * kDT;
  if (dim < kTermsDim) {  // one CTA a tile
    l1_tile_by_terms(s, emb, ld, m, dim, r0, c0, dist);
    return;
  }

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int g = lane >> 2, q = lane & 3;
  const int wi = (warp >> 1) * 8, wj = (warp & 1) * 32;  // the warp's rows and columns in the tile
  const int n_chunks = (dim + kDK - 1) / kDK;
  const int beg = (int)((int64_t)n_chunks * rank / ranks);
  const int end = (int)((int64_t)n_chunks * (rank + 1) / ranks);

  // lane (g, q) keeps rows q and q + 4 of the warp's eight against columns 8 jj + g
  float run[2][4] = {};
  float nrm = 0.f;  // sum of |e| of row 8 warp + g of the 128
  if (threadIdx.x == 0) s.n_close = 0;
  // the sums of the warp's 8 of the 128 rows over stage c (product rows 0-7) and of their
  // magnitudes (rows 8-15)
  auto row_sums = [&](int c) {
    const int row = 8 * warp + g;
#pragma unroll
    for (int sub = 0; sub < 2; ++sub) {
      float d[4];
#pragma unroll
      for (int e = 0; e < 2; ++e) {
        const uint4 x = s.stage[c % kDStages][row][l1_chunk(row, 8 * sub + 4 * e + q)];
        add_rows(d, x.x, x.x & 0x7fff7fffu, x.y, x.y & 0x7fff7fffu, e == 0);
        add_rows(d, x.z, x.z & 0x7fff7fffu, x.w, x.w & 0x7fff7fffu, false);
      }
      if (q == 0) s.h[c & 1][sub][row] = 0.5f * d[0];
      nrm += d[2];
    }
  };
  if (beg < end) {
    l1_load(s, beg % kDStages, beg, emb, ld, m, dim, r0, c0);
    l1_commit();
    if (beg + 1 < end) l1_load(s, (beg + 1) % kDStages, beg + 1, emb, ld, m, dim, r0, c0);
    l1_commit();
    l1_wait();
    __syncthreads();
    row_sums(beg);
  }
  // a tile most of whose pairs are close after an eighth of the values is
  // computed term by term from there
  const int look = ranks == 1 && n_chunks >= 16 ? n_chunks / 8 : -1;
  bool by_terms = false;
  for (int c = beg; c < end; ++c) {
    // one barrier a stage: stage c + 1 and the row sums of stage c are there,
    // stage c - 1 is done with; the row sums of stage c + 1 follow now
    if (c == look && q == 0) s.norm[8 * warp + g] = nrm;
    l1_wait_all();
    __syncthreads();
    if (c + 2 < end) l1_load(s, (c + 2) % kDStages, c + 2, emb, ld, m, dim, r0, c0);
    if (c + 1 < end) row_sums(c + 1);
    const auto& st = s.stage[c % kDStages];
#pragma unroll 1
    for (int sub = 0; sub < 2; ++sub) {
      float acc[8][2][4];
#pragma unroll
      for (int e = 0; e < 2; ++e) {
        uint4 b[4];
#pragma unroll
        for (int jj = 0; jj < 4; ++jj) {
          const int row = kDT + wj + 8 * jj + g;
          b[jj] = st[row][l1_chunk(row, 8 * sub + 4 * e + q)];
        }
#pragma unroll
        for (int i = 0; i < 8; ++i) {
          const uint4 a = st[wi + i][l1_chunk(wi + i, 8 * sub + 4 * e + q)];
#pragma unroll
          for (int p = 0; p < 2; ++p) {
            add_rows(acc[i][p], max_bf16x2(a.x, b[2 * p].x), max_bf16x2(a.x, b[2 * p + 1].x),
                     max_bf16x2(a.y, b[2 * p].y), max_bf16x2(a.y, b[2 * p + 1].y), e == 0);
            add_rows(acc[i][p], max_bf16x2(a.z, b[2 * p].z), max_bf16x2(a.z, b[2 * p + 1].z),
                     max_bf16x2(a.w, b[2 * p].w), max_bf16x2(a.w, b[2 * p + 1].w), false);
          }
        }
      }
#pragma unroll
      for (int u = 0; u < 2; ++u) {
        const float hi = s.h[c & 1][sub][wi + 4 * u + q];
#pragma unroll
        for (int jj = 0; jj < 4; ++jj) {
          const int p = jj >> 1, w = 2 * (jj & 1);
          const float m01 = q & 1 ? acc[4 * u + 1][p][w] : acc[4 * u][p][w];
          const float m23 = q & 1 ? acc[4 * u + 3][p][w] : acc[4 * u + 2][p][w];
          run[u][jj] += (q & 2 ? m23 : m01) - (hi + s.h[c & 1][sub][kDT + wj + 8 * jj + g]);
        }
      }
    }
    if (c == look) {
      int close = 0;
#pragma unroll
      for (int u = 0; u < 2; ++u)
#pragma unroll
        for (int jj = 0; jj < 4; ++jj)
          close += !(2.f * close_ratio * run[u][jj] >=
                     s.norm[wi + 4 * u + q] + s.norm[kDT + wj + 8 * jj + g]);
      if (__syncthreads_count(close > 4) > kDThreads / 2) {
        by_terms = true;
        break;
      }
    }
  }
  l1_wait_all();
  __syncthreads();
  if (q == 0) s.norm[8 * warp + g] = nrm;
  if (ranks > 1) {
    float(*part)[kDThreads] = reinterpret_cast<float(*)[kDThreads]>(&s.stage[0][0][0]);
    if (rank > 0) {
#pragma unroll
      for (int u = 0; u < 2; ++u)
#pragma unroll
        for (int jj = 0; jj < 4; ++jj) part[4 * u + jj][threadIdx.x] = run[u][jj];
    }
    cluster.sync();
    if (rank == 0) {
      for (int o = 1; o < ranks; ++o) {
        const float(*there)[kDThreads] = cluster.map_shared_rank(part, o);
#pragma unroll
        for (int u = 0; u < 2; ++u)
#pragma unroll
          for (int jj = 0; jj < 4; ++jj) run[u][jj] += there[4 * u + jj][threadIdx.x];
        if (threadIdx.x < 2 * kDT) s.norm[threadIdx.x] += cluster.map_shared_rank(s.norm, o)[threadIdx.x];
      }
    }
    cluster.sync();
    if (rank > 0) return;
  } else {
    __syncthreads();
  }
  if (!by_terms) {
    // of a tile on the diagonal its upper half
#pragma unroll
    for (int u = 0; u < 2; ++u)
#pragma unroll
      for (int jj = 0; jj < 4; ++jj) {
        const int li = wi + 4 * u + q, lj = wj + 8 * jj + g;
        const int i = r0 + li, j = c0 + lj;
        if (i > j || j >= m) continue;
        const float d = 2.f * run[u][jj];
        const float n = s.norm[li] + s.norm[kDT + lj];
        if (!((i == j || close_ratio * d >= n) && n < 1e37f)) {
          const int at = atomicAdd(&s.n_close, 1);
          if (at < kListed) s.close[at] = (uint16_t)(li * kDT + lj);
        }
        dist[(int64_t)i * m + j] = d;
        dist[(int64_t)j * m + i] = d;
      }
    __syncthreads();
    by_terms = s.n_close > kListed;
  }
  if (by_terms) {
    l1_tile_by_terms(s, emb, ld, m, dim, r0, c0, dist);
    return;
  }
  // the close pairs one by one, a warp each
  for (int e = warp; e < s.n_close; e += kDThreads / 32) {
    const int i = r0 + s.close[e] / kDT, j = c0 + s.close[e] % kDT;
    const __nv_bfloat16 *ei = emb + (int64_t)i * ld, *ej = emb + (int64_t)j * ld;
    float acc = 0.f;
#pragma unroll 4
    for (int k = 8 * lane; k + 8 <= dim; k += 256)
      acc = add_abs_diff8(acc, *reinterpret_cast<const uint4*>(ei + k),
                          *reinterpret_cast<const uint4*>(ej + k));
    for (int k = (dim & ~7) + lane; k < dim; k += 32)
      acc += fabsf(__bfloat162float(ei[k]) - __bfloat162float(ej[k]));
    for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
    if (lane == 0) {
      dist[(int64_t)i * m + j] = acc;
      dist[(int64_t)j * m + i] = acc;
    }
  }
}

constexpr int kMThreads = 256;
constexpr int kMWarps = kMThreads / 32;

__global__ void __launch_bounds__(kMThreads)
    mmd_trials_kernel(const float* __restrict__ dist, int m, const int8_t* __restrict__ labels,
                      double* __restrict__ mmd_out) {
  extern __shared__ int8_t lab[];  // this trial's labels, m bytes
  __shared__ double red[kMWarps][4];
  __shared__ int count[2];
  const int t = blockIdx.x;
  const int8_t* lt = labels + (int64_t)t * m;
  if (threadIdx.x < 2) count[threadIdx.x] = 0;
  __syncthreads();
  int nx = 0, ny = 0;
  for (int j = threadIdx.x; j < m; j += kMThreads) {
    const int8_t l = lt[j];
    lab[j] = l;
    nx += l == 0;
    ny += l == 1;
  }
  for (int o = 16; o > 0; o >>= 1) {
    nx += __shfl_xor_sync(0xffffffffu, nx, o);
    ny += __shfl_xor_sync(0xffffffffu, ny, o);
  }
  if ((threadIdx.x & 31) == 0) {
    atomicAdd(&count[0], nx);  // integer counts: exact in any order
    atomicAdd(&count[1], ny);
  }
  __syncthreads();
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  // s[a][b]: sum of d(i, j) over rows i with label a and columns j with label b
  double s[2][2] = {{0.0, 0.0}, {0.0, 0.0}};
  for (int i = warp; i < m; i += kMWarps) {
    const int li = lab[i];
    if (li != 0 && li != 1) continue;
    const float* row = dist + (int64_t)i * m;
    float r0 = 0.f, r1 = 0.f;
    for (int j = lane; j < m; j += 32) {
      const int lj = lab[j];
      const float d = row[j];
      r0 += lj == 0 ? d : 0.f;
      r1 += lj == 1 ? d : 0.f;
    }
    for (int o = 16; o > 0; o >>= 1) {
      r0 += __shfl_xor_sync(0xffffffffu, r0, o);
      r1 += __shfl_xor_sync(0xffffffffu, r1, o);
    }
    s[li][0] += (double)r0;
    s[li][1] += (double)r1;
  }
  if (lane == 0) {
    red[warp][0] = s[0][0];
    red[warp][1] = s[0][1];
    red[warp][2] = s[1][0];
    red[warp][3] = s[1][1];
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    double sxx = 0.0, sxy = 0.0, syx = 0.0, syy = 0.0;
    for (int w = 0; w < kMWarps; ++w) {
      sxx += red[w][0];
      sxy += red[w][1];
      syx += red[w][2];
      syy += red[w][3];
    }
    const double fx = (double)count[0], fy = (double)count[1];
    mmd_out[t] = (count[0] > 0 && count[1] > 0)
                     ? (sxy + syx) / (fx * fy) - sxx / (fx * fx) - syy / (fy * fy)
                     : 0.0;
  }
}

// The launch of `tiles` clusters of n CTAs.
void l1_config(cudaLaunchConfig_t& cfg, cudaLaunchAttribute* at, int n, int64_t tiles,
               cudaStream_t st) {
  cfg.gridDim = dim3((unsigned)(tiles * n));
  cfg.blockDim = dim3(kDThreads);
  cfg.dynamicSmemBytes = sizeof(L1Smem);
  cfg.stream = st;
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim.x = (unsigned)n;
  at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
  cfg.attrs = at;
  cfg.numAttrs = 1;
}

// Clusters of 1, 2, 4 and 8 CTAs that the current device holds at once,
// asked for (and the shared-memory size set) on a device's first use.
using L1Resident = std::array<int, 4>;
cudaError_t l1_resident(L1Resident& out) {
  static std::mutex mu;
  static std::map<int, L1Resident> held;
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  std::lock_guard<std::mutex> lock(mu);
  const auto it = held.find(dev);
  if (it != held.end()) {
    out = it->second;
    return cudaSuccess;
  }
  e = cudaFuncSetAttribute(l1_distance_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                           (int)sizeof(L1Smem));
  for (int l = 0; l < 4 && e == cudaSuccess; ++l) {
    cudaLaunchConfig_t cfg = {};
    cudaLaunchAttribute at[1];
    l1_config(cfg, at, 1 << l, 1, nullptr);
    e = cudaOccupancyMaxActiveClusters(&out[l], l1_distance_kernel, &cfg);
  }
  if (e == cudaSuccess) held.emplace(dev, out);
  return e;
}

}  // namespace

cudaError_t launch_l1_distances(const __nv_bfloat16* emb, int64_t ld, int m, int dim, float* dist,
                                cudaStream_t st) {
  if (m <= 0) return cudaSuccess;
  const int64_t nb = (m + kDT - 1) / kDT, tiles = nb * (nb + 1) / 2;
  const int n_chunks = (dim + kDK - 1) / kDK;
  if (tiles * kMaxCluster > INT_MAX) return cudaErrorInvalidValue;
  L1Resident held;
  const cudaError_t e = l1_resident(held);
  if (e != cudaSuccess) return e;
  // CTAs per tile: the time is the waves of clusters over their share of the
  // chunks; a cluster's start and its reduction cost about four chunks' time
  int best = 1;
  double best_t = 0.0;
  for (int n = 1, l = 0; n <= kMaxCluster; n *= 2, ++l) {
    if (held[l] < 1 || (n > 1 && (n_chunks < 4 * n || dim < kTermsDim))) continue;
    const double waves = (double)((tiles + held[l] - 1) / held[l]);
    const double t = waves * ((double)n_chunks / n + (n > 1 ? 4.0 : 0.0));
    if (best_t == 0.0 || t < best_t) { best = n; best_t = t; }
  }
  cudaLaunchConfig_t cfg = {};
  cudaLaunchAttribute at[1];
  l1_config(cfg, at, best, tiles, st);
  const float close_ratio = std::min(kCloseRatio, (float)dim / kDimPerRatio);  // see Precision above
  return cudaLaunchKernelEx(&cfg, l1_distance_kernel, emb, ld, m, dim, dist, close_ratio);
}

cudaError_t launch_mmd_trials(const float* dist, int m, const int8_t* labels, int trials,
                              double* mmd, cudaStream_t st) {
  if (trials <= 0) return cudaSuccess;
  if ((size_t)m > 48 * 1024) return cudaErrorInvalidValue;
  mmd_trials_kernel<<<trials, kMThreads, (size_t)m, st>>>(dist, m, labels, mmd);
  return cudaGetLastError();
}

}  // namespace synth
