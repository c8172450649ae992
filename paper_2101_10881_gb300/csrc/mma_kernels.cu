// mma_kernels.cu -- the convolution kernels of the integer arithmetic, on the
// tensor cores: exact products of 9- or 10-bit slices (slices.cuh).
//
// A truncated series product z_j = sum_i x_i y_{j-i} (Eq. eqconvform) of slice
// vectors is a sum over i of matrix products C[r][j] += T(x_i)[r][q] Y[q][j-i]: rows r
// the slices of the result, T(x_i)[r][q] = x_i[r - q] the Toeplitz matrix of x_i's
// slices, columns j.  The correlation of the VJP, r_j = sum_i x_{j+i} y_i, is the
// same with y_i in the Toeplitz matrix and column rows x_{j+i}.
//
// What bounds it: the f16 mma.sync (m16n8k16, fp32 accumulators; 301 T
// multiply-adds/s measured on this GPU, where 32x32->64-bit integer products run
// at 10 T/s and one of them is worth about nine slice products) as long as the
// fragments cost less than it does.  They do because
// - the Toeplitz fragments need no matrix in memory: with the rows of a 16-row
//   block dealt as r = 16 b + 2 g + rho - 1 (g the fragment row, rho the half of the
//   tile), the two slices a lane holds are consecutive and start rho slices into a
//   word, so every fragment register is one byte permute of two neighbouring words
//   of x_i, and all blocks of all rows of x_i come from 4 NB words per lane (NB
//   16-row blocks);
// - a term whose grids lie delta digits below the column's reference grid is the
//   same column read delta words early (rows of zeros lie between the coefficients),
//   so every lane shifts its own column by an address;
// - blocks above the diagonal (rows whose slices all lie above the column slices)
//   are zero and not issued.
// tcgen05 has three times the rate, but needs the Toeplitz matrix in shared memory
// (one copy of x per row of a core matrix) and 128 rows for every k; reading that
// operand (32 cycles a step against 16 to 40 for the columns here) would bound it at
// about the time of this form.
//
// The sums: fp32 accumulators are exact up to 2^24 (in units of a slice product).
// The upper part of every accumulator is moved into a second fp32 number (four
// additions) before its terms could pass that, by the Cauchy-Schwarz bound from the
// largest slice norms of the two series (or the largest possible products, whichever
// allows more).  The rows are then carried into digits by the lanes that hold them
// (warp shuffles move the carries), the top digit is found, and L digits are stored
// on a grid of their own.  Rows beyond 16 NB - 1 slices are not formed; for every k
// what is dropped weighs no more, against the smallest possible leading digits, than
// the products the 28-bit form drops (p + q >= L28): 2^-239, 2^-382, 2^-526, 2^-585 of
// the product for k = 4, 5, 8, 10 against 2^-221, 2^-277, 2^-445, 2^-529.
//
// Measured (one GB300, convolution kernel): p2-like d = 152, k = 10, 9.28 ms in the integer
// pipe's best shape and 10.1 ms in its default one, 5.8 ms here; all pairs of 48 variables
// with every third a triple, d = 152, k = 4 / 5 / 8 / 10: 0.57 / 0.73 / 1.74 / 1.75 ms ->
// 0.39 / 0.62 / 0.83 / 0.95 ms, with exponential series 0.54 / 0.70 / 1.69 / 1.74 ->
// 0.37 / 0.56 / 0.99 / 1.12.
#include <cuda_runtime.h>

#include <cstdint>

#include "dag_sync.cuh"
#include "kernels.hpp"
#include "slices.cuh"

namespace pes {

namespace {

// Shared memory of one buffer, in words: eight rows of zeros and the column
// operand's rows behind them, the Toeplitz operand's rows, and the grids of both; the
// column grids have kPad entries of kZeroGrid on either side (columns before the series
// have no term there).  A row of the Toeplitz operand holds, for every word u from
// -8 to L - 1, the two fragment words that start at slices 2 u and 2 u + 1 (zeros up to
// u = -2, which also follow the row before), so that a lane gets both with one 64-bit
// load; it takes twice the room of the words themselves, which are staged in place first.
// (One word a digit, the fragment words formed as they are read, for degrees without room
// for the pairs: 0.57 to 0.9 of the integer pipe's speed, and of the tiles' that take them.)
constexpr int kPairLead = 8;
constexpr int kPad = 48;               // > 7 + 8 (NT - 1): how far before the series a group's columns run
constexpr int kZeroGrid = -(1 << 24);  // staged grid (four times the grid) of a zero coefficient
constexpr int32_t kZeroMeta = -(1 << 30);  // the meta of a zero coefficient
struct BufLayout {
  int y, x, ga, gb, mx, my, words;  // (mx, my: the metas as copied)
};
__host__ __device__ constexpr BufLayout buf_layout(int L, int sw, int xrows, int yrows) {
  BufLayout b{};
  b.y = 8 * sw;
  b.x = b.y + (yrows + 1) * sw;  // (a row of zeros, before the Toeplitz operand's coefficient 0 and after the columns)
  b.ga = b.x + xrows * 2 * (L + kPairLead) + sw;
  b.gb = b.ga + xrows;
  b.mx = b.gb + kPad + yrows + kPad;
  b.my = b.mx + xrows;
  b.words = (b.my + yrows + 31) / 32 * 32;
  return b;
}

// Words from one staged column coefficient to the next: 4 mod 8, so that the 8 x 4 words
// a warp reads of 8 columns fall in 32 banks.  For k = 4 and 5 twice the digits, so that
// every term that reaches a column at all reads it from zeros in front of it (series
// whose coefficients fall over hundreds of bits, as exponential ones do, took 1.25 times
// as long with the lanes of deeper terms handled apart); at k = 8 and 10 that would cost
// a CTA an SM, and fewer of their terms lie so deep.
__host__ __device__ constexpr int mma_stride(int k) {
  return k <= 4 ? 36 : k <= 5 ? 44 : 8 * ((slice_digits(k) + 7) / 8) + 4;
}

constexpr int kMiscWords = 32;
constexpr int kRangeWord = 8;  // where a Range starts in the misc words

template <int K>
struct Mma {
  static constexpr int W = slice_bits(K);
  static constexpr int L = slice_digits(K);
  static constexpr int KS = (L + 7) / 8;          // 16-slice blocks of a column
  static constexpr int NB = KS;                   // 16-row blocks of the result
  static constexpr int SW = mma_stride(K);
  static constexpr int G = L < 16 ? 16 : 32;      // lanes that take a row in the passes over staged rows
  // Columns are staged shifted down to the largest grid of their series, by up to SP
  // digits, where that reaches every coefficient: a term's address then does not
  // depend on its column coefficient's grid.  At least PZ zero words lie before a
  // coefficient's digits, and columns may be read up to RA words late.
  static constexpr int SP = G - L < 4 ? G - L : 4;
  static constexpr int PZ = SW - L - SP;
  static constexpr int RA = SW - 8 * KS < 4 ? SW - 8 * KS : 4;
  static constexpr int PS = L + kPairLead;        // pairs of a Toeplitz row
  static constexpr int NT = kMmaGroupTiles;       // column tiles of 8 coefficients a warp accumulates at once
  // terms whose slice products stay within 2^24 whatever the slices are
  static constexpr int kDrain = ((1 << 24) - 512) / (2 * L << (2 * W - 2));
  // terms between two carries of the accumulators (their upper parts stay exact
  // to 2^33)
  static constexpr int kLimit = ((1 << (33 - (2 * W - 2))) - 64) / (2 * L);
  static_assert(8 * NB - L <= 8, "the fragments read no further than the zeros after a row of pairs");
  static_assert(SW - L >= 4 && PZ >= 0 && SP >= 0 && SP <= RA, "zeros between the staged coefficients");
  static_assert(kDrain >= 1, "one term must fit the accumulators");
  static_assert(4 * (kMiscWords + buf_layout(L, SW, kLimit + 1, kLimit + 1).words) > 227 * 1024,
                "whole series that fit in shared memory are never carried in between");
  static_assert(kPad > 8 * NT, "pads of the column grids");
};


// All of the kernels' shared memory: kMiscWords words, then the buffers.  Staged rows
// and grids are addressed by byte offsets into it (word indices would cost a shift at
// every use), and the staged grids are kept as four times the grid, the bytes a column
// is shifted by.
extern __shared__ __align__(128) uint32_t sm[];
__device__ __forceinline__ uint32_t lds(int off) {
  return *reinterpret_cast<const uint32_t*>(reinterpret_cast<const char*>(sm) + off);
}
__device__ __forceinline__ uint2 lds2(int off) {
  return *reinterpret_cast<const uint2*>(reinterpret_cast<const char*>(sm) + off);
}

__device__ __forceinline__ uint32_t smem_addr(const void* p) {
  return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}
__device__ __forceinline__ void copy4(void* dst, const void* src) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(smem_addr(dst)), "l"(src) : "memory");
}
__device__ __forceinline__ void copies_wait() { asm volatile("cp.async.wait_all;" ::: "memory"); }

// acc += a b: 16 rows x 16 slices times 16 slices x 8 columns, f16, fp32 sums
__device__ __forceinline__ void mma_f16(float (&c)[4], uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3, uint32_t b0,
                                        uint32_t b1) {
  asm("mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0,%1,%2,%3},{%4,%5,%6,%7},{%8,%9},{%0,%1,%2,%3};"
      : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
      : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}

// Copy the words (STEP words apart, rows STRIDE words apart, `rev`: last row first) and
// the metas of coefficients [c0, c0 + n) of a series.
template <int K, int STRIDE, int STEP>
__device__ __forceinline__ void stage_rows(uint32_t* rows, int32_t* metas, const int32_t* series, int S, int c0, int n,
                                           bool rev) {
  constexpr int L = Mma<K>::L, G = Mma<K>::G;
  const int p = threadIdx.x % G, r = threadIdx.x / G, per = blockDim.x / G;
  if (p < L) {
    const int32_t* src = series + static_cast<long long>(c0) * L + p;
    uint32_t* dst = rows + p * STEP;
#pragma unroll 4
    for (int c = r; c < n; c += per) copy4(dst + (rev ? n - 1 - c : c) * STRIDE, src + c * L);
  }
  const int32_t* g = series + static_cast<long long>(S) * L + c0;
  for (int t = threadIdx.x; t < n; t += blockDim.x) copy4(metas + (rev ? n - 1 - t : t), g + t);
}

// The claimed sub-job (in the misc words).
struct Claim {
  int32_t claimed, failed, ready;
};

// What a warp finds in the staged metas.
struct Found {
  int qx, qy;          // largest norms
  int gmax, gmin;      // largest and smallest grid of a nonzero column coefficient, times four
  int x0, x1, y0, y1;  // [x0, x1), [y0, y1): first to last nonzero coefficient of either operand
  int spread;          // how far apart the grids of two products can lie, times four
};

// Every warp looks through the metas of the nx Toeplitz and ny column coefficients (that
// saves a barrier over sharing what it finds); together they leave four times the grids
// in ga and gb.  Where the nonzero coefficients lie is looked for when there are zeros, or
// column coefficients 16 digits apart.
__device__ __forceinline__ Found split_metas(const int32_t* mx, int32_t* ga, int nx, const int32_t* my, int32_t* gb,
                                             int ny) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, warps = blockDim.x >> 5;
  Found f{0, 0, -(1 << 30), 1 << 30, 0, nx, 0, ny, 0};
  bool zeros = false;
  for (int c = lane, u = 0; c < nx; c += 32, ++u) {
    const int32_t w = mx[c];
    if (u % warps == warp) ga[c] = 4 * meta_grid(w);
    f.qx = max(f.qx, w & 255);
    zeros |= (w & 255) == 0;
  }
  for (int c = lane, u = 0; c < ny; c += 32, ++u) {
    const int32_t w = my[c], g = 4 * meta_grid(w);
    if (u % warps == warp) gb[c] = g;
    f.qy = max(f.qy, w & 255);
    f.gmax = max(f.gmax, g > kZeroGrid ? g : f.gmax);
    f.gmin = min(f.gmin, g > kZeroGrid ? g : f.gmin);
    zeros |= (w & 255) == 0;
  }
  f.qx = __reduce_max_sync(0xffffffffu, f.qx);
  f.qy = __reduce_max_sync(0xffffffffu, f.qy);
  f.gmax = __reduce_max_sync(0xffffffffu, f.gmax);
  f.gmin = __reduce_min_sync(0xffffffffu, f.gmin);
  if (__any_sync(0xffffffffu, zeros) || f.gmax - f.gmin >= 64) {
    int x0 = 1 << 20, x1 = 0, y0 = 1 << 20, y1 = 0, xmax = -(1 << 30), xmin = 1 << 30;
    for (int c = lane; c < nx; c += 32) {
      const int g = 4 * meta_grid(mx[c]);
      if (g > kZeroGrid) {
        x0 = min(x0, c);
        x1 = c + 1;
        xmax = max(xmax, g);
        xmin = min(xmin, g);
      }
    }
    for (int c = lane; c < ny; c += 32)
      if (4 * meta_grid(my[c]) > kZeroGrid) {
        y0 = min(y0, c);
        y1 = c + 1;
      }
    f.x0 = __reduce_min_sync(0xffffffffu, x0);
    f.x1 = __reduce_max_sync(0xffffffffu, x1);
    f.y0 = __reduce_min_sync(0xffffffffu, y0);
    f.y1 = __reduce_max_sync(0xffffffffu, y1);
    xmax = __reduce_max_sync(0xffffffffu, xmax);
    xmin = __reduce_min_sync(0xffffffffu, xmin);
    f.spread = f.x1 > 0 && f.y1 > 0 ? xmax - xmin + f.gmax - f.gmin : 0;
  }
  return f;
}

// The same of a chunk in the tiled kernel, whose range tile_range has found.  (Whole warps
// run through both loops: with those above, the kernel of k = 10 spills and takes 12 %
// longer.)
__device__ __forceinline__ Found split_chunk(const int32_t* mx, int32_t* ga, int nx, const int32_t* my, int32_t* gb,
                                             int ny) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, warps = blockDim.x >> 5;
  Found f{0, 0, -(1 << 30), 1 << 30, 0, nx, 0, ny, 0};
  for (int c0 = 0, u = 0; c0 < nx; c0 += 32, ++u) {
    const int c = c0 + lane;
    const int32_t w = c < nx ? mx[c] : kZeroMeta;
    if (c < nx && u % warps == warp) ga[c] = 4 * meta_grid(w);
    f.qx = max(f.qx, w & 255);
  }
  for (int c0 = 0, u = 0; c0 < ny; c0 += 32, ++u) {
    const int c = c0 + lane;
    const int32_t w = c < ny ? my[c] : kZeroMeta;
    const int g = 4 * meta_grid(w);
    if (c < ny && u % warps == warp) gb[c] = g;
    f.qy = max(f.qy, w & 255);
    f.gmax = max(f.gmax, g > kZeroGrid ? g : f.gmax);
    f.gmin = min(f.gmin, g > kZeroGrid ? g : f.gmin);
  }
  f.qx = __reduce_max_sync(0xffffffffu, f.qx);
  f.qy = __reduce_max_sync(0xffffffffu, f.qy);
  f.gmax = __reduce_max_sync(0xffffffffu, f.gmax);
  f.gmin = __reduce_min_sync(0xffffffffu, f.gmin);
  return f;
}

// Where the nonzero coefficients of the two operands lie: [x0, x1) and [y0, y1); far:
// products can lie L digits below the largest of their column.
struct Range {
  int x0, x1, y0, y1, far;
};

// The terms [begin, end) that meet nonzero coefficients in the columns jlo to jhi.
__device__ __forceinline__ void nonzero_terms(const volatile Range* r, int jlo, int jhi, int& begin, int& end) {
  begin = max(r->x0, jlo - r->y1 + 1);
  end = min(r->x1, jhi - r->y0 + 1);
}

// The terms [x0, x1) that meet nonzero coefficients in the columns [c0, terms) of an
// output tile (into the Range of the misc words), by the whole CTA.  `either`: either
// operand may be the Toeplitz one; true if it is better the second, which has fewer.  (Not
// inlined: the kernel around it has no register to spare.)
__device__ __noinline__ bool tile_range(const int32_t* gx, const int32_t* gy, int step, int terms, int c0,
                                        bool either) {
  Range* r = reinterpret_cast<Range*>(sm + kRangeWord);
  if (threadIdx.x == 0) *r = Range{terms, 0, terms, 0, 0};
  __syncthreads();
  int x0 = terms, x1 = 0, y0 = terms, y1 = 0;
  for (int i = threadIdx.x; i < terms; i += blockDim.x) {
    const bool nx = 4 * meta_grid(__ldcg(gx + i)) > kZeroGrid, ny = 4 * meta_grid(__ldcg(gy + i * step)) > kZeroGrid;
    x0 = nx ? min(x0, i) : x0;
    x1 = nx ? i + 1 : x1;
    y0 = ny ? min(y0, i) : y0;
    y1 = ny ? i + 1 : y1;
  }
  x0 = __reduce_min_sync(0xffffffffu, x0);
  x1 = __reduce_max_sync(0xffffffffu, x1);
  y0 = __reduce_min_sync(0xffffffffu, y0);
  y1 = __reduce_max_sync(0xffffffffu, y1);
  if ((threadIdx.x & 31) == 0) {
    atomicMin(&r->x0, x0);
    atomicMax(&r->x1, x1);
    atomicMin(&r->y0, y0);
    atomicMax(&r->y1, y1);
  }
  __syncthreads();
  x0 = r->x0, x1 = r->x1, y0 = r->y0, y1 = r->y1;
  const bool swap = either && y1 - y0 < x1 - x0;
  __syncthreads();
  if (threadIdx.x == 0) {
    r->x0 = max(swap ? y0 : x0, c0 - (swap ? x1 : y1) + 1);
    r->x1 = min(swap ? y1 : x1, terms - (swap ? x0 : y0));
  }
  __syncthreads();
  return swap;
}

// The columns' grids lie close enough for their rows to be shifted to the largest.
template <int K>
__device__ __forceinline__ bool is_flat(const Found& f) {
  return f.gmax > kZeroGrid && f.gmax - f.gmin <= 4 * Mma<K>::SP;
}

// The passes over the staged rows, G lanes a row: the fragment pairs of nx Toeplitz
// rows, and the ny column rows shifted by gmax minus their grid (`flat`; the
// words behind a row's digits are cleared either way).
template <int K>
__device__ __forceinline__ void form_rows(uint32_t* x, int nx, uint32_t* y, const int32_t* my, int ny, bool flat,
                                          int gmax) {
  using M = Mma<K>;
  constexpr int L = M::L, G = M::G, U = 4;  // rows in flight per lane
  const int p = threadIdx.x % G, r = threadIdx.x / G;
  const int per = blockDim.x / G;
  const bool word = p < L;
  {
    uint32_t* at = x + (r * M::PS + kPairLead + p) * 2;
    const int step = per * M::PS * 2;
    const bool follows = p < G - 1;  // (the last lane's shuffle returns its own word)
    auto row = [&](uint32_t* to, uint32_t w, bool live) {
      const uint32_t s = __shfl_down_sync(0xffffffffu, w, 1, G);
      const uint32_t next = follows ? s : 0u;
      if (live && word) {
        *reinterpret_cast<uint2*>(to) = make_uint2(__byte_perm(w, next, 0x1032), __byte_perm(w, next, 0x7610));
        if (p == 0) to[-1] = __byte_perm(0u, w, 0x7610);
      }
    };
    int c0 = 0;
    for (; c0 + U * per <= nx; c0 += U * per, at += U * step) {
      uint32_t w[U];
#pragma unroll
      for (int u = 0; u < U; ++u) w[u] = word ? at[u * step] : 0u;
#pragma unroll
      for (int u = 0; u < U; ++u) row(at + u * step, w[u], true);
    }
    for (; c0 < nx; c0 += per, at += step) {
      const bool live = c0 + r < nx;
      row(at, live && word ? *at : 0u, live);
    }
  }
  uint32_t* at = y + r * M::SW + p;
  const int step = per * M::SW;
  auto row = [&](uint32_t* to, uint32_t w, int32_t meta, bool live) {
    int sh = flat ? (gmax - 4 * meta_grid(meta)) >> 2 : 0;
    sh = static_cast<unsigned>(sh) <= static_cast<unsigned>(M::SP) ? sh : 0;  // (zero coefficients stay)
    const uint32_t v = __shfl_sync(0xffffffffu, w, p - sh, G);
    if (live && p < L + M::SP) *to = p >= sh ? v : 0u;
  };
  int c0 = 0;
  for (; c0 + U * per <= ny; c0 += U * per, at += U * step) {
    uint32_t w[U];
    int32_t m[U];
#pragma unroll
    for (int u = 0; u < U; ++u) {
      w[u] = word ? at[u * step] : 0u;
      m[u] = my[c0 + u * per + r];
    }
#pragma unroll
    for (int u = 0; u < U; ++u) row(at + u * step, w[u], m[u], true);
  }
  for (; c0 < ny; c0 += per, at += step) {
    const bool live = c0 + r < ny;
    row(at, live && word ? *at : 0u, live ? my[c0 + r] : 0, live);
  }
}

// Terms whose slice products stay within 2^24 (less the 2^8 an accumulator keeps
// between moves), from the largest norms of the two operands.
template <int K>
__device__ __forceinline__ int drain_terms(const Found& f) {
  const float r = sqrtf(meta_norm(f.qx)) * sqrtf(meta_norm(f.qy)) * 1.0001f;
  return max(Mma<K>::kDrain, min(64, static_cast<int>(16776704.f / r)));
}

// Where a group's operands are staged (byte offsets): Toeplitz row 0 and its grid, the
// column row that the lane's column of tile 0 meets at term 0 (from the lane's word on)
// and its grid; and what the passes found.
struct Terms {
  int x, ga, y, gb, zero;
  int every;  // terms between two moves of the upper parts
  bool flat;  // columns staged on one grid, gmax
  int gmax;
};

// From the first to the last of the terms [begin, end) whose product reaches a column: its
// grid lies above the column's `least` (three tiles; four times the grids at ga, and, of
// the lane's columns, at gb).
__device__ __forceinline__ int2 reaching_terms(int ga, int gb, int begin, int end, int3 least) {
  int first = end, last = begin;
#pragma unroll 2
  for (int i = begin + static_cast<int>(threadIdx.x & 3); i < end; i += 4) {
    const int gx = static_cast<int>(lds(ga + 4 * i)), at = gb - 4 * i;
    const int y0 = static_cast<int>(lds(at)), y1 = static_cast<int>(lds(at - 32)), y2 = static_cast<int>(lds(at - 64));
    if (gx + y0 > least.x || gx + y1 > least.y || gx + y2 > least.z) {
      first = min(first, i);
      last = i + 1;
    }
  }
  return make_int2(__reduce_min_sync(0xffffffffu, first), __reduce_max_sync(0xffffffffu, last));
}

// A group of up to NT column tiles of one warp: tile t holds the columns 8 t before those
// of tile 0.
template <int K>
struct Group {
  using M = Mma<K>;
  static constexpr int W = M::W, L = M::L, KS = M::KS, NB = M::NB, SW = M::SW, PZ = M::PZ, NT = M::NT;
  static constexpr int B = 2 * W;
  static constexpr float kUnit = 281474976710656.f;    // 2^48: one slice product
  static constexpr float kUnitHi = 549755813888.f;     // 2^39: the unit of the upper parts, 2^9 products
  static constexpr float kSplit = 1.5f / 65536.f;      // 1.5 2^23 units of the upper parts
  static constexpr int kLow = 4 * slice_grid_low(K);   // sums of grids below: zero
  float acc[NT][NB][4];  // rows 2 g - 1 (elements 0, 1: columns 2 tl, 2 tl + 1) and 2 g (2, 3) of each block
  float up[NT][NB][4];   // the upper parts
  int gs[NT];            // four times the reference grid of column g of each tile
  int gs_lo, gs_hi;      // the smallest and largest of them

  __device__ __forceinline__ void clear() {
#pragma unroll
    for (int t = 0; t < NT; ++t)
#pragma unroll
      for (int b = 0; b < NB; ++b)
#pragma unroll
        for (int e = 0; e < 4; ++e) acc[t][b][e] = up[t][b][e] = 0.f;
  }

  // Move the upper parts of the accumulators of tile t (exact: every step is a sum of
  // multiples of one unit within 24 bits), two at a time.
  __device__ __forceinline__ void drain(int t) {
#pragma unroll
    for (int b = 0; b < NB; ++b)
#pragma unroll
      for (int e = 0; e < 4; e += 2) {
        asm("{\n .reg .b64 a, u, h, s, m;\n mov.b64 a, {%0, %1};\n mov.b64 u, {%2, %3};\n mov.b64 s, {%4, %4};\n"
            " mov.b64 m, {%5, %5};\n add.rn.f32x2 h, a, s;\n add.rn.f32x2 h, h, m;\n add.rn.f32x2 u, u, h;\n"
            " mov.b64 m, {%6, %6};\n fma.rn.f32x2 a, h, m, a;\n mov.b64 {%0, %1}, a;\n mov.b64 {%2, %3}, u;\n}"
            : "+f"(acc[t][b][e]), "+f"(acc[t][b][e + 1]), "+f"(up[t][b][e]), "+f"(up[t][b][e + 1])
            : "f"(kSplit), "f"(-kSplit), "f"(-1.f));
      }
  }

  // The columns' reference grids, from the largest sums gm of four times the grids of
  // their terms (the lanes of a column agree); columns without a nonzero term take one
  // of the others, as every term of theirs reads zeros.
  __device__ __forceinline__ void set_grids(const int (&gm)[NT]) {
    int lo = 1 << 30, hi = -(1 << 30);
#pragma unroll
    for (int t = 0; t < NT; ++t) {
      const bool some = gm[t] >= kLow;
      lo = min(lo, some ? gm[t] : lo);
      hi = max(hi, some ? gm[t] : hi);
    }
    gs_lo = __reduce_min_sync(0xffffffffu, lo);
    gs_hi = __reduce_max_sync(0xffffffffu, hi);
#pragma unroll
    for (int t = 0; t < NT; ++t) gs[t] = gm[t] >= kLow ? gm[t] : max(gs_hi, kLow);
  }

  // the Toeplitz fragments of the row at xr: word offset 4 (kap - 1), slice rho
  __device__ __forceinline__ static void fragments(uint32_t (&A)[2 * NB][2], int xr) {
#pragma unroll
    for (int kap = 0; kap < 2 * NB; ++kap) {
      const uint2 w = lds2(xr + 32 * (kap - 1));
      A[kap][0] = w.x;
      A[kap][1] = w.y;
    }
  }

  __device__ __forceinline__ void multiply(int t, const uint32_t (&A)[2 * NB][2], const uint32_t (&Bf)[KS][2]) {
    // (blocks downwards: the products of one accumulator lie as far apart as they can)
#pragma unroll
    for (int c = 0; c < KS; ++c)
#pragma unroll
      for (int b = NB - 1; b >= c; --b)
        mma_f16(acc[t][b], A[2 * (b - c) + 1][0], A[2 * (b - c) + 1][1], A[2 * (b - c)][0], A[2 * (b - c)][1], Bf[c][0],
                Bf[c][1]);
  }

  // Byte offset from the row a column meets of what tile t reads of it, but for the
  // term's grid (columns staged on gmax).
  __device__ __forceinline__ int column(int t, const Terms& a) const { return a.gmax - gs[t] - 32 * t * SW; }

  __device__ __forceinline__ static void load(uint32_t (&Bf)[KS][2], int at) {
#pragma unroll
    for (int c = 0; c < KS; ++c) {
      Bf[c][0] = lds(at + 32 * c);
      Bf[c][1] = lds(at + 32 * c + 16);
    }
  }

  // The terms i in [i0, i1) of the first NA tiles, every column by its own grid.
  template <int NA>
  __device__ __forceinline__ void run_any(int i0, int i1, const Terms& a, int& left) {
    const int lane = threadIdx.x & 31, la = (lane >> 2) - (lane & 3) - 1, wl = lane & 3;
    int xr = a.x + (i0 * M::PS + kPairLead + la) * 8;
    int yr = a.y - i0 * SW * 4, gb = a.gb - i0 * 4;
    const int near = 4 * (a.flat ? PZ : SW - L);
    const int end = a.ga + 4 * i1;
#pragma unroll 1
    for (int ga = a.ga + 4 * i0; ga != end; ga += 4) {
      const int gx = static_cast<int>(lds(ga));
      uint32_t A[2 * NB][2];
      fragments(A, xr);
#pragma unroll
      for (int t = 0; t < NA; ++t) {
        // bytes the column is shifted by: 4 for every digit the term lies below the
        // column's reference grid
        const int delta = gs[t] - gx - static_cast<int>(lds(gb - 32 * t));
        const int bn = a.flat ? yr + gx + column(t, a) : yr - delta - 32 * t * SW;
        const bool ok = static_cast<unsigned>(delta) <= static_cast<unsigned>(near);
        const bool far = !ok && static_cast<unsigned>(delta) < static_cast<unsigned>(4 * L);
        uint32_t Bf[KS][2];
        load(Bf, ok ? bn : a.zero);
        if (SW - L - M::SP < L - 1 && __any_sync(0xffffffffu, far)) {
          if (far) {
            // word w of the shifted column is word w - delta / 4 of the coefficient
#pragma unroll
            for (int c = 0; c < KS; ++c)
#pragma unroll
              for (int h = 0; h < 2; ++h)
                Bf[c][h] = 4 * (8 * c + 4 * h + wl) >= delta ? lds(bn + 32 * c + 16 * h) : 0u;
          }
          __syncwarp();
        }
        multiply(t, A, Bf);
      }
      xr += 8 * M::PS;
      yr -= 4 * SW;
      gb -= 4;
      if (--left == 0) {
        left = a.every;
#pragma unroll
        for (int t = 0; t < NA; ++t) drain(t);
      }
    }
  }

  // The same where every term's Toeplitz grid is at least lo (or that of a zero
  // coefficient) and reads every column between PZ words early and RA words late: the
  // address of a column row is one sum.  The fragments of the next term and the next
  // column rows are loaded while the products of the present ones issue; without that
  // the loads' latency, not the mma, bounds the loop (2 to 4 warps per scheduler).
  template <int NA>
  __device__ __forceinline__ void run_flat(int i0, int i1, int lo, const Terms& a, int& left) {
    const int lane = threadIdx.x & 31, la = (lane >> 2) - (lane & 3) - 1;
    constexpr int XS = 8 * M::PS;
    int xr = a.x + (i0 * M::PS + kPairLead + la) * 8;
    int yr = a.y - i0 * SW * 4;
    int yt[NA];
#pragma unroll
    for (int t = 0; t < NA; ++t) yt[t] = column(t, a);
    const int last = a.ga + 4 * (i1 - 1);
    int ga = a.ga + 4 * i0;
    uint32_t A[2][2 * NB][2], Bf[2][KS][2];
    int yg = yr + max(static_cast<int>(lds(ga)), lo);
    fragments(A[0], xr);
    load(Bf[0], yg + yt[0]);
    for (;;) {
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        // (after the last term, the last term's again)
        const bool more = ga != last;
        ga = more ? ga + 4 : ga;
        xr = more ? xr + XS : xr;
        yr = more ? yr - 4 * SW : yr;
        const int yn = yr + max(static_cast<int>(lds(ga)), lo);
        fragments(A[h ^ 1], xr);
#pragma unroll
        for (int t = 0; t < NA; ++t) {
          load(Bf[(h * NA + t + 1) & 1], t + 1 < NA ? yg + yt[t + 1 < NA ? t + 1 : 0] : yn + yt[0]);
          multiply(t, A[h], Bf[(h * NA + t) & 1]);
        }
        yg = yn;
        if (--left == 0) {
          left = a.every;
#pragma unroll
          for (int t = 0; t < NA; ++t) drain(t);
        }
        if (!more) return;
      }
    }
  }

  // Add the terms [0, n[t]) of every tile, n not increasing (tiles without terms last).
  __device__ __forceinline__ void terms(const int (&n)[NT], const Terms& a) {
    // terms from `from` on take the flat loop
    const int lo = gs_hi - a.gmax - 4 * PZ, hi = gs_lo - a.gmax + 4 * M::RA;
    int from = n[0];
    if (a.flat && gs_hi >= kLow && lo <= hi) {
      from = 0;
      for (int u = threadIdx.x & 31; u < n[0]; u += 32) {
        const int gx = static_cast<int>(lds(a.ga + 4 * u));
        if (gx > kZeroGrid && (gx < lo || gx > hi)) from = u + 1;
      }
      from = __reduce_max_sync(0xffffffffu, from);
    }
    int left = a.every, i = 0;
    segment<NT>(n, i, from, lo, a, left);
#pragma unroll
    for (int t = 0; t < NT; ++t) drain(t);
  }
  template <int NA>
  __device__ __forceinline__ void segment(const int (&n)[NT], int& i, int from, int lo, const Terms& a, int& left) {
    if (n[NA - 1] > i) {
      const int mid = min(max(i, from), n[NA - 1]);
      if (mid > i) run_any<NA>(i, mid, a, left);
      if (n[NA - 1] > mid) run_flat<NA>(mid, n[NA - 1], lo, a, left);
      i = n[NA - 1];
    }
    if constexpr (NA > 1) segment<NA - 1>(n, i, from, lo, a, left);
  }

  // The rows of every tile and column 2 tl + cc as words of one digit and what lies above
  // them: the digit 8 b + g is v[t][cc][b] + hi[t][cc][b] of the next one, |v| <= 2^(B-1).
  __device__ __forceinline__ void words(int (&v)[NT][2][NB], int (&hi)[NT][2][NB]) const {
    constexpr int HALF = 1 << (B - 1);
#pragma unroll
    for (int t = 0; t < NT; ++t)
#pragma unroll
      for (int cc = 0; cc < 2; ++cc)
#pragma unroll
        for (int b = 0; b < NB; ++b) {
          // digit = (2^9 u0 + a0) 2^W + 2^9 u1 + a1, in units of 2^B and a rest below 2^(B+1):
          // u0 = 2^(B-W-9) h0 + l0, u1 = 2^(B-9) h1 + l1
          const int u0 = __float2int_rn(up[t][b][cc] * kUnitHi), u1 = __float2int_rn(up[t][b][2 + cc] * kUnitHi);
          const int a0 = __float_as_int(__fmaf_rn(acc[t][b][cc], kUnit, 12582912.f)) - 0x4b400000;
          const int a1 = __float_as_int(__fmaf_rn(acc[t][b][2 + cc], kUnit, 12582912.f)) - 0x4b400000;
          const int r =
              ((u0 & ((1 << (B - W - 9)) - 1)) << (W + 9)) + (a0 << W) + ((u1 & ((1 << (B - 9)) - 1)) << 9) + a1;
          const int c = (r + HALF) >> B;
          hi[t][cc][b] = (u0 >> (B - W - 9)) + (u1 >> (B - 9)) + c;
          v[t][cc][b] = r - c * (1 << B);
        }
  }

  // Carry the words into balanced digits (all tiles together: the chains of shuffles of
  // one column alone would be waited for); top: the digit -1 (added to, in the lanes of
  // g = 7).
  __device__ __forceinline__ static void carry_words(int (&v)[NT][2][NB], int (&hi)[NT][2][NB], int (&top)[NT][2]) {
    constexpr int HALF = 1 << (B - 1);
    const int lane = threadIdx.x & 31, g = lane >> 2;
    const int src = (lane + 4) & 31;  // the lane of digit s + 1 (g = 7: of the next block's first digit)
    for (;;) {
      int any = 0;
#pragma unroll
      for (int t = 0; t < NT; ++t)
#pragma unroll
        for (int cc = 0; cc < 2; ++cc) {
          int r[NB];
#pragma unroll
          for (int b = 0; b < NB; ++b) r[b] = __shfl_sync(0xffffffffu, hi[t][cc][b], src);
          if (g == 7) top[t][cc] += r[0];
#pragma unroll
          for (int b = 0; b < NB; ++b) {
            const int in = g < 7 ? r[b] : (b + 1 < NB ? r[b + 1] : 0);
            const int s = v[t][cc][b] + in;
            hi[t][cc][b] = (s + HALF) >> B;
            v[t][cc][b] = s - hi[t][cc][b] * (1 << B);
            any |= hi[t][cc][b];
          }
        }
      if (!__any_sync(0xffffffffu, any != 0)) break;
    }
  }

  // Carry every accumulator into digits and put the digits back (each in the last
  // slice row of its digit), so that the sums can go on; top[t][cc] collects what
  // leaves the rows at the top.
  __device__ __forceinline__ void carry(int (&top)[NT][2]) {
    int v[NT][2][NB], hi[NT][2][NB];
    words(v, hi);
    carry_words(v, hi, top);
#pragma unroll
    for (int t = 0; t < NT; ++t) {
#pragma unroll
      for (int cc = 0; cc < 2; ++cc)
#pragma unroll
        for (int b = 0; b < NB; ++b) {
          acc[t][b][cc] = up[t][b][cc] = up[t][b][2 + cc] = 0.f;
          acc[t][b][2 + cc] = static_cast<float>(v[t][cc][b]) * (1.f / kUnit);
        }
      drain(t);
    }
  }

  // Round the columns of the first nt tiles (tile t: j0 - 8 t + 0..7, those within
  // [jlo, d]) to L digits on grids of their own and store them, column j as coefficient j
  // (`rev`: d - j).  v, top: their digits.
  __device__ __forceinline__ void store(int nt, int j0, int jlo, int d, bool rev, int32_t* zrows, int32_t* zmeta,
                                        const int (&v)[NT][2][NB], const int (&top)[NT][2]) const {
    const int lane = threadIdx.x & 31, g = lane >> 2, tl = lane & 3;
#pragma unroll
    for (int t = 0; t < NT; ++t) {
      if (t >= nt) break;
#pragma unroll
      for (int cc = 0; cc < 2; ++cc) {
        const int gsj = __shfl_sync(0xffffffffu, gs[t], 4 * (2 * tl + cc)) >> 2;
        // z: index of the first nonzero digit of the column, -1 (top) .. 8 NB (none)
        int z = 8 * NB;
#pragma unroll
        for (int b = NB - 1; b >= 0; --b) {
          const unsigned nz = (__ballot_sync(0xffffffffu, v[t][cc][b] != 0) >> tl) & 0x11111111u;
          z = nz ? 8 * b + ((__ffs(nz) - 1) >> 2) : z;
        }
        if ((__ballot_sync(0xffffffffu, g == 7 && top[t][cc] != 0) >> tl) & 0x10000000u) z = -1;
        const int j = j0 - 8 * t + 2 * tl + cc, jo = rev ? d - j : j;
        const bool live = j >= jlo && j <= d;
        int32_t* row = zrows + static_cast<long long>(jo) * L + (g - z);
        int sq = 0;  // squared slices of the digits kept
#pragma unroll
        for (int b = 0; b < NB; ++b) {
          const uint32_t w = slice_encode<W>(v[t][cc][b]);
          const bool kept = static_cast<unsigned>(8 * b + g - z) < static_cast<unsigned>(L);
          sq += kept ? slice_square(w) : 0;
          if (kept && live) row[8 * b] = static_cast<int32_t>(w);
        }
        if (z < 0 && g == 7) {
          const uint32_t w = slice_encode<W>(top[t][cc]);
          sq += slice_square(w);
          if (live) row[z - g] = static_cast<int32_t>(w);
        }
#pragma unroll
        for (int o = 4; o <= 16; o <<= 1) sq += __shfl_xor_sync(0xffffffffu, sq, o);
        // (the digits beyond the rows formed)
        if (live)
          for (int b = NB; 8 * b + g - z < L; ++b) row[8 * b] = 0;
        if (live && g == 0) zmeta[jo] = z == 8 * NB ? slice_meta(GRID_ZERO, 0) : slice_meta(gsj - z, sq);
      }
    }
  }
};

// out = in1 +- in2 of coefficient j, exactly, cut to L digits
template <int K>
__device__ __forceinline__ void add_rows(const int32_t* xs, const int32_t* ys, int S, int j, long long sgn,
                                         int32_t* zrows) {
  constexpr int W = Mma<K>::W, L = Mma<K>::L, B = 2 * W;
  const int32_t gx = meta_grid(__ldcg(xs + static_cast<long long>(S) * L + j));
  const int32_t gy = meta_grid(__ldcg(ys + static_cast<long long>(S) * L + j));
  const int32_t* rx = xs + static_cast<long long>(j) * L;
  const int32_t* ry = ys + static_cast<long long>(j) * L;
  int32_t* row = zrows + static_cast<long long>(j) * L;
  const int32_t g = max(gx, gy);
  int32_t o[L];
  int32_t gz = GRID_ZERO;
  if (g < slice_grid_low(K)) {
#pragma unroll
    for (int p = 0; p < L; ++p) o[p] = 0;
  } else {
    const int sx = g - gx, sy = g - gy;  // digits below the common grid's top
    int64_t E[L + 1];
    E[0] = 0;
#pragma unroll
    for (int q = 0; q < L; ++q) {
      const long long xv = q >= sx ? slice_decode<W>(static_cast<uint32_t>(__ldcg(rx + q - sx))) : 0;
      const long long yv = q >= sy ? slice_decode<W>(static_cast<uint32_t>(__ldcg(ry + q - sy))) : 0;
      E[q + 1] = xv + sgn * yv;
    }
    gz = sum_to_digits<L, B>(E, g + 1, o);
  }
  int sq = 0;
#pragma unroll
  for (int p = 0; p < L; ++p) {
    const uint32_t w = slice_encode<W>(o[p]);
    sq += slice_square(w);
    row[p] = static_cast<int32_t>(w);
  }
  zrows[static_cast<long long>(S) * L + j] = slice_meta(gz, sq);
}

// ---------------------------------------------------------------------------
// whole series in shared memory
// ---------------------------------------------------------------------------

// The nt tiles from the o-th longest on of a job whose series are staged, by one warp:
// tile o holds the columns d - 7 - 8 o to d - 8 o, so that the ragged tile is the one
// with fewest terms.  Terms at either end that reach no column (zero coefficients, or
// products L digits below the largest of every column) are left out, as the integer pipe
// leaves out every such term.  All pairs of 128 variables, d = 152, k = 4 (integer pipe;
// all terms; here): coefficients of degree 0 1.87; 2.40; 1.56 ms, inputs of degree 1 1.34;
// 2.41; 1.27 ms, exponential inputs 2.01; 2.36; 1.62 ms.  The range of the nonzero
// coefficients is read from shared memory for every group: registers are what the term
// loop has fewest of.  (128 products of 64, k = 10, uniform series: 6.13 ms without the
// ranges, 6.20 with them.)
template <int K>
__device__ __forceinline__ void columns(int d, int o, int nt, Terms a, bool rev, int32_t* zrows, int32_t* zmeta) {
  constexpr int SW = Mma<K>::SW, NT = Mma<K>::NT, NB = Mma<K>::NB;
  const int lane = threadIdx.x & 31, g = lane >> 2, tl = lane & 3;
  Group<K> grp;
  const int j0 = d - 7 - 8 * o;
  a.y += 4 * ((j0 + g) * SW + tl);
  a.gb += 4 * (j0 + g);
  a.zero += 4 * tl;
  // the largest grid of every column's terms (columns of the later tiles find no term
  // past their last one)
  int n[NT], gm[NT];
#pragma unroll
  for (int t = 0; t < NT; ++t) {
    n[t] = t < nt ? d + 1 - 8 * (o + t) : 0;
    gm[t] = 2 * kZeroGrid;
  }
#pragma unroll 2
  for (int i = tl; i < n[0]; i += 4) {
    const int gx = static_cast<int>(lds(a.ga + 4 * i));
#pragma unroll
    for (int t = 0; t < NT; ++t) gm[t] = __viaddmax_s32(gx, static_cast<int>(lds(a.gb - 4 * i - 32 * t)), gm[t]);
  }
#pragma unroll
  for (int t = 0; t < NT; ++t) {
    gm[t] = max(gm[t], __shfl_xor_sync(0xffffffffu, gm[t], 1));
    gm[t] = max(gm[t], __shfl_xor_sync(0xffffffffu, gm[t], 2));
    if (t >= nt) gm[t] = 2 * kZeroGrid;
  }
  grp.set_grids(gm);
  const volatile Range* range = reinterpret_cast<const volatile Range*>(sm + kRangeWord);
  int begin, end;
  nonzero_terms(range, max(0, j0 - 8 * (nt - 1)), j0 + 7, begin, end);
  if (range->far != 0 && begin < min(end, n[0])) {
    static_assert(NT == 3, "reaching_terms takes three tiles");
    const int reach = 4 * Mma<K>::L;
    const int2 r = reaching_terms(a.ga, a.gb, begin, min(end, n[0]),
                                  make_int3(grp.gs[0] - reach, nt > 1 ? grp.gs[1] - reach : 1 << 30,
                                            nt > 2 ? grp.gs[2] - reach : 1 << 30));
    begin = r.x;
    end = r.y;
  }
#pragma unroll
  for (int t = 0; t < NT; ++t) n[t] = min(n[t], end) - begin;
  a.x += begin * 8 * Mma<K>::PS;
  a.ga += 4 * begin;
  a.y -= 4 * begin * SW;
  a.gb -= 4 * begin;
  grp.clear();
  grp.terms(n, a);
  int v[NT][2][NB], hi[NT][2][NB], top[NT][2] = {};
  grp.words(v, hi);
  grp.carry_words(v, hi, top);
  grp.store(nt, j0, 0, d, rev, zrows, zmeta, v, top);
}

// One persistent launch runs every job of every layer: jobs are claimed in layer
// order from a counter, a job waits (bounded) for the flags of the jobs that
// produce its operands, and sets its own.  Part p of a job split into `split`
// parts takes its share of the column tiles.  The tiles are taken in groups of
// consecutive ones (which share the Toeplitz fragments of their terms), dealt to the
// warps of all parts longest first, back and forth, so that every warp has about the
// same number of terms.  A correlation is run as a convolution with the series x reversed,
// and its result stored backwards.  Staging depth 2 claims the next job early and copies its
// operands into a second buffer, if they are complete, while this one is computed.
template <int K>
__global__ void __launch_bounds__(mma_max_threads(K)) dag_mma_kernel(DagArgs a) {
  using M = Mma<K>;
  constexpr int SW = M::SW, NT = M::NT, L = M::L;
  const int tid = threadIdx.x, T = blockDim.x;
  const BufLayout lay = buf_layout(L, SW, a.dmax + 1, a.dmax + 1);
  Claim* next = reinterpret_cast<Claim*>(sm);
  uint32_t* buf0 = sm + kMiscWords;
  const int nbuf = a.depth >= 2 ? 2 : 1;
  for (int t = tid; t < nbuf * lay.words; t += T) buf0[t] = 0u;
  __syncthreads();
  for (int t = tid; t < nbuf * kPad; t += T)
    reinterpret_cast<int32_t*>(buf0 + t / kPad * lay.words + lay.gb)[t % kPad] = kZeroGrid;
  __syncthreads();
  const int epoch = *reinterpret_cast<volatile int32_t*>(&a.ctrl->epoch);
  const int split = parts(a);
  const int nsub = a.njobs * split;
  const int warps = T >> 5, WT = warps * split;
  const bool ahead = a.depth >= 2;

  // next->claimed: the claimed sub-job, ->ready: its operands are complete
  auto claim = [&]() {
    next->claimed = atomicAdd(&a.ctrl->next[a.counter], 1);
    next->failed = 0;
    next->ready = 0;
  };
  auto ready = [&](bool blocking) {
    const int sj = next->claimed;
    if (sj >= nsub) return;
    const int job = sj / split;
    const ConvJob jb = a.jobs[job];
    if (blocking) {
      if (wait_done(a, jb.dep1, epoch, job) && wait_done(a, jb.dep2, epoch, job))
        next->ready = 1;
      else
        next->failed = 1;
    } else if (is_done(a, jb.dep1, epoch) && is_done(a, jb.dep2, epoch)) {
      next->ready = 1;
    }
  };
  auto stage = [&](const ConvJob& jb, uint32_t* buf) {
    if (jb.kind == JOB_ADD || jb.kind == JOB_SUB) return;  // read where they lie
    const InstInfo in = a.inst[jb.inst];
    const int32_t* s1 = a.ws + in.ws_base + static_cast<long long>(jb.in1) * in.ws_sstride;
    const int32_t* s2 = a.ws + in.ws_base + static_cast<long long>(jb.in2) * in.ws_sstride;
    const bool conv = jb.kind == JOB_CONV;
    int32_t* mx = reinterpret_cast<int32_t*>(buf + lay.mx);
    int32_t* my = reinterpret_cast<int32_t*>(buf + lay.my);
    stage_rows<K, SW, 1>(buf + lay.y, my, conv ? s2 : s1, in.S, 0, in.d + 1, !conv);
    stage_rows<K, 2 * M::PS, 2>(buf + lay.x + 2 * kPairLead, mx, conv ? s1 : s2, in.S, 0, in.d + 1, false);
  };

  bool claimed = false, staged = false;
  int cur = 0;
  for (;;) {
    if (tid == 0) {
      if (!claimed) claim();
      if (!next->ready) ready(true);
    }
    __syncthreads();
    const int sj = next->claimed;
    if (sj >= nsub || next->failed) break;
    const int job = sj / split;
    const int part = sj - job * split;
    const ConvJob jb = a.jobs[job];
    const InstInfo in = a.inst[jb.inst];
    const int d = in.d;
    uint32_t* buf = buf0 + cur * lay.words;
    if (!staged) stage(jb, buf);
    copies_wait();
    __syncthreads();
    staged = false;
    const bool elementwise = jb.kind == JOB_ADD || jb.kind == JOB_SUB;
    if (ahead) {
      if (tid == 0) {
        claim();
        ready(false);
      }
      __syncthreads();
      const int nj = next->claimed;
      if (nj < nsub && next->ready) {
        stage(a.jobs[nj / split], buf0 + (cur ^ 1) * lay.words);
        staged = true;
      }
    }
    int32_t* zrows = a.ws + in.ws_base + static_cast<long long>(jb.out) * in.ws_sstride;
    int32_t* zmeta = zrows + static_cast<long long>(in.S) * L;
    if (elementwise) {
      const int32_t* s1 = a.ws + in.ws_base + static_cast<long long>(jb.in1) * in.ws_sstride;
      const int32_t* s2 = a.ws + in.ws_base + static_cast<long long>(jb.in2) * in.ws_sstride;
      for (int j = part * T + tid; j <= d; j += T * split)
        add_rows<K>(s1, s2, in.S, j, jb.kind == JOB_SUB ? -1 : 1, zrows);
    } else {
      const int32_t* my = reinterpret_cast<const int32_t*>(buf + lay.my);
      const Found f =
          split_metas(reinterpret_cast<const int32_t*>(buf + lay.mx), reinterpret_cast<int32_t*>(buf + lay.ga), d + 1,
                      my, reinterpret_cast<int32_t*>(buf + lay.gb) + kPad, d + 1);
      Terms at{};
      at.flat = is_flat<K>(f);
      at.gmax = at.flat ? f.gmax : 0;
      at.every = drain_terms<K>(f);
      if (tid == 0)
        *reinterpret_cast<Range*>(sm + kRangeWord) = Range{f.x0, f.x1, f.y0, f.y1, f.spread >= 4 * L};
      form_rows<K>(buf + lay.x, d + 1, buf + lay.y, my, d + 1, at.flat, at.gmax);
      __syncthreads();
      const int base = 4 * (kMiscWords + cur * lay.words);
      at.x = base + 4 * lay.x;
      at.ga = base + 4 * lay.ga;
      at.y = base + 4 * lay.y;
      at.gb = base + 4 * (lay.gb + kPad);
      at.zero = base;
      const int ntiles = (d + 8) / 8;
      const bool corr = jb.kind == JOB_CORR;
      // groups of gsz consecutive tiles, so many that every warp gets two, a long and
      // a short one
      const int gsz = min(NT, (ntiles + 2 * WT - 1) / (2 * WT));
      const int ngroups = (ntiles + gsz - 1) / gsz;
      const int wk = (tid >> 5) * split + part;
      for (int q = 0; q * WT < ngroups; ++q) {
        const int og = q * WT + ((q & 1) ? WT - 1 - wk : wk);
        if (og >= ngroups) continue;
        const int o = og * gsz;  // the o-th longest tile
        columns<K>(d, o, min(gsz, ntiles - o), at, corr, zrows, zmeta);
      }
    }
    __syncthreads();
    if (tid == 0) st_release(a.flags + sj, epoch);
    claimed = ahead;
    if (ahead) cur ^= 1;
  }
  copies_wait();
}

// ---------------------------------------------------------------------------
// output tiles, for degrees whose whole series do not fit in shared memory
// ---------------------------------------------------------------------------

// Sub-job j * split + t computes the coefficients [tD, tD + D) of job j, D =
// a.tile.  The Toeplitz operand is staged a.xrows coefficients at a time with the
// window of the column operand they meet; the accumulators stay in registers over
// the whole series, carried into digits before their upper parts could pass 24 bits.
// The reference grids are those of the whole series, so the results are the
// whole-series kernel's, bit for bit.
template <int K>
__global__ void __launch_bounds__(mma_max_threads(K)) dag_mma_tiled_kernel(DagArgs a) {
  using M = Mma<K>;
  constexpr int SW = M::SW, NT = M::NT, L = M::L;
  const int tid = threadIdx.x, T = blockDim.x, lane = tid & 31, g = lane >> 2, tl = lane & 3;
  const int D = a.tile, XR = a.xrows;
  const BufLayout lay = buf_layout(L, SW, XR, D + XR);
  Claim* next = reinterpret_cast<Claim*>(sm);
  uint32_t* buf = sm + kMiscWords;
  for (int t = tid; t < lay.words; t += T) buf[t] = 0u;
  __syncthreads();
  int32_t* ga = reinterpret_cast<int32_t*>(buf + lay.ga);
  int32_t* mx = reinterpret_cast<int32_t*>(buf + lay.mx);
  int32_t* my = reinterpret_cast<int32_t*>(buf + lay.my);
  int32_t* gb = reinterpret_cast<int32_t*>(buf + lay.gb) + kPad;
  for (int t = tid; t < kPad; t += T) gb[t - kPad] = kZeroGrid;
  const int epoch = *reinterpret_cast<volatile int32_t*>(&a.ctrl->epoch);
  const int tiles = parts(a);
  const int nsub = a.njobs * tiles;
  const int warps = T >> 5, warp = tid >> 5;

  for (;;) {
    __syncthreads();
    if (tid == 0) {
      next->claimed = atomicAdd(&a.ctrl->next[a.counter], 1);
      next->failed = 0;
    }
    __syncthreads();
    const int sj = next->claimed;
    if (sj >= nsub) break;
    const int job = sj / tiles;
    const int tile = sj - job * tiles;
    const ConvJob jb = a.jobs[job];
    const InstInfo in = a.inst[jb.inst];
    const int d = in.d, S = in.S;
    const int jn = min(D, d + 1 - tile * D);  // output coefficients of this tile (<= 0: none)
    const bool elementwise = jb.kind == JOB_ADD || jb.kind == JOB_SUB;
    const bool conv = jb.kind == JOB_CONV;
    if (jn > 0) {
      if (tid == 0) {
        const int t_lo = elementwise ? tile : 0;
        const int t_hi = (elementwise || conv) ? tile : d / D;
        bool ok = true;
        for (int t = t_lo; ok && t <= t_hi; ++t) {
          if (jb.dep1 >= 0) ok = wait_flag(a, jb.dep1 * tiles + t, epoch, job);
          if (ok && jb.dep2 >= 0) ok = wait_flag(a, jb.dep2 * tiles + t, epoch, job);
        }
        next->failed = ok ? 0 : 1;
      }
      __syncthreads();
      if (next->failed) break;
      const int32_t* s1 = a.ws + in.ws_base + static_cast<long long>(jb.in1) * in.ws_sstride;
      const int32_t* s2 = a.ws + in.ws_base + static_cast<long long>(jb.in2) * in.ws_sstride;
      int32_t* zrows = a.ws + in.ws_base + static_cast<long long>(jb.out) * in.ws_sstride;
      int32_t* zmeta = zrows + static_cast<long long>(S) * L;
      if (elementwise) {
        for (int j = tile * D + tid; j < tile * D + jn; j += T)
          add_rows<K>(s1, s2, S, j, jb.kind == JOB_SUB ? -1 : 1, zrows);
      } else {
        // columns [c0, c0 + jn); of a correlation, those of the reversed result, whose
        // column operand is the reversed first series
        const int c0 = conv ? tile * D : d + 1 - tile * D - jn;
        const int terms = c0 + jn;  // of the tile's longest coefficient
        // Only chunks of terms that meet nonzero coefficients in a column of the tile are
        // staged, and the operand with fewer of them is the Toeplitz one (inputs of degree 1;
        // integer pipe, all chunks, here: 8 products of 16, d = 1023, k = 10: 3.1, 8.8,
        // 2.0 ms; 40 products of 4, d = 600, k = 10: 0.74, 1.53, 0.69 ms).
        volatile Range* range = reinterpret_cast<volatile Range*>(sm + kRangeWord);
        const long long metas = static_cast<long long>(S) * L;
        const bool first = tile_range((conv ? s1 : s2) + metas, conv ? s2 + metas : s1 + metas + d, conv ? 1 : -1,
                                      terms, c0, conv) != conv;
        const int32_t* xs = first ? s1 : s2;  // the Toeplitz operand
        const int32_t* ys = first ? s2 : s1;
        const int32_t* gX = xs + metas;
        const int32_t* gY = ys + metas;
        const int ntiles = (jn + 7) / 8;
        // groups of consecutive column tiles, longest first, in passes of one per warp
        const int gsz = min(NT, (ntiles + warps - 1) / warps);
        const int ngroups = (ntiles + gsz - 1) / gsz;
        for (int p0 = 0; p0 < ngroups; p0 += warps) {
          Group<K> grp;
          const int o = (p0 + warp) * gsz;
          const int j0 = c0 + jn - 8 * (o + 1);  // first column of tile 0
          int cnt[NT], top[NT][2], gm[NT];
#pragma unroll
          for (int t = 0; t < NT; ++t) {
            const bool exists = t < gsz && o + t < ntiles;
            cnt[t] = exists ? j0 - 8 * t + 8 : 0;
            top[t][0] = top[t][1] = 0;
            gm[t] = 2 * kZeroGrid;
            const int j = j0 - 8 * t + g;
            if (exists) {
#pragma unroll 4
              for (int i = tl; i <= j; i += 4) {
                const int m = j - i;
                gm[t] = max(gm[t], 4 * (meta_grid(__ldcg(gX + i)) + meta_grid(__ldcg(gY + (conv ? m : d - m)))));
              }
            }
            gm[t] = max(gm[t], __shfl_xor_sync(0xffffffffu, gm[t], 1));
            gm[t] = max(gm[t], __shfl_xor_sync(0xffffffffu, gm[t], 2));
          }
          grp.set_grids(gm);
          grp.clear();
          int held = 0;  // terms since the last carry
          for (int i0 = 0; i0 < terms; i0 += XR) {
            const int xn = min(XR, terms - i0);
            if (i0 + xn <= range->x0 || i0 >= range->x1) continue;
            // the column rows those terms meet: [y0, y1)
            const int y0 = max(0, c0 - (i0 + xn - 1)), y1 = min(d + 1, c0 + jn - i0);
            __syncthreads();  // the rows staged before are no longer read
            stage_rows<K, SW, 1>(buf + lay.y, my, ys, S, conv ? y0 : d + 1 - y1, y1 - y0, !conv);
            stage_rows<K, 2 * M::PS, 2>(buf + lay.x + 2 * kPairLead, mx, xs, S, i0, xn, false);
            copies_wait();
            __syncthreads();
            const Found f = split_chunk(mx, ga, xn, my, gb, y1 - y0);
            Terms at{};
            at.flat = is_flat<K>(f);
            at.gmax = at.flat ? f.gmax : 0;
            at.every = drain_terms<K>(f);
            form_rows<K>(buf + lay.x, xn, buf + lay.y, my, y1 - y0, at.flat, at.gmax);
            __syncthreads();
            if (held + xn > M::kLimit) {
              grp.carry(top);
              held = 0;
            }
            held += xn;
            int n[NT];
#pragma unroll
            for (int t = 0; t < NT; ++t) n[t] = max(0, min(xn, cnt[t] - i0));
            const int m = j0 + g - i0 - y0;
            constexpr int base = 4 * kMiscWords;
            at.x = base + 4 * lay.x;
            at.ga = base + 4 * lay.ga;
            at.y = base + 4 * (lay.y + m * SW + tl);
            at.gb = base + 4 * (lay.gb + kPad + m);
            at.zero = base + 4 * tl;
            grp.terms(n, at);
          }
          int v[NT][2][M::NB], hi[NT][2][M::NB];
          grp.words(v, hi);
          grp.carry_words(v, hi, top);
          grp.store(min(gsz, ntiles - o), j0, c0, d, !conv, zrows, zmeta, v, top);
        }
      }
    }
    __syncthreads();
    if (tid == 0) st_release(a.flags + sj, epoch);
  }
}

template <int K>
void* mma_fn(bool tiled) {
  return tiled ? reinterpret_cast<void*>(&dag_mma_tiled_kernel<K>) : reinterpret_cast<void*>(&dag_mma_kernel<K>);
}

}  // namespace

// The line is the work of an average layer in terms (of one coefficient with one column
// tile): a job's passes around its products (fragment pairs, grids, carries, fewer warps in
// flight per job) take about 10 us however short it is, so a table needs layers wide enough
// to keep every SM on several jobs, and more of them where the staged series leave an SM one
// CTA.  At k <= 3 a coefficient's slices fill too little of a 16-slice block (20 % slower at
// k = 2, d = 152).  Degrees whose whole series fit in shared memory only as 28-bit digits
// stay there, and so do those of k = 4 and 5 with one CTA an SM, but the widest of k = 4.
//
// Integer pipe's time over this form's, 7226 random polynomials (monomials of 2 to 16
// variables), tenth percentile / median for uniform series; exponential ones with
// coefficients of degree 0; coefficients falling by 2 bits a degree:
//   k = 10, d 56-248, work 250-330 k   1.14 / 1.32   1.04 / 1.17   0.98 / 1.13
//           d 249-471, 400-500 k       1.17 / 1.35   1.34 / 1.55   1.02 / 1.15
//           tiles, 500-750 k           1.33 / 1.43   1.35 / 1.60   (zeros from d = 450 on)
//   k = 8,  d 72-252, 330-400 k        1.12 / 1.23   0.99 / 1.10   0.94 / 1.07
//           d 253-513, 750-1120 k      1.18 / 1.40   1.31 / 1.65   1.01 / 1.20
//           tiles, 1.75-3.25 M         1.05 / 1.25   1.41 / 1.85
//   k = 4,  d 136-199, 640-800 k       1.10 / 1.16   1.03 / 1.08   0.93 / 1.04
//           d 200-329, 1.2-1.8 M       1.19 / 1.33   1.25 / 1.47   1.00 / 1.13
//           d 330-669, 2.8-5.2 M       1.25 / 1.32   1.45 / 1.80   0.98 / 1.14
//           tiles, 640-800 k           1.05 / 1.10   1.77 / 2.20
//   k = 5,  d 256-277, 1.2-1.8 M       1.18 / 1.37   1.40 / 1.46   1.04 / 1.16
// and below the lines: k = 4, d 200-329, 400-640 k 0.88 / 0.98, d 330-660, 0.4-1.8 M 0.80 /
// 0.97; k = 5, d 278-556 0.80 / 0.95, tiles 0.90 / 0.97; k = 8, d 253-507, 250-400 k 0.93 /
// 1.05, tiles of exponential series 0.71 / 0.78.
bool mma_takes(int k, int d, const int32_t* supp_ptr, int32_t m0, int32_t m1, bool whole, size_t optin) {
  if (m0 >= m1 || !mma_has(k)) return false;
  if (d < (k == 4 ? 136 : k == 5 ? 256 : k == 8 ? 72 : 56)) return false;
  if (whole && mma_smem_bytes(k, d, 1) > optin) return false;
  // products and layers of the monomials (3 n - 3 and n of one of n >= 2 variables)
  int64_t jobs = 0;
  int32_t layers = 1;
  for (int32_t m = m0; m < m1; ++m) {
    const int32_t n = supp_ptr[m + 1] - supp_ptr[m];
    jobs += n < 2 ? 1 : 3 * n - 3;
    layers = n > layers ? n : layers;
  }
  const double tiles = (d + 8) / 8, terms = 0.5 * (d + 1);
  const double work = static_cast<double>(jobs) / layers * tiles * terms;
  const bool two = 2 * (mma_smem_bytes(k, d, 1) + 1024) <= 228 * 1024;  // two CTAs fit an SM
  constexpr double kNever = 1e30;
  double least = kNever;
  switch (k) {
    case 4: least = !whole ? 640e3 : !two ? 2.8e6 : d < 173 ? 640e3 : 3.7e3 * d; break;
    case 5: least = !whole || !two ? kNever : d < 266 ? 750e3 + 45e3 * (d - 256) : 1.2e6; break;
    case 8: least = !whole ? 1.75e6 : two ? 350e3 : 750e3; break;
    case 10: least = !whole ? 600e3 : two ? 250e3 : 400e3; break;
  }
  return work >= least;
}

void* mma_kernel(int k, bool tiled) {
  switch (k) {
    case 4: return mma_fn<4>(tiled);
    case 5: return mma_fn<5>(tiled);
    case 8: return mma_fn<8>(tiled);
    case 10: return mma_fn<10>(tiled);
    default: return nullptr;
  }
}

size_t mma_smem_bytes(int k, int dmax, int depth) {
  const BufLayout lay = buf_layout(slice_digits(k), mma_stride(k), dmax + 1, dmax + 1);
  const size_t buffers = depth >= 2 ? 2 : 1;
  return 4 * (kMiscWords + buffers * static_cast<size_t>(lay.words));
}

// Threads per CTA for degree dmax: as many warps as fill the registers with the CTAs that
// fit in an SM's shared memory (12, 16 or 20 warps an SM), at most one per column tile.
// (k = 10, d = 127: three CTAs of four warps instead of three take 0.87 of the time.)
int mma_threads(int k, int dmax) {
  const int warps = mma_max_threads(k) / 32;
  const int ctas = static_cast<int>((228 * 1024) / (mma_smem_bytes(k, dmax, 1) + 1024));
  const int most = (dmax + 8) / 8;
  auto filled = [&](int w) { return w * (ctas < warps / w ? ctas : warps / w); };
  int full = 0;
  for (int w = 1; w <= warps && w <= most; ++w) full = filled(w) > full ? filled(w) : full;
  // (more CTAs rather than the last warps: one stages while others multiply)
  int best = 1;
  while (20 * filled(best) < 17 * full) ++best;
  return 32 * best;
}

size_t mma_tiled_smem_bytes(int k, int tile, int xrows) {
  return 4 * (static_cast<size_t>(kMiscWords) +
              static_cast<size_t>(buf_layout(slice_digits(k), mma_stride(k), xrows, tile + xrows).words));
}

}  // namespace pes
