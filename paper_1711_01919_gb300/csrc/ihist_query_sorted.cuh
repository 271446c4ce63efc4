// ihist_query_sorted.cuh -- Eq. 2 region histograms for large rectangle
// batches on a bin-major H, with the corner lookups put in row order first.
//
// Eq. 2 reads four words of H per (rectangle, bin).  In the bin-major layout
// a bin plane is h x w words, so the lookups of random rectangles land on
// random DRAM lines: each 4-byte corner costs a whole line fetch (one
// thread per (rectangle, bin) runs at the random-gather rate of the GPU).
// Here the lookups are first bucketed by row (a counting sort), then made
// bucket after bucket: the corners of one row of one plane are read at about
// the same time, so every line of H they touch comes from DRAM once and
// serves all of them from L2.  The order is the same for every bin, so the
// sort is paid once per batch.
//
// What is sorted is a row's pair of corners, not a corner: Eq. 2 is
//   (H[y1][x1] - H[y1][x0-1]) - (H[y0-1][x1] - H[y0-1][x0-1]),
// one difference per row, so a rectangle has two lookups (one when it starts
// at row 0) and the values kept between the two passes over a group of bins
// are half as many -- 64 MB for 2^20 rectangles and 8 bins, which L2 holds,
// where one value per corner took 128 MB and went through DRAM.
//
//   1. pair_rank     per valid rectangle and row: its rank in the row's
//                    bucket, cnt[y]++ (the one atomic of a pair)
//   2. row_offsets   exclusive scan of cnt over the h rows (one CTA)
//   3. pair_scatter  pair -> position off[y] + rank: pts[pos] = (y, x1, x0-1)
//   4. pair_gather   per group of nb bins: val[pos][j] = H[b0 + j][y][x1] -
//                    H[b0 + j][y][x0-1]
//   5. pair_combine  out[r][b0 + j] = val[lower row][j] - val[upper row][j]
// in uint32 modular arithmetic, as Eq. 2 is evaluated everywhere.
//
// Pairs within a row bucket come in atomic order, which changes the
// positions but not the result: each output word is the same four terms.
#pragma once

#include "ihist_device.cuh"

namespace ihist {

// A load that takes no more than 64 bytes from DRAM: by default a miss
// fetches the whole 128-byte line (126 bytes per random 4-byte load measured,
// 63 with the hint).
__device__ __forceinline__ uint32_t ld_64b(const uint32_t *p) {
  uint32_t v;
  asm("ld.global.nc.L2::64B.b32 %0, [%1];" : "=r"(v) : "l"(p));
  return v;
}

constexpr uint32_t kNoPair = 0xffffffffu;  // a pair that Eq. 2 does not have
constexpr uint32_t kNoColumn = 0xffffu;    // column -1 (w <= 65535, so no column has this index)

__device__ __forceinline__ bool rect_ok(const int32_t *rects, unsigned int r, int H, int W, int &x0, int &y0,
                                        int &x1, int &y1) {
  const int32_t *p = rects + 4 * (size_t)r;  // 4-byte aligned rows: four scalar loads
  x0 = __ldg(p);
  y0 = __ldg(p + 1);
  x1 = __ldg(p + 2);
  y1 = __ldg(p + 3);
  return (0 <= x0) & (x0 <= x1) & (x1 < W) & (0 <= y0) & (y0 <= y1) & (y1 < H);
}

// 1. slot[r] = the ranks of rectangle r's lower (y1) and upper (y0 - 1) row
// pairs; kNoPair for a pair it does not have (bad rectangles latch the status).
__global__ void __launch_bounds__(256) pair_rank_kernel(const int32_t *__restrict__ rects, unsigned int n, int H,
                                                        int W, unsigned int *cnt, uint2 *__restrict__ slot,
                                                        Ctrl *ctrl) {
  for (unsigned int r = blockIdx.x * blockDim.x + threadIdx.x; r < n; r += gridDim.x * blockDim.x) {
    int x0, y0, x1, y1;
    uint2 s = make_uint2(kNoPair, kNoPair);
    if (rect_ok(rects, r, H, W, x0, y0, x1, y1)) {
      s.x = atomicAdd(cnt + y1, 1u);
      if (y0 > 0) s.y = atomicAdd(cnt + y0 - 1, 1u);
    } else {
      latch_status(ctrl, kStatusBadRect);
    }
    slot[r] = s;
  }
}

// 2. off[y] = sum of cnt[0..y), off[H] = the number of pairs; one CTA of
// 1024 threads, each scanning a contiguous run of rows.
__global__ void __launch_bounds__(1024) row_offsets_kernel(const unsigned int *__restrict__ cnt, int H,
                                                           unsigned int *off) {
  __shared__ unsigned int s_part[1024];
  const int t = threadIdx.x;
  const int per = (H + 1023) / 1024;
  const int y0 = min(H, t * per), y1 = min(H, y0 + per);
  unsigned int sum = 0u;
  for (int y = y0; y < y1; ++y) sum += cnt[y];
  s_part[t] = sum;
  __syncthreads();
  // inclusive scan of the 1024 partial sums (Hillis-Steele in shared memory)
  for (int d = 1; d < 1024; d <<= 1) {
    const unsigned int v = t >= d ? s_part[t - d] : 0u;
    __syncthreads();
    s_part[t] += v;
    __syncthreads();
  }
  unsigned int run = s_part[t] - sum;
  for (int y = y0; y < y1; ++y) {
    off[y] = run;
    run += cnt[y];
  }
  if (t == 1023) off[H] = s_part[1023];
}

// 3. each pair goes to its position; slot[r] becomes the positions.
__global__ void __launch_bounds__(256) pair_scatter_kernel(const int32_t *__restrict__ rects, unsigned int n, int H,
                                                           int W, const unsigned int *__restrict__ off,
                                                           uint2 *__restrict__ pts, uint2 *__restrict__ slot) {
  for (unsigned int r = blockIdx.x * blockDim.x + threadIdx.x; r < n; r += gridDim.x * blockDim.x) {
    int x0, y0, x1, y1;
    if (!rect_ok(rects, r, H, W, x0, y0, x1, y1)) continue;
    uint2 s = slot[r];
    const uint32_t xs = (uint32_t)x1 << 16 | (x0 > 0 ? (uint32_t)(x0 - 1) : kNoColumn);
    s.x += off[y1];
    pts[s.x] = make_uint2((uint32_t)y1, xs);
    if (y0 > 0) {
      s.y += off[y0 - 1];
      pts[s.y] = make_uint2((uint32_t)(y0 - 1), xs);
    }
    slot[r] = s;
  }
}

// 4. one thread per pair: the nb differences of bins b0 .. b0+nb-1,
// val[pos][0..nb).  NB is the compile-time group width (the last group may
// hold fewer bins, nb <= NB).
//
// Bound by DRAM reads of H in 64-byte pieces, about 63% of them touched by
// 2^20 random rectangles on 8192 x 8192.  The CTAs are as many as the pairs
// need and run in row order, so that at any time only the rows of the pairs
// in flight are open: 2^20 rectangles x 128 bins, 8 per pass, 7.26 ms with a
// capped grid striding over all rows and whole-line misses, 6.16 with 64-byte
// misses, 4.74 with both.  One thread per (pair, bin) is as fast there (4.56
// ms) but slower where rows are short (1187 x 1510 x 25, 2^20 rectangles: 775
// against 530 us), where neighbouring pairs share lines in L1.
__host__ __device__ constexpr int gather_threads(int nb) { return nb == 16 ? 1024 : 512; }

template <int NB>
__global__ void __launch_bounds__(gather_threads(NB)) pair_gather_kernel(const uint32_t *__restrict__ hist, int H, int W, int b0,
                                                          int nb, const uint2 *__restrict__ pts,
                                                          const unsigned int *__restrict__ off,
                                                          uint32_t *__restrict__ val) {
  const unsigned int pos = blockIdx.x * blockDim.x + threadIdx.x;
  if (pos >= off[H]) return;
  const size_t plane = (size_t)H * (size_t)W;
  const uint2 pt = __ldg(pts + pos);
  const uint32_t *row = hist + (size_t)b0 * plane + (size_t)pt.x * W;
  const uint32_t *hi = row + (pt.y >> 16), *lo = row + (pt.y & 0xffffu);
  const bool left = (pt.y & 0xffffu) != kNoColumn;
  uint32_t v[NB], u[NB];
#pragma unroll
  for (int j = 0; j < NB; ++j) {
    v[j] = j < nb ? ld_64b(hi + (size_t)j * plane) : 0u;
    u[j] = j < nb && left ? ld_64b(lo + (size_t)j * plane) : 0u;
  }
  uint32_t *dst = val + (size_t)pos * NB;
#pragma unroll
  for (int j = 0; j < NB; j += 4)
    *reinterpret_cast<uint4 *>(dst + j) =
        make_uint4(v[j] - u[j], v[j + 1] - u[j + 1], v[j + 2] - u[j + 2], v[j + 3] - u[j + 3]);
}

// 5. out[r][b0 + j]: NB / 4 consecutive threads per rectangle, four bins
// each, so the two val rows and the output piece are whole sectors.  VEC:
// the output piece is 16-byte aligned and holds NB bins.
template <int NB, bool VEC>
__global__ void __launch_bounds__(256) pair_combine_kernel(const uint2 *__restrict__ slot, unsigned int n, int B,
                                                           int b0, int nb, const uint32_t *__restrict__ val,
                                                           uint32_t *__restrict__ out) {
  constexpr int T = NB / 4;
  const unsigned long long total = (unsigned long long)n * T;
  for (unsigned long long p = (unsigned long long)blockIdx.x * blockDim.x + threadIdx.x; p < total;
       p += (unsigned long long)gridDim.x * blockDim.x) {
    const unsigned int r = (unsigned int)(p / T);
    const int j = 4 * (int)(p % T);
    const uint2 s = __ldg(slot + r);
    uint4 v = make_uint4(0u, 0u, 0u, 0u), u = v;
    if (s.x != kNoPair) v = __ldcg(reinterpret_cast<const uint4 *>(val + (size_t)s.x * NB + j));
    if (s.y != kNoPair) u = __ldcg(reinterpret_cast<const uint4 *>(val + (size_t)s.y * NB + j));
    v = make_uint4(v.x - u.x, v.y - u.y, v.z - u.z, v.w - u.w);
    uint32_t *o = out + (size_t)r * B + b0 + j;
    if (VEC) {
      st_stream_v4(o, v.x, v.y, v.z, v.w);
    } else {
      const uint32_t vv[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
      for (int i = 0; i < 4; ++i)
        if (j + i < nb) st_stream(o + i, vv[i]);
    }
  }
}

}  // namespace ihist
