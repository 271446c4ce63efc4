// ihist_bands.cuh -- the integral histogram of one frame in two launches
// that wait on nothing inside themselves: band_count_kernel reads the frame
// once and leaves the counts that every band starts from, band_emit_kernel
// writes H (Eq. 1 of arXiv 1711.01919).
//
// What it is for: the look-back kernel (ihist_scan.cuh) carries counts from
// band to band through flags in global memory, and a frame that fills only a
// wave or two of CTAs spends as long on that chain (ticket, count, publish,
// look back, publish again) as on its stores.  Counting needs no chain: the
// number of pixels of a bin above a band, in one column, is a sum of the
// column's counts in the bands above, and those depend on the frame alone.
// Measured per frame, back to back, look-back kernel -> these two (uniform
// pixels, GB300): 320x240 x 16 16.9 -> 6.2 us, 640x480 x 32 21.4 -> 11.4,
// 1280x720 x 32 36 -> 26, 1920x1080 x 64 104.9 -> 85.5 (a plain fill of the
// same bytes takes 78.5), 1921x1081 x 64 160 -> 92, 3840x2160 x 64 355 -> 329;
// quad-major 1920x1080 x 64 108 -> 90, 1921x1081 x 64 582 -> 116; pixel-major
// 640x480 x 64 61 -> 22, 1920x1080 x 64 150 -> 92, 1921x1081 x 37 300 -> 74,
// 3840x2160 x 64 521 -> 348.
//
// Superband: 4 bands of R rows (R = 8, 16 or 32).  A group is 4 bins, packed
// as the bytes of one word; a chunk is 128 columns.  The count kernel leaves
//   q    [H][chunks * 128]           each pixel's bin, one byte
//   pb   [band][group][column]       counts of the column in the bands above
//                                    this one within its superband (bytes)
//   sb   [superband][group][column]  counts of the column in the superband
//   rl   [chunk][group][row]         counts of the row inside the chunk
//   rls  [chunk][3][group][row]      counts of the row inside the chunk's first
//                                    32, 64 and 96 columns (pixel-major only)
//   ct   [group][chunk][band]        counts of the band inside the chunk
//                                    (16-bit lanes; only when a band is split
//                                    into width segments)
// and a band's first row of H follows from pb, the sb above and a scan along
// the columns.
#pragma once

#include "ihist_device.cuh"

namespace ihist {

constexpr int kSuper = 4;            // bands per superband
constexpr int kCountThreads = 512;
constexpr int kHalf = kChunk / 2;    // columns of a column tile
constexpr int kColPitch = kHalf + 4;  // bytes between rows of a column tile
constexpr int kRowPitch = kChunk + 4;  // of a row tile: rows one bank apart, so a warp reads down a column of words without conflicts
constexpr int kSegWarps = 8;         // chunks of one emit CTA at most

struct BandDesc {
  const uint8_t *in;
  long long pitch;
  uint32_t *out;
  const uint32_t *lut;  // table plans: 8 * bin of each intensity, or the no-bin mark
  int jc, jmul[4], jstride[4];  // joint plans: channels, their bins and digit weights (see ihist_joint.cuh)
  int H, W, B, qmul;
  int early;            // 1: the frame may be read before the previous grid has completed
  int R, nbands, nsb, nq, nchunks, nsegs, cps;
  int split;     // a count thread counts R >> split pixels
  int wpg, gpc;  // emit CTAs: warps of one group, and groups
  uint8_t *q;
  int bpb, nblk;  // pixel-major: bins of one CTA (a multiple of 4, at most 64) and blocks of them
  uint32_t *pb, *sb, *rl, *rls;
  uint2 *ct;
  Ctrl *ctrl;  // checked builds: where a failed store check is latched
};

// Elements of the workspace's arrays.
__host__ __device__ inline size_t q_size(const BandDesc &f) { return (size_t)f.H * f.nchunks * kChunk; }
__host__ __device__ inline size_t pb_size(const BandDesc &f) { return (size_t)f.nbands * f.nq * f.nchunks * kChunk; }
__host__ __device__ inline size_t sb_size(const BandDesc &f) { return (size_t)f.nsb * f.nq * f.nchunks * kChunk; }
__host__ __device__ inline size_t rl_size(const BandDesc &f) { return (size_t)f.nchunks * f.nq * f.nsb * kSuper * f.R; }
__host__ __device__ inline size_t rls_size(const BandDesc &f) { return 3 * rl_size(f); }
__host__ __device__ inline size_t ct_size(const BandDesc &f) { return (size_t)f.nbands * f.nq * f.nchunks; }

// Checked builds: whether the n elements at p lie in array a of the workspace.
#define IHIST_IN(f, a, p, n) IHIST_GUARD((f).ctrl, (p) >= (f).a && (p) + (n) <= (f).a + a##_size(f))

__device__ __forceinline__ void griddep_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void griddep_release() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }

// 16 bytes from global to shared memory, past L1 (both addresses aligned).
__device__ __forceinline__ void copy_async16(void *dst, const void *src) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(smem_u32(dst)), "l"(src) : "memory");
}
__device__ __forceinline__ void copy_async_wait() { asm volatile("cp.async.wait_all;" ::: "memory"); }

// One more in a byte counter of this thread's own (shared memory address).
__device__ __forceinline__ void bump_byte(uint32_t a) {
  asm volatile(
      "{\n\t.reg .u32 n;\n\t"
      "ld.shared.u8 n, [%0];\n\t"
      "add.u32 n, n, 1;\n\t"
      "st.shared.u8 [%0], n;\n\t}" ::"r"(a)
      : "memory");
}

enum { kBinUniform = 0, kBinTable = 1, kBinJoint = 2 };

// Bins of four pixels, one byte each.
template <int MODE>
__device__ __forceinline__ uint32_t bins4(const BandDesc &f, const uint8_t *s_lut, uint32_t v) {
  if constexpr (MODE == kBinTable) {
    return (uint32_t)s_lut[v & 0xffu] | (uint32_t)s_lut[(v >> 8) & 0xffu] << 8 |
           (uint32_t)s_lut[(v >> 16) & 0xffu] << 16 | (uint32_t)s_lut[v >> 24] << 24;
  } else {
    // floor(v * B / 256): two products in 16-bit lanes, v * B <= 255 * 256
    const uint32_t e = (v & 0x00ff00ffu) * (uint32_t)f.qmul, o = ((v >> 8) & 0x00ff00ffu) * (uint32_t)f.qmul;
    return ((e >> 8) & 0x00ff00ffu) | (o & 0xff00ff00u);
  }
}

// Joint bins of the four pixels of C channels at src, loaded as C words (4 C
// byte loads, in both roles of the count kernel, cost a 1920x1080 RGB frame 6
// us: 94.5 -> 88.6).
template <int C>
__device__ __forceinline__ uint32_t joint4(const BandDesc &f, const uint8_t *src) {
  uint32_t v[C], q = 0u;
#pragma unroll
  for (int c = 0; c < C; ++c) v[c] = __ldcg(reinterpret_cast<const unsigned int *>(src) + c);
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    uint32_t k = 0u;
#pragma unroll
    for (int c = 0; c < C; ++c) {
      const int at = i * C + c;
      k += ((__byte_perm(v[at >> 2], 0u, 0x4440u + (at & 3)) * (uint32_t)f.jmul[c]) >> 8) * (uint32_t)f.jstride[c];
    }
    q |= k << (8 * i);
  }
  return q;
}

// Put the bins of rows r, r + step, .. < nrows (of the rows from y0 on) at
// columns x .. x+3 into a tile column (and, with to_q, into the plane of
// bins).  Columns past the frame get bin 0: they lie right of every column
// that is stored, so no result depends on them.
template <int MODE>
__device__ __forceinline__ void load_tile(const BandDesc &f, const uint8_t *s_lut, int y0, int r, int step, int nrows,
                                          int x, uint32_t *tp, int tstep, bool to_q) {
  const size_t wpad = (size_t)f.nchunks * kChunk;
  const uint8_t *src = f.in + (long long)(y0 + r) * f.pitch;
  uint8_t *qp = f.q + (size_t)(y0 + r) * wpad + x;
  const long long sstep = (long long)step * f.pitch;
  const size_t qstep = (size_t)step * wpad;
  if constexpr (MODE == kBinJoint) {
    const bool words = x + 3 < f.W && ((reinterpret_cast<uintptr_t>(f.in) | (uintptr_t)f.pitch) & 3u) == 0;
    src += x * f.jc;
#pragma unroll 2
    for (; r < nrows; r += step) {
      uint32_t q = 0u;
      if (words) {
        q = f.jc == 3 ? joint4<3>(f, src) : f.jc == 4 ? joint4<4>(f, src) : f.jc == 2 ? joint4<2>(f, src) : joint4<1>(f, src);
      } else {
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          if (x + i < f.W) {
            uint32_t k = 0u;
            for (int c = 0; c < f.jc; ++c)
              k += (((uint32_t)__ldg(src + i * f.jc + c) * (uint32_t)f.jmul[c]) >> 8) * (uint32_t)f.jstride[c];
            q |= k << (8 * i);
          }
        }
      }
      *tp = q;
      if (to_q && IHIST_IN(f, q, qp, 4)) *reinterpret_cast<uint32_t *>(qp) = q;
      src += sstep;
      tp += tstep;
      qp += qstep;
    }
  } else {
    const bool words = x + 3 < f.W && ((reinterpret_cast<uintptr_t>(f.in) | (uintptr_t)f.pitch) & 3u) == 0;
    src += x;
    if (words) {
#pragma unroll 8
      for (; r < nrows; r += step) {
        const uint32_t q = bins4<MODE>(f, s_lut, __ldcg(reinterpret_cast<const unsigned int *>(src)));
        *tp = q;
        if (to_q && IHIST_IN(f, q, qp, 4)) *reinterpret_cast<uint32_t *>(qp) = q;
        src += sstep;
        tp += tstep;
        qp += qstep;
      }
    } else {
#pragma unroll 2
      for (; r < nrows; r += step) {
        uint32_t v = 0u;
#pragma unroll
        for (int i = 0; i < 4; ++i)
          if (x + i < f.W) v |= (uint32_t)__ldg(src + i) << (8 * i);
        const uint32_t q = bins4<MODE>(f, s_lut, v);
        *tp = q;
        if (to_q && IHIST_IN(f, q, qp, 4)) *reinterpret_cast<uint32_t *>(qp) = q;
        src += sstep;
        tp += tstep;
        qp += qstep;
      }
    }
  }
}

// Shared memory of the count kernel: the tile's bins, then one byte counter
// per bin and thread, as words of 4 bins [nq + 1][512] (thread t's word of
// group g in bank t mod 32 whatever the pixel, so no access conflicts; the
// extra word takes values that are in no bin).  A column tile is 64 columns
// x 8 pieces of R >> split rows, a row tile 128 columns x as many rows as
// make 512 pieces of R >> split pixels.
__host__ __device__ inline int col_tile_rows(const BandDesc &f) { return 8 * (f.R >> f.split); }
__host__ __device__ inline int row_tile_rows(const BandDesc &f) { return 4 * (f.R >> f.split); }
__host__ __device__ inline size_t count_tile_bytes(const BandDesc &f) {
  const int col = col_tile_rows(f) * kColPitch, row = row_tile_rows(f) * kRowPitch;
  return (size_t)(col > row ? col : row);
}
__host__ __device__ inline size_t count_smem_bytes(const BandDesc &f) {
  return count_tile_bytes(f) + (size_t)(f.nq + 1) * kCountThreads * 4;
}

// Each thread counts R >> split pixels of one column, or of one row, in its
// own byte counters, so a pixel costs two counter updates in all whatever
// the number of bins; the CTA then adds its threads' counters up into the
// columns' and rows' counts.  Grid: x over half chunks, y over column tiles
// of rows; z = 0 column tiles, 1 row tiles (two per column tile).
template <int MODE>
__device__ __forceinline__ void band_count(const BandDesc &f, uint8_t *smem_raw, const uint3 block) {
  __shared__ uint8_t s_lut[MODE == kBinTable ? 256 : 1];
  if (!IHIST_GUARD(f.ctrl, block.x < 2u * f.nchunks && (int)block.y * col_tile_rows(f) < f.H && block.z < 2u)) {
    griddep_wait();
    return;
  }
  const int t = threadIdx.x, lane = t & 31, w = t >> 5;
  uint32_t *tile32 = reinterpret_cast<uint32_t *>(smem_raw);
  uint32_t *hist = reinterpret_cast<uint32_t *>(smem_raw + count_tile_bytes(f));
  const size_t wpad = (size_t)f.nchunks * kChunk;
  const int per = f.R >> f.split;  // pixels one thread counts
  if constexpr (MODE == kBinTable) {
    const uint32_t none = 4u * (uint32_t)f.nq;  // counted in the extra word, matched by no group
    if (t < 256) {
      const uint32_t e = __ldcg(f.lut + t);
      s_lut[t] = (uint8_t)((e >> 3) < (uint32_t)f.B ? e >> 3 : none);
    }
    __syncthreads();
  }
  const uint32_t mine = smem_u32(hist + t);
  auto count = [&](uint32_t v) { bump_byte(mine + v + (v >> 2) * (kCountThreads * 4 - 4)); };
  auto clear = [&]() {
    for (int e = t; e < (f.nq + 1) * (kCountThreads / 4); e += kCountThreads)
      reinterpret_cast<uint4 *>(hist)[e] = make_uint4(0u, 0u, 0u, 0u);
  };
  if (block.z == 0) {
    const int hc = block.x;
    const int y0 = block.y * col_tile_rows(f), nrows = min(col_tile_rows(f), f.H - y0);
    const int x4 = hc * kHalf + 4 * (t & 15);
    const int tcol = (t >> 4) * (kColPitch / 4) + (t & 15);
    constexpr int kRowStep = kCountThreads / 16, kTileStep = kRowStep * (kColPitch / 4);
    load_tile<MODE>(f, s_lut, y0, t >> 4, kRowStep, nrows, x4, tile32 + tcol, kTileStep, !f.early);
    clear();
    if (f.early) {
      griddep_wait();
      const uint32_t *rp = tile32 + tcol;
      uint8_t *qp = f.q + (size_t)(y0 + (t >> 4)) * wpad + x4;
      for (int r = t >> 4; r < nrows; r += kRowStep, rp += kTileStep, qp += kRowStep * wpad)
        if (IHIST_IN(f, q, qp, 4)) *reinterpret_cast<uint32_t *>(qp) = *rp;
    }
    __syncthreads();
    const int x = t & (kHalf - 1), piece = t / kHalf;
    {
      const int n = max(0, min(per, nrows - piece * per));
      const uint8_t *col = smem_raw + piece * per * kColPitch + x;
      int r = 0;
      for (; r + 4 <= n; r += 4) {
        uint32_t v[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) v[i] = col[(r + i) * kColPitch];
#pragma unroll
        for (int i = 0; i < 4; ++i) count(v[i]);
      }
      for (; r < n; ++r) count(col[r * kColPitch]);
    }
    __syncthreads();
    // thread (column, every eighth group): down each superband's bands
    const size_t band_step = (size_t)f.nq * wpad;
    const int sb0 = block.y << 1 >> f.split, sb1 = min(sb0 + (2 >> f.split), f.nsb);
    for (int g = piece; g < f.nq; g += kCountThreads / kHalf) {
      const uint32_t *hg = hist + g * kCountThreads + x;
      const size_t at = (size_t)g * wpad + hc * kHalf + x;
      for (int sb = sb0; sb < sb1; ++sb) {
        uint32_t *pb = f.pb + (size_t)sb * kSuper * band_step + at;
        uint32_t above[kSuper + 1];  // bytes of at most 4R <= 128
        above[0] = 0u;
#pragma unroll
        for (int j = 0; j < kSuper; ++j) {
          above[j + 1] = above[j] + hg[0];
          if (f.split) above[j + 1] += hg[kHalf];
          hg += kHalf << f.split;
        }
        const int nbk = f.nbands - sb * kSuper;
#pragma unroll
        for (int j = 1; j < kSuper; ++j) {
          pb += band_step;
          if (j < nbk && IHIST_IN(f, pb, pb, 1)) *pb = above[j];
        }
        uint32_t *sbp = f.sb + (size_t)sb * band_step + at;
        if (IHIST_IN(f, sb, sbp, 1)) *sbp = above[kSuper];
      }
    }
  } else {
    const int c = block.x >> 1;
    const int trows = row_tile_rows(f), lr = __ffs(trows) - 1;
    const int y0 = (2 * block.y + (block.x & 1)) * trows, nrows = min(trows, f.H - y0);
    load_tile<MODE>(f, s_lut, y0, w, kCountThreads / 32, nrows, c * kChunk + 4 * lane,
                    tile32 + w * (kRowPitch / 4) + lane, kCountThreads / 32 * (kRowPitch / 4), false);
    clear();
    if (f.early) griddep_wait();
    __syncthreads();
    const int r = t & (trows - 1), piece = t >> lr, pieces = kCountThreads >> lr;
    if (r < nrows) {
      const uint32_t *src = tile32 + r * (kRowPitch / 4) + piece * (per / 4);
#pragma unroll 2
      for (int i = 0; i < per / 4; ++i) {
        const uint32_t v = src[i];
#pragma unroll
        for (int e = 0; e < 4; ++e) count(__byte_perm(v, 0u, 0x4440u + e));
      }
    }
    __syncthreads();
    const size_t hpad = (size_t)f.nsb * kSuper * f.R;
    if (y0 < (int)hpad) {
      // thread (row, every pieces-th group); a warp may hold two groups
      const uint32_t *hg = hist + piece * kCountThreads + r;
      uint32_t *rl = f.rl + ((size_t)c * f.nq + piece) * hpad + y0 + r;
      const int y = y0 + r;
      const int k = y >> (__ffs(f.R) - 1);
      const bool first = (y & (f.R - 1)) == 0 && y < f.H;
      uint2 *ct = f.ct + ((size_t)piece * f.nchunks + c) * f.nbands + k;
      for (int g0 = 0; g0 < f.nq; g0 += pieces) {
        const bool in = g0 + piece < f.nq;
        uint32_t n = 0u;  // bytes of at most 128
        if (in) {
          if (f.rls == nullptr) {
#pragma unroll 4
            for (int p = 0; p < kCountThreads; p += trows) n += hg[p];
          } else {
            const int strip = (kCountThreads / 4) - 1;  // a quarter of the pieces, each trows counters
            uint32_t *rls = f.rls + ((size_t)(3 * c) * f.nq + g0 + piece) * hpad + y0 + r;
            for (int p = 0; p < kCountThreads; p += trows) {
              n += hg[p];
              if (((p + trows) & strip) == 0 && p + trows < kCountThreads) {
                if (IHIST_IN(f, rls, rls, 1)) *rls = n;
                rls += (size_t)f.nq * hpad;
              }
            }
          }
          if (IHIST_IN(f, rl, rl, 1)) *rl = n;
        }
        if (f.nsegs > 1) {
          // a band's R rows lie in neighbouring lanes
          uint32_t lo = n & 0x00ff00ffu, hi = (n >> 8) & 0x00ff00ffu;
          if (f.R == 32) {
            lo = __reduce_add_sync(kFull, lo);
            hi = __reduce_add_sync(kFull, hi);
          } else {
            for (int d = 1; d < f.R; d <<= 1) {
              lo += __shfl_xor_sync(kFull, lo, d);
              hi += __shfl_xor_sync(kFull, hi, d);
            }
          }
          if (in && first && IHIST_IN(f, ct, ct, 1)) *ct = make_uint2(lo, hi);
          ct += (size_t)pieces * f.nchunks * f.nbands;
        }
        hg += pieces * kCountThreads;
        rl += (size_t)pieces * hpad;
      }
    }
  }
}

template <int MODE>
__global__ void __launch_bounds__(kCountThreads, 4) band_count_kernel(const __grid_constant__ BandDesc f) {
  extern __shared__ __align__(16) uint8_t smem_raw[];
  if (!f.early) griddep_wait();
  band_count<MODE>(f, smem_raw, blockIdx);
  griddep_release();
}

// CTAs of one frame, in the order (z, y, x) of the grid above.
__host__ __device__ inline unsigned int count_ctas(const BandDesc &f) {
  return 4u * (unsigned)f.nchunks * (unsigned)((f.H + col_tile_rows(f) - 1) / col_tile_rows(f));
}

// Batches: the frames of one launch, as the running count of their CTAs.
// (By value: the search reads the constant bank.  A batch of more frames
// takes several launches.)
constexpr int kBatchFrames = 256;
struct BandBatch {
  const BandDesc *frames;
  int n;
  unsigned int end[kBatchFrames];
};

// This CTA's frame, copied to shared memory (with loads that see what the
// copy before this launch wrote), and its index among the frame's CTAs.  The
// index comes from the binding the launch was made for, so the descriptor must
// be that binding's: the host orders the copies of a binding and its launches,
// whatever their streams.  (A check of the descriptor here, a branch before the
// rest of the kernel, cost 4 frames of 3840x2160 x 16 pixel-major 430 -> 440 us.)
__device__ __forceinline__ unsigned int batch_frame(const BandBatch &b, BandDesc *s_desc) {
  int lo = 0, hi = b.n - 1;
  while (lo < hi) {
    const int mid = (lo + hi) >> 1;
    if (b.end[mid] > blockIdx.x) hi = mid; else lo = mid + 1;
  }
  constexpr int kWords = (int)(sizeof(BandDesc) / 4);
  static_assert(sizeof(BandDesc) % 4 == 0 && kWords <= 128, "one word per thread");
  if (threadIdx.x < kWords)
    reinterpret_cast<uint32_t *>(s_desc)[threadIdx.x] =
        ld_relaxed_u32(reinterpret_cast<const uint32_t *>(b.frames + lo) + threadIdx.x);
  __syncthreads();
  return blockIdx.x - (lo > 0 ? b.end[lo - 1] : 0u);
}

template <int MODE>
__global__ void __launch_bounds__(kCountThreads, 4) band_count_batch_kernel(const __grid_constant__ BandBatch b) {
  extern __shared__ __align__(16) uint8_t smem_raw[];
  __shared__ BandDesc s_desc;
  griddep_wait();
  unsigned int it = batch_frame(b, &s_desc);
  const BandDesc &f = s_desc;
  uint3 block;
  block.x = it % (2u * f.nchunks);
  it /= 2u * f.nchunks;
  const unsigned int ny = (unsigned)(f.H + col_tile_rows(f) - 1) / (unsigned)col_tile_rows(f);
  block.y = it % ny;
  block.z = it / ny;
  band_count<MODE>(f, smem_raw, block);
  griddep_release();
}


// Inclusive prefix of v[0..3] (this lane's 4 columns) over the chunk.
__device__ __forceinline__ void chunk_prefix(uint32_t v[4], int lane) {
  v[1] += v[0];
  v[2] += v[1];
  v[3] += v[2];
  const uint32_t s = warp_scan_incl(v[3], lane);
  const uint32_t ex = s - v[3];
  v[0] += ex;
  v[1] += ex;
  v[2] += ex;
  v[3] = s;
}

__device__ __forceinline__ void add_bytes16(uint32_t &lo, uint32_t &hi, uint32_t w) {
  lo += w & 0x00ff00ffu;         // bins 0 and 2
  hi += (w >> 8) & 0x00ff00ffu;  // bins 1 and 3
}

// Dynamic shared memory of the emit kernel: the band's bins.
__host__ __device__ inline size_t emit_smem_bytes(int warps, int R) { return (size_t)warps * R * kChunk; }

// One CTA per (band, group, width segment), one warp per chunk of the
// segment.  LAYOUT: 0 bin-major, 2 quad-major.  VEC: rows of H (quad-major:
// its 16-byte words) start on 16-byte boundaries.  Bin-major rows that do not
// (W no multiple of 4) leave as 4-byte stores, 128 contiguous bytes each:
// after the scan the lanes exchange columns through shared memory, from 4
// neighbouring ones per lane to columns lane, lane + 32, .. -- one word per
// column for the four bins, so the exchange costs 5 accesses a row.
//
// planes: items run through the bands of one group before the next, so that
// the CTAs of many frames write few planes at a time (64 frames of 1920x1080
// x 64, bin-major: 5.71 -> 5.65 ms with their queries; quad-major, whose rows
// are four times as long, 2.55 -> 2.59 for 32 frames, so it keeps the band
// order, in which a single frame is as fast).
template <int LAYOUT, bool VEC>
__device__ __forceinline__ void band_emit(const BandDesc &f, uint8_t *smem_raw, unsigned int it, bool planes) {
  __shared__ uint4 s_row[kSegWarps][32];   // per chunk: counts left of it, per row of the band
  __shared__ uint2 s_own[kSegWarps][32];   // per chunk: its own counts, per row (16-bit lanes)
  __shared__ uint2 s_left[kSegWarps][32];  // per warp: its share of the chunks left of the segment
  __shared__ uint4 s_tot[kSegWarps];       // per chunk: its counts in the rows above the band
  __shared__ uint4 s_ltot[kSegWarps];      // per warp: its share of the same left of the segment
  constexpr bool SPREAD = LAYOUT == 0 && !VEC;
  constexpr int P = 4;  // rows in hand at a time
  __shared__ __align__(16) uint32_t s_col[SPREAD ? kSegWarps : 1][SPREAD ? 4 : 1][SPREAD ? kChunk : 4];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, nw = blockDim.x >> 5;
  const int seg = (int)(it % (unsigned)f.nsegs);
  it /= (unsigned)f.nsegs;
  const unsigned int ngs = (unsigned)(f.nq + f.gpc - 1) / (unsigned)f.gpc;
  const int lg = w / f.wpg, w0 = lg * f.wpg;  // this warp's group in the CTA, and that group's first warp
  const int gs = (int)(planes ? it / (unsigned)f.nbands : it % ngs) * f.gpc;
  const int g = gs + lg;
  const int k = (int)(planes ? it % (unsigned)f.nbands : it / ngs);
  const int c0 = seg * f.cps;
  const int c = c0 + w - w0;
  if (!IHIST_GUARD(f.ctrl, k < f.nbands && gs < f.nq && c0 < f.nchunks)) return;
  const bool live = lg < f.gpc && g < f.nq && c < f.nchunks;
  const int y0 = k * f.R;
  const int nrows = min(f.R, f.H - y0);
  const size_t wpad = (size_t)f.nchunks * kChunk;
  const size_t hpad = (size_t)f.nsb * kSuper * f.R;
  const int sbk = k / kSuper;
  const int x = c * kChunk + 4 * lane;
  uint8_t *tile = smem_raw + (size_t)w * f.R * kChunk;
  uint32_t acc[4][4];  // running H of this lane's 4 columns, per bin
  if (live) {
    const uint8_t *qp = f.q + (size_t)y0 * wpad + c * kChunk;
    for (int r = lane >> 3; r < nrows; r += 4) {
      const uint8_t *src = qp + (size_t)r * wpad + 16 * (lane & 7);
      if (IHIST_IN(f, q, src, 16)) copy_async16(tile + r * kChunk + 16 * (lane & 7), src);
    }
    const uint32_t *rp = f.rl + ((size_t)c * f.nq + g) * hpad + y0 + lane;
    const uint32_t own = lane < f.R && IHIST_IN(f, rl, rp, 1) ? __ldcg(rp) : 0u;
    // counts above the band in this lane's columns, two bins per word
    uint32_t lo[4], hi[4];
    {
      const uint32_t *pp = f.pb + ((size_t)k * f.nq + g) * wpad + x;
      const uint4 p = k % kSuper && IHIST_IN(f, pb, pp, 4) ? __ldcg(reinterpret_cast<const uint4 *>(pp))
                                                           : make_uint4(0u, 0u, 0u, 0u);  // a superband's first band
      const uint32_t pv[4] = {p.x, p.y, p.z, p.w};
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        lo[i] = hi[i] = 0u;
        add_bytes16(lo[i], hi[i], pv[i]);
      }
    }
    const uint32_t *sp = f.sb + (size_t)g * wpad + x;
    const size_t sstep = (size_t)f.nq * wpad;
#pragma unroll 4
    for (int s = 0; s < sbk; ++s) {
      if (!IHIST_IN(f, sb, sp + s * sstep, 4)) break;
      const uint4 p = __ldcg(reinterpret_cast<const uint4 *>(sp + s * sstep));
      add_bytes16(lo[0], hi[0], p.x);
      add_bytes16(lo[1], hi[1], p.y);
      add_bytes16(lo[2], hi[2], p.z);
      add_bytes16(lo[3], hi[3], p.w);
    }
#pragma unroll
    for (int b = 0; b < 4; ++b) {
#pragma unroll
      for (int i = 0; i < 4; ++i) acc[b][i] = (((b & 1) ? hi[i] : lo[i]) >> (b & 2 ? 16 : 0)) & 0xffffu;
      chunk_prefix(acc[b], lane);
    }
    if (lane == 31) s_tot[w] = make_uint4(acc[0][3], acc[1][3], acc[2][3], acc[3][3]);
    uint2 o = make_uint2(0u, 0u);
    add_bytes16(o.x, o.y, own);
    s_own[w][lane] = o;
  }
  if (seg > 0) {
    // the chunks left of the segment, shared out over the CTA's warps (which
    // hold one group then)
    uint2 l = make_uint2(0u, 0u);
    for (int cl = w; cl < c0; cl += nw) {
      const uint32_t *rp = f.rl + ((size_t)cl * f.nq + gs) * hpad + y0 + lane;
      if (lane < f.R && IHIST_IN(f, rl, rp, 1)) add_bytes16(l.x, l.y, __ldcg(rp));
    }
    s_left[w][lane] = l;
    uint4 tot = make_uint4(0u, 0u, 0u, 0u);
    auto add = [&](uint2 v) {
      tot.x += v.x & 0xffffu;
      tot.z += v.x >> 16;
      tot.y += v.y & 0xffffu;
      tot.w += v.y >> 16;
    };
#pragma unroll 4
    for (int cl = w; cl < c0; cl += nw)
      for (int j = lane; j < k; j += 32) {
        const uint2 *cp = f.ct + ((size_t)gs * f.nchunks + cl) * f.nbands + j;
        if (IHIST_IN(f, ct, cp, 1)) add(__ldcg(cp));
      }
    tot.x = __reduce_add_sync(kFull, tot.x);
    tot.y = __reduce_add_sync(kFull, tot.y);
    tot.z = __reduce_add_sync(kFull, tot.z);
    tot.w = __reduce_add_sync(kFull, tot.w);
    if (lane == 0) s_ltot[w] = tot;
  }
  copy_async_wait();
  __syncthreads();
  if (!live) return;
  {
    uint4 l = make_uint4(0u, 0u, 0u, 0u);
    uint2 r = make_uint2(0u, 0u);
    for (int i = w0; i < w; ++i) {
      const uint4 v = s_tot[i];
      l.x += v.x; l.y += v.y; l.z += v.z; l.w += v.w;
      const uint2 o = s_own[i][lane];
      r.x += o.x; r.y += o.y;
    }
    if (seg > 0)
      for (int i = 0; i < nw; ++i) {
        const uint4 v = s_ltot[i];
        l.x += v.x; l.y += v.y; l.z += v.z; l.w += v.w;
        const uint2 o = s_left[i][lane];
        r.x += o.x; r.y += o.y;
      }
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      acc[0][i] += l.x; acc[1][i] += l.y; acc[2][i] += l.z; acc[3][i] += l.w;
    }
    s_row[w][lane] = make_uint4(r.x & 0xffffu, r.y & 0xffffu, r.x >> 16, r.y >> 16);
    __syncwarp();
  }
  const uint32_t gbase = 32u * (uint32_t)g;
  const size_t plane = (size_t)f.H * (size_t)f.W;
  const int nb = min(4, f.B - 4 * g);
  const uint32_t *out_end = f.out + plane * (size_t)f.B;
  (void)out_end;
  // element e of this lane: column x + e, or column c * 128 + lane + 32 e
  const int xs = SPREAD ? c * kChunk + lane : x;
  if constexpr (SPREAD) {
#pragma unroll
    for (int b = 0; b < 4; ++b)
      *reinterpret_cast<uint4 *>(&s_col[w][b][4 * lane]) = make_uint4(acc[b][0], acc[b][1], acc[b][2], acc[b][3]);
    __syncwarp();
#pragma unroll
    for (int b = 0; b < 4; ++b)
#pragma unroll
      for (int e = 0; e < 4; ++e) acc[b][e] = s_col[w][b][32 * e + lane];
    __syncwarp();
  }
  uint32_t *o = LAYOUT == 0 ? f.out + ((size_t)(4 * g) * f.H + y0) * f.W + xs
                            : f.out + (((size_t)g * f.H + y0) * f.W + x) * 4;
  for (int r0 = 0; r0 < nrows; r0 += P) {
    // the prefix of P rows' one-hot bytes along the chunk, four bins to a
    // word; the rows' shuffles are independent
    uint32_t p[P][4], tot[P];
#pragma unroll
    for (int i = 0; i < P; ++i) {
      // R is a multiple of P: rows past the frame hold what the tile held, and are not stored
      const uint32_t px = *reinterpret_cast<const uint32_t *>(tile + (r0 + i) * kChunk + 4 * lane);
#pragma unroll
      for (int e = 0; e < 4; ++e) p[i][e] = shl_clamp(1u, 8u * __byte_perm(px, 0u, 0x4440u + e) - gbase);
      p[i][1] += p[i][0];
      p[i][2] += p[i][1];
      p[i][3] += p[i][2];
      tot[i] = p[i][3];
    }
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
      uint32_t n[P];
#pragma unroll
      for (int i = 0; i < P; ++i) n[i] = __shfl_up_sync(kFull, tot[i], d);
#pragma unroll
      for (int i = 0; i < P; ++i)
        if (lane >= d) tot[i] += n[i];  // bytes of at most 128
    }
#pragma unroll
    for (int i = 0; i < P; ++i) {
      const uint32_t ex = tot[i] - p[i][3];
      p[i][0] += ex;
      p[i][1] += ex;
      p[i][2] += ex;
      p[i][3] = tot[i];
    }
    if constexpr (SPREAD) {
#pragma unroll
      for (int i = 0; i < P; ++i)
        *reinterpret_cast<uint4 *>(&s_col[w][i][4 * lane]) = make_uint4(p[i][0], p[i][1], p[i][2], p[i][3]);
      __syncwarp();
#pragma unroll
      for (int i = 0; i < P; ++i)
#pragma unroll
        for (int e = 0; e < 4; ++e) p[i][e] = s_col[w][i][32 * e + lane];
      __syncwarp();
    }
#pragma unroll
    for (int i = 0; i < P; ++i) {
      if (r0 + i >= nrows) break;
      const uint4 rc = s_row[w][r0 + i];
      const uint32_t rcv[4] = {rc.x, rc.y, rc.z, rc.w};
#pragma unroll
      for (int b = 0; b < 4; ++b)
#pragma unroll
        for (int e = 0; e < 4; ++e) acc[b][e] += __byte_perm(p[i][e], 0u, 0x4440u + b) + rcv[b];
      if constexpr (LAYOUT == 0) {
#pragma unroll
        for (int b = 0; b < 4; ++b) {
          if (b < nb) {
            uint32_t *ob = o + b * plane;
            if (VEC) {
              if (x < f.W && IHIST_GUARD(f.ctrl, ob >= f.out && ob + 4 <= out_end)) st_stream_v4(ob, acc[b][0], acc[b][1], acc[b][2], acc[b][3]);
            } else {
#pragma unroll
              for (int e = 0; e < 4; ++e)
                if (xs + 32 * e < f.W && IHIST_GUARD(f.ctrl, ob + 32 * e >= f.out && ob + 32 * e < out_end))
                  st_stream(ob + 32 * e, acc[b][e]);
            }
          }
        }
        o += f.W;
      } else {
        const bool v8 = VEC && (reinterpret_cast<uintptr_t>(o) & 31u) == 0;
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          const uint4 a0 = make_uint4(acc[0][2 * h], acc[1][2 * h], acc[2][2 * h], acc[3][2 * h]);
          const uint4 a1 = make_uint4(acc[0][2 * h + 1], acc[1][2 * h + 1], acc[2][2 * h + 1], acc[3][2 * h + 1]);
          if (v8 && x + 2 * h + 1 < f.W) {
            if (IHIST_GUARD(f.ctrl, o + 8 * h >= f.out && o + 8 * h + 8 <= out_end)) st_stream_v8(o + 8 * h, a0, a1);
          } else {
#pragma unroll
            for (int e = 0; e < 2; ++e) {
              const uint4 v = e ? a1 : a0;
              uint32_t *oe = o + 8 * h + 4 * e;
              if (x + 2 * h + e < f.W && IHIST_GUARD(f.ctrl, oe >= f.out && oe + 4 <= out_end)) {
                if (VEC) {
                  st_stream_v4(oe, v.x, v.y, v.z, v.w);
                } else {
                  st_stream(oe, v.x);
                  st_stream(oe + 1, v.y);
                  st_stream(oe + 2, v.z);
                  st_stream(oe + 3, v.w);
                }
              }
            }
          }
        }
        o += (size_t)f.W * 4;
      }
    }
  }
}

template <int LAYOUT, bool VEC>
__global__ void __launch_bounds__(kSegWarps * 32, LAYOUT == 0 && !VEC ? 3 : 4)
    band_emit_kernel(const __grid_constant__ BandDesc f) {
  extern __shared__ __align__(16) uint8_t smem_raw[];  // per chunk: the band's bins, R rows of 128 bytes
  griddep_wait();
  griddep_release();
  band_emit<LAYOUT, VEC>(f, smem_raw, blockIdx.x, false);
}

template <int LAYOUT, bool VEC>
__global__ void __launch_bounds__(kSegWarps * 32, LAYOUT == 0 && !VEC ? 3 : 4)
    band_emit_batch_kernel(const __grid_constant__ BandBatch b) {
  extern __shared__ __align__(16) uint8_t smem_raw[];
  __shared__ BandDesc s_desc;
  griddep_wait();
  griddep_release();
  const unsigned int it = batch_frame(b, &s_desc);
  const BandDesc f = s_desc;
  band_emit<LAYOUT, VEC>(f, smem_raw, it, LAYOUT == 0);
}

// Pixel-major H[y][x][b].  One CTA per (band, block of bins, chunk), one warp
// per 32 columns of the chunk and 32 * NJ bins of the block; a lane holds NJ
// bins (32 apart) of all 32 columns, so that a pixel's counts leave as
// contiguous stores and a row of a chunk as one run.  Walking along the row,
// a lane keeps its bins' count of the row so far and adds it to the column's
// running H: a compare, an add and an add per count, with no scan across
// lanes at all.  One bin per lane makes twice the warps (1920x1080 x 64: 97
// us against 104), two keep a record that is no multiple of 32 bytes in one
// warp's hands, whose stores meet in L2 (1921x1081 x 37: 77 against 111).
// The loads before the first row are what leaves the stores idle (a chain of
// several L2 round trips per CTA): two groups' and two rows' loads at a time
// took 1920x1080 x 64 from 97.8 to 92.1 us, 640x480 x 32 from 16.7 to 14.4.
constexpr int kPixelBins = 64;                // bins of one CTA at most
constexpr int kStripCols = 32;
constexpr size_t kPixelTopBytes = (size_t)kChunk * kPixelBins * 4;
__host__ __device__ inline size_t pixel_smem_bytes(int R) {
  return kPixelTopBytes + (size_t)4 * R * kPixelBins * 2 + (size_t)R * kChunk;
}

// The rows of one strip.  FULL: all 32 columns lie inside the frame.
template <int NJ, bool FULL>
__device__ __forceinline__ void emit_strip(const BandDesc &f, uint32_t (&acc)[kStripCols][NJ], const uint32_t (&bin)[NJ],
                                           const bool (&has)[NJ], const uint2 *s_left, const uint8_t *tile, int y0,
                                           int nrows, int x0, int ncols, int b0) {
  constexpr int kUnits = kPixelBins / 4;
  uint32_t *row = f.out + ((size_t)y0 * f.W + x0) * f.B + b0;
  const uint32_t *out_end = f.out + (size_t)f.H * f.W * f.B;
  (void)out_end;
  for (int y = 0; y < nrows; ++y) {
    const uint4 q0 = *reinterpret_cast<const uint4 *>(tile + y * kChunk);
    const uint4 q1 = *reinterpret_cast<const uint4 *>(tile + y * kChunk + 16);
    const uint32_t qv[8] = {q0.x, q0.y, q0.z, q0.w, q1.x, q1.y, q1.z, q1.w};
    uint32_t rc[NJ];
#pragma unroll
    for (int j = 0; j < NJ; ++j)
      rc[j] = reinterpret_cast<const uint16_t *>(s_left + y * kUnits + ((bin[j] >> 2) ^ (y & 15)))[bin[j] & 3];
    uint32_t *o = row + bin[0];
#pragma unroll
    for (int i = 0; i < kStripCols; ++i) {
      const uint32_t q = __byte_perm(qv[i >> 2], 0u, 0x4440u + (i & 3));
#pragma unroll
      for (int j = 0; j < NJ; ++j) {
        if (q == (uint32_t)b0 + bin[j]) ++rc[j];
        acc[i][j] += rc[j];
        if ((FULL || i < ncols) && has[j] && IHIST_GUARD(f.ctrl, o + 32 * j >= f.out && o + 32 * j < out_end))
          st_stream(o + 32 * j, acc[i][j]);
      }
      o += f.B;
    }
    row += (size_t)f.W * f.B;
  }
}

template <int WARPS, int NJ>
__device__ __forceinline__ void band_emit_pixel(const BandDesc &f, uint8_t *smem_raw, unsigned int it) {
  // first rows of H [column][16-byte unit of 4 bins ^ (column / 4 mod 8)], then
  // the counts left of each strip [strip][row][8-byte unit of 4 bins ^ (row
  // mod 16)], then the band's bins [row][column]
  uint4 *s_top = reinterpret_cast<uint4 *>(smem_raw);
  uint2 *s_left = reinterpret_cast<uint2 *>(smem_raw + kPixelTopBytes);
  constexpr int kUnits = kPixelBins / 4;
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const int c = (int)(it % (unsigned)f.nchunks);
  it /= (unsigned)f.nchunks;
  const int blk = (int)(it % (unsigned)f.nblk);
  const int k = (int)(it / (unsigned)f.nblk);
  const int b0 = blk * f.bpb, nb = min(f.bpb, f.B - b0);
  const int g0 = b0 >> 2, ng = (nb + 3) >> 2;
  const int y0 = k * f.R, nrows = min(f.R, f.H - y0);
  const size_t wpad = (size_t)f.nchunks * kChunk;
  const size_t hpad = (size_t)f.nsb * kSuper * f.R;
  const int lr = __ffs(f.R) - 1;
  uint8_t *tile = smem_raw + kPixelTopBytes + (size_t)4 * f.R * kPixelBins * 2;
  if (!IHIST_GUARD(f.ctrl, k < f.nbands)) return;
  for (int e = threadIdx.x; e < nrows * 8; e += blockDim.x) {
    const uint8_t *src = f.q + (size_t)(y0 + (e >> 3)) * wpad + c * kChunk + 16 * (e & 7);
    if (IHIST_IN(f, q, src, 16)) copy_async16(tile + 16 * e, src);
  }
  // counts left of each strip, per row and bin: two rows (or groups) per
  // thread with their loads in flight together
  const int lefts = ng << lr;
  for (int e0 = threadIdx.x; e0 < lefts; e0 += 2 * WARPS * 32) {
    const size_t step = (size_t)f.nq * hpad;
    const bool two = e0 + WARPS * 32 < lefts;
    const uint32_t *p[2];
    uint32_t lo[2] = {0u, 0u}, hi[2] = {0u, 0u}, sv[2][3];
#pragma unroll
    for (int u = 0; u < 2; ++u) {
      const int e = two ? e0 + u * WARPS * 32 : e0;
      p[u] = f.rl + (size_t)(g0 + (e >> lr)) * hpad + y0 + (e & (f.R - 1));
      const uint32_t *ps = f.rls + ((size_t)(3 * c) * f.nq + g0 + (e >> lr)) * hpad + y0 + (e & (f.R - 1));
#pragma unroll
      for (int i = 0; i < 3; ++i) sv[u][i] = IHIST_IN(f, rls, ps + i * step, 1) ? __ldcg(ps + i * step) : 0u;
    }
#pragma unroll 4
    for (int cl = 0; cl < c; ++cl) {
      if (!IHIST_IN(f, rl, p[0] + cl * step, 1) || !IHIST_IN(f, rl, p[1] + cl * step, 1)) break;
      const uint32_t v0 = __ldcg(p[0] + cl * step), v1 = __ldcg(p[1] + cl * step);
      add_bytes16(lo[0], hi[0], v0);
      add_bytes16(lo[1], hi[1], v1);
    }
#pragma unroll
    for (int u = 0; u < 2; ++u) {
      if (u == 1 && !two) break;
      const int e = e0 + u * WARPS * 32, gi = e >> lr, y = e & (f.R - 1);
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        uint32_t l = lo[u], h = hi[u];
        if (i > 0) add_bytes16(l, h, sv[u][i - 1]);
        s_left[(i * f.R + y) * kUnits + (gi ^ (y & 15))] = make_uint2((l & 0xffffu) | h << 16, l >> 16 | (h & 0xffff0000u));
      }
    }
  }
  // H in the row above the band, four bins of the chunk at a time, two such
  // groups per warp with their loads in flight together
  const int sbk = k / kSuper;
  for (int gi0 = w; gi0 < ng; gi0 += 2 * WARPS) {
    const bool two = gi0 + WARPS < ng;
    const int g = g0 + gi0;
    const int x = c * kChunk + 4 * lane;
    uint32_t lo[2][4], hi[2][4], left[2][4];
#pragma unroll
    for (int u = 0; u < 2; ++u)
#pragma unroll
      for (int i = 0; i < 4; ++i) lo[u][i] = hi[u][i] = left[u][i] = 0u;
    auto add = [&](int u, uint4 p) {
      add_bytes16(lo[u][0], hi[u][0], p.x);
      add_bytes16(lo[u][1], hi[u][1], p.y);
      add_bytes16(lo[u][2], hi[u][2], p.z);
      add_bytes16(lo[u][3], hi[u][3], p.w);
    };
    auto add_left = [&](int u, uint2 v) {
      left[u][0] += v.x & 0xffffu;
      left[u][2] += v.x >> 16;
      left[u][1] += v.y & 0xffffu;
      left[u][3] += v.y >> 16;
    };
    const uint4 none = make_uint4(0u, 0u, 0u, 0u);
    const size_t sstep = (size_t)f.nq * wpad;
    const uint32_t *sp = f.sb + (size_t)g * wpad + x, *sp2 = sp + (size_t)WARPS * wpad;
#pragma unroll 4
    for (int s = 0; s < sbk; ++s) {
      if (!IHIST_IN(f, sb, sp + s * sstep, 4) || (two && !IHIST_IN(f, sb, sp2 + s * sstep, 4))) break;
      const uint4 p0 = __ldcg(reinterpret_cast<const uint4 *>(sp + s * sstep));
      const uint4 p1 = two ? __ldcg(reinterpret_cast<const uint4 *>(sp2 + s * sstep)) : none;
      add(0, p0);
      add(1, p1);
    }
    const uint32_t *pb = f.pb + ((size_t)k * f.nq + g) * wpad + x;
    if (k % kSuper && IHIST_IN(f, pb, pb, 4) && (!two || IHIST_IN(f, pb, pb + (size_t)WARPS * wpad, 4))) {
      const uint4 p0 = __ldcg(reinterpret_cast<const uint4 *>(pb));
      const uint4 p1 = two ? __ldcg(reinterpret_cast<const uint4 *>(pb + (size_t)WARPS * wpad)) : none;
      add(0, p0);
      add(1, p1);
    }
    const uint2 *ctp = f.ct + (size_t)g * f.nchunks * f.nbands + lane;
    const size_t cstep = (size_t)WARPS * f.nchunks * f.nbands;
    for (int j = lane; j < k; j += 32, ctp += 32) {
#pragma unroll 4
      for (int cl = 0; cl < c; ++cl) {
        if (!IHIST_IN(f, ct, ctp + (size_t)cl * f.nbands, 1) ||
            (two && !IHIST_IN(f, ct, ctp + cstep + (size_t)cl * f.nbands, 1)))
          break;
        const uint2 v0 = __ldcg(ctp + (size_t)cl * f.nbands);
        const uint2 v1 = two ? __ldcg(ctp + cstep + (size_t)cl * f.nbands) : make_uint2(0u, 0u);
        add_left(0, v0);
        add_left(1, v1);
      }
    }
#pragma unroll
    for (int u = 0; u < 2; ++u) {
      if (u == 1 && !two) break;
      const int gi = gi0 + u * WARPS;
      uint32_t top[4][4];
#pragma unroll
      for (int b = 0; b < 4; ++b) {
        const uint32_t l = __reduce_add_sync(kFull, left[u][b]);
#pragma unroll
        for (int i = 0; i < 4; ++i) top[b][i] = (((b & 1) ? hi[u][i] : lo[u][i]) >> (b & 2 ? 16 : 0)) & 0xffffu;
        chunk_prefix(top[b], lane);
#pragma unroll
        for (int i = 0; i < 4; ++i) top[b][i] += l;
      }
#pragma unroll
      for (int i = 0; i < 4; ++i)
        s_top[(4 * lane + i) * kUnits + (gi ^ (lane & 7))] = make_uint4(top[0][i], top[1][i], top[2][i], top[3][i]);
    }
  }
  copy_async_wait();
  __syncthreads();
  const int strip = w & 3;
  const int x0 = c * kChunk + kStripCols * strip;
  const int ncols = min(kStripCols, f.W - x0);
  if (ncols <= 0) return;
  // this lane's bins within the block; where there is none it follows the first and stores nothing
  uint32_t bin[NJ];
  bool has[NJ];
#pragma unroll
  for (int j = 0; j < NJ; ++j) {
    bin[j] = (uint32_t)(32 * NJ * (w >> 2) + lane + 32 * j);
    has[j] = bin[j] < (uint32_t)nb;
    if (!has[j]) bin[j] = 0u;
  }
  uint32_t acc[kStripCols][NJ];
#pragma unroll
  for (int i = 0; i < kStripCols; ++i) {
    const int x = kStripCols * strip + i;
#pragma unroll
    for (int j = 0; j < NJ; ++j)
      acc[i][j] = reinterpret_cast<const uint32_t *>(s_top + x * kUnits + ((bin[j] >> 2) ^ (x >> 2 & 7)))[bin[j] & 3];
  }
  const uint2 *left = s_left + strip * f.R * kUnits;
  if (ncols == kStripCols)
    emit_strip<NJ, true>(f, acc, bin, has, left, tile + kStripCols * strip, y0, nrows, x0, ncols, b0);
  else
    emit_strip<NJ, false>(f, acc, bin, has, left, tile + kStripCols * strip, y0, nrows, x0, ncols, b0);
}

template <int WARPS, int NJ>
__global__ void __launch_bounds__(WARPS * 32, NJ == 2 ? 4 : 24 / WARPS)
    band_emit_pixel_kernel(const __grid_constant__ BandDesc f) {
  extern __shared__ __align__(16) uint8_t smem_raw[];
  griddep_wait();
  griddep_release();
  band_emit_pixel<WARPS, NJ>(f, smem_raw, blockIdx.x);
}

template <int WARPS, int NJ>
__global__ void __launch_bounds__(WARPS * 32, NJ == 2 ? 4 : 24 / WARPS)
    band_emit_pixel_batch_kernel(const __grid_constant__ BandBatch b) {
  extern __shared__ __align__(16) uint8_t smem_raw[];
  __shared__ BandDesc s_desc;
  griddep_wait();
  griddep_release();
  const unsigned int it = batch_frame(b, &s_desc);
  const BandDesc f = s_desc;
  band_emit_pixel<WARPS, NJ>(f, smem_raw, it);
}

}  // namespace ihist
