// ihist_bands.cu -- host side of the two-launch path (ihist_bands.cuh):
// which frames take it, its workspace and its launches.
#include <algorithm>
#include <cstring>

#include "ihist_bands.cuh"
#include "ihist_bands_host.h"

namespace ihist {
namespace host {

namespace {

using CountFn = void (*)(const BandDesc);
using EmitFn = void (*)(const BandDesc);

CountFn count_fn(int mode) {
  return mode == kBinJoint ? band_count_kernel<kBinJoint>
         : mode == kBinTable ? band_count_kernel<kBinTable>
                             : band_count_kernel<kBinUniform>;
}

// vec: the kernel's VEC, or for pixel-major that pixel records are whole
// 32-byte sectors (one bin per lane).
EmitFn emit_fn(const BandDesc &f, int layout, bool vec) {
  if (layout == IHIST_PIXEL_MAJOR)
    return f.bpb <= 32 ? band_emit_pixel_kernel<4, 1> : vec ? band_emit_pixel_kernel<8, 1> : band_emit_pixel_kernel<4, 2>;
  if (layout == IHIST_QUAD_MAJOR) return vec ? band_emit_kernel<2, true> : band_emit_kernel<2, false>;
  return vec ? band_emit_kernel<0, true> : band_emit_kernel<0, false>;
}

}  // namespace

size_t bands_layout(BandDesc *f, char *base) {
  const size_t wpad = (size_t)f->nchunks * kChunk;
  const size_t hpad = (size_t)f->nsb * kSuper * f->R;
  size_t off = 0;
  auto take = [&](size_t bytes) {
    char *p = base ? base + off : nullptr;
    off = align_up(off + bytes, 256);
    return p;
  };
  f->q = reinterpret_cast<uint8_t *>(take((size_t)f->H * wpad));
  f->pb = reinterpret_cast<uint32_t *>(take((size_t)f->nbands * f->nq * wpad * 4));
  f->sb = reinterpret_cast<uint32_t *>(take((size_t)f->nsb * f->nq * wpad * 4));
  f->rl = reinterpret_cast<uint32_t *>(take((size_t)f->nchunks * f->nq * hpad * 4));
  f->rls = reinterpret_cast<uint32_t *>(take(f->nblk ? (size_t)f->nchunks * 3 * f->nq * hpad * 4 : 0));
  if (!f->nblk) f->rls = nullptr;
  f->ct = reinterpret_cast<uint2 *>(take(f->nsegs > 1 ? (size_t)f->nbands * f->nq * f->nchunks * 8 : 0));
  return off;
}

bool bands_shape(int h, int w, int nbins, int layout, int sms, BandDesc *f) {
  const bool pixel = layout == IHIST_PIXEL_MAJOR;
  // Larger frames run the look-back kernel for many waves, where its chain is
  // hidden, and here the counts outgrow L2 (bin-major: 3840x2160 x 64 1.08x
  // faster here, 4096x4096 x 128 and 8192x8192 x 16 0.96x and 0.94x; quad-
  // major 7680x4320 x 32 1.11x, pixel-major 1.82x).  A tall frame's bands add up one word per
  // superband above them (256x16384 x 16 1.07x, 2000x65535 x 16 0.70x).
  const long long pixels = (long long)h * w;
  if (h > 8192 || pixels > (layout == IHIST_BIN_MAJOR ? 12000000ll : 40000000ll)) return false;
  std::memset(f, 0, sizeof(*f));
  f->H = h;
  f->W = w;
  f->B = nbins;
  f->nq = (nbins + 3) / 4;
  f->nchunks = (w + kChunk - 1) / kChunk;
  f->nsegs = pixel ? f->nchunks : (f->nchunks + kSegWarps - 1) / kSegWarps;  // a pixel-major CTA holds one chunk
  f->cps = (f->nchunks + f->nsegs - 1) / f->nsegs;
  // Rows per band: long bands write fewer counts, short ones make more warps
  // (each emits one chunk of one band).  640x480 x 32 at R = 8, 16, 32: 11.6,
  // 11.3, 11.4 us; 320x240 x 16: 5.7, 6.9, 9.2; 1920x1080 x 64 with 1000
  // queries behind it: 106, 95, 103; 3840x2160 x 64: 488, 343, 329.
  if (pixel) {
    f->nblk = (nbins + kPixelBins - 1) / kPixelBins;
    f->bpb = ((nbins + f->nblk - 1) / f->nblk + 3) / 4 * 4;
    f->nblk = (nbins + f->bpb - 1) / f->bpb;
  }
  const long long per_band = (long long)f->nq * f->nchunks;
  auto warps = [&](int R) { return (h + R - 1) / R * per_band; };
  f->R = warps(32) >= 16000 || h > 2048 ? 32 : warps(16) >= 600 ? 16 : 8;
  if (pixel) {
    // by CTAs: 1920x1080 x 64 at R = 32 (510 CTAs) and 16: 97, 100 us; 640x480
    // x 64 at 32, 16 (150 CTAs) and 8: 27.8, 23.9, 25.8; 320x240 x 16 at 16
    // and 8 (90 CTAs): 10.2, 8.6
    auto ctas = [&](int R) { return (long long)((h + R - 1) / R) * f->nblk * f->nchunks; };
    f->R = ctas(32) >= 400 || h > 2048 ? 32 : ctas(16) >= 120 ? 16 : 8;
  }
  // Count threads take R pixels each, or R / 2 where that leaves less than
  // two CTAs per SM (640x480 x 32: 14.9 -> 14.7 us with its queries; above
  // it, 1920x1080 x 64, R pixels: 96.4 -> 95.3).
  const long long row_tiles = (h + col_tile_rows(*f) - 1) / col_tile_rows(*f);
  f->split = 4 * f->nchunks * row_tiles < 2 * sms ? 1 : 0;
  f->nbands = (h + f->R - 1) / f->R;
  f->nsb = (f->nbands + kSuper - 1) / kSuper;
  return (long long)f->nbands * (pixel ? f->nblk : f->nq) * f->nsegs < 0x7fffffffll;
}

int bands_prepare(const BandDesc &f, int mode, int layout, size_t optin) {
  const size_t smem = count_smem_bytes(f);
  cudaFuncAttributes a;
  if (cudaFuncGetAttributes(&a, count_fn(mode)) != cudaSuccess) {
    cudaGetLastError();
    return IHIST_ERR_CUDA;
  }
  if (smem + a.sharedSizeBytes > optin) return IHIST_ERR_UNSUPPORTED;
  // the attribute belongs to the function, so every plan sets the same limit
  if (cudaFuncSetAttribute(count_fn(mode), cudaFuncAttributeMaxDynamicSharedMemorySize,
                           (int)(optin - a.sharedSizeBytes)) != cudaSuccess) {
    cudaGetLastError();
    return IHIST_ERR_CUDA;
  }
  for (int v = 0; v < 2; ++v) {
    const bool pixel = f.nblk > 0;
    if (cudaFuncSetAttribute(emit_fn(f, layout, v != 0),
                             cudaFuncAttributeMaxDynamicSharedMemorySize,
                             (int)(pixel ? pixel_smem_bytes(32) : emit_smem_bytes(kSegWarps, 32))) != cudaSuccess) {
      cudaGetLastError();
      return IHIST_ERR_CUDA;
    }
  }
  return IHIST_OK;
}

int launch_bands(const BandDesc &f, int mode, int layout, void *stream) {
  cudaLaunchConfig_t cfg;
  std::memset(&cfg, 0, sizeof(cfg));
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  cfg.stream = (cudaStream_t)stream;
  cfg.gridDim = dim3(2u * f.nchunks, (unsigned)((f.H + col_tile_rows(f) - 1) / col_tile_rows(f)), 2u);
  cfg.blockDim = dim3(kCountThreads);
  cfg.dynamicSmemBytes = count_smem_bytes(f);
  cudaError_t e = cudaLaunchKernelEx(&cfg, count_fn(mode), f);
  if (e == cudaSuccess) {
    bool vec = ((uintptr_t)f.out & 15u) == 0;
    if (layout == IHIST_PIXEL_MAJOR) {
      vec = f.B % 8 == 0 && ((uintptr_t)f.out & 31u) == 0;
      cfg.gridDim = dim3((unsigned)f.nbands * (unsigned)f.nblk * (unsigned)f.nchunks);
      cfg.blockDim = dim3(f.bpb <= 32 || !vec ? 128 : 256);
      cfg.dynamicSmemBytes = pixel_smem_bytes(f.R);
    } else {
      vec = vec && (layout == IHIST_QUAD_MAJOR || f.W % 4 == 0);
      cfg.gridDim = dim3((unsigned)f.nbands * (unsigned)f.nq * (unsigned)f.nsegs);
      cfg.blockDim = dim3((unsigned)std::min(f.cps, f.nchunks) * 32u);
      cfg.dynamicSmemBytes = emit_smem_bytes(cfg.blockDim.x / 32u, f.R);
    }
    e = cudaLaunchKernelEx(&cfg, emit_fn(f, layout, vec), f);
  }
  if (e != cudaSuccess) {
    cudaGetLastError();
    return IHIST_ERR_CUDA;
  }
  return IHIST_OK;
}

}  // namespace host
}  // namespace ihist
