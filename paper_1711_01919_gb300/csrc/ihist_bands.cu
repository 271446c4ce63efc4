// ihist_bands.cu -- host side of the two-launch path (ihist_bands.cuh):
// which frames take it, its workspace and its launches.
#include <algorithm>
#include <cstring>

#include "ihist_bands.cuh"
#include "ihist_bands_host.h"

namespace ihist {
namespace host {

namespace {

using BandFn = void (*)(const BandDesc);
using BandBatchFn = void (*)(const BandBatch);

BandFn count_fn(int mode) {
  return mode == kBinJoint ? band_count_kernel<kBinJoint>
         : mode == kBinTable ? band_count_kernel<kBinTable>
                             : band_count_kernel<kBinUniform>;
}
BandBatchFn count_batch_fn(int mode) {
  return mode == kBinJoint ? band_count_batch_kernel<kBinJoint>
         : mode == kBinTable ? band_count_batch_kernel<kBinTable>
                             : band_count_batch_kernel<kBinUniform>;
}

BandFn emit_fn(int kind) {
  switch (kind) {
    case 0: return band_emit_kernel<0, true>;
    case 1: return band_emit_kernel<0, false>;
    case 2: return band_emit_kernel<2, true>;
    case 3: return band_emit_kernel<2, false>;
    case 4: return band_emit_pixel_kernel<4, 1>;
    case 5: return band_emit_pixel_kernel<8, 1>;
    default: return band_emit_pixel_kernel<4, 2>;
  }
}
BandBatchFn emit_batch_fn(int kind) {
  switch (kind) {
    case 0: return band_emit_batch_kernel<0, true>;
    case 1: return band_emit_batch_kernel<0, false>;
    case 2: return band_emit_batch_kernel<2, true>;
    case 3: return band_emit_batch_kernel<2, false>;
    case 4: return band_emit_pixel_batch_kernel<4, 1>;
    case 5: return band_emit_pixel_batch_kernel<8, 1>;
    default: return band_emit_pixel_batch_kernel<4, 2>;
  }
}

unsigned int emit_ctas(const BandDesc &f, int kind) {
  return kind >= 4 ? (unsigned)f.nbands * (unsigned)f.nblk * (unsigned)f.nchunks
                   : (unsigned)f.nbands * (unsigned)((f.nq + f.gpc - 1) / f.gpc) * (unsigned)f.nsegs;
}
size_t emit_smem(const BandDesc &f, int kind) {
  return kind >= 4 ? pixel_smem_bytes(f.R) : emit_smem_bytes(f.wpg * f.gpc, f.R);
}

template <typename Arg>
cudaError_t launch(void (*fn)(const Arg), unsigned int x, unsigned int y, unsigned int z, unsigned int threads,
                   size_t smem, const Arg &arg, void *stream) {
  cudaLaunchConfig_t cfg;
  std::memset(&cfg, 0, sizeof(cfg));
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  cfg.stream = (cudaStream_t)stream;
  cfg.gridDim = dim3(x, y, z);
  cfg.blockDim = dim3(threads);
  cfg.dynamicSmemBytes = smem;
  return cudaLaunchKernelEx(&cfg, fn, arg);
}

// Let fn use `smem` bytes of dynamic shared memory.  The attribute belongs to
// the function, so every plan asks for the same amount, the most any frame
// needs.
template <typename Fn>
int allow_smem(Fn fn, size_t smem) {
  if (cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem) == cudaSuccess) return IHIST_OK;
  cudaGetLastError();
  return IHIST_ERR_CUDA;
}

size_t max_count_smem() {
  BandDesc f;
  bands_describe(1, 1, 256, IHIST_BIN_MAJOR, 32, 0, &f);
  return count_smem_bytes(f);  // 150 KB
}
size_t max_emit_smem(int kind) { return kind >= 4 ? pixel_smem_bytes(32) : emit_smem_bytes(kSegWarps, 32); }

}  // namespace

size_t bands_layout(BandDesc *f, char *base, bool any_layout) {
  const bool pixel = f->nblk > 0;
  size_t off = 0;
  auto take = [&](size_t bytes) {
    char *p = base && bytes ? base + off : nullptr;
    off = align_up(off + bytes, 256);
    return p;
  };
  f->q = reinterpret_cast<uint8_t *>(take(q_size(*f)));
  f->pb = reinterpret_cast<uint32_t *>(take(pb_size(*f) * 4));
  f->sb = reinterpret_cast<uint32_t *>(take(sb_size(*f) * 4));
  f->rl = reinterpret_cast<uint32_t *>(take(rl_size(*f) * 4));
  f->ct = reinterpret_cast<uint2 *>(take(f->nsegs > 1 || any_layout ? ct_size(*f) * 8 : 0));
  f->rls = reinterpret_cast<uint32_t *>(take(pixel || any_layout ? rls_size(*f) * 4 : 0));
  if (!pixel) f->rls = nullptr;
  return off;
}

void bands_describe(int h, int w, int nbins, int layout, int R, int split, BandDesc *f) {
  const bool pixel = layout == IHIST_PIXEL_MAJOR;
  std::memset(f, 0, sizeof(*f));
  f->H = h;
  f->W = w;
  f->B = nbins;
  f->qmul = nbins;
  f->nq = (nbins + 3) / 4;
  f->nchunks = (w + kChunk - 1) / kChunk;
  f->nsegs = pixel ? f->nchunks : (f->nchunks + kSegWarps - 1) / kSegWarps;  // a pixel-major CTA holds one chunk
  f->cps = (f->nchunks + f->nsegs - 1) / f->nsegs;
  f->wpg = f->cps;
  f->gpc = 1;
  if (pixel) {
    f->nblk = (nbins + kPixelBins - 1) / kPixelBins;
    f->bpb = ((nbins + f->nblk - 1) / f->nblk + 3) / 4 * 4;
    f->nblk = (nbins + f->bpb - 1) / f->bpb;
  }
  f->R = R;
  f->split = split;
  f->nbands = (h + R - 1) / R;
  f->nsb = (f->nbands + kSuper - 1) / kSuper;
}

bool bands_fit(int h, int w, int layout) {
  // Larger frames run the look-back kernel for many waves, where its chain is
  // hidden, and here the counts outgrow L2 (bin-major: 3840x2160 x 64 1.08x
  // faster here, 4096x4096 x 128 and 8192x8192 x 16 0.96x and 0.94x; quad-
  // major 7680x4320 x 32 1.11x, pixel-major 1.82x).  A tall frame's bands add
  // up one word per superband above them (256x16384 x 16 1.07x, 2000x65535 x
  // 16 0.70x).
  return h <= 8192 && (long long)h * w <= (layout == IHIST_BIN_MAJOR ? 12000000ll : 40000000ll);
}

// Rows per band: long bands write fewer counts, short ones make more warps
// (each emits one chunk of one band).  640x480 x 32 at R = 8, 16, 32: 11.6,
// 11.3, 11.4 us; 320x240 x 16: 5.7, 6.9, 9.2; 1920x1080 x 64 with 1000
// queries behind it: 106, 95, 103; 3840x2160 x 64: 488, 343, 329.  Where pixels
// are many and bins few, there are not that many warps, but the count kernel is
// what takes the time, and it is the faster the more pixels share a thread's
// counters: at R = 16 and 32 12000x1000 x 4 takes 62 and 57 us, 65532x183 x 8
// 121 and 98, 24 frames of 1920x1080 x 1 188 and 137, 64 of 640x480 x 4 98 and
// 85 (below that, the order changes with the last wave: 2400x2000 x 8 44 and 47,
// 16 frames of 640x480 x 12 51 and 59, x 4 28 and 26).
int bands_rows(long long warps32, long long warps16, long long pixels, int h_max) {
  if (warps32 >= 16000 || h_max > 2048 || pixels >= 11000000) return 32;
  return warps16 >= 600 ? 16 : 8;
}

// Frames within those sizes that the look-back kernel still does faster.
static bool look_back_faster(const BandDesc &f, int layout, bool table) {
  const long long px = (long long)f.H * f.W;
  if (layout == IHIST_PIXEL_MAJOR)
    // records of one or two whole sectors, which that kernel stores complete:
    // 4320x7680 x 8 440 us against 460 here, 400x65532 x 8 and x 16 1.16x and
    // 1.07x faster (x 12 0.8x; here a CTA also adds up the counts of all chunks
    // to its left), 4320x5800 x 8 0.94x, 600x65535 x 8 (rows off 16 bytes) 0.97x
    return (f.B == 8 && f.W % 4 == 0 && px > (f.W > 48000 ? 16000000 : 30000000)) ||
           (f.B == 16 && f.W > 62000 && px > 24000000);
  // Four bins only, counted in a pass as long as their stores: 4800x8192 x 4 168
  // us here, 161 there, 7680x4320 x 4 0.93x.
  if (layout == IHIST_QUAD_MAJOR && f.B == 4 && f.W % 16 == 0 && px > 38000000) return true;
  // Bins and counts that L2 does not hold, where its own loads are whole (rows
  // of 16-byte multiples): bin-major 3840x2160 x 128 (58 MB) 660 us here, 663
  // there, x 192 (83 MB) 998 / 967, 3200x2500 x 160 (68 MB) 788 / 808, 4000x3000
  // x 64 (48 MB) 483 / 487, x 256 (156 MB) 1960 / 1820; up to 16 chunks wide
  // 1456x8192 x 160 (101 MB) the same, x 192 1.03x; quad-major 7680x4320 x 96
  // (182 MB) 0.99x, x 128 (232 MB) 1.02x, 4800x8192 x 192 5743 / 4986.  Rows of
  // other widths are faster here at any size (1464x8192 x 256 0.79x).  With
  // tables, which cost that kernel more, the lines lie higher (bin-major
  // 4000x3000 x 128 the same, x 192 1.03x, quad-major 4800x8192 x 128 0.97x, x
  // 192 1.06x).
  const long long mb = layout == IHIST_QUAD_MAJOR ? (table ? 335 : 190)
                       : f.nchunks > 16           ? (table ? 110 : 72)
                                                  : (table ? 160 : 105);
  return f.W % 16 == 0 && (long long)(q_size(f) + 4 * (pb_size(f) + sb_size(f) + rl_size(f))) > mb * 1000000;
}

bool bands_shape(int h, int w, int nbins, int layout, bool table, int sms, BandDesc *f) {
  if (!bands_fit(h, w, layout)) return false;
  bands_describe(h, w, nbins, layout, 32, 0, f);
  const long long per_band = (long long)f->nq * f->nchunks;
  auto bands = [&](int R) { return (long long)((h + R - 1) / R); };
  int R = bands_rows(bands(32) * per_band, bands(16) * per_band, (long long)h * w, h);
  if (layout == IHIST_PIXEL_MAJOR) {
    // by CTAs: 1920x1080 x 64 at R = 32 (510 CTAs) and 16: 97, 100 us; 640x480
    // x 64 at 32, 16 (150 CTAs) and 8: 27.8, 23.9, 25.8; 320x240 x 16 at 16
    // and 8 (90 CTAs): 10.2, 8.6
    const long long ctas = (long long)f->nblk * f->nchunks;
    R = bands(32) * ctas >= 400 || h > 2048 ? 32 : bands(16) * ctas >= 120 ? 16 : 8;
  }
  bands_describe(h, w, nbins, layout, R, 0, f);
  if (look_back_faster(*f, layout, table)) return false;
  // Count threads take R pixels each, or R / 2 where that leaves fewer than
  // 7/4 CTAs per SM, 2 when rows are also counted by strips (1280x720 x 32,
  // 240 CTAs: 27.3 -> 26.0 us; 1920x1080 with 300 CTAs: x 128 bin-major slower
  // split, 159.3 -> 162.8, x 64 pixel-major with its queries faster, 108.6 ->
  // 102).
  if (4u * count_ctas(*f) < (f->nblk ? 8u : 7u) * (unsigned)sms) f->split = 1;
  return (long long)f->nbands * (f->nblk ? f->nblk : f->nq) * f->nsegs < 0x7fffffffll;
}

int bands_kind(const BandDesc &f, int layout) {
  const uintptr_t out = reinterpret_cast<uintptr_t>(f.out);
  // pixel-major: one bin per lane where records are whole 32-byte sectors
  if (layout == IHIST_PIXEL_MAJOR) return f.bpb <= 32 ? 4 : f.B % 8 == 0 && (out & 31u) == 0 ? 5 : 6;
  const bool vec = (out & 15u) == 0;
  return layout == IHIST_QUAD_MAJOR ? (vec ? 2 : 3) : vec && f.W % 4 == 0 ? 0 : 1;
}

int bands_prepare(int mode, int layout) {
  int rc = allow_smem(count_fn(mode), max_count_smem());
  for (int kind = 0; kind < kBandKinds && rc == IHIST_OK; ++kind)
    if (bands_kind_layout(kind) == layout) rc = allow_smem(emit_fn(kind), max_emit_smem(kind));
  return rc;
}

int bands_prepare_batch() {
  int rc = IHIST_OK;
  for (int mode = kBinUniform; mode <= kBinJoint && rc == IHIST_OK; ++mode)
    rc = allow_smem(count_batch_fn(mode), max_count_smem());
  for (int kind = 0; kind < kBandKinds && rc == IHIST_OK; ++kind)
    rc = allow_smem(emit_batch_fn(kind), max_emit_smem(kind));
  return rc;
}

int launch_bands(const BandDesc &f, int mode, int layout, void *stream) {
  const int kind = bands_kind(f, layout);
  cudaError_t e = launch(count_fn(mode), 2u * f.nchunks, (unsigned)((f.H + col_tile_rows(f) - 1) / col_tile_rows(f)), 2u,
                         kCountThreads, count_smem_bytes(f), f, stream);
  if (e == cudaSuccess)
    e = launch(emit_fn(kind), emit_ctas(f, kind), 1u, 1u, bands_threads(f, kind), emit_smem(f, kind), f, stream);
  if (e != cudaSuccess) {
    cudaGetLastError();
    return IHIST_ERR_CUDA;
  }
  return IHIST_OK;
}

unsigned int bands_threads(const BandDesc &f, int kind) {
  return kind == 5 ? 256u : kind >= 4 ? 128u : 32u * (unsigned)(f.wpg * f.gpc);
}

// A count launch gives every CTA the shared memory of its largest frame, and
// shared memory is what limits its CTAs per SM (up to 72 bins four, 108 three,
// 180 two, above that one, at 32 rows per band), so frames share a launch only
// with frames that allow as many (where they are more than a few waves): 255
// frames of 320x240 x 8 and one of x 256, with their emit launch, took 268 us
// in one launch and take 182 in two, 31 of 1280x720 x 32 and one of x 256 810
// and 740.
int bands_count_class(const BandDesc &f) {
  constexpr size_t kSm = 228u << 10, kOther = 2048;  // an SM's shared memory; static and reserved bytes of a CTA
  return (int)std::min<size_t>(4, kSm / (count_smem_bytes(f) + kOther));
}

BandRun bands_run(bool count, int kernel, const BandDesc *d_desc) {
  BandRun r;
  r.count = count;
  r.kernel = kernel;
  r.threads = count ? (unsigned)kCountThreads : kernel == 5 ? 256u : kernel >= 4 ? 128u : 32u * kSegWarps;
  r.smem = !count && kernel < 4 ? emit_smem_bytes(kSegWarps, 32) : 0;
  r.batch.frames = d_desc;
  r.batch.n = 0;
  return r;
}

bool bands_run_add(BandRun *r, const BandDesc &f) {
  BandBatch &b = r->batch;
  if (b.n == kBatchFrames) return false;
  const unsigned int ctas = r->count ? count_ctas(f) : emit_ctas(f, r->kernel);
  b.end[b.n] = ctas + (b.n > 0 ? b.end[b.n - 1] : 0u);
  ++b.n;
  if (r->count || r->kernel >= 4) r->smem = std::max(r->smem, r->count ? count_smem_bytes(f) : emit_smem(f, r->kernel));
  return true;
}

int launch_bands_batch(const BandRun *runs, int nruns, void *stream) {
  for (const BandRun *r = runs; r < runs + nruns; ++r)
    if (launch(r->count ? count_batch_fn(r->kernel) : emit_batch_fn(r->kernel), r->batch.end[r->batch.n - 1], 1u, 1u,
               r->threads, r->smem, r->batch, stream) != cudaSuccess) {
      cudaGetLastError();
      return IHIST_ERR_CUDA;
    }
  return IHIST_OK;
}

}  // namespace host
}  // namespace ihist
