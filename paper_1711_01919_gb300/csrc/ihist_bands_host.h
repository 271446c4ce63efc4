// ihist_bands_host.h -- host interface of the two-launch path
// (ihist_bands.cu), used by plans (ihist_api.cu) and batches
// (ihist_batch_api.cu).
#pragma once

#include "ihist_bands.cuh"
#include "ihist_host.h"

namespace ihist {
namespace host {

// Emit kernels: 0, 1 bin-major (rows 16-byte aligned or not), 2, 3 quad-major
// (likewise), 4, 5, 6 pixel-major (at most 32 bins a block, one bin per lane,
// two bins per lane).
constexpr int kBandKinds = 7;
inline int bands_kind_layout(int kind) {
  return kind < 2 ? IHIST_BIN_MAJOR : kind < 4 ? IHIST_QUAD_MAJOR : IHIST_PIXEL_MAJOR;
}
int bands_kind(const BandDesc &f, int layout);
unsigned int bands_threads(const BandDesc &f, int kind);

// Whether the two-launch path is the faster one for a frame of this size.
bool bands_fit(int h, int w, int layout);

// Rows per band of bin- or quad-major frames: emit warps at 32 and 16 rows per
// band, pixels, and the tallest frame.
int bands_rows(long long warps32, long long warps16, long long pixels, int h_max);

// The shape fields of a frame with R rows per band.
void bands_describe(int h, int w, int nbins, int layout, int R, int split, BandDesc *f);

// Whether a plan's frames take the two-launch path, and their shape in *f
// (table: they bin through a value -> bin table).
bool bands_shape(int h, int w, int nbins, int layout, bool table, int sms, BandDesc *f);

// Workspace bytes of the shape; with a base (256-byte aligned), also the
// pointers into it.  any_layout: enough for the same shape in every layout.
size_t bands_layout(BandDesc *f, char *base, bool any_layout = false);

// Let the kernels of this binning and layout (or all batch kernels) use the
// shared memory they need.
int bands_prepare(int mode, int layout);
int bands_prepare_batch();

// Both launches of one frame, with programmatic stream serialization.
int launch_bands(const BandDesc &f, int mode, int layout, void *stream);

// Count CTAs per SM that a frame's shared memory allows (1..4).
int bands_count_class(const BandDesc &f);

// One launch of a batch: at most kBatchFrames frames through the count kernel of
// a binning or the emit kernel of a kind, whose descriptors the launch must find
// on the device from d_desc on.
struct BandRun {
  bool count;
  int kernel;
  unsigned int threads;
  size_t smem;
  BandBatch batch;
};
BandRun bands_run(bool count, int kernel, const BandDesc *d_desc);
bool bands_run_add(BandRun *r, const BandDesc &f);  // false: the launch is full
int launch_bands_batch(const BandRun *runs, int nruns, void *stream);

}  // namespace host
}  // namespace ihist
