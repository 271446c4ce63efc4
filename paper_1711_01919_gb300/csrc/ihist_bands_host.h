// ihist_bands_host.h -- host interface of the two-launch path
// (ihist_bands.cu), used by plans (ihist_api.cu).
#pragma once

#include "ihist_bands.cuh"
#include "ihist_host.h"

namespace ihist {
namespace host {

// Whether a frame takes the two-launch path, and its shape fields in *f.
bool bands_shape(int h, int w, int nbins, int layout, int sms, BandDesc *f);

// Workspace bytes of the shape; with a base (256-byte aligned), also the
// pointers into it.
size_t bands_layout(BandDesc *f, char *base);

// Let the kernels of this binning and layout use their shared memory (optin: the
// largest a CTA may have).
int bands_prepare(const BandDesc &f, int mode, int layout, size_t optin);

// Both launches, with programmatic stream serialization.
int launch_bands(const BandDesc &f, int mode, int layout, void *stream);

}  // namespace host
}  // namespace ihist
