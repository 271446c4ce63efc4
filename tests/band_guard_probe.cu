// One frame through the checked count and emit kernels with more CTAs than it
// has: the surplus ones' indices lie outside the frame's workspace arrays (not
// outside the buffers, which the caller makes larger).  Built by
// test_gpu_checked_bands.py with -DIHIST_CHECKED.
#include "ihist_bands.cu"

using namespace ihist;
using namespace ihist::host;

extern "C" size_t probe_workspace(int h, int w, int nbins, int layout, int R) {
  BandDesc f;
  bands_describe(h, w, nbins, layout, R, 0, &f);
  return bands_layout(&f, nullptr);
}

// Returns the latched status, or minus a CUDA error.  chunks, bands: surplus
// chunks of the count grid and bands of the emit grid.
extern "C" int probe_run(int h, int w, int nbins, int layout, int R, const uint8_t *in, uint32_t *out, char *ws,
                         int *ctrl, int chunks, int bands) {
  BandDesc f;
  bands_describe(h, w, nbins, layout, R, 0, &f);
  bands_layout(&f, ws);
  f.in = in;
  f.pitch = w;
  f.out = out;
  f.ctrl = reinterpret_cast<Ctrl *>(ctrl);
  if (bands_prepare(kBinUniform, layout) != IHIST_OK) return -1;
  const int kind = bands_kind(f, layout);
  cudaError_t e = launch(count_fn(kBinUniform), 2u * (f.nchunks + chunks),
                         (unsigned)((h + col_tile_rows(f) - 1) / col_tile_rows(f)) + (unsigned)chunks, 2u, kCountThreads,
                         count_smem_bytes(f), f, nullptr);
  if (e == cudaSuccess)
    e = launch(emit_fn(kind), emit_ctas(f, kind) / f.nbands * (f.nbands + bands), 1u, 1u, bands_threads(f, kind),
               emit_smem(f, kind), f, nullptr);
  if (e == cudaSuccess) e = cudaDeviceSynchronize();
  Ctrl c;
  if (e == cudaSuccess) e = cudaMemcpy(&c, ctrl, sizeof(c), cudaMemcpyDeviceToHost);
  return e == cudaSuccess ? c.status : -(int)e;
}
