// Internal accessors of the context for translation units other than mk_api.cu.
#pragma once

#include <cuda_runtime.h>

#include <cstdint>
#include <vector>

#include "../../include/mockskewer.h"

namespace mkhost {
cudaStream_t ctx_stream(mk_ctx *c);
int ctx_device(mk_ctx *c);
int ctx_fail(mk_ctx *c, int code, const char *msg);
int ctx_sms(mk_ctx *c);
// Device scratch of at least `bytes` bytes, shared by the calls that take it
// (each finishes with it, and calls ctx_trim_scratch, before it returns).
// MK_ENOMEM when it cannot grow.
int ctx_scratch(mk_ctx *c, size_t bytes, unsigned char **p);
// Gives the scratch back if it is larger than kScratchKept, the most that a
// context holds between calls (the draw of a 1024^3 box takes 151 MB of it).
constexpr size_t kScratchKept = size_t(256) << 20;
void ctx_trim_scratch(mk_ctx *c);
// FP64 cosmology of the context (Sec. 2): z(D_C), G(z), D_C(z)
double ctx_z_of(mk_ctx *c, double r);
double ctx_growth(mk_ctx *c, double z);
double ctx_distance(mk_ctx *c, double z);
// Pixel redshifts z_J of the tables for pixel size dr and, per J, the number
// of pixels of the n_sk skewers d_sk at J (synchronous; GPU time added to *ms).
int ctx_pixel_histogram(mk_ctx *c, double dr, const mk_skewer *d_sk, int64_t n_sk, std::vector<double> &z,
                        std::vector<int64_t> &count, double *ms);
}  // namespace mkhost
