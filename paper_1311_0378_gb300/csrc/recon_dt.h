// Distance transform: internal launcher (see recon_dt.cu). Not part of the C ABI.
#pragma once
#include <cuda_runtime.h>
#include <stddef.h>
#include <stdint.h>

enum { DT_OK = 0, DT_ECUDA = 1 };

// Scratch starts with 32 words, 128 bytes apart, that say in which call background
// was last seen. Cleared when the scratch is allocated; the rest needs no
// initialisation.
constexpr size_t DT_HEADER = 4096;
// Device scratch bytes for an H x W image (those words, column masks, column distances).
size_t dt_scratch_bytes(int H, int W);

// Queues the whole transform on stream st. B: device H x W bytes (nonzero =
// foreground); d2: device uint32 H x W out; site: device int32 H x W out, or
// NULL; scratch: dt_scratch_bytes(H, W) device bytes; call: nonzero, another number
// than in the scratch's calls before.
int dt_run(const uint8_t *B, int H, int W, int *site, unsigned *d2, void *scratch, unsigned call, int sms, cudaStream_t st);
