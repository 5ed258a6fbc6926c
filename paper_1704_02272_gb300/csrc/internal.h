// Host-side table object and error reporting shared by the library's
// translation units.
#pragma once
#include <cuda_runtime.h>
#include <stdarg.h>
#include <stddef.h>
#include <stdint.h>

#include <vector>

#include "../../include/pfac.h"
#include "table.h"

struct pfac_table {
    pfac::DevTable dev;
    void *d_blob = nullptr;
    uint64_t blob_bytes = 0;
    // host-only tables keep their blob here (the DevTable's pointers point
    // into it; no kernel reads them: every match call refuses such a table)
    std::vector<uint8_t> h_blob;
    pfac_table_info_t info{};
    uint32_t kmin = 0, kmax = 0;  // prefix nodes exist for depths kmin..kmax
    int device = 0;
    // autotuned defaults (0 = none)
    uint32_t tuned_variant = 0;
    uint32_t tuned_k = 0;
    uint32_t tuned_copies = 0;
    uint32_t tuned_masks = 0;
    uint32_t tuned_gram = 0;
    uint32_t tuned_bytes = 0;
    uint32_t tuned_nw = 0;
    uint32_t tuned_kernel = 0;
    uint32_t tuned_records = 0;
    uint32_t tuned_resolver = 0;
    double match_density = 0.0;  // expected matches per position of uniform text
};

namespace pfac {

int set_error(int status, const char *fmt, ...);
void clear_error();

// PFAC_OK when the current device and, for a non-NULL stream, the stream's
// device are the device the table was uploaded to; otherwise PFAC_EINVAL
// (with a message naming `who`), so that no kernel is launched on one GPU
// with another GPU's pointers.
int check_table_device(const pfac_table *t, void *cuda_stream, const char *who);

// Shared-memory wavefronts of one warp-wide load of random words with 2^i
// copies interleaved over the banks: lanes that share a copy collide.
constexpr double LOAD_WAVEFRONTS[6] = {3.7, 3.4, 3.1, 2.85, 2.0, 1.0};

// Bytes of a workspace that do not grow with the input, at most: a fixed
// scratch or pool of N bytes is made this much larger, so that it holds what
// takes N bytes for its input alone.
constexpr uint64_t WS_FIXED_BYTES = 32 << 10;

// The options that need the least scratch: the library's choice of the rest,
// 32 records a slice, and no buffer for a resolver launch.
inline pfac_match_opts lean_opts(const pfac_match_opts *opts) {
    pfac_match_opts o{};
    if (opts) o = *opts;
    if (!o.records_per_slice) o.records_per_slice = 32;
    if (!o.resolver) o.resolver = 1;
    return o;
}

// Stream-ordered scratch from the library's own pool of the current context
// (freed with cudaFreeAsync), and giving back what the pool keeps (waits for
// the device first; nothing where there is no pool).
cudaError_t scratch_alloc(void **p, size_t bytes, cudaStream_t st);
void scratch_trim();

// Id of the current CUDA context, one that no other context of the process
// has or gets (0 when it cannot be told).
uint64_t current_context_id();

}  // namespace pfac
