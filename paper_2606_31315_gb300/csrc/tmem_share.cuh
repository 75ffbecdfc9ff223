// How CTAs of different launches share the tensor memory of one SM.  Plain C++ (no CUDA types), so that the
// arithmetic is checked on the host.
#pragma once

namespace bp {

constexpr int kTmemColumns = 512;  // tensor-memory columns of an SM
constexpr int kTmemGrain = 32;     // an allocation is a power of two of at least 32 columns

// The columns allocated for n of them.
constexpr int tmem_columns(int n) {
    int c = kTmemGrain;
    while (c < n) c <<= 1;
    return c;
}

// Shared memory (in all: dynamic, static and the system's share) that a CTA with `columns` of tensor memory takes
// of an SM that has sm_smem bytes.  tcgen05.alloc waits without a limit for columns that others hold, and a CTA
// whose cluster or grid waits for its peers holds its own meanwhile: two calls on two streams that meet on two SMs
// in opposite orders would never end.  With shared memory in proportion to columns the allocation never waits,
// whatever launches meet: CTAs whose columns add up to more than 512, so to 544 at least, need more shared memory
// than the SM has.  (A bound per launch, 1 / (512 / columns + 1) of the SM, kept only CTAs of one column count to
// 512: one of 256 columns and five of 64 fitted an SM.)
constexpr int tmem_smem_share(int columns, int sm_smem) {
    return (int)((long long)columns * sm_smem / (kTmemColumns + kTmemGrain)) + 1;
}

}  // namespace bp
