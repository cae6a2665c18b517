// A kernel's device status word, the abort flag that its CTA's roles share,
// and the bounded wait that watches the flag.
#pragma once

#include "bsr_internal.h"
#include "ptx.cuh"

namespace bsr {

// Records `code` unless an earlier error is recorded.
__device__ __forceinline__ void set_status(int *status, int code) { atomicCAS(status, DEV_OK, code); }
__device__ __forceinline__ bool aborted(const int *flag) { return *reinterpret_cast<const volatile int *>(flag) != 0; }

// Bounded wait that also gives up when another role of the CTA stopped. With
// `beat`, the limit begins anew while that word changes (a role for which every
// other one waits in the end reports that it is at work).
__device__ __forceinline__ bool wait_or_abort(uint64_t *bar, uint32_t parity, uint64_t limit_ns, const int *flag,
                                              const int *beat = nullptr) {
    if (ptx::mbar_try_wait(bar, parity)) return true;
    uint64_t t0 = ptx::globaltimer();
    int seen = 0;
    while (true) {
        if (ptx::mbar_try_wait(bar, parity)) return true;
        if (aborted(flag)) return false;
        const uint64_t t = ptx::globaltimer();
        if (t - t0 <= limit_ns) continue;
        const int now = beat ? *reinterpret_cast<const volatile int *>(beat) : 0;
        if (now == seen) return false;
        seen = now;
        t0 = t;
    }
}

}  // namespace bsr
