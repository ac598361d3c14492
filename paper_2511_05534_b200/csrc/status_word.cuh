// Status word of a call that starts its own word: one kernel's blocks report to it, in whatever order they run, on a
// workspace that held anything before.  64 bits: the status code below (what the reader returns), the number of the call
// that wrote it above.  Clearing and reporting both look at the number: a report made before the call's first block has
// come to clear the word stays, a word of any other call goes.
#pragma once
#include <stdint.h>

#ifdef __CUDACC__
#define FLOWMM_STATUS_FN __host__ __device__ __forceinline__
#else
#define FLOWMM_STATUS_FN inline
#endif

namespace flowmm {

// The word after call `call` has cleared it: what the call itself has reported stays.
FLOWMM_STATUS_FN unsigned long long status_cleared(unsigned long long word, uint32_t call) {
    return (uint32_t)(word >> 32) == call ? word : (unsigned long long)call << 32;
}
// The word after call `call` has reported `code`: the call's first report stays.
FLOWMM_STATUS_FN unsigned long long status_reported(unsigned long long word, uint32_t call, int code) {
    const unsigned long long mine = status_cleared(word, call);
    return (uint32_t)mine != 0u ? mine : mine | (uint32_t)code;
}

#ifdef __CUDACC__
// Clears the word (code 0) or reports.  Within a call the word changes twice at most, so the exchange is tried three times at most.
__device__ __forceinline__ void status_write(int *status, uint32_t call, int code) {
    unsigned long long *word = reinterpret_cast<unsigned long long *>(status), seen = *reinterpret_cast<volatile unsigned long long *>(word);
    for (int tries = 0; tries < 3; ++tries) {
        const unsigned long long next = code == 0 ? status_cleared(seen, call) : status_reported(seen, call, code);
        if (next == seen) return;
        const unsigned long long prev = atomicCAS(word, seen, next);
        if (prev == seen) return;
        seen = prev;
    }
}
#endif

}  // namespace flowmm
