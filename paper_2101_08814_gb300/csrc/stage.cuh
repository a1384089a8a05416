// Staged blocks that leave shared memory by bulk copies.
#pragma once

#include "tcgen05.cuh"

namespace rascal {

// Position (in floats, 0..3) at which a staged block must start in a 16-byte aligned buffer so that the staged and
// the global addresses agree modulo 16 bytes.
__device__ inline int stage_shift(const float* dst) { return (int)((reinterpret_cast<uintptr_t>(dst) >> 2) & 3); }

// Writes count floats staged at st (st and dst congruent mod 16 bytes) to dst: thread 0 issues one bulk copy for
// the aligned body, threads 0..6 store the ragged head and tail. Call after the fence and barrier that publish st.
__device__ inline void store_staged(float* dst, const float* st, int count) {
    if (threadIdx.x >= 32) return;  // warp 0 does all of it: the other warps skip the address arithmetic
    const int head = min((4 - stage_shift(dst)) & 3, count);
    const int body = (count - head) & ~3;
    const int tail = count - head - body;
    const int t = threadIdx.x;
    if (t == 0) {  // one bulk group per call, possibly empty, so that waits can count calls
        if (body > 0) bulk_store(dst + head, st + head, (uint32_t)body * 4u);
        bulk_commit();
    }
    if (t < head) dst[t] = st[t];
    if (t >= 4 && t < 4 + tail) dst[head + body + t - 4] = st[head + body + t - 4];
}

}  // namespace rascal
