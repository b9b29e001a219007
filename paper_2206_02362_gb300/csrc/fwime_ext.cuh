// Device helpers shared by the extension kernels (scatter, imaging): walking the (step, shot) pairs of a
// segment, asynchronous copies.
#pragma once
#include "fwime_kernels.cuh"

namespace fwk {

// ---- asynchronous global -> shared copies (LDGSTS)
__device__ __forceinline__ void cpa_commit() { asm volatile("cp.async.commit_group;\n" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cpa_wait() { asm volatile("cp.async.wait_group %0;\n" ::"n"(N) : "memory"); }
// 16 bytes, past L1 (both addresses 16-byte aligned); valid = false zero-fills and reads nothing
__device__ __forceinline__ void cpa16(unsigned dst, const float *src, bool valid)
{
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;\n" ::"r"(dst), "l"(src), "r"(valid ? 16 : 0) : "memory");
}

// Row pointers of N rings at the (step, shot) pairs of a segment in order (shot fastest): one addition per ring
// and pair, a multiply only when the time slot changes.  What stays the same along the segment is read from the
// kernel's parameters again instead of kept in registers.
template <int N>
struct PairRows {
    const float *row[N];
    int slot[N], s;
    // starting at the first pair
    __device__ __forceinline__ void init(const RingRef *const (&r)[N], int n0, long long rowoff)
    {
        s = 0;
#pragma unroll
        for (int k = 0; k < N; ++k) {
            slot[k] = r[k]->mod > 0 ? (n0 + r[k]->shift) % r[k]->mod : r[k]->shift;
            row[k] = r[k]->base + rowoff + (long long)slot[k] * r[k]->slot_stride;
        }
    }
    __device__ __forceinline__ void next(const RingRef *const (&r)[N], int S, long long P, long long rowoff)
    {
        if (++s == S) {
            s = 0;
#pragma unroll
            for (int k = 0; k < N; ++k) {
                if (++slot[k] == r[k]->mod) slot[k] = 0;   // mod == 0 (direct rings) never wraps
                row[k] = r[k]->base + rowoff + (long long)slot[k] * r[k]->slot_stride;
            }
        } else {
#pragma unroll
            for (int k = 0; k < N; ++k) row[k] += P;
        }
    }
};

}  // namespace fwk
