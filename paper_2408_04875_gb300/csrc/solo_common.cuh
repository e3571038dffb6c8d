// Pieces shared by the two kernels that run FP32 lanes on groups of CTAs in one cooperative
// launch (solo.cu: any storage; sell_lane.cu: the sliced storage): the bounded group barrier
// and the Alg. 2 row epilogue.
#pragma once

#include "gemv_rows.cuh"

namespace ubqp {

__device__ __forceinline__ unsigned long long ld_acquire_u64(const unsigned long long* p)
{
    unsigned long long v;
    asm volatile("ld.acquire.gpu.global.u64 %0, [%1];" : "=l"(v) : "l"(p) : "memory");
    return v;
}

// Group barrier on a monotonic 64-bit arrival counter: barrier number gen + 1 of the group is
// complete when the counter reaches nc * (gen + 1).  A CTA adds its arrival without waiting for
// the result and polls the counter (bounded); nobody resets anything, so a barrier costs one
// round trip after the last arrival.
__device__ __forceinline__ bool solo_grid_sync(const SoloArgs& A, unsigned long long* bar, int nc,
                                               unsigned long long& gen, int* s_ok)
{
    __syncthreads();
    if (nc == 1) return *s_ok != 0;
    if (threadIdx.x == 0) {
        const unsigned long long target = (gen + 1ull) * (unsigned long long)nc;
        __threadfence();
        asm volatile("red.relaxed.gpu.global.add.u64 [%0], 1;" ::"l"(bar) : "memory");
        const long long t0 = clock64();
        while (ld_acquire_u64(bar) < target) {
            if (clock64() - t0 > (long long)A.wait_cycles) {
                atomicExch(A.err, 1);
                *s_ok = 0;
                break;
            }
        }
        gen += 1ull;
    }
    __syncthreads();
    return *s_ok != 0;
}

// Alg. 2 row epilogue of the single-barrier step for row i: x_k, x_{k-1}, d - p, d + b' and
// g_{k-1} of the row given, g_k written to gnew[i] and returned; the arithmetic of row_epilogue
// (PH_INNER)
__device__ __forceinline__ float solo_inner_row(const LaneDev& L, int k, int i, float v, float x, float xp, float dmp,
                                                float tsum, float gold, float* gnew, Acc& a)
{
    const float g = fmaf(dmp, 2.f * x - 1.f, fmaf(2.f, v, tsum));
    if (k >= 1) {
        const float sd = x - xp;
        const float y = g - gold;
        csum_add(a.s[0], sd * sd);
        csum_add(a.s[1], sd * y);
        csum_add(a.s[2], y * y);
    } else {
        a.m[1] = fmaxf(a.m[1], fabsf(dmp));
        a.m[2] = fmaxf(a.m[2], fabsf(L.vec[V_BBAR * L.ld + i]));
        a.m[3] = fmaxf(a.m[3], L.oabs[i] + fabsf(dmp));
    }
    gnew[i] = g;
    const float viol = (x > 0.f && x < 1.f) ? fabsf(g) : (x <= 0.f ? fmaxf(-g, 0.f) : fmaxf(g, 0.f));
    a.m[0] = fmaxf(a.m[0], viol);
    return g;
}

__device__ __forceinline__ unsigned long long solo_item_bytes(const LaneDev& L, int blk, int row0, int rows)
{
    if (L.spv)
        return 6ull * (unsigned long long)(L.spo[(row0 + rows + 31) >> 5] - L.spo[row0 >> 5]) +
               (blk == 0 ? 4ull * L.n : 0ull) + 16ull * rows;
    return (unsigned long long)rows * L.n * 4ull + (blk == 0 ? 4ull * L.n : 0ull) + 16ull * rows;
}

}  // namespace ubqp
