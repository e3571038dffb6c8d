// What the kernels that run FP32 lanes on groups of CTAs (sell_lane.cu, sym_lane.cu) exchange
// within a step, and how: tagged words in global memory that the readers poll, instead of a
// barrier, a record array and the vectors.
//
// A word is two 64-bit pairs of a value and the step's tag; a pair is read and written whole, so
// nothing is fenced and nobody counts arrivals: a word is there when both its tags are.  (Three
// values and one tag in a 128-bit access would be a third less to read, but a record with the
// step's tag and the previous value was seen with such words.)  Words alternate between two
// buffers by the step's parity; each kernel says why that is enough.  A hop takes 1,700 cycles
// between 16 CTAs and 2,800 between 79 (a barrier and the loads after it 3,400 and 4,700).
#pragma once

#include "solo_common.cuh"

namespace ubqp {

namespace {

// the eigen-solver's twelve Gram sums (a word each): products of the row vectors x, Ax, w, Aw, p, Ap
// (0 .. 5) in row_epilogue's order, sum t in nibble t
constexpr int kGramWords = 12;
constexpr unsigned long long kGramLeft = 0x422000422000ull, kGramRight = 0x442420553531ull;

// warp-level result of a reduction: the sums and maxima of one phase
struct WarpRed {
    float2 s[12];
    float m[4];
};

// two values, each with the tag in its own 64 bits (the unit that is read and written whole)
__device__ __forceinline__ void st_word(ulonglong2* p, float a, float b, uint32_t tag)
{
    const unsigned long long t = (unsigned long long)tag << 32;
    asm volatile("st.relaxed.gpu.global.v2.u64 [%0], {%1, %2};" ::"l"(p), "l"(t | __float_as_uint(a)),
                 "l"(t | __float_as_uint(b))
                 : "memory");
}

// one warp stores a slice's words, lane t word t; the warp is whole again before it waits
__device__ __forceinline__ void publish(ulonglong2* p, bool mine, int lane, float2 v, uint32_t tag)
{
    if (mine) st_word(p + lane, v.x, v.y, tag);
    __syncwarp();
}

__device__ __forceinline__ ulonglong2 ld_word(const ulonglong2* p)
{
    ulonglong2 v;
    asm volatile("ld.relaxed.gpu.global.v2.u64 {%0, %1}, [%2];" : "=l"(v.x), "=l"(v.y) : "l"(p) : "memory");
    return v;
}

__device__ __forceinline__ bool has_tag(ulonglong2 v, uint32_t tag)
{
    return (uint32_t)(v.x >> 32) == tag && (uint32_t)(v.y >> 32) == tag;
}
__device__ __forceinline__ float2 word_values(ulonglong2 v)
{
    return make_float2(__uint_as_float((uint32_t)v.x), __uint_as_float((uint32_t)v.y));
}

// Waits until the N words p[h] of every thread of the warp carry `tag` (threads without words of
// their own pass another's).  The warp leaves the loop as a whole: with a loop that each thread
// left by itself, the threads still waiting ran one after another, a trip to L2 each (20,000
// cycles a wait with 16 of them, against 1,700).
template <int N>
__device__ __forceinline__ void wait_words(const SoloArgs& A, const ulonglong2* const (&p)[N], uint32_t tag,
                                           ulonglong2 (&v)[N], volatile int* s_ok)
{
    const long long t0 = clock64();
    for (;;) {
#pragma unroll
        for (int h = 0; h < N; ++h) v[h] = ld_word(p[h]);
        bool all = true;
#pragma unroll
        for (int h = 0; h < N; ++h) all &= has_tag(v[h], tag);
        if (__all_sync(0xffffffffu, all)) return;
        const bool late = clock64() - t0 > (long long)A.wait_cycles || !*s_ok;
        if (__any_sync(0xffffffffu, late)) {
            atomicExch(A.err, 1);
            *s_ok = 0;
            return;
        }
    }
}

// the butterfly of N compensated sums and M maxima, level by level (acc_shfl_reduce's order)
template <int N, int M>
__device__ __forceinline__ void butterfly(float2* s, float* m)
{
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        float2 w[N > 0 ? N : 1];
        float wm[M > 0 ? M : 1];
#pragma unroll
        for (int t = 0; t < N; ++t) {
            w[t].x = __shfl_xor_sync(0xffffffffu, s[t].x, o);
            w[t].y = __shfl_xor_sync(0xffffffffu, s[t].y, o);
        }
#pragma unroll
        for (int t = 0; t < M; ++t) wm[t] = __shfl_xor_sync(0xffffffffu, m[t], o);
#pragma unroll
        for (int t = 0; t < N; ++t) s[t] = csum_merge(s[t], w[t]);
#pragma unroll
        for (int t = 0; t < M; ++t) m[t] = fmaxf(m[t], wm[t]);
    }
}

// where g_{k-1} of a subproblem stopped before step k is kept (solo.cu alternates the two)
__device__ __forceinline__ int g_buf(int k) { return (k & 1) ? V_G : V_W; }

// two of the 32 values held one per lane, for the word `lane` of a slice's row words
__device__ __forceinline__ float2 row_word(float g, int lane)
{
    const float a = __shfl_sync(0xffffffffu, g, (2 * lane) & 31);
    return make_float2(a, __shfl_sync(0xffffffffu, g, (2 * lane + 1) & 31));
}

// the first W words of every block of buffer w (stride words per block) into dst, 2 W values per
// block, by threads tid of nt (whole warps)
template <int W>
__device__ __forceinline__ void gather_rows(const SoloArgs& A, const ulonglong2* w, int stride, int nblk, uint32_t tag,
                                            float* dst, int tid, int nt, volatile int* s_ok)
{
    constexpr int kFly = 8;
    const int nq = W * nblk;
    for (int base = tid & ~31; base < nq; base += kFly * nt) {
        const int q0 = base + (tid & 31);
        const ulonglong2* p[kFly];
        ulonglong2 v[kFly];
#pragma unroll
        for (int h = 0; h < kFly; ++h) {
            int q = q0 + h * nt;
            if (q >= nq) q = min(q0, nq - 1);
            p[h] = w + (size_t)(q / W) * stride + q % W;
        }
        wait_words<kFly>(A, p, tag, v, s_ok);
#pragma unroll
        for (int h = 0; h < kFly; ++h)
            if (q0 + h * nt < nq) reinterpret_cast<float2*>(dst)[q0 + h * nt] = word_values(v[h]);
    }
}

}  // namespace

}  // namespace ubqp
