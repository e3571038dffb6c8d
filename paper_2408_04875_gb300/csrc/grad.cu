// The penalized objective of Sec. 4.1, problem (p), its gradient and its backward, for a batch of
// points sharing Q, b, p (ubqp_penalized_eval, ubqp_penalized_eval_noalloc, ubqp_penalized_vjp):
//     h_r = x_r^T Q x_r + b^T x_r + sum_i p_i (x_ri - x_ri^2),  g_r = 2 (Q - Diag p) x_r + b + p
//
// grad_kernel computes a tile of 32 rows x TN points per CTA.  Thread = row (lane) of one of eight
// warps; each warp takes an eighth of the columns of every staged chunk for all TN points, so a
// thread reads an entry of Q once from shared memory for TN products and the points' entries by
// broadcast.  Chunks of 32 rows of Q and TN points (512 bytes a row) arrive by cp.async, three
// deep.  Bound: a few points read Q once (memory); from about TN = 8 on the arithmetic, which in
// FP32 is 11 operations for four products (a chain of FMAs, added to a TwoSum-compensated sum: the
// accuracy of the inner loop's row dots) and in FP64 the FP64 pipe.  The eight warps' sums are
// merged in order and the epilogue forms g and the point's share of h.
//
// Measured (device time per call, before: one point's rows per work item, Q read once per point):
// n = 1000, 64 points FP32 36 -> 14 us; n = 1001, 37 points FP64 165 -> 85 us; n = 8192, 128 points
// FP32 2110 -> 970 us, i.e. 24 T FP32 operations/s of the 36 T that packed additions alone reach
// here (two rows a thread, 16 points a CTA or FMAs in place of subtractions: no faster).
//
// The FP32 epilogue works in error-free pairs (TwoSum, FMA product errors) and rounds g once.  Against
// FP64 at n = 8192, 128 points, relative root mean square (before: row products rounded to FP32, then
// FP64): h 5.0e-8 either way, g 5.95e-8 -> 4.76e-8.  FP64
// adds chains of eight products in two levels (four chains, then those), which keeps its rounding
// at that of a row dot spread over 64 accumulators.
#include <algorithm>

#include "gemv_rows.cuh"

namespace ubqp {

namespace {

constexpr int kRowT = 32;          // rows per tile
constexpr int kChunkBytes = 512;   // bytes of a row per stage
constexpr int kRowStride = kChunkBytes + 16;   // in shared memory: 16-byte loads of 8 rows meet no bank twice
constexpr int kStages = 3;
constexpr int kTilesPerCta = 4;    // up to this many row tiles one CTA takes them all and writes h itself

struct GradArgs {
    const void *Q, *b, *p, *x;
    void *g, *h;
    double* part;    // [point][tile] shares of h (more than kTilesPerCta tiles), else null
    int32_t n;
    int64_t batch;
    int32_t tiles;
};

template <int BYTES>
__device__ __forceinline__ void cp_async(uint32_t dst, const void* src, bool in)
{
    const int sz = in ? BYTES : 0;   // 0: zero-fill
    if constexpr (BYTES == 16) asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst), "l"(src), "r"(sz) : "memory");
    else asm volatile("cp.async.ca.shared.global [%0], [%1], %3, %2;" ::"r"(dst), "l"(src), "r"(sz), "n"(BYTES) : "memory");
}

// ROWS rows (row stride n entries, the first `valid` exist) of columns k0 .. k0 + chunk into dst;
// a thread copies the same column of every kThreads / per-th row
template <typename T, int CP, int ROWS>
__device__ __forceinline__ void stage_rows(uint32_t dst, const T* src, int64_t n, int k0, int valid)
{
    constexpr int per = kChunkBytes / CP, E = CP / (int)sizeof(T), step = kThreads / per;
    const int c = (int)threadIdx.x % per, r0 = (int)threadIdx.x / per;
    const bool in_k = k0 + c * E < n;
    const T* p = src + (int64_t)r0 * n + k0 + c * E;
    dst += r0 * kRowStride + c * CP;
#pragma unroll
    for (int i = 0; i < (ROWS + step - 1) / step; ++i) {
        const int r = r0 + i * step;
        if (ROWS % step == 0 || r < ROWS) {
            const bool in = in_k && r < valid;
            cp_async<CP>(dst + i * step * kRowStride, in ? p : src, in);
        }
        p += (int64_t)step * n;
    }
}

// Packed FP32 pairs (one instruction, two lanes of the same rate)
__device__ __forceinline__ unsigned long long mul2(unsigned long long a, unsigned long long b)
{
    unsigned long long d;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
    return d;
}
__device__ __forceinline__ unsigned long long fma2(unsigned long long a, unsigned long long b, unsigned long long c)
{
    unsigned long long d;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
    return d;
}
__device__ __forceinline__ unsigned long long add2(unsigned long long a, unsigned long long b)
{
    unsigned long long d;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
    return d;
}
__device__ __forceinline__ unsigned long long sub2(unsigned long long a, unsigned long long b)
{
    unsigned long long d;
    asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
    return d;
}

// accumulators of one (row, point)
template <typename T> struct GradAcc;
template <> struct GradAcc<float> {
    // two compensated sums side by side: the even and the odd products of every eight, each four a
    // chain of FMAs (cacc4's operations on both at once: half the instructions)
    unsigned long long s, e;
    __device__ void zero() { s = e = 0ull; }
    __device__ __forceinline__ void add8(ulonglong2 q0, ulonglong2 q1, ulonglong2 u0, ulonglong2 u1)
    {
        unsigned long long t = mul2(q0.x, u0.x);
        t = fma2(q0.y, u0.y, t);
        t = fma2(q1.x, u1.x, t);
        t = fma2(q1.y, u1.y, t);
        const unsigned long long n = add2(s, t), bb = sub2(n, s);   // TwoSum
        e = add2(e, add2(sub2(s, sub2(n, bb)), sub2(t, bb)));
        s = n;
    }
    __device__ __forceinline__ float2 sum() const
    {
        return csum_merge(make_float2(__uint_as_float((uint32_t)s), __uint_as_float((uint32_t)e)),
                          make_float2(__uint_as_float((uint32_t)(s >> 32)), __uint_as_float((uint32_t)(e >> 32))));
    }
};
template <> struct GradAcc<double> {
    double lo, hi;   // the chains of the current four chunks, and of all before
    __device__ void zero() { lo = hi = 0.0; }
};

}  // namespace

template <typename T, int TN, int CP>
__global__ void __launch_bounds__(kThreads, 2) grad_kernel(GradArgs A)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    constexpr int KT = kChunkBytes / (int)sizeof(T);
    constexpr int KW = KT / kWarps;   // columns of a chunk per warp: 16 (FP32) or 8 (FP64)
    constexpr int kStageBytes = (kRowT + TN) * kRowStride;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int64_t n = A.n;
    const int64_t p0 = (int64_t)blockIdx.x * TN;
    const int64_t np = min((int64_t)TN, A.batch - p0);
    const T* Q = static_cast<const T*>(A.Q);
    const T* x = static_cast<const T*>(A.x) + p0 * n;
    const uint32_t base = (uint32_t)__cvta_generic_to_shared(smem_raw);
    const int nchunk = (int)((n + KT - 1) / KT);
    const bool all = A.tiles <= kTilesPerCta;   // this CTA takes every row tile
    const int t0 = all ? 0 : (int)blockIdx.y, t1 = all ? A.tiles : t0 + 1;
    constexpr int NJ = (TN + kWarps - 1) / kWarps;   // points whose epilogue a warp runs
    double hsum[NJ];
#pragma unroll
    for (int q = 0; q < NJ; ++q) hsum[q] = 0.0;

    for (int t = t0; t < t1; ++t) {
        const int64_t row0 = (int64_t)t * kRowT;
        auto stage = [&](int c) {
            if (c < nchunk) {
                const uint32_t s = base + (uint32_t)(c % kStages) * kStageBytes;
                stage_rows<T, CP, kRowT>(s, Q + row0 * n, n, c * KT, (int)min((int64_t)kRowT, n - row0));
                stage_rows<T, CP, TN>(s + kRowT * kRowStride, x, n, c * KT, (int)np);
            }
            asm volatile("cp.async.commit_group;" ::: "memory");
        };
        GradAcc<T> acc[TN];
#pragma unroll
        for (int j = 0; j < TN; ++j) acc[j].zero();
#pragma unroll
        for (int c = 0; c < kStages - 1; ++c) stage(c);
        for (int c = 0; c < nchunk; ++c) {
            asm volatile("cp.async.wait_group %0;" ::"n"(kStages - 2) : "memory");
            __syncthreads();   // chunk c is there; everybody has left chunk c - 1, whose stage is next
            stage(c + kStages - 1);
            const unsigned char* s = smem_raw + (size_t)(c % kStages) * kStageBytes;
            const unsigned char* sq = s + lane * kRowStride + warp * (KW * (int)sizeof(T));
            const unsigned char* sx = s + kRowT * kRowStride + warp * (KW * (int)sizeof(T));
            if constexpr (sizeof(T) == 4) {
#pragma unroll
                for (int k = 0; k < KW / 8; ++k) {
                    const ulonglong2* q = reinterpret_cast<const ulonglong2*>(sq) + 2 * k;
                    const ulonglong2 q0 = q[0], q1 = q[1];
#pragma unroll
                    for (int j = 0; j < TN; ++j) {
                        const ulonglong2* u = reinterpret_cast<const ulonglong2*>(sx + j * kRowStride) + 2 * k;
                        acc[j].add8(q0, q1, u[0], u[1]);
                    }
                }
            } else {
                double2 q[KW / 2];
#pragma unroll
                for (int k = 0; k < KW / 2; ++k) q[k] = reinterpret_cast<const double2*>(sq)[k];
#pragma unroll
                for (int j = 0; j < TN; ++j) {
                    const double2* u = reinterpret_cast<const double2*>(sx + j * kRowStride);
                    double v = q[0].x * u[0].x;
                    v = fma(q[0].y, u[0].y, v);
#pragma unroll
                    for (int k = 1; k < KW / 2; ++k) {
                        v = fma(q[k].x, u[k].x, v);
                        v = fma(q[k].y, u[k].y, v);
                    }
                    acc[j].lo += v;
                    if ((c & 3) == 3) {
                        acc[j].hi += acc[j].lo;
                        acc[j].lo = 0.0;
                    }
                }
            }
        }
        asm volatile("cp.async.wait_all;" ::: "memory");
        __syncthreads();
        // ---- the warps' sums side by side: [point][warp][row]
        if constexpr (sizeof(T) == 4) {
            float2* red = reinterpret_cast<float2*>(smem_raw);
#pragma unroll
            for (int j = 0; j < TN; ++j) red[(j * kWarps + warp) * 32 + lane] = acc[j].sum();
        } else {
            double* red = reinterpret_cast<double*>(smem_raw);
#pragma unroll
            for (int j = 0; j < TN; ++j) red[(j * kWarps + warp) * 32 + lane] = acc[j].hi + acc[j].lo;
        }
        __syncthreads();
        // ---- epilogue: warp w finishes points w, w + 8, ...; lane = row
        const int64_t row = row0 + lane;
        const bool in = row < n;
        const T bi = in && A.b ? static_cast<const T*>(A.b)[row] : T(0);
        const T pi = in && A.p ? static_cast<const T*>(A.p)[row] : T(0);
#pragma unroll
        for (int q = 0; q < NJ; ++q) {
            const int j = warp + kWarps * q;
            if (j >= np) break;
            const T xi = in ? x[(int64_t)j * n + row] : T(0);
            T* gp = A.g ? static_cast<T*>(A.g) + (p0 + j) * n + row : nullptr;
            double hj;
            if constexpr (sizeof(T) == 4) {
                const float2* red = reinterpret_cast<const float2*>(smem_raw) + j * kWarps * 32 + lane;
                float2 v = red[0];
#pragma unroll
                for (int w = 1; w < kWarps; ++w) v = csum_merge(v, red[32 * w]);
                // a + ae = v + b + p - p x,  g = 2 a - (b + p), the share of h = x a
                float c, ce, s, e1, a, e2, gs, e3;
                two_sum(bi, pi, c, ce);
                const float px = __fmul_rn(pi, xi), pe = fmaf(pi, xi, -px);
                two_sum(v.x, c, s, e1);
                two_sum(s, -px, a, e2);
                const float ae = ((v.y + ce) + (e1 + e2)) - pe;
                two_sum(2.f * a, -c, gs, e3);
                float gi = gs + (fmaf(2.f, ae, e3) - ce);
                const float vf = v.x + v.y;
                if (!isfinite(gi)) gi = 2.f * vf - 2.f * pi * xi + bi + pi;   // the pairs lose infinities
                if (in && gp) *gp = gi;
                const float th = __fmul_rn(xi, a);
                const float2 h1 = make_float2(th, fmaf(xi, ae, fmaf(xi, a, -th)));
                const float2 hs = csum_shfl_reduce(h1);
                hj = (double)hs.x + (double)hs.y;
                // FP64 where the pairs have left FP32's range: a share of h that is itself beyond it, or
                // shares (finite ones) whose sums are, on the way or in the end
                if (__any_sync(0xffffffffu, !isfinite(hj))) {
                    const bool ok = isfinite(h1.x) && isfinite(h1.y);
                    hj = dsum_shfl_reduce(ok ? (double)h1.x + (double)h1.y
                                             : (double)xi * ((double)vf + (double)bi + (double)pi - (double)pi * (double)xi));
                }
            } else {
                const double* red = reinterpret_cast<const double*>(smem_raw) + j * kWarps * 32 + lane;
                const double v = ((red[0] + red[32]) + (red[64] + red[96])) + ((red[128] + red[160]) + (red[192] + red[224]));
                if (in && gp) *gp = 2.0 * v - 2.0 * pi * xi + bi + pi;
                hj = dsum_shfl_reduce(xi * (v + bi + pi - pi * xi));
            }
            if (all) hsum[q] += hj;
            else if (A.part && lane == 0) A.part[(p0 + j) * A.tiles + t] = hj;
        }
        __syncthreads();   // the sums are read: the stages may be filled again
    }
    if (all && A.h && lane == 0) {
#pragma unroll
        for (int q = 0; q < NJ; ++q) {
            const int j = warp + kWarps * q;
            if (j < np) static_cast<T*>(A.h)[p0 + j] = (T)hsum[q];
        }
    }
}

// h of each point from its tiles' shares, one warp per point (a fixed order)
template <typename T>
__global__ void __launch_bounds__(kThreads) grad_h_kernel(const double* part, int tiles, int64_t batch, T* h)
{
    const int lane = threadIdx.x & 31;
    const int64_t r = (int64_t)blockIdx.x * kWarps + (threadIdx.x >> 5);
    if (r >= batch) return;
    double s = 0.0;
    for (int t = lane; t < tiles; t += 32) s += part[r * tiles + t];
    s = dsum_shfl_reduce(s);
    if (lane == 0) h[r] = (T)s;
}

static int grad_tiles(int64_t n) { return (int)((n + kRowT - 1) / kRowT); }

// scratch of one call: the shares of h
size_t grad_scratch_bytes(int64_t n, int64_t batch)
{
    const int tiles = grad_tiles(n);
    return tiles <= kTilesPerCta ? 0 : (size_t)batch * (size_t)tiles * sizeof(double);
}

template <typename T, int TN, int CP>
static cudaError_t grad_run(const GradArgs& a, cudaStream_t s)
{
    const size_t smem = std::max((size_t)kStages * (kRowT + TN) * kRowStride, (size_t)TN * kWarps * 32 * 8);
    cudaError_t e = cudaFuncSetAttribute(grad_kernel<T, TN, CP>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    const dim3 grid((unsigned)((a.batch + TN - 1) / TN), (unsigned)(a.tiles <= kTilesPerCta ? 1 : a.tiles));
    grad_kernel<T, TN, CP><<<grid, kThreads, smem, s>>>(a);
    return cudaGetLastError();
}

template <typename T, int TN>
static cudaError_t grad_run_aligned(const GradArgs& a, cudaStream_t s)
{
    // 16-byte copies where every row of Q and x starts on a 16-byte boundary, else one per element
    const bool al = a.n % (16 / (int)sizeof(T)) == 0 && reinterpret_cast<uintptr_t>(a.Q) % 16 == 0 &&
                    reinterpret_cast<uintptr_t>(a.x) % 16 == 0;
    return al ? grad_run<T, TN, 16>(a, s) : grad_run<T, TN, (int)sizeof(T)>(a, s);
}

// h and grad h of `batch` points on stream s; scratch: grad_scratch_bytes(n, batch) of device memory
// (may be null when that is 0 or h is not wanted)
cudaError_t launch_grad(const void* Q, const void* b, const void* p, const void* x, int64_t n, int64_t batch, int dtype,
                        void* h, void* g, void* scratch, int sms, cudaStream_t s)
{
    GradArgs a;
    a.Q = Q;
    a.b = b;
    a.p = p;
    a.x = x;
    a.g = g;
    a.h = h;
    a.part = h ? static_cast<double*>(scratch) : nullptr;
    a.n = (int32_t)n;
    a.batch = batch;
    a.tiles = grad_tiles(n);
    // points per CTA: the width whose last wave of CTAs wastes least, counting a CTA's staging of
    // its rows as three points' arithmetic (FP32; half a point's in FP64, whose products take
    // longer than the copies).  Device time by width 1, 2, 4, 8 (and 16, which is never the best):
    // n = 1000, 64 points FP32 32, 23, 16, 14 (15) us; n = 8192, 128 points 2.86, 1.72, 1.18, 0.97
    // (0.99) ms; n = 4099, one point 15, 18, 22, 32 us; n = 1001, 37 points FP64 92, 85, 123, 160 us
    const bool f64 = dtype == 1;
    int tn = 1;
    double best = 1e300;
    for (int c = 1; c <= 8; c *= 2) {
        const int64_t ctas = (a.tiles <= kTilesPerCta ? 1 : a.tiles) * ((batch + c - 1) / c);
        const double cost = (double)((ctas + sms - 1) / sms) * (c + (f64 ? 0.5 : 3.0));
        if (cost <= best) {
            best = cost;
            tn = c;
        }
    }
    cudaError_t e;
    if (f64) {
        e = tn == 1 ? grad_run_aligned<double, 1>(a, s)
            : tn == 2 ? grad_run_aligned<double, 2>(a, s)
            : tn == 4 ? grad_run_aligned<double, 4>(a, s) : grad_run_aligned<double, 8>(a, s);
    } else {
        e = tn == 1 ? grad_run_aligned<float, 1>(a, s)
            : tn == 2 ? grad_run_aligned<float, 2>(a, s)
            : tn == 4 ? grad_run_aligned<float, 4>(a, s) : grad_run_aligned<float, 8>(a, s);
    }
    if (e != cudaSuccess) return e;
    if (h && a.tiles > kTilesPerCta) {
        const unsigned blocks = (unsigned)((batch + kWarps - 1) / kWarps);
        if (f64) grad_h_kernel<double><<<blocks, kThreads, 0, s>>>(a.part, a.tiles, batch, (double*)h);
        else grad_h_kernel<float><<<blocks, kThreads, 0, s>>>(a.part, a.tiles, batch, (float*)h);
        e = cudaGetLastError();
    }
    return e;
}

// ---------------------------------------------------------------------------------
// Vector-Jacobian product of h (backward of the penalized objective) for `batch` points:
//   gx[r][i] = go[r] g[r][i],  gp[i] = sum_r go[r] (x_ri - x_ri^2),  gb[i] = sum_r go[r] x_ri
// A CTA takes 16 coordinates.  Its threads read 64 points' pieces at a time (all loads in flight
// together), write gx and leave x and go in shared memory as FP64, where one warp adds the chunk's
// terms to the two sums in order r = 0, 1, ... (lanes 0-15 gp's, 16-31 gb's) while the others go on
// with the next chunk.  Bound: the FP64 pipe, two instructions a point; all 32 lanes of the adding
// warp carry a sum, and the conversions are spread over the other warps.
constexpr int kVjpRows = 64, kVjpCols = 16;

template <typename T>
__global__ void __launch_bounds__(kThreads) penalized_vjp_kernel(const T* x, const T* g, const T* go, int64_t n, int64_t batch,
                                                                 T* gx, T* gp, T* gb)
{
    __shared__ double sx[2][kVjpRows][kVjpCols];
    __shared__ double sw[2][kVjpRows];
    constexpr int kPass = kThreads / kVjpCols, U = kVjpRows / kPass;
    const int col = threadIdx.x % kVjpCols, rr = threadIdx.x / kVjpCols;
    const int64_t i = (int64_t)blockIdx.x * kVjpCols + col;
    const bool in = i < n;
    const bool sums = gp || gb;
    const bool pen = (threadIdx.x & 31) < kVjpCols;   // warp 0: this lane's sum is gp's
    double acc = 0.0;
    int buf = 0;
    for (int64_t r0 = 0; r0 < batch; r0 += kVjpRows, buf ^= 1) {
        T xv[U], gv[U], wv[U];
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const int64_t r = r0 + rr + kPass * u;
            const bool ok = r < batch;
            wv[u] = ok ? go[r] : T(0);
            xv[u] = ok && in && sums ? x[r * n + i] : T(0);
            gv[u] = ok && in && gx ? g[r * n + i] : T(0);
        }
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const int64_t r = r0 + rr + kPass * u;
            if (gx && in && r < batch) gx[r * n + i] = wv[u] * gv[u];
            if (sums) {
                sx[buf][rr + kPass * u][col] = (double)xv[u];
                if (col == 0) sw[buf][rr + kPass * u] = (double)wv[u];
            }
        }
        if (!sums) continue;
        __syncthreads();   // (one barrier a chunk: a buffer is written again two chunks later)
        if (threadIdx.x < 32) {
            const int m = (int)min((int64_t)kVjpRows, batch - r0);
#pragma unroll 8
            for (int q = 0; q < m; ++q) {
                const double xi = sx[buf][q][col];
                acc = fma(sw[buf][q], pen ? fma(-xi, xi, xi) : xi, acc);
            }
        }
    }
    if (threadIdx.x < 32 && in) {
        if (pen && gp) gp[i] = (T)acc;
        if (!pen && gb) gb[i] = (T)acc;
    }
}

cudaError_t launch_penalized_vjp(const void* x, const void* g, const void* go, int64_t n, int64_t batch, int dtype,
                                 void* gx, void* gp, void* gb, cudaStream_t s)
{
    const unsigned blocks = (unsigned)((n + kVjpCols - 1) / kVjpCols);
    if (dtype == 1)
        penalized_vjp_kernel<double><<<blocks, kThreads, 0, s>>>((const double*)x, (const double*)g, (const double*)go, n,
                                                                 batch, (double*)gx, (double*)gp, (double*)gb);
    else
        penalized_vjp_kernel<float><<<blocks, kThreads, 0, s>>>((const float*)x, (const float*)g, (const float*)go, n, batch,
                                                                (float*)gx, (float*)gp, (float*)gb);
    return cudaGetLastError();
}

}  // namespace ubqp
