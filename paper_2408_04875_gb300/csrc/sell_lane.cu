// FP32 lanes on the sliced storage, each on its own group of CTAs, many steps of Alg. 3 per
// cooperative launch.  The groups and the lanes they run are those of solo.cu; this kernel has
// the two steps that a solve repeats most written for latency:
//
//   Alg. 2 (PABB) step    products, row epilogue, ONE exchange, decision, whole x_{k+1}
//   LOBPCG iteration      products, Gram sums, one exchange, Rayleigh-Ritz, own rows' update,
//                         a second exchange of the next input u
//
// What bounds a step is a chain of dependent latencies, not bytes: a lane of n = 2500 has 4 MB
// of stored entries on 79 CTAs.  Therefore
//   * a CTA keeps the entries of its slices in shared memory for the whole launch (as many
//     slices as fit, the rest is read from L2), repacked so that a thread's groups of four
//     values and columns are one 16-byte and one 8-byte load;
//   * the rows a CTA owns live in registers of the warp that finishes them (x_{k-1}, g_{k-1},
//     d - p, d + b'; for the eigen-solver its six vectors), x_k and g_k of every row in shared
//     memory;
//   * CTAs exchange a step's results in one hop, a slice's 32 gradient entries and its partial sums
//     as tagged words (lane_words.cuh).  Words alternate between two buffers by the step's parity: a
//     CTA stores the words of step j + 2 only after it has received all of step j + 1, and a CTA
//     sends those only after it has read all of step j;
//   * the scalar step (KKT test, BB step) is taken by every thread from the reduced sums,
//     without a round through one thread and shared memory.
//
// Measured (cycles per Alg. 2 step at n = 500, 1000 in the mixed batch of twelve, 2500; one group
// of 16, 11, 79 CTAs): products 710, 3000, 1940; epilogue 1480, 1800, 1310; exchange 2290, 2700,
// 3240; decision 390, 400, 690; x_{k+1} 150, 160, 330.  Device time of whole runs against the
// barrier-and-records form this replaced: n = 50 to the end 13.7 -> 6.0 ms, n = 500 to the end
// 303 -> 136 ms, n = 2500 (40 subproblems) 82 -> 42 ms, the batch of twelve 241 -> 116 ms.
//
// The arithmetic and its order are those of the other schedulers (item_rows_sell's shares,
// row_epilogue, the record of a 32-row block, reduce_partials, decide, lane_apply), so a lane's
// results do not depend on the kernel that runs it.  All other phases run the shared functions
// with group barriers.  Every wait is bounded; when one runs out the CTA sets the error flag
// and leaves, and the others leave at their own next wait.
//
// Lane vectors written by one CTA are read by others within the launch: plain loads of this
// file are cached in L2 only (-dlcm=cg).
#include "lane_words.cuh"

namespace ubqp {

namespace {

constexpr int kRowWords = 16;                 // 32 values, two to a word
constexpr int kRecWords = 5;                  // the ten numbers of an Alg. 2 record
constexpr int kStepWords = kRowWords + kRecWords;
static_assert(kGramWords <= kStepWords && kSellWordsPerBlock == 2 * (kStepWords + kRowWords), "exchange words per block");

// sum of the shared-memory copy of one share (cnt entries of a slice, thread = row): groups of four
// products as FMA chains, added to a compensated sum, the up to seven entries left over one by
// one; the operations of item_rows_sell.  (The missing ones of the seven add zero, which changes
// nothing and costs less than branching around them.)
__device__ __forceinline__ float2 share_smem(const float* mv, const uint16_t* mc, int cnt, const float* su, int lane)
{
    const int ng = (cnt >> 3) * 2, rest = cnt & 7;
    const float4* v4 = reinterpret_cast<const float4*>(mv) + lane;
    const uint2* c4 = reinterpret_cast<const uint2*>(mc) + lane;
    const float* v1 = mv + 128 * ng + lane;
    const uint16_t* c1 = mc + 128 * ng + lane;
    float r[7];
#pragma unroll
    for (int e = 0; e < 7; ++e) r[e] = e < rest ? __fmul_rn(v1[32 * e], su[c1[32 * e]]) : 0.f;
    float2 acc = make_float2(0.f, 0.f);
    auto group = [&](float4 q, uint2 c) {
        float t = __fmul_rn(q.x, su[c.x & 0xffffu]);
        t = fmaf(q.y, su[c.x >> 16], t);
        t = fmaf(q.z, su[c.y & 0xffffu], t);
        return fmaf(q.w, su[c.y >> 16], t);
    };
    int j = 0;
    for (; j + 4 <= ng; j += 4) {
        float4 q[4];
        uint2 c[4];
        float t[4];
#pragma unroll
        for (int h = 0; h < 4; ++h) {
            q[h] = v4[32 * (j + h)];
            c[h] = c4[32 * (j + h)];
        }
#pragma unroll
        for (int h = 0; h < 4; ++h) t[h] = group(q[h], c[h]);
#pragma unroll
        for (int h = 0; h < 4; ++h) csum_add(acc, t[h]);
    }
    if (j < ng) {   // two groups (ng is even)
        const float t0 = group(v4[32 * j], c4[32 * j]), t1 = group(v4[32 * (j + 1)], c4[32 * (j + 1)]);
        csum_add(acc, t0);
        csum_add(acc, t1);
    }
#pragma unroll
    for (int e = 0; e < 7; ++e) csum_add(acc, r[e]);
    return acc;
}

// the same from the stored slice (L2), sixteen entries of the share in flight per thread
__device__ __forceinline__ float2 share_gmem(const float* V, const uint16_t* C, int k0, int k1, const float* su)
{
    V += 32 * (int64_t)k0;
    C += 32 * (int64_t)k0;
    const int ng = ((k1 - k0) >> 3) * 2;
    float2 acc = make_float2(0.f, 0.f);
    int j = 0;
    for (; j + 4 <= ng; j += 4) {
        float q[16];
        int c[16];
#pragma unroll
        for (int e = 0; e < 16; ++e) {
            q[e] = __ldg(V + 32 * (4 * j + e));
            c[e] = __ldg(C + 32 * (4 * j + e));
        }
#pragma unroll
        for (int h = 0; h < 4; ++h) {
            float t = __fmul_rn(q[4 * h], su[c[4 * h]]);
            t = fmaf(q[4 * h + 1], su[c[4 * h + 1]], t);
            t = fmaf(q[4 * h + 2], su[c[4 * h + 2]], t);
            t = fmaf(q[4 * h + 3], su[c[4 * h + 3]], t);
            csum_add(acc, t);
        }
    }
    for (; j < ng; ++j) {
        float q[4];
        int c[4];
#pragma unroll
        for (int e = 0; e < 4; ++e) {
            q[e] = __ldg(V + 32 * (4 * j + e));
            c[e] = __ldg(C + 32 * (4 * j + e));
        }
        float t = __fmul_rn(q[0], su[c[0]]);
        t = fmaf(q[1], su[c[1]], t);
        t = fmaf(q[2], su[c[2]], t);
        t = fmaf(q[3], su[c[3]], t);
        csum_add(acc, t);
    }
    for (int k = 4 * ng; k < k1 - k0; ++k) csum_add(acc, __fmul_rn(__ldg(V + 32 * k), su[__ldg(C + 32 * k)]));
    return acc;
}

// the slices of a lane that this CTA owns: rank, rank + nc, ... (`one`: every slice of a lane of
// one block, the CTA's warps shared out over them)
struct Slices {
    int rank, nc, n;
    __device__ __forceinline__ int at(int b) const { return rank + b * nc; }
};

// one slice of a CTA: first stored entry, width, and where its copy in shared memory starts (-1: none)
struct SliceAt {
    int64_t base;
    int width, at;
};
// one warp's share of a slice: first entry and count, and where the copy's values (in floats) and
// columns (in 16-bit units) start
struct __align__(16) ShareAt {
    int k0, cnt, v, c;
};

}  // namespace

// kPer CTAs share an SM (1: up to 255 registers a thread; 2: 128).  kTight: what the owner of a slice
// leaves for the other warps (the eigen-solver's vectors at its 32 rows, or the rows' products in FP64)
// lies over the slice's shares, which the owner has read by then, instead of in 8 KB of its own.  Two CTAs
// on an SM then hold vectors up to ld = 12,416 instead of 11,392; shorter ones keep the other form,
// which is up to 1.5 % faster on lanes of one CTA.  Three and four lanes of n = 12000, density 0.002,
// two subproblems, device time: 5.0 and 5.7 ms, against 7.8 and 8.8 ms on solo.cu.
template <int kPer, bool kTight>
__global__ void __launch_bounds__(kThreads, kPer) sell_lane_kernel(SoloArgs A)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    __shared__ double s_sv[kTight ? 1 : kThreads];
    __shared__ LaneState S;
    __shared__ Partial R;
    __shared__ Decision D;
    __shared__ int s_ok, s_g;
    __shared__ unsigned long long s_gen0;
    __shared__ float2 s_share[kSoloMaxSl * kThreads];
    __shared__ WarpRed s_red[kWarps];
    __shared__ WarpRed s_rec[kSoloMaxSl];   // records of a one-CTA group
    __shared__ float s_basis[kTight ? 1 : kWarps][6 * 32];   // the eigen-solver's vectors at the CTA's rows
    __shared__ SliceAt s_sl[kWarps];
    __shared__ ShareAt s_sh[kWarps][kWarps];
    __shared__ __align__(16) LaneDev sL;
    __shared__ Params sP;

    // ---- this CTA's group, its rank in the group and the group's barrier (as in solo.cu)
    if (threadIdx.x == 0) {
        int lo = 0, hi = A.ngroups - 1;   // the last group whose first CTA is <= blockIdx.x
        while (lo < hi) {
            const int mid = (lo + hi + 1) >> 1;
            if (A.gcta[mid] <= (int)blockIdx.x) lo = mid;
            else hi = mid - 1;
        }
        s_g = lo;
        s_ok = 1;
    }
    __syncthreads();
    const int g = s_g;
    const int c0 = A.gcta[g];
    const int nc = A.gcta[g + 1] - c0;
    const int rank = (int)blockIdx.x - c0;
    unsigned long long* bar = reinterpret_cast<unsigned long long*>(A.bar + (size_t)g * kSoloBarStride);
    if (threadIdx.x == 0) {
        s_gen0 = ld_acquire_u64(bar) / (unsigned long long)nc;
        sP = A.P;
        if (rank != 0) sP.hist = nullptr;
    }
    __syncthreads();
    unsigned long long gen = s_gen0;
    const Params& P = sP;
    const int tid = (int)threadIdx.x, lane = tid & 31, warp = tid >> 5;
    int steps_left = A.budget;

    for (int li = A.gfirst[g]; li < A.gfirst[g + 1] && steps_left > 0; ++li) {
        const int lane_id = A.glanes[li];
        __syncthreads();   // shared state of the previous lane no longer in use
        if (tid < (int)(sizeof(LaneDev) / 8))
            reinterpret_cast<int2*>(&sL)[tid] = __ldg(reinterpret_cast<const int2*>(A.lane + lane_id) + tid);
        __syncthreads();
        const LaneDev& L = sL;
        if (tid == 0) S = *L.st;
        __syncthreads();
        if (S.phase == PH_DONE) continue;
        const int n = L.n, ld = L.ld, nblk = L.nblk;
        const bool pabb = L.method == 0;
        const int nq4 = ld >> 2;
        const int qa = (int)((int64_t)nq4 * rank / nc), qb = (int)((int64_t)nq4 * (rank + 1) / nc);
        const int ia = min(4 * qa, n), ib = min(4 * qb, n);
        float* su = reinterpret_cast<float*>(smem_raw);   // the product's input (x_k in Alg. 2)
        float* sg = su + ld;                              // g_k of every row
        float* vec = L.vec;

        // ---- this CTA's slices.  A lane of one block (up to 256 rows, one CTA): its 32-row slices
        // side by side, wps warps each.  Otherwise one slice per block, eight warps each.
        const bool one = nblk == 1 && nc == 1 && A.rows_per_item >= n;
        const int wps = one ? L.spwps : kWarps;
        Slices sl{rank, nc, 0};
        if (one) sl = Slices{0, 1, (n + 31) >> 5};
        else sl.n = rank < nblk ? (nblk - rank + nc - 1) / nc : 0;

        // ---- as many of them as fit in shared memory: thread r of a warp's share takes its entries
        // in groups of four (one 16-byte and one 8-byte load), the remainder one by one.  What a
        // warp needs of each slice (its share's bounds, where the entries lie) is kept in s_sl.
        if (tid < sl.n) {
            const int64_t o0 = L.spo[sl.at(tid)];
            s_sl[tid] = SliceAt{o0, (int)((L.spo[sl.at(tid) + 1] - o0) >> 5), 0};
        }
        __syncthreads();
        unsigned char* mat = smem_raw + 2 * (size_t)ld * sizeof(float);
        if (tid == 0) {
            int used = 0;
            for (int b = 0; b < sl.n; ++b) {
                const int bytes = s_sl[b].width * 32 * 6;
                s_sl[b].at = used + bytes <= A.mat_bytes ? used : -1;   // -1: read from L2
                if (s_sl[b].at >= 0) used += bytes;
            }
        }
        __syncthreads();
        for (int b = 0; b < sl.n; ++b) {
            const SliceAt q = s_sl[b];
            if (warp >= wps) continue;   // (with wps < 8 the other warps idle here)
            const int k0 = q.width * warp / wps, cnt = q.width * (warp + 1) / wps - k0;
            const int v0 = q.at / 4 + 32 * k0, c0 = q.at / 2 + 64 * q.width + 32 * k0;
            if (lane == 0) s_sh[b][warp] = ShareAt{k0, cnt, v0, c0};
            if (q.at < 0) continue;
            float* mv = reinterpret_cast<float*>(mat) + v0;
            uint16_t* mc = reinterpret_cast<uint16_t*>(mat) + c0;
            const float* V = L.spv + q.base + 32 * (int64_t)k0 + lane;
            const uint16_t* C = L.spc + q.base + 32 * (int64_t)k0 + lane;
            const int ng = (cnt >> 3) * 2;
            for (int e = 0; e < cnt; ++e) {
                const int at = e < 4 * ng ? 32 * (e & ~3) + 4 * lane + (e & 3) : 32 * e + lane;
                mv[at] = __ldg(V + 32 * e);
                mc[at] = __ldg(C + 32 * e);
            }
        }
        // ---- the row this thread finishes: row `tid` of a one-block lane, or row `lane` of the
        // slice of this warp
        const bool own_warp = one ? 32 * warp < n : warp < sl.n;
        const int row = one ? tid : 32 * sl.at(warp) + lane;
        const bool own = own_warp && row < n;
        const int rc = own ? row : n - 1;
        const float2* my_sh = s_share + (one ? warp * wps * 32 : warp * kThreads) + lane;   // share p at 32 p

        // where the owner of slice b leaves its vectors and its rows' products.  A lane of one block has its
        // shares in the first kThreads entries of s_share and the rest free.
        constexpr int kOwn = 6 * 32 / 2;   // float2 entries
        static_assert(kThreads + kWarps * kOwn <= kSoloMaxSl * kThreads && kOwn <= kThreads, "room for what the owners leave");
        auto basis = [&](int b) -> float* {
            if constexpr (kTight) return reinterpret_cast<float*>(s_share + (one ? kThreads + b * kOwn : b * kThreads));
            else return s_basis[b];
        };
        auto prods = [&](int b) -> double* {
            if constexpr (kTight) return reinterpret_cast<double*>(s_share + (one ? kThreads + b * 32 : b * kThreads));
            else return s_sv + 32 * b;
        };

        // the products of every slice of this CTA, shares into s_share; then v of the own row
        auto share = [&](int b, int part) -> float2 {
            const ShareAt h = s_sh[b][part];
            if (s_sl[b].at < 0) {
                const int64_t o0 = s_sl[b].base + lane;
                return share_gmem(L.spv + o0, L.spc + o0, h.k0, h.k0 + h.cnt, su);
            }
            return share_smem(reinterpret_cast<const float*>(mat) + h.v, reinterpret_cast<const uint16_t*>(mat) + h.c, h.cnt,
                              su, lane);
        };
        auto products = [&]() {
            if (one) {
                const int q = warp / wps, part = warp - q * wps;
                s_share[warp * 32 + lane] = q < sl.n ? share(q, part) : make_float2(0.f, 0.f);
            } else {
                for (int b = 0; b < sl.n; ++b) s_share[b * kThreads + warp * 32 + lane] = share(b, warp);
            }
        };
        auto own_product = [&]() -> float {   // the shares merged in share order
            float2 a = my_sh[0];
            if (wps == kWarps) {
                float2 h[kWarps];
#pragma unroll
                for (int p = 1; p < kWarps; ++p) h[p] = my_sh[32 * p];
#pragma unroll
                for (int p = 1; p < kWarps; ++p) a = csum_merge(a, h[p]);
            } else {
                for (int p = 1; p < wps; ++p) a = csum_merge(a, my_sh[32 * p]);
            }
            return a.x + a.y;
        };
        auto count_bytes = [&]() {   // profiling only
            if (P.bytes && own_warp && lane == 0 && (!one || warp == 0)) {
                const int blk = one ? 0 : sl.at(warp), row0 = one ? 0 : 32 * blk;
                atomicAdd(P.bytes, solo_item_bytes(L, blk, row0, one ? n : min(32, n - row0)));
            }
        };
        const int nw = one ? (n + 31) >> 5 : min(kWarps, (nblk + 31) >> 5);   // warps with records
        const int gw0 = nw < kWarps ? nw : 0;   // the others collect the gradient
        ulonglong2* const xa = L.xch;                                            // step words: [2][nblk][21]
        ulonglong2* const xb = L.xch + (size_t)2 * nblk * kStepWords;               // row words: [2][nblk][16]
        __syncthreads();

        for (; steps_left > 0; ) {
            const int ph = S.phase;
            if (ph == PH_DONE) break;
            if (ph == PH_INNER && pabb) {
                // ================= Alg. 2 until the subproblem or the launch's budget ends
                int k = S.k;
                const int k_in = k;
                float rho = S.rho, alpha = S.alpha;
                uint32_t upd = (uint32_t)S.updates;
                item_load_u(L, su);
                float r_dmp = 0.f, r_ts = 0.f, r_xp = 0.f, r_g = 0.f;
                if (own_warp) {
                    r_dmp = vec[(size_t)V_DMP * ld + rc];
                    r_ts = L.tsum[rc];
                    if (k >= 1) {
                        r_xp = vec[(size_t)V_XPREV * ld + rc];
                        r_g = vec[(size_t)g_buf(k) * ld + rc];
                    }
                }
                const float tol = P.tol_inner, qmax = L.qmax_off, amin = P.alpha_min, amax = P.alpha_max;
                const int kmax = P.max_inner, tlen = L.trace_len;
                int exit_code = -1;
                float2 t3[3];
                float tm[4];
                __syncthreads();
                while (steps_left > 0) {
                    products();
                    __syncthreads();
                    const uint32_t tag = 2u * upd + 1u;
                    ulonglong2* const w = xa + (size_t)(upd & 1u) * nblk * kStepWords;
                    if (own_warp) {
                        const float v = own_product();
                        const float x = su[rc];
                        float gk = fmaf(r_dmp, 2.f * x - 1.f, fmaf(2.f, v, r_ts));
                        float2 s[3];
                        float m[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
                        for (int t = 0; t < 3; ++t) s[t] = make_float2(0.f, 0.f);
                        if (own) {
                            if (k >= 1) {
                                const float sd = x - r_xp;
                                const float y = gk - r_g;
                                csum_add(s[0], sd * sd);
                                csum_add(s[1], sd * y);
                                csum_add(s[2], y * y);
                            } else {
                                m[1] = fmaxf(0.f, fabsf(r_dmp));
                                m[2] = fmaxf(0.f, fabsf(vec[(size_t)V_BBAR * ld + rc]));
                                m[3] = fmaxf(0.f, L.oabs[rc] + fabsf(r_dmp));
                            }
                            const float viol =
                                (x > 0.f && x < 1.f) ? fabsf(gk) : (x <= 0.f ? fmaxf(-gk, 0.f) : fmaxf(gk, 0.f));
                            m[0] = fmaxf(0.f, viol);
                        } else {
                            gk = 0.f;
                        }
                        r_xp = x;
                        r_g = gk;
                        if (k >= 1) butterfly<3, 1>(s, m);   // the other maxima belong to step 0, the sums to the rest
                        else butterfly<0, 4>(s, m);
                        if (nc == 1) {
                            sg[row] = gk;   // row < 32 * slices <= ld
                            WarpRed& r = one ? s_red[warp] : s_rec[warp];
                            if (lane == 0) {
#pragma unroll
                                for (int t = 0; t < 3; ++t) r.s[t] = s[t];
#pragma unroll
                                for (int t = 0; t < 4; ++t) r.m[t] = m[t];
                            }
                        } else {
                            float2 p = row_word(gk, lane);
                            if (lane == kRowWords) p = s[0];
                            if (lane == kRowWords + 1) p = s[1];
                            if (lane == kRowWords + 2) p = s[2];
                            if (lane == kRowWords + 3) p = make_float2(m[0], m[1]);
                            if (lane == kRowWords + 4) p = make_float2(m[2], m[3]);
                            publish(w + (size_t)sl.at(warp) * kStepWords, lane < kStepWords, lane, p, tag);
                        }
                        count_bytes();
                    }
                    // ---- every row's g_k into sg, the block records reduced in reduce_partials' order
                    // (the barrier also keeps the other warps from polling, and so from taking issue slots,
                    // while the epilogue runs)
                    __syncthreads();
                    if (!one) {
                        if (warp < nw) {
                            float2 s[3];
                            float m[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
                            for (int t = 0; t < 3; ++t) s[t] = make_float2(0.f, 0.f);
                            for (int blk0 = 32 * warp; blk0 < nblk; blk0 += kThreads) {   // whole warps
                                const bool mine = blk0 + lane < nblk;
                                const int blk = min(blk0 + lane, nblk - 1);
                                float2 p[3];
                                float pm[4];
                                if (nc == 1) {
#pragma unroll
                                    for (int t = 0; t < 3; ++t) p[t] = s_rec[blk].s[t];
#pragma unroll
                                    for (int t = 0; t < 4; ++t) pm[t] = s_rec[blk].m[t];
                                } else {
                                    const ulonglong2* src = w + (size_t)blk * kStepWords + kRowWords;
                                    const ulonglong2* const pp[kRecWords] = {src, src + 1, src + 2, src + 3, src + 4};
                                    ulonglong2 v[kRecWords];
                                    wait_words<kRecWords>(A, pp, tag, v, &s_ok);
#pragma unroll
                                    for (int t = 0; t < 3; ++t) p[t] = word_values(v[t]);
                                    const float2 m01 = word_values(v[3]), m23 = word_values(v[4]);
                                    pm[0] = m01.x;
                                    pm[1] = m01.y;
                                    pm[2] = m23.x;
                                    pm[3] = m23.y;
                                }
                                if (mine) {
#pragma unroll
                                    for (int t = 0; t < 3; ++t) s[t] = csum_merge(s[t], p[t]);
#pragma unroll
                                    for (int t = 0; t < 4; ++t) m[t] = fmaxf(m[t], pm[t]);
                                }
                            }
                            __syncwarp();
                            if (k >= 1) butterfly<3, 1>(s, m);   // the other maxima belong to step 0, the sums to the rest
                            else butterfly<0, 4>(s, m);
                            if (lane == 0) {
#pragma unroll
                                for (int t = 0; t < 3; ++t) s_red[warp].s[t] = s[t];
#pragma unroll
                                for (int t = 0; t < 4; ++t) s_red[warp].m[t] = m[t];
                            }
                        }
                        if (nc > 1 && warp >= gw0)
                            gather_rows<kRowWords>(A, w, kStepWords, nblk, tag, sg, tid - 32 * gw0, kThreads - 32 * gw0, &s_ok);
                        __syncthreads();
                    }
                    if (!s_ok) break;
                    // ---- the scalar step, by every thread
#pragma unroll
                    for (int t = 0; t < 3; ++t) t3[t] = s_red[0].s[t];
#pragma unroll
                    for (int t = 0; t < 4; ++t) tm[t] = s_red[0].m[t];
                    for (int q = 1; q < nw; ++q) {
#pragma unroll
                        for (int t = 0; t < 3; ++t) t3[t] = csum_merge(t3[t], s_red[q].s[t]);
#pragma unroll
                        for (int t = 0; t < 4; ++t) tm[t] = fmaxf(tm[t], s_red[q].m[t]);
                    }
                    const float rho_k = rho, alpha_k = alpha;
                    exit_code = inner_scalar(0, k, kmax, tol, amin, amax, qmax, tm, csum_value(t3[0]),
                                             csum_value(t3[1]), csum_value(t3[2]), rho, alpha);
                    if (exit_code >= 0) {   // the general update takes the step from the state before it
                        rho = rho_k;
                        alpha = alpha_k;
                        break;
                    }
                    if (k < tlen) {
                        for (int i = ia + tid; i < ib; i += kThreads) L.trace_x[(size_t)k * n + i] = su[i];
                        if (rank == 0 && tid == 0 && L.trace_alpha) L.trace_alpha[k] = alpha;
                        __syncthreads();
                    }
                    // x_{k+1} = P(x_k - alpha g_k), every row, in place
                    {
                        float4* x4 = reinterpret_cast<float4*>(su);
                        const float4* g4 = reinterpret_cast<const float4*>(sg);
                        for (int q = tid; q < nq4; q += kThreads) {
                            float4 xv = x4[q];
                            const float4 gv = g4[q];
                            xv.x = fminf(fmaxf(fmaf(-alpha, gv.x, xv.x), 0.f), 1.f);
                            xv.y = fminf(fmaxf(fmaf(-alpha, gv.y, xv.y), 0.f), 1.f);
                            xv.z = fminf(fmaxf(fmaf(-alpha, gv.z, xv.z), 0.f), 1.f);
                            xv.w = fminf(fmaxf(fmaf(-alpha, gv.w, xv.w), 0.f), 1.f);
                            x4[q] = xv;
                        }
                    }
                    ++k;
                    ++upd;
                    --steps_left;
                    __syncthreads();
                }
                if (!s_ok) break;
                if (tid == 0) {
                    const int done = k - k_in;
                    S.k = k;
                    S.rho = rho;
                    S.alpha = alpha;
                    S.inner_iters += done;
                    S.inner_steps += done;
                    S.updates += done;
                }
                if (exit_code < 0) {
                    // the launch ends inside the subproblem: x_k (also the next u) and, per owned row,
                    // x_{k-1} and g_{k-1} back to the lane
                    for (int i = ia + tid; i < ib; i += kThreads) {
                        vec[(size_t)V_X * ld + i] = su[i];
                        vec[(size_t)V_U * ld + i] = su[i];
                    }
                    if (own) {
                        vec[(size_t)V_XPREV * ld + row] = r_xp;
                        vec[(size_t)g_buf(k) * ld + row] = r_g;
                    }
                    break;
                }
                // the subproblem has ended: the general update from x_k
                for (int i = ia + tid; i < ib; i += kThreads) vec[(size_t)V_X * ld + i] = su[i];
                if (tid == 0) {
#pragma unroll
                    for (int t = 0; t < 12; ++t) R.s[t] = t < 3 ? t3[t < 3 ? t : 0] : make_float2(0.f, 0.f);
#pragma unroll
                    for (int t = 0; t < 6; ++t) R.m[t] = t < 4 ? tm[t < 4 ? t : 0] : 0.f;
                    R.f = 0.0;
                    decide(L, S, R, P, D);
                }
                __syncthreads();
            } else if (ph == PH_LOB) {
                // ================= LOBPCG until it converges or the launch's budget ends
                item_load_u(L, su);
                float r_d = 0.f, r_dmp = 0.f, r_t = 0.f, lx = 0.f, lax = 0.f, lp = 0.f, lap = 0.f, lw = 0.f;
                if (own) {
                    r_d = vec[(size_t)V_D * ld + row];
                    r_dmp = vec[(size_t)V_DMP * ld + row];
                    r_t = vec[(size_t)V_T * ld + row];
                    lx = vec[(size_t)V_LX * ld + row];
                    lax = vec[(size_t)V_LAX * ld + row];
                    lp = vec[(size_t)V_LP * ld + row];
                    lap = vec[(size_t)V_LAP * ld + row];
                    lw = vec[(size_t)V_LW * ld + row];
                }
                uint32_t upd = (uint32_t)S.updates;
                bool more = true;
                __syncthreads();
                while (steps_left > 0) {
                    products();
                    __syncthreads();
                    ulonglong2* const w = xa + (size_t)(upd & 1u) * nblk * kStepWords;
                    const uint32_t tag = 2u * upd + 1u;
                    float aw = 0.f;
                    if (own_warp) {
                        const float v = own_product();
                        if (own && r_d != 0.f) aw = r_d * fmaf(r_dmp, r_d * lw, v);
                        if constexpr (kTight) __syncwarp();   // the shares are read
                        float* q = basis(warp) + lane;   // rows beyond n hold zeros
                        q[0] = lx;
                        q[32] = lax;
                        q[64] = lw;
                        q[96] = aw;
                        q[128] = lp;
                        q[160] = lap;
                        count_bytes();
                    }
                    __syncthreads();
                    // ---- the twelve Gram sums of every slice, two per warp and turn
                    for (int task = warp; task < 6 * sl.n; task += kWarps) {
                        const int b = task / 6, t = 2 * (task - 6 * b);
                        const float* q = basis(b) + lane;
                        float2 s[2];
#pragma unroll
                        for (int h = 0; h < 2; ++h) {
                            const int l = (int)(kGramLeft >> (4 * (t + h))) & 15, r = (int)(kGramRight >> (4 * (t + h))) & 15;
                            s[h] = make_float2(0.f, 0.f);
                            csum_add(s[h], q[32 * l] * q[32 * r]);
                        }
                        butterfly<2, 0>(s, nullptr);
                        if (nc == 1) {
                            WarpRed& r = one ? s_red[b] : s_rec[b];
                            if (lane < 2) r.s[t + lane] = lane ? s[1] : s[0];
                        } else {
                            publish(w + (size_t)sl.at(b) * kStepWords + t, lane < 2, lane, lane ? s[1] : s[0], tag);
                        }
                    }
                    if (nc == 1) __syncthreads();
                    // ---- over the blocks, in reduce_partials' order: block b belongs to group b / 32 (mod 8),
                    // the groups' sums are merged in order
                    if (one) {
                        if (tid < 12) {
                            float2 v = s_red[0].s[tid];
                            for (int q = 1; q < nw; ++q) v = csum_merge(v, s_red[q].s[tid]);
                            R.s[tid] = v;
                        }
                    } else if (warp < 6) {
                        const int t = 2 * warp;
                        float2 sum[2];
                        for (int g0 = 0; g0 < nw; g0 += 4) {
                            float2 s[8];   // groups g0 .. g0 + 3, two sums each
#pragma unroll
                            for (int h = 0; h < 8; ++h) s[h] = make_float2(0.f, 0.f);
                            for (int blk0 = 32 * g0; blk0 < nblk; blk0 += kThreads) {
                                float2 v[8];
                                if (nc == 1) {
#pragma unroll
                                    for (int h = 0; h < 4; ++h) {
                                        const int blk = min(blk0 + 32 * h + lane, nblk - 1);
                                        v[2 * h] = s_rec[blk].s[t];
                                        v[2 * h + 1] = s_rec[blk].s[t + 1];
                                    }
                                } else {
                                    const ulonglong2* pp[8];
                                    ulonglong2 wv[8];
#pragma unroll
                                    for (int h = 0; h < 4; ++h) {
                                        pp[2 * h] = w + (size_t)min(blk0 + 32 * h + lane, nblk - 1) * kStepWords + t;
                                        pp[2 * h + 1] = pp[2 * h] + 1;
                                    }
                                    wait_words<8>(A, pp, tag, wv, &s_ok);
#pragma unroll
                                    for (int h = 0; h < 8; ++h) v[h] = word_values(wv[h]);
                                }
#pragma unroll
                                for (int h = 0; h < 8; ++h)
                                    if (g0 + h / 2 < nw && blk0 + 32 * (h / 2) + lane < nblk) s[h] = csum_merge(s[h], v[h]);
                            }
                            if (nw == 1) butterfly<2, 0>(s, nullptr);
                            else butterfly<8, 0>(s, nullptr);
#pragma unroll
                            for (int h = 0; h < 4; ++h) {
                                if (g0 + h >= nw) break;
#pragma unroll
                                for (int e = 0; e < 2; ++e) sum[e] = g0 + h == 0 ? s[e] : csum_merge(sum[e], s[2 * h + e]);
                            }
                        }
                        if (lane < 2) R.s[t + lane] = lane ? sum[1] : sum[0];
                    }
                    __syncthreads();
                    if (!s_ok) break;
                    if (tid == 0) decide(L, S, R, P, D);
                    __syncthreads();
                    if (D.act != (A_LOB_UPDATE | A_RESID)) {
                        more = false;
                        break;
                    }
                    // ---- the own rows' update (lane_apply's operations) and the next input everywhere
                    const float np = fmaf(D.cw, lw, D.cp * lp);
                    const float nap = fmaf(D.cw, aw, D.cp * lap);
                    lx = fmaf(D.cx, lx, np);
                    lax = fmaf(D.cx, lax, nap);
                    lp = np;
                    lap = nap;
                    const float r = lax - D.lam * lx;
                    lw = r_t * r;
                    const float u = own ? r_d * lw : 0.f;
                    if (nc == 1) {
                        if (own_warp) su[row] = u;
                    } else {
                        ulonglong2* const wu = xb + (size_t)(upd & 1u) * nblk * kRowWords;
                        if (own_warp) {
                            const float2 p = row_word(u, lane);
                            publish(wu + (size_t)sl.at(warp) * kRowWords, lane < kRowWords, lane, p, tag + 1u);
                        }
                        gather_rows<kRowWords>(A, wu, kRowWords, nblk, tag + 1u, su, tid, kThreads, &s_ok);
                    }
                    if (tid == 0) S.updates += 1;
                    ++upd;
                    --steps_left;
                    __syncthreads();
                    if (!s_ok) break;
                }
                if (!s_ok) break;
                if (more) {   // the launch ends inside the eigen-solve
                    if (own) {
                        vec[(size_t)V_LX * ld + row] = lx;
                        vec[(size_t)V_LAX * ld + row] = lax;
                        vec[(size_t)V_LP * ld + row] = lp;
                        vec[(size_t)V_LAP * ld + row] = lap;
                        vec[(size_t)V_LW * ld + row] = lw;
                    }
                    for (int i = ia + tid; i < ib; i += kThreads) vec[(size_t)V_U * ld + i] = su[i];
                    break;
                }
            } else {
                // ================= every other step: the shared functions between group barriers
                item_load_u(L, su);
                __syncthreads();
                if (ph == PH_EVAL) {
                    double* sv = kTight ? reinterpret_cast<double*>(s_share) : s_sv;
                    for (int blk = rank; blk < nblk; blk += nc) {
                        const int row0 = blk * A.rows_per_item;
                        const int rows = min(A.rows_per_item, n - row0);
                        item_rows_eval(L, row0, rows, su, sv, lane, warp);
                        __syncthreads();
                        item_finish(L, ph, S.k, blk, row0, rows, sv, P);
                        __syncthreads();
                    }
                } else {
                    // the products of all slices first, then the blocks' epilogues
                    products();
                    __syncthreads();
                    if constexpr (kTight) {
                        if (own_warp) {
                            const float v = own_product();
                            __syncwarp();   // the shares are read
                            prods(warp)[lane] = (double)v;
                        }
                    } else if (own_warp) {
                        s_sv[tid] = (double)own_product();
                    }
                    __syncthreads();
                    for (int b = 0; b < (one ? 1 : sl.n); ++b) {
                        const int blk = one ? 0 : sl.at(b), row0 = 32 * blk;
                        item_finish(L, ph, S.k, blk, row0, one ? n : min(32, n - row0), prods(b), P);
                        __syncthreads();
                    }
                }
                if (!solo_grid_sync(A, bar, nc, gen, &s_ok)) break;
                reduce_partials(L.part, nblk, ph, R);
                if (tid == 0) decide(L, S, R, P, D);
                __syncthreads();
            }
            // ---- the element-wise update of the step just decided, by slices
            lane_apply(L, P, D, ia, ib, qa, qb, tid, kThreads);
            if (tid == 0) {
                S.updates += 1;
                if (rank == 0 && (D.act & A_TRACE) && L.trace_alpha) L.trace_alpha[D.trace_k] = D.alpha;
            }
            --steps_left;
            if (!solo_grid_sync(A, bar, nc, gen, &s_ok)) break;
        }
        __syncthreads();
        if (rank == 0 && tid == 0) *L.st = S;
        if (!s_ok) break;
    }
    // ---- the group's lanes still unfinished (rank 0 wrote the state of every lane it ran)
    __syncthreads();
    if (rank == 0 && tid == 0) {
        int left = 0;
        for (int li = A.gfirst[g]; li < A.gfirst[g + 1]; ++li) left += A.lane[A.glanes[li]].st->phase != PH_DONE ? 1 : 0;
        if (left) atomicAdd(A.active_after, left);
    }
}

static const void* sell_fn(int per, bool tight)
{
    if (per == 1) return (const void*)sell_lane_kernel<1, false>;
    return tight ? (const void*)sell_lane_kernel<2, true> : (const void*)sell_lane_kernel<2, false>;
}

static size_t sell_limit(const void* fn, int per)
{
    int dev = 0, sm = 0, res = 0;
    size_t most = 0;
    cudaFuncAttributes fa;
    if (cudaGetDevice(&dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&sm, cudaDevAttrMaxSharedMemoryPerMultiprocessor, dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&res, cudaDevAttrReservedSharedMemoryPerBlock, dev) != cudaSuccess ||
        cudaFuncGetAttributes(&fa, fn) != cudaSuccess || smem_limit(fn, &most) != cudaSuccess) {
        cudaGetLastError();
        return 0;
    }
    const int64_t a = (int64_t)sm / per - res - (int64_t)fa.sharedSizeBytes;
    const int64_t v = std::min(a, (int64_t)most) / 1024 * 1024;
    return v > 0 ? (size_t)v : 0;
}

// the largest dynamic shared memory of a CTA when `per` (1 or 2) of them share an SM and `vecs` bytes
// of it are vectors: the tight form where the other does not hold them
size_t sell_smem_limit(int per, size_t vecs, bool* tight)
{
    *tight = false;
    const size_t v = sell_limit(sell_fn(per, false), per);
    if (per == 1 || vecs <= v) return v;
    *tight = true;
    return sell_limit(sell_fn(per, true), per);
}

// whether `per` CTAs with this much dynamic shared memory are resident on an SM
bool sell_fits(int per, bool tight, size_t smem)
{
    int got = 0;
    const void* fn = sell_fn(per, tight);
    if (open_smem(fn, smem) != cudaSuccess ||
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&got, fn, kThreads, smem) != cudaSuccess) {
        cudaGetLastError();
        got = 0;
    }
    return got >= per;
}

cudaError_t launch_sell(const SoloArgs& a, int per, bool tight, size_t smem, cudaStream_t s)
{
    SoloArgs args = a;
    void* params[] = {&args};
    return cudaLaunchCooperativeKernel(sell_fn(per, tight), dim3((unsigned)a.grid), dim3(kThreads), params, smem, s);
}

}  // namespace ubqp
