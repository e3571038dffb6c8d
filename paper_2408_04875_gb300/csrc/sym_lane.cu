// FP32 lanes on the symmetric tiles, each on its own group of CTAs, many steps of Alg. 3 per
// cooperative launch: what sell_lane.cu is for the sliced storage.
//
// CTA c of a group of C owns the stored 128 x 128 tiles c, c + C, ... of its lane (as many as fit
// stay in shared memory for the whole launch, the rest is read from L2) and, if c < nb, row block
// c (C is at least nb).  A product takes one exchange: every tile's row and column products go out
// as tagged words (lane_words.cuh), the owner of a row block collects the nb partial vectors of its
// rows and sums them.  An Alg. 2 step then has the row epilogue at the block's owner and one
// exchange of g and the records to every CTA; a LOBPCG iteration one of the Gram sums and one of the
// next input.  The lane loop that ran these lanes paid, per 128 x 128 tile and step, a pop from the
// ring, the descriptor, the tile from L2 and a counter, and then the same per row block.
//
// Bound: latency (two exchanges through L2 per Alg. 2 step of about 1.7k cycles each, the tile
// products and the sums over nb partial vectors between them).  Measured against the lane loop,
// whole calls: six lanes of n = 200 to 1500, density 0.5, 50 subproblems of 20 steps 85-93 -> 25-28
// ms; device time of 4 lanes of n = 2000 6.4 -> 2.3 ms, 4 of n = 4500 (18 tiles a CTA) 10.4 -> 7.5 ms.
//
// Buffers by the step's parity: tile words of step j + 2 overwrite those of step j.  Their sender
// has the gradient (or input) words of step j + 1 of every row block, and an owner sends those only
// after it has read its tile words of step j + 1, so of step j too.  Block words of step j + 2: their
// sender has all block words of step j + 1, so every tile's words of step j + 1 had been sent, by
// CTAs that had read the block words of step j before.  (Every CTA owns a tile.)
//
// The arithmetic and its order are those of the lane loop (sym_tile_part, sym_group_item,
// sym_block_sums, row_epilogue, the record of a 128-row block, reduce_partials, decide,
// lane_apply): the same bits.  Every wait is bounded.  Plain loads are cached in L2 only (-dlcm=cg).
#include "lane_words.cuh"

namespace ubqp {

namespace {

constexpr int kBlkRows = kSymT;                    // 128
constexpr int kValWords = kBlkRows / 2;            // a block's values
constexpr int kTileWords = 2 * kValWords;          // row products, column products
constexpr int kRecWords = 5;                       // the ten numbers of an Alg. 2 record
constexpr int kBlkWords = kValWords + kGramWords;  // values, then the record or the Gram sums
constexpr int kRowWarps = kBlkRows / 32;
constexpr int kTileBytes = kSymT * kSymT * 4;

// One tile: its row products into s_row and the column products of this thread's warp into s_colw
// (merged by the caller); sym_tile_part's mapping and operations, u in shared memory.
template <bool kShared>
__device__ __forceinline__ void tile_products(const float4* tile, const float* su, int I, int J, float (*s_colw)[kSymT],
                                              float* s_row)
{
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const float4 uj = reinterpret_cast<const float4*>(su + J * kSymT)[lane];
    float c0 = 0.f, c1 = 0.f, c2 = 0.f, c3 = 0.f;
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        const int r0 = warp * 16 + h * 8;
        float4 q[8];
#pragma unroll
        for (int r = 0; r < 8; ++r) {
            const float4* p = tile + (size_t)(r0 + r) * (kSymT / 4) + lane;
            if constexpr (kShared) q[r] = *p;
            else q[r] = ldg_stream(p);
        }
        const float4 ui0 = reinterpret_cast<const float4*>(su + I * kSymT + r0)[0];
        const float4 ui1 = reinterpret_cast<const float4*>(su + I * kSymT + r0)[1];
        const float uis[8] = {ui0.x, ui0.y, ui0.z, ui0.w, ui1.x, ui1.y, ui1.z, ui1.w};
        float v[8];
#pragma unroll
        for (int r = 0; r < 8; ++r) {
            float a = __fmul_rn(q[r].x, uj.x);
            a = fmaf(q[r].y, uj.y, a);
            a = fmaf(q[r].z, uj.z, a);
            v[r] = fmaf(q[r].w, uj.w, a);
            const float ui = uis[r];
            c0 = fmaf(q[r].x, ui, c0);
            c1 = fmaf(q[r].y, ui, c1);
            c2 = fmaf(q[r].z, ui, c2);
            c3 = fmaf(q[r].w, ui, c3);
        }
        {
            const bool up = lane & 16;
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                const float keep = up ? v[j + 4] : v[j], send = up ? v[j] : v[j + 4];
                v[j] = keep + __shfl_xor_sync(0xffffffffu, send, 16);
            }
        }
        {
            const bool up = lane & 8;
#pragma unroll
            for (int j = 0; j < 2; ++j) {
                const float keep = up ? v[j + 2] : v[j], send = up ? v[j] : v[j + 2];
                v[j] = keep + __shfl_xor_sync(0xffffffffu, send, 8);
            }
        }
        {
            const bool up = lane & 4;
            const float keep = up ? v[1] : v[0], send = up ? v[0] : v[1];
            v[0] = keep + __shfl_xor_sync(0xffffffffu, send, 4);
        }
        v[0] += __shfl_xor_sync(0xffffffffu, v[0], 2);
        v[0] += __shfl_xor_sync(0xffffffffu, v[0], 1);
        if ((lane & 3) == 0) s_row[r0 + ((lane >> 2) & 7)] = v[0];
    }
    s_colw[warp][4 * lane + 0] = c0;
    s_colw[warp][4 * lane + 1] = c1;
    s_colw[warp][4 * lane + 2] = c2;
    s_colw[warp][4 * lane + 3] = c3;
}

}  // namespace

__global__ void __launch_bounds__(kThreads, 1) sym_lane_kernel(SoloArgs A)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    __shared__ double sv[kThreads];
    __shared__ LaneState S;
    __shared__ Partial R;
    __shared__ Decision D;
    __shared__ int s_ok, s_g;
    __shared__ unsigned long long s_gen0;
    __shared__ float s_colw[2][kWarps][kSymT];
    __shared__ float2 s_row2[2][kSymT / 2];
    __shared__ WarpRed s_red[kWarps];
    __shared__ WarpRed s_rec[kRowWarps];
    __shared__ float s_basis[kRowWarps][6 * 32];
    __shared__ int2 s_ij[kSymMaxTiles];
    __shared__ __align__(16) LaneDev sL;
    __shared__ Params sP;

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
        const float* Qsym = A.sym[lane_id].Qsym;
        const int n = L.n, ld = L.ld, nb = L.nblk, ntiles = nb * (nb + 1) / 2;
        const bool pabb = L.method == 0;
        const int nq4 = ld >> 2;
        const int qa = (int)((int64_t)nq4 * rank / nc), qb = (int)((int64_t)nq4 * (rank + 1) / nc);
        const int ia = min(4 * qa, n), ib = min(4 * qb, n);
        float* su = reinterpret_cast<float*>(smem_raw);
        float* sg = su + ld;
        float* s_part = sg + ld;   // [K][row]: the own block's partial vectors
        float* vec = L.vec;
        // ---- this CTA's tiles; the first nres of them in shared memory
        const int my_t = rank < ntiles ? (ntiles - rank + nc - 1) / nc : 0;
        const int nres = min(my_t, A.mat_bytes / kTileBytes);
        float4* mat = reinterpret_cast<float4*>(s_part + (size_t)nb * kBlkRows);
        if (tid < my_t) {
            int I, J;
            sym_tile_ij(rank + tid * nc, nb, I, J);
            s_ij[tid] = make_int2(I, J);
        }
        for (int b = 0; b < nres; ++b) {
            const float4* src = reinterpret_cast<const float4*>(Qsym + (size_t)(rank + b * nc) * kSymT * kSymT);
            for (int e = tid; e < kTileBytes / 16; e += kThreads) mat[(size_t)b * (kTileBytes / 16) + e] = __ldg(src + e);
        }
        // ---- the row block this CTA owns, if any; thread = row for the first four warps
        const bool has_blk = rank < nb;
        const bool row_warp = has_blk && warp < kRowWarps;
        const int row = rank * kBlkRows + tid;
        const bool own = row_warp && row < n;
        const int rc = own ? row : n - 1;
        ulonglong2* const x1 = L.xch;                                          // [2][tile][128]
        ulonglong2* const x2 = x1 + (size_t)2 * ntiles * kTileWords;           // [2][block][76]
        ulonglong2* const x3 = x2 + (size_t)2 * nb * kBlkWords;                // [2][block][64]
        const int nw = min(kWarps, (nb + 31) >> 5);   // warps with records
        const int gw0 = nw < kWarps ? nw : 0;
        __syncthreads();

        // the products with su of every row of the own block (this thread's row for tid < 128)
        auto product = [&](uint32_t upd) -> float {
            const uint32_t tag = 4u * upd + 1u;
            ulonglong2* const w = x1 + (size_t)(upd & 1u) * ntiles * kTileWords;
            for (int t0 = 0; t0 < my_t; t0 += 2) {
                if (t0 > 0) __syncthreads();   // the previous pair's products have been sent
#pragma unroll 1
                for (int k = 0; k < 2 && t0 + k < my_t; ++k) {
                    const int2 ij = s_ij[t0 + k];
                    float* sr = reinterpret_cast<float*>(s_row2[k]);
                    if (t0 + k < nres) tile_products<true>(mat + (size_t)(t0 + k) * (kTileBytes / 16), su, ij.x, ij.y, s_colw[k], sr);
                    else tile_products<false>(reinterpret_cast<const float4*>(Qsym + (size_t)(rank + (t0 + k) * nc) * kSymT * kSymT),
                                              su, ij.x, ij.y, s_colw[k], sr);
                    if (P.bytes && tid == 0) {
                        const unsigned long long ri = (unsigned long long)min(kSymT, n - ij.x * kSymT);
                        const unsigned long long cj = (unsigned long long)min(kSymT, n - ij.y * kSymT);
                        atomicAdd(P.bytes, ri * cj * 4ull + 2ull * kSymT * 4ull + (ij.x != ij.y ? 2ull : 1ull) * kSymT * 4ull);
                    }
                }
                __syncthreads();
                const int k = tid / kSymT, e = tid % kSymT;   // one half of the CTA per tile
                const bool mine = t0 + k < my_t;
                float2 acc = make_float2(0.f, 0.f);
#pragma unroll
                for (int q = 0; q < kWarps; ++q) csum_add(acc, s_colw[k][q][e]);
                const float c = acc.x + acc.y, cn = __shfl_down_sync(0xffffffffu, c, 1);
                if (mine) {
                    ulonglong2* const wt = w + (size_t)(rank + (t0 + k) * nc) * kTileWords;
                    const int2 ij = s_ij[t0 + k];
                    if (ij.x != ij.y && !(e & 1)) st_word(wt + kValWords + e / 2, c, cn, tag);
                    if (e < kValWords) st_word(wt + e, s_row2[k][e].x, s_row2[k][e].y, tag);
                }
                __syncwarp();
            }
            float v = 0.f;
            if (has_blk) {
                // the partial vectors K = 0 .. nb - 1 of the block's rows: row products of tile (b, K),
                // K >= b, column products of tile (K, b) below
                const int q = tid / kValWords, e = tid % kValWords, b = rank;
                for (int K0 = 0; K0 < nb; K0 += 16) {
                    const ulonglong2* p[4];
                    ulonglong2 wv[4];
#pragma unroll
                    for (int h = 0; h < 4; ++h) {
                        const int K = min(K0 + 4 * h + q, nb - 1);
                        const int i = min(b, K), j = max(b, K);
                        p[h] = w + (size_t)(i * nb - i * (i - 1) / 2 + j - i) * kTileWords + (K >= b ? 0 : kValWords) + e;
                    }
                    wait_words<4>(A, p, tag, wv, &s_ok);
#pragma unroll
                    for (int h = 0; h < 4; ++h) {
                        const int K = K0 + 4 * h + q;
                        if (K < nb) reinterpret_cast<float2*>(s_part)[K * kValWords + e] = word_values(wv[h]);
                    }
                }
                __syncthreads();
                if (tid < kBlkRows) {
                    float2 acc = make_float2(0.f, 0.f);
                    for (int K = 0; K < nb; ++K) csum_add(acc, s_part[K * kBlkRows + tid]);
                    v = acc.x + acc.y;
                }
            }
            return v;
        };
        auto count_block = [&]() {   // profiling only
            if (P.bytes && has_blk && tid == 0) {
                const unsigned long long rows = (unsigned long long)min(kBlkRows, n - rank * kBlkRows);
                atomicAdd(P.bytes, rows * (unsigned long long)nb * 4ull + 16ull * rows);
            }
        };

        for (; steps_left > 0;) {
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
                if (row_warp) {
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
                    const float v = product(upd);
                    const uint32_t tag = 4u * upd + 2u;
                    ulonglong2* const w = x2 + (size_t)(upd & 1u) * nb * kBlkWords;
                    if (row_warp) {
                        const float x = su[rank * kBlkRows + tid];
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
                        publish(w + (size_t)rank * kBlkWords + 16 * warp, lane < 16, lane, row_word(gk, lane), tag);
                        if (k >= 1) butterfly<3, 1>(s, m);   // the other maxima belong to step 0, the sums to the rest
                        else butterfly<0, 4>(s, m);
                        if (lane == 0) {
#pragma unroll
                            for (int t = 0; t < 3; ++t) s_rec[warp].s[t] = s[t];
#pragma unroll
                            for (int t = 0; t < 4; ++t) s_rec[warp].m[t] = m[t];
                        }
                        count_block();
                    }
                    __syncthreads();
                    if (has_blk && warp == 0) {   // the block's record: its warps merged in order
                        float2 p = make_float2(0.f, 0.f);
                        if (lane < 3) {
                            p = s_rec[0].s[lane];
#pragma unroll
                            for (int q = 1; q < kRowWarps; ++q) p = csum_merge(p, s_rec[q].s[lane]);
                        } else if (lane < kRecWords) {
                            const int t = 2 * (lane - 3);
                            p = make_float2(s_rec[0].m[t], s_rec[0].m[t + 1]);
#pragma unroll
                            for (int q = 1; q < kRowWarps; ++q)
                                p = make_float2(fmaxf(p.x, s_rec[q].m[t]), fmaxf(p.y, s_rec[q].m[t + 1]));
                        }
                        publish(w + (size_t)rank * kBlkWords + kValWords, lane < kRecWords, lane, p, tag);
                    }
                    // ---- every row's g_k into sg, the block records reduced in reduce_partials' order
                    if (warp < nw) {
                        float2 s[3];
                        float m[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
                        for (int t = 0; t < 3; ++t) s[t] = make_float2(0.f, 0.f);
                        for (int blk0 = 32 * warp; blk0 < nb; blk0 += kThreads) {   // whole warps
                            const ulonglong2* src = w + (size_t)min(blk0 + lane, nb - 1) * kBlkWords + kValWords;
                            const ulonglong2* const pp[kRecWords] = {src, src + 1, src + 2, src + 3, src + 4};
                            ulonglong2 wv[kRecWords];
                            wait_words<kRecWords>(A, pp, tag, wv, &s_ok);
                            if (blk0 + lane < nb) {
#pragma unroll
                                for (int t = 0; t < 3; ++t) s[t] = csum_merge(s[t], word_values(wv[t]));
                                const float2 m01 = word_values(wv[3]), m23 = word_values(wv[4]);
                                m[0] = fmaxf(m[0], m01.x);
                                m[1] = fmaxf(m[1], m01.y);
                                m[2] = fmaxf(m[2], m23.x);
                                m[3] = fmaxf(m[3], m23.y);
                            }
                        }
                        __syncwarp();
                        if (k >= 1) butterfly<3, 1>(s, m);
                        else butterfly<0, 4>(s, m);
                        if (lane == 0) {
#pragma unroll
                            for (int t = 0; t < 3; ++t) s_red[warp].s[t] = s[t];
#pragma unroll
                            for (int t = 0; t < 4; ++t) s_red[warp].m[t] = m[t];
                        }
                    }
                    if (warp >= gw0)
                        gather_rows<kValWords>(A, w, kBlkWords, nb, tag, sg, tid - 32 * gw0, kThreads - 32 * gw0, &s_ok);
                    __syncthreads();
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
                    exit_code = inner_scalar(0, k, kmax, tol, amin, amax, qmax, tm, csum_value(t3[0]), csum_value(t3[1]),
                                             csum_value(t3[2]), rho, alpha);
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
                    // the launch ends inside the subproblem
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
                    const float v = product(upd);
                    const uint32_t tag = 4u * upd + 2u;
                    ulonglong2* const w = x2 + (size_t)(upd & 1u) * nb * kBlkWords;
                    float aw = 0.f;
                    if (row_warp) {
                        if (own && r_d != 0.f) aw = r_d * fmaf(r_dmp, r_d * lw, v);
                        float* q = s_basis[warp] + lane;   // rows beyond n hold zeros
                        q[0] = lx;
                        q[32] = lax;
                        q[64] = lw;
                        q[96] = aw;
                        q[128] = lp;
                        q[160] = lap;
                        count_block();
                    }
                    __syncthreads();
                    if (has_blk) {
                        // the twelve Gram sums of the block's four warps of rows, then merged in order
                        for (int task = warp; task < 6 * kRowWarps; task += kWarps) {
                            const int b = task / 6, t = 2 * (task - 6 * b);
                            const float* q = s_basis[b] + lane;
                            float2 s[2];
#pragma unroll
                            for (int h = 0; h < 2; ++h) {
                                const int l = (int)(kGramLeft >> (4 * (t + h))) & 15, r = (int)(kGramRight >> (4 * (t + h))) & 15;
                                s[h] = make_float2(0.f, 0.f);
                                csum_add(s[h], q[32 * l] * q[32 * r]);
                            }
                            butterfly<2, 0>(s, nullptr);
                            if (lane < 2) s_rec[b].s[t + lane] = lane ? s[1] : s[0];
                        }
                        __syncthreads();
                        if (warp == 0) {
                            float2 p = make_float2(0.f, 0.f);
                            if (lane < kGramWords) {
                                p = s_rec[0].s[lane];
#pragma unroll
                                for (int q = 1; q < kRowWarps; ++q) p = csum_merge(p, s_rec[q].s[lane]);
                            }
                            publish(w + (size_t)rank * kBlkWords + kValWords, lane < kGramWords, lane, p, tag);
                        }
                    }
                    // ---- over the blocks, in reduce_partials' order (as in sell_lane.cu)
                    if (warp < 6) {
                        const int t = 2 * warp;
                        float2 sum[2];
                        for (int g0 = 0; g0 < nw; g0 += 4) {
                            float2 s[8];   // groups g0 .. g0 + 3, two sums each
#pragma unroll
                            for (int h = 0; h < 8; ++h) s[h] = make_float2(0.f, 0.f);
                            for (int blk0 = 32 * g0; blk0 < nb; blk0 += kThreads) {
                                const ulonglong2* pp[8];
                                ulonglong2 wv[8];
#pragma unroll
                                for (int h = 0; h < 4; ++h) {
                                    pp[2 * h] = w + (size_t)min(blk0 + 32 * h + lane, nb - 1) * kBlkWords + kValWords + t;
                                    pp[2 * h + 1] = pp[2 * h] + 1;
                                }
                                wait_words<8>(A, pp, tag, wv, &s_ok);
#pragma unroll
                                for (int h = 0; h < 8; ++h)
                                    if (g0 + h / 2 < nw && blk0 + 32 * (h / 2) + lane < nb)
                                        s[h] = csum_merge(s[h], word_values(wv[h]));
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
                    ulonglong2* const wu = x3 + (size_t)(upd & 1u) * nb * kValWords;
                    if (row_warp)
                        publish(wu + (size_t)rank * kValWords + 16 * warp, lane < 16, lane, row_word(u, lane), tag + 1u);
                    gather_rows<kValWords>(A, wu, kValWords, nb, tag + 1u, su, tid, kThreads, &s_ok);
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
                // ================= every other step: the shared functions between group barriers; the
                // evaluation reads dense rows, the others take their products from the tiles
                const int rows = has_blk ? min(kBlkRows, n - rank * kBlkRows) : 0;
                item_load_u(L, su);
                __syncthreads();
                if (ph == PH_EVAL) {
                    if (has_blk) item_rows_eval(L, rank * kBlkRows, rows, su, sv, lane, warp);
                } else {
                    const float v = product((uint32_t)S.updates);
                    if (tid < rows) sv[tid] = (double)v;
                }
                __syncthreads();
                if (!s_ok) break;
                if (has_blk) item_finish(L, ph, S.k, rank, rank * kBlkRows, rows, sv, P, ph == PH_EVAL ? 0 : nb);
                __syncthreads();
                if (!solo_grid_sync(A, bar, nc, gen, &s_ok)) break;
                reduce_partials(L.part, nb, ph, R);
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

// exchange words of a lane of nb row blocks
size_t sym_lane_words(int nb)
{
    return 2 * ((size_t)nb * (nb + 1) / 2 * kTileWords + (size_t)nb * (kBlkWords + kValWords));
}

// shared memory of a CTA: two vectors, the partial vectors of its row block and up to `tiles` tiles;
// 0 when even those vectors do not fit.  mat_bytes: the tiles' part
size_t sym_lane_smem(int ld, int tiles, int32_t* mat_bytes)
{
    size_t most = 0;
    if (smem_limit((const void*)sym_lane_kernel, &most) != cudaSuccess) {
        cudaGetLastError();
        return 0;
    }
    const int64_t base = 2 * (int64_t)ld * 4 + (int64_t)(ld / kSymT) * kBlkRows * 4;
    const int64_t room = (int64_t)most - base;
    if (room < 0) return 0;
    const int64_t fit = std::min<int64_t>(tiles, room / kTileBytes);
    *mat_bytes = (int32_t)(fit * kTileBytes);
    const size_t smem = (size_t)(base + fit * kTileBytes);
    if (open_smem((const void*)sym_lane_kernel, smem) != cudaSuccess) {
        cudaGetLastError();
        return 0;
    }
    return smem;
}

cudaError_t launch_sym(const SoloArgs& a, size_t smem, cudaStream_t s)
{
    SoloArgs args = a;
    void* params[] = {&args};
    return cudaLaunchCooperativeKernel((const void*)sym_lane_kernel, dim3((unsigned)a.grid), dim3(kThreads), params, smem, s);
}

}  // namespace ubqp
