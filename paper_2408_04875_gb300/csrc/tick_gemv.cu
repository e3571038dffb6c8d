// Phase A on CUDA cores, lock-step scheduler: one launch per tick in which every active
// lane advances by one step.  v = Q_off u for each (lane, row block) item, then the per-row
// epilogue of the lane's phase (gradient of Alg. 2, eigen-solver matvec, Jacobi sweep,
// exact evaluation); the last CTA of a lane runs its update.  Persistent CTAs of 256
// threads pull items from a queue and stream rows from HBM into registers with 16-byte
// loads while u sits in shared memory.  The kernel is bound by the bytes of Q it reads:
// n * ld * 4 per lane per tick (FP32), 8 per entry for the evaluation tick.
#include "gemv_rows.cuh"

namespace ubqp {

// ---------------------------------------------------------------------------------
__global__ void __launch_bounds__(kThreads, 4) phase_a_gemv_kernel(TickArgs A)
{
    // Persistent: CTAs pull (lane, row-block) items from a queue until it is empty; the
    // items of the largest lanes come first.  u stays in shared memory while consecutive
    // items belong to the same lane.
    extern __shared__ __align__(16) unsigned char smem_raw[];
    float* su = reinterpret_cast<float*>(smem_raw);
    __shared__ double sv[kThreads];
    __shared__ int s_item, s_ulane, is_last;
    if (threadIdx.x == 0) s_ulane = -1;
    for (;;) {
        if (threadIdx.x == 0) s_item = atomicAdd(A.work, 1);
        __syncthreads();
        const int item = s_item;
        if (item >= A.nitems) break;
        const int2 it = A.items[item];
        const LaneDev& L = A.lanes[it.x];
        const int ph = L.st->phase;
        if (ph == PH_DONE) {
            __syncthreads();
            continue;
        }
        const int k = L.st->k;
        const int row0 = it.y * A.rows_per_item;
        const int rows = min(A.rows_per_item, L.n - row0);
        if (s_ulane != it.x) item_load_u(L, su);   // consecutive items of one lane share u
        __syncthreads();
        if (threadIdx.x == 0) s_ulane = it.x;
        item_rows_solver(L, ph, row0, rows, su, sv, threadIdx.x & 31, threadIdx.x >> 5);
        __syncthreads();
        item_finish(L, ph, k, it.y, row0, rows, sv, A.P);
        if (A.fused) {
            // every CTA publishes its partial and epilogue writes, then counts itself in; the
            // CTA that completes the lane's count runs the lane's update.  No CTA waits.
            __threadfence();
            __syncthreads();
            if (threadIdx.x == 0) is_last = (atomicAdd(L.counter, 1u) == (unsigned)(L.nblk - 1));
            __syncthreads();
            if (is_last) {
                __threadfence();
                lane_update(L, A.P, A.active_count);
                if (threadIdx.x == 0) {
                    *L.counter = 0u;
                    s_ulane = -1;
                }
            }
        }
        __syncthreads();
    }
    // the last CTA to leave resets the queue for the next tick
    if (threadIdx.x == 0 && atomicAdd(A.done, 1) == (int)gridDim.x - 1) {
        *A.work = 0;
        *A.done = 0;
    }
}

cudaError_t prepare_phase_a_gemv(int max_ld)
{
    // always opted in: the static shared memory counts against the 48 KB default as well
    return open_smem((const void*)phase_a_gemv_kernel, (size_t)max_ld * sizeof(float));
}

// persistent grid: every CTA that fits on the GPU at once, never more CTAs than items
int gemv_grid(int max_ld, int nitems)
{
    int dev = 0, sms = 148, per = 1;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    cudaError_t e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, phase_a_gemv_kernel, kThreads,
                                                                  (size_t)max_ld * sizeof(float));
    if (e != cudaSuccess || per < 1) {
        cudaGetLastError();
        per = 1;
    }
    int g = sms * per;
    return nitems < g ? nitems : g;
}

cudaError_t launch_phase_a_gemv_f32(const TickArgs& a, cudaStream_t s)
{
    // shared: u of the widest lane (ld floats); rows_per_item <= kThreads
    size_t smem = (size_t)a.max_ld * sizeof(float);
    phase_a_gemv_kernel<<<a.grid, kThreads, smem, s>>>(a);
    return cudaGetLastError();
}

}  // namespace ubqp
