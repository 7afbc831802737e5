// ccmc_step.cu -- the kernels of one CCMC time step (Spencer et al.,
// arXiv:1807.03749, Sec. II and Sec. IV.B-C) that do not depend on the
// Hamiltonian kind or the precision, the dispatch of a step to its
// instantiation (ccmc_step_<kind>_<precision>.cu) and the allocation-free
// sort-and-reduce entry point.  The device building blocks are in ccmc_kernels.cuh.
//
//  f3  k_local_table / k_local_scan      batch: k_sample_plan
//  ccmc_reduce_records_noalloc (end of file): the sort and reduction as a
//      standalone call on a static scratch array
#include <mutex>

#include "../../include/ccmc.h"
#include "ccmc_kernels.cuh"

namespace ccmc {

// Batch work plan for the sampler: virtual blocks per replica from its
// sample count, their prefix, the reset work counter, and zeroed E_num
// partials for the slots a replica does not use this step (the final
// reduction reads wmax of them).  One block.
__global__ void __launch_bounds__(1024) k_sample_plan(const StepArgs *__restrict__ A, int nrep, FlatPlan fp,
                                                       int enum_base)
{
    __shared__ int sm[32];
    __shared__ int carry;
    if (threadIdx.x == 0) carry = 0;
    __syncthreads();
    for (int r0 = 0; r0 < nrep; r0 += blockDim.x) {
        const int r = r0 + threadIdx.x;
        int want = 0;
        if (r < nrep) {
            const i64 ns = A[r].st->n_sel;
            const i64 w = (ns + fp.per_block - 1) / fp.per_block;
            want = (int)(w < 1 ? 1 : (w > fp.wmax ? fp.wmax : w));
        }
        int tot;
        const int incl = block_incl_scan(want, sm, tot);
        if (r < nrep) fp.vstart[r] = carry + incl - want;
        __syncthreads();
        if (threadIdx.x == 0) carry += tot;
        __syncthreads();
    }
    if (threadIdx.x == 0) {
        fp.vstart[nrep] = carry;
        *fp.counter = 0u;
    }
    __syncthreads();
    // unused E_num slots of every replica
    for (int r = 0; r < nrep; r++) {
        const i64 ns = A[r].st->n_sel;
        const i64 w = (ns + fp.per_block - 1) / fp.per_block;
        const int used = (int)(w < 1 ? 1 : (w > fp.wmax ? fp.wmax : w));
        u64 *ep = A[r].wa.enum_part;
        for (int q = used + (int)threadIdx.x; q < fp.wmax; q += blockDim.x) {
            ep[2 * (enum_base + q)] = 0;
            ep[2 * (enum_base + q) + 1] = 0;
        }
    }
}

__global__ void __launch_bounds__(SCAN_THREADS) k_local_scan(const StepArgs *__restrict__ A)
{
    const StepArgs &a = A[blockIdx.y];
    d_local_scan(a.st, a.p, a.wa);
}

template <int K>
__global__ void __launch_bounds__(WORK_THREADS) k_local_table(const StepArgs *__restrict__ A)
{
    REPLICA;
    d_local_table<K>(a.s, a.list[cur_], a.st, a.p, a.wa);
}

void launch_local_table(const StepArgs *A, int K, dim3 grid, cudaStream_t sm)
{
    switch (K) {
    case 1: k_local_table<1><<<grid, WORK_THREADS, 0, sm>>>(A); break;
    case 2: k_local_table<2><<<grid, WORK_THREADS, 0, sm>>>(A); break;
    case 3: k_local_table<3><<<grid, WORK_THREADS, 0, sm>>>(A); break;
    case 4: k_local_table<4><<<grid, WORK_THREADS, 0, sm>>>(A); break;
    case 5: k_local_table<5><<<grid, WORK_THREADS, 0, sm>>>(A); break;
    default: k_local_table<6><<<grid, WORK_THREADS, 0, sm>>>(A); break;
    }
}

// ---------------------------------------------------------------------------
// Launcher
// ---------------------------------------------------------------------------

int bits_for(u64 bound)
{
    int b = 1;
    while (b < 64 && (bound - 1) >> b) b++;
    return b;
}

int sort_passes(const Shapes &sh)
{
    return (sh.key_bits + sh.digit_bits - 1) / sh.digit_bits;
}

// instantiated in ccmc_step_<kind>_<precision>.cu
#define CCMC_EXTERN_LAUNCH(R, GAS)                                                                            \
    extern template cudaError_t launch_phases<R, GAS>(const StepArgs *, int, int, const Shapes &, bool,       \
                                                      cudaStream_t, i64 *, const cudaEvent_t *, const FlatPlan *)
CCMC_EXTERN_LAUNCH(double, true);
CCMC_EXTERN_LAUNCH(double, false);
CCMC_EXTERN_LAUNCH(float, true);
CCMC_EXTERN_LAUNCH(float, false);

cudaError_t launch_group(const StepArgs *A, int nrep, int K, bool gas, bool fp32, const Shapes &sh, bool multi_att,
                         cudaStream_t sm, i64 *launches, const cudaEvent_t *ev, const FlatPlan *plan)
{
    if (fp32)
        return gas ? launch_phases<float, true>(A, nrep, K, sh, multi_att, sm, launches, ev, plan)
                   : launch_phases<float, false>(A, nrep, K, sh, multi_att, sm, launches, ev, plan);
    return gas ? launch_phases<double, true>(A, nrep, K, sh, multi_att, sm, launches, ev, plan)
               : launch_phases<double, false>(A, nrep, K, sh, multi_att, sm, launches, ev, plan);
}

cudaError_t launch_step(StepCtx &c)
{
    cudaError_t e = launch_group(c.d_args, 1, c.K, c.gas, c.fp32, c.sh, c.prm.fnc || c.prm.multispawn, c.stream,
                                 c.launches, c.profile ? c.events : nullptr);
    c.sorted_buf = sort_passes(c.sh) & 1;
    c.cur ^= 1;
    return e;
}

}  // namespace ccmc

// ---------------------------------------------------------------------------
// Sort-and-reduce of spawned records without any allocation
//
// For callers that may not allocate device memory: plugins whose host
// application owns the device allocator, and loops that must keep a fixed
// device-memory footprint once set up.  The scratch lives in one file-scope
// device array that every GPU loading this library holds until the process
// exits; every call on a device shares it and leaves its contents behind
// (the barriers are left as found and the output weights are zeroed before the
// per-run atomics).  One launch sorts and reduces: 65,536 records of 27 bits
// took 16 launches and 119 us, now 56 us; 3,001 of 33 bits 19 launches and
// 130 us, now 50 us.
// ---------------------------------------------------------------------------

namespace ccmc {
namespace {

constexpr size_t NOALLOC_MAX = (size_t)1 << 16;   // records per call
constexpr int NOALLOC_GRID = (int)(NOALLOC_MAX / (2 * SORT_THREADS));   // blocks of the largest call

struct NoAllocResult {
    i64 n_keys;
    int unfinished;        // a wait ran out (set by the block that gave up; n_keys may be written all the same)
    NoAllocResult *next;   // of the free ones
};

struct NoAllocScratch {
    u64 key[2][NOALLOC_MAX];
    i64 pop[2][NOALLOC_MAX];
    __align__(16) unsigned hist[(1 << SORT_DIGIT_BITS) * NOALLOC_GRID];
    i64 part[4 * NOALLOC_GRID];
    unsigned bar[2];
    DevStep st;
};

__device__ __align__(256) NoAllocScratch g_noalloc;

constexpr int NOALLOC_SLOTS = 64;   // results allocated at a time

std::mutex g_noalloc_mutex;
NoAllocScratch *g_noalloc_ptr[256];
// Page-locked, mapped words, one per call under way: the kernel writes its
// call's result there.  Calls of several threads can follow each other on the
// GPU (one stream, or streams ordered by events) while their host parts
// overlap, so a word belongs to one call from its launch until it is read.
NoAllocResult *g_noalloc_free[256];

// The whole call (its blocks wait for each other: a cooperative launch when
// there are several).
__global__ void __launch_bounds__(SORT_THREADS, 1) k_noalloc(const u64 *keys_in, const i64 *pops_in, i64 n, int key_bits,
                                                             u64 *keys_out, i64 *pops_out, NoAllocScratch *N,
                                                             NoAllocResult *res)
{
    SortSmem &S = *(SortSmem *)dyn_smem;
    __shared__ i64 sm[64];
    __shared__ unsigned err;
    const Team t = {(int)blockIdx.x, (int)gridDim.x};
    if (t.n > 1) {
        // a wait of an earlier call that has not cleared the barriers yet ran out
        if (threadIdx.x == 0) err = N->st.err;
        __syncthreads();
        if (err & ERRB_TIMEOUT) {
            res->unfinished = 1;
            return;
        }
    }
    u64 *key[2] = {N->key[0], N->key[1]};
    i64 *pop[2] = {N->pop[0], N->pop[1]};
    i64 m = -1;
    if (team_sort(keys_in, pops_in, key, pop, n, key_bits, SORT_DIGIT_BITS, N->hist, N->bar, t, &N->st, S)) {
        const int src = ((key_bits + SORT_DIGIT_BITS - 1) / SORT_DIGIT_BITS) & 1;
        m = team_reduce(key[src], pop[src], n, keys_out, pops_out, N->part, N->bar, t, &N->st, sm);
    }
    if (m < 0) res->unfinished = 1;
    else if (t.id == 0 && threadIdx.x == 0) res->n_keys = m;
}

// Device address of the scratch on the current device dev, looked up once per
// device (host code cannot use the symbol itself as a device address), with
// the kernel's shared memory size set, and a page-locked word for the result
// that the caller gives back.
cudaError_t noalloc_scratch(int &dev, NoAllocScratch **out, NoAllocResult **res)
{
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    if (dev < 0 || dev >= 256) return cudaErrorInvalidDevice;
    std::lock_guard<std::mutex> lock(g_noalloc_mutex);
    if (!g_noalloc_ptr[dev]) {
        void *p = nullptr;
        e = cudaGetSymbolAddress(&p, g_noalloc);
        if (e != cudaSuccess) return e;
        e = cudaFuncSetAttribute(k_noalloc, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(SortSmem));
        if (e != cudaSuccess) return e;
        g_noalloc_ptr[dev] = (NoAllocScratch *)p;
    }
    if (!g_noalloc_free[dev]) {
        NoAllocResult *r = nullptr;
        e = cudaHostAlloc((void **)&r, NOALLOC_SLOTS * sizeof(NoAllocResult), cudaHostAllocMapped);
        if (e != cudaSuccess) return e;
        for (int q = 0; q < NOALLOC_SLOTS; q++) r[q].next = q + 1 < NOALLOC_SLOTS ? r + q + 1 : nullptr;
        g_noalloc_free[dev] = r;
    }
    *out = g_noalloc_ptr[dev];
    *res = g_noalloc_free[dev];
    g_noalloc_free[dev] = (*res)->next;
    return cudaSuccess;
}

void noalloc_done(int dev, NoAllocResult *res)
{
    std::lock_guard<std::mutex> lock(g_noalloc_mutex);
    res->next = g_noalloc_free[dev];
    g_noalloc_free[dev] = res;
}

}  // namespace

}  // namespace ccmc

extern "C" ccmc_status ccmc_reduce_records_noalloc(const uint64_t *keys_in, const int64_t *pops_in, size_t n,
                                                   int32_t key_bits, uint64_t *keys_out, int64_t *pops_out,
                                                   size_t *n_out, void *cuda_stream)
{
    using namespace ccmc;
    if (!n_out) return CCMC_ERR_ARG;
    *n_out = 0;
    if (n > NOALLOC_MAX || key_bits < 1 || key_bits > 64) return CCMC_ERR_ARG;
    if (n == 0) return CCMC_OK;
    if (!keys_in || !pops_in || !keys_out || !pops_out) return CCMC_ERR_ARG;
    cudaStream_t sm = (cudaStream_t)cuda_stream;
    int dev = 0;
    NoAllocScratch *S = nullptr;
    NoAllocResult *res = nullptr;
    if (noalloc_scratch(dev, &S, &res) != cudaSuccess) return CCMC_ERR_CUDA;
    res->n_keys = 0;
    res->unfinished = 0;
    cudaError_t e = launch_blocks(k_noalloc, dim3((unsigned)sort_blocks((i64)n)), n > SORT_TILE, SORT_THREADS,
                                  sizeof(SortSmem), sm, (const u64 *)keys_in, (const i64 *)pops_in, (i64)n, (int)key_bits,
                                  (u64 *)keys_out, (i64 *)pops_out, S, res);
    if (e == cudaSuccess) e = cudaStreamSynchronize(sm);
    const i64 m = *(volatile i64 *)&res->n_keys;
    const bool unfinished = *(volatile int *)&res->unfinished != 0;
    if (e == cudaSuccess && unfinished) {   // a wait ran out: the next call starts clean
        cudaMemsetAsync(S->bar, 0, sizeof(S->bar) + sizeof(S->st), sm);
        cudaStreamSynchronize(sm);
    }
    noalloc_done(dev, res);
    if (e != cudaSuccess) return CCMC_ERR_CUDA;
    if (unfinished) return CCMC_ERR_TIMEOUT;
    *n_out = (size_t)m;
    return CCMC_OK;
}
