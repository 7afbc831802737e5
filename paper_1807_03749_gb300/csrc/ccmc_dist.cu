// ccmc_dist.cu -- co-location statistics of the paper's distribution of
// excitors over processors (Sec. III, Eq. ccmc_dist, Fig. excitdistrib),
// simulated on one GPU: the owner of every excitor at every iteration, then,
// for every pair of excitors, the number of iterations they shared a
// processor, summed (with its square) over pairs at each checkpoint.

#include "../../include/ccmc.h"
#include "ccmc_device.cuh"

namespace ccmc {
namespace {

constexpr int MAX_CHECKPOINTS = 64;
constexpr int TILE_I = 32, TILE_J = 64;   // excitors per side of a pair tile
constexpr int CHUNK = 1024;               // iterations whose owners a warp stages at a time
constexpr int MAX_PLANES = 16;            // bits of an owner (n_ranks <= 65535)

// V, one entry of a plane, holds a group of iterations: 128 (uint4), or 32
// (unsigned) for a call of at most 32, which then reads and compares a quarter
// (30,000 excitors, 65,535 processors, one iteration: 1.2 ms, 3.7 with 128).
template <typename V>
constexpr int group_of = 8 * (int)sizeof(V);

__device__ __forceinline__ void set_entry(uint4 &v, const unsigned (&w)[4]) { v = make_uint4(w[0], w[1], w[2], w[3]); }
__device__ __forceinline__ void set_entry(unsigned &v, const unsigned (&w)[1]) { v = w[0]; }

// The owners as bit planes over time: bit t of planes[(g nb + b) npad + i] is
// bit b of excitor i's owner at iteration t of group g, so that two excitors'
// owners are compared 32 iterations at a time, one three-input logic
// operation per bit.  One warp per excitor and 1024 iterations: an owner lasts
// 2^nu_move iterations (Eq. ccmc_dist), so each is hashed once (the lanes take
// the runs) and spread over its iterations by ballots.
template <typename V>
__global__ void __launch_bounds__(256) k_owner_planes(const u64 *dets, i64 n, i64 npad, int nw, i64 t_max, int nu_move,
                                                      u64 n_ranks, int nb, V *planes)
{
    constexpr int GROUP = group_of<V>, W = GROUP / 32;
    __shared__ unsigned short own[8][CHUNK + 8];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const i64 chunks = (t_max + CHUNK - 1) / CHUNK;
    const bool moves = nu_move < 64;
    const u64 omask = moves && nu_move > 0 ? ~0ULL >> nu_move : ~0ULL;   // owners' phases wrap with the 64-bit sum
    for (i64 q = (i64)blockIdx.x * 8 + wid; q < n * chunks; q += (i64)gridDim.x * 8) {
        const i64 c = q / n, i = q - c * n, t0 = c * CHUNK;
        const i64 tn = t_max - t0 < CHUNK ? t_max - t0 : (i64)CHUNK;
        const u64 *d = dets + i * nw;
        const u64 h = words_hash(d, nw);
        const u64 r0 = moves ? (h + (u64)t0) >> nu_move : 0;
        const int runs = moves ? (int)((((h + (u64)(t0 + tn - 1)) >> nu_move) - r0) & omask) + 1 : 1;
        for (int r = lane; r < runs; r += 32) {
            u64 x[6];
            for (int w = 0; w < nw; w++) x[w] = d[w];
            x[0] ^= moves ? (r0 + (u64)r) & omask : 0;
            own[wid][r] = (unsigned short)(words_hash(x, nw) % n_ranks);
        }
        __syncwarp();
        for (int g = 0; g * GROUP < tn; g++) {
            unsigned word[W] = {};   // of the plane of this lane's bit
#pragma unroll
            for (int w = 0; w < W; w++) {
                const int t = g * GROUP + w * 32 + lane;
                unsigned o = 0;
                if (t < tn) o = own[wid][moves ? (int)((((h + (u64)(t0 + t)) >> nu_move) - r0) & omask) : 0];
                for (int b = 0; b < nb; b++) {
                    const unsigned m = __ballot_sync(0xFFFFFFFFu, (o >> b) & 1u);
                    if (lane == b) word[w] = m;
                }
            }
            if (lane < nb) set_entry(planes[((t0 / GROUP + g) * nb + lane) * npad + i], word);
        }
        __syncwarp();
    }
}

// carry-save addition of two bits to a column: the sum stays, the carry is returned
__device__ __forceinline__ unsigned csa(unsigned &sum, unsigned a, unsigned b)
{
    const unsigned u = sum ^ a, carry = (sum & a) | (u & b);
    sum = u ^ b;
    return carry;
}

// the iterations at which two owners' bits differ
__device__ __forceinline__ void differ(uint4 &d, const uint4 &a, const uint4 &b)
{
    d.x |= a.x ^ b.x;
    d.y |= a.y ^ b.y;
    d.z |= a.z ^ b.z;
    d.w |= a.w ^ b.w;
}
__device__ __forceinline__ void differ(unsigned &d, unsigned a, unsigned b) { d |= a ^ b; }

// A pair's count of equal owners: 4 cnt + 2 popc(twos) + popc(ones)
struct PairCount {
    unsigned ones, twos, cnt;
};

// adds a group's equal iterations, of those in the mask m
__device__ __forceinline__ void count_equal(PairCount &c, const uint4 &d, const unsigned (&m)[4])
{
    const unsigned ta = csa(c.ones, ~d.x & m[0], ~d.y & m[1]), tb = csa(c.ones, ~d.z & m[2], ~d.w & m[3]);
    c.cnt += __popc(csa(c.twos, ta, tb));
}
__device__ __forceinline__ void count_equal(PairCount &c, unsigned d, const unsigned (&m)[1])
{
    c.ones = ~d & m[0];   // (the only group)
}

// One 32 x 64 tile of pairs (i in the row tile, j in the column tile, j > i)
// per block of 8 warps: each thread walks 4 x 2 pairs through the iterations,
// a group at a time, and adds C and C^2 of its pairs at each checkpoint.  Bound
// by integer logic: nb operations per 32 iterations of a pair, two more for
// the carry-save columns that replace three of four population counts (8
// issue slots each); the next group's planes are copied meanwhile.  3,813
// excitors, 4,096 iterations, 32 processors: 0.71 ms (19.2 ms comparing and
// adding one owner at a time).
template <typename V>
__global__ void __launch_bounds__(256) k_pairs(const V *planes, i64 n, i64 npad, int nb, i64 t_max, const i64 *ck,
                                               int nck, u64 *sum_c, u64 *sum_c2)
{
    constexpr int GROUP = group_of<V>, W = GROUP / 32;
    const i64 i0 = (i64)blockIdx.y * TILE_I, j0 = (i64)blockIdx.x * TILE_J;
    if (j0 + TILE_J - 1 <= i0) return;
    extern __shared__ uint4 tiles[];   // two stages of [bit][TILE_I + TILE_J] entries
    constexpr int PER = 4 / W, ROW = (TILE_I + TILE_J) / PER;   // entries per 16 bytes, 16-byte pieces of a bit's row
    const int pieces = nb * ROW;
    __shared__ i64 sck[MAX_CHECKPOINTS];
    __shared__ u64 part[8][2];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    if (threadIdx.x < nck) sck[threadIdx.x] = ck[threadIdx.x];
    PairCount pc[8];
#pragma unroll
    for (int q = 0; q < 8; q++) pc[q] = {0, 0, 0};
    int k = 0;
    // the next group's planes are copied while this one's are compared
    auto copy = [&](i64 g) {
        if (g * GROUP < t_max)
            for (int q = threadIdx.x; q < pieces; q += 256) {
                const int b = q / ROW, e = (q - b * ROW) * PER;
                // (16-byte aligned: the tiles begin at multiples of four excitors)
                const V *src = planes + (g * nb + b) * npad + (e < TILE_I ? i0 + e : j0 + e - TILE_I);
                const unsigned dst = (unsigned)__cvta_generic_to_shared(tiles + (g & 1) * pieces + q);
                asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst), "l"(src) : "memory");
            }
        asm volatile("cp.async.commit_group;" ::: "memory");
    };
    copy(0);
    for (i64 t0 = 0, g = 0; t0 < t_max; t0 += GROUP, g++) {
        copy(g + 1);
        asm volatile("cp.async.wait_group 1;" ::: "memory");
        __syncthreads();
        const V *tile = (const V *)(tiles + (g & 1) * pieces);
        V diff[8] = {};
#pragma unroll 1
        for (int b = 0; b < nb; b++) {
            const V *row = tile + b * (TILE_I + TILE_J);
            const V ja = row[TILE_I + lane], jb = row[TILE_I + 32 + lane];
#pragma unroll
            for (int a = 0; a < 4; a++) {
                const V ii = row[wid * 4 + a];
                differ(diff[2 * a], ii, ja);
                differ(diff[2 * a + 1], ii, jb);
            }
        }
        // checkpoints T in (t0, t0 + GROUP]: the count so far and the first
        // T - t0 iterations of this group
        while (k < nck && sck[k] <= t0 + GROUP) {
            const int T = (int)(sck[k] - t0);
            unsigned m[W];
#pragma unroll
            for (int w = 0; w < W; w++) {
                const int left = T - 32 * w;
                m[w] = left >= 32 ? 0xFFFFFFFFu : (left <= 0 ? 0u : (1u << left) - 1u);
            }
            u64 s1 = 0, s2 = 0;
#pragma unroll
            for (int q = 0; q < 8; q++) {
                const i64 i = i0 + wid * 4 + (q >> 1), j = j0 + (q & 1) * 32 + lane;
                PairCount p = pc[q];
                count_equal(p, diff[q], m);
                const u64 c = 4ULL * p.cnt + 2 * __popc(p.twos) + __popc(p.ones);
                if (j < n && j > i) {
                    s1 += c;
                    s2 += c * c;
                }
            }
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) {
                s1 += __shfl_xor_sync(0xFFFFFFFFu, s1, o);
                s2 += __shfl_xor_sync(0xFFFFFFFFu, s2, o);
            }
            __syncthreads();
            if (lane == 0) {
                part[wid][0] = s1;
                part[wid][1] = s2;
            }
            __syncthreads();
            if (threadIdx.x < 2) {
                u64 s = 0;
                for (int w = 0; w < 8; w++) s += part[w][threadIdx.x];
                atomicAdd((unsigned long long *)&(threadIdx.x ? sum_c2 : sum_c)[k], (unsigned long long)s);
            }
            k++;
        }
        if constexpr (W > 1) {
            const unsigned all[4] = {~0u, ~0u, ~0u, ~0u};
#pragma unroll
            for (int q = 0; q < 8; q++) count_equal(pc[q], diff[q], all);
        }
        __syncthreads();   // this stage is free for the copy after next
    }
}

// Owners and pairs with entries of V; d: determinants, ck: checkpoints, s1 and s2: sums, on the device.
template <typename V>
cudaError_t launch_colocation(const u64 *d, i64 n, i64 npad, int nw, i64 t_max, int nu_move, u64 n_ranks, int nb, void *planes,
                              const i64 *ck, int nck, u64 *s1, u64 *s2, cudaStream_t sm)
{
    const int entry = (TILE_I + TILE_J) * (int)sizeof(V);
    // the limit belongs to the kernel, not to the launch: every call sets the
    // same one, so that a call of another thread cannot lower it in between
    const cudaError_t e = cudaFuncSetAttribute(k_pairs<V>, cudaFuncAttributeMaxDynamicSharedMemorySize, 2 * MAX_PLANES * entry);
    if (e != cudaSuccess) return e;
    k_owner_planes<V><<<1216, 256, 0, sm>>>(d, n, npad, nw, t_max, nu_move, n_ranks, nb, (V *)planes);
    k_pairs<V><<<dim3((unsigned)(npad / TILE_J), (unsigned)((n + TILE_I - 1) / TILE_I)), 256, 2 * nb * entry, sm>>>(
        (const V *)planes, n, npad, nb, t_max, ck, nck, s1, s2);
    return cudaGetLastError();
}

}  // namespace
}  // namespace ccmc

extern "C" ccmc_status ccmc_colocation(const uint64_t *dets, size_t n, int32_t n_words, int64_t n_ranks,
                                       int32_t nu_move, const int64_t *checkpoints, int32_t n_checkpoints,
                                       uint64_t *sum_c, uint64_t *sum_c2, void *cuda_stream)
{
    using namespace ccmc;
    if (!dets || !checkpoints || !sum_c || !sum_c2 || n < 2 || n > ((size_t)1 << 20) || n_words < 1 ||
        n_words > MAXK || n_ranks < 1 || n_ranks > 65535 || nu_move < 0 || n_checkpoints < 1 ||
        n_checkpoints > MAX_CHECKPOINTS)
        return CCMC_ERR_ARG;
    for (int k = 0; k < n_checkpoints; k++)
        if (checkpoints[k] < 1 || (k > 0 && checkpoints[k] <= checkpoints[k - 1])) return CCMC_ERR_ARG;
    const i64 t_max = checkpoints[n_checkpoints - 1];
    if (t_max > ((i64)1 << 20)) return CCMC_ERR_ARG;
    cudaStream_t sm = (cudaStream_t)cuda_stream;
    ccmc_status st = CCMC_OK;
    const size_t nn = n, nw = (size_t)n_words, nck = (size_t)n_checkpoints;
    int nb = 1;
    while ((n_ranks - 1) >> nb) nb++;
    // one block of device memory: planes (padded to whole tiles), determinants, sums, checkpoints
    const size_t npad = (nn + TILE_J - 1) / TILE_J * TILE_J;
    const bool narrow = t_max <= group_of<unsigned>;
    const size_t groups = ((size_t)t_max + group_of<uint4> - 1) / group_of<uint4>;
    const size_t planes_bytes = groups * (size_t)nb * npad * (narrow ? sizeof(unsigned) : sizeof(uint4));
    void *mem = nullptr;
    // (from the device's stream-ordered pool: a cudaMalloc and cudaFree cost a
    // small call 90 us more; the pool keeps nothing past the next synchronisation)
    if (cudaMallocAsync(&mem, planes_bytes + 8 * (nn * nw + 3 * nck), sm) != cudaSuccess) {
        cudaGetLastError();
        return CCMC_ERR_OOM;
    }
    u64 *d_dets = (u64 *)((unsigned char *)mem + planes_bytes), *d_s1 = d_dets + nn * nw, *d_s2 = d_s1 + nck;
    i64 *d_ck = (i64 *)(d_s2 + nck);
    if (cudaMemcpyAsync(d_dets, dets, nn * nw * 8, cudaMemcpyHostToDevice, sm) != cudaSuccess ||
        cudaMemcpyAsync(d_ck, checkpoints, nck * 8, cudaMemcpyHostToDevice, sm) != cudaSuccess ||
        cudaMemsetAsync(d_s1, 0, 2 * nck * 8, sm) != cudaSuccess) {
        st = CCMC_ERR_CUDA;
    } else {
        auto *launch = narrow ? launch_colocation<unsigned> : launch_colocation<uint4>;
        if (launch(d_dets, (i64)n, (i64)npad, n_words, t_max, nu_move, (u64)n_ranks, nb, mem, d_ck, n_checkpoints, d_s1, d_s2,
                   sm) != cudaSuccess ||
            cudaMemcpyAsync(sum_c, d_s1, nck * 8, cudaMemcpyDeviceToHost, sm) != cudaSuccess ||
            cudaMemcpyAsync(sum_c2, d_s2, nck * 8, cudaMemcpyDeviceToHost, sm) != cudaSuccess ||
            cudaStreamSynchronize(sm) != cudaSuccess)
            st = CCMC_ERR_CUDA;
    }
    if (st != CCMC_OK) cudaStreamSynchronize(sm);   // no copy may still use the caller's arrays
    cudaFreeAsync(mem, sm);
    return st;
}
