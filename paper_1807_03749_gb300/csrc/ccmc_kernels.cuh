// ccmc_kernels.cuh -- device code of one CCMC time step (Spencer et al.,
// arXiv:1807.03749, Sec. II and Sec. IV.B-C): the building blocks a1-a10,
// the kernels templated on the Hamiltonian kind and the precision R of the
// matrix elements, and the template that issues a whole step.  Each (kind, R)
// pair is instantiated in its own translation unit (ccmc_step_<kind>_<R>.cu)
// so that they compile in parallel; the kernels that depend on neither are
// defined once, in ccmc_step.cu.
//
//  a1  k_scan      : |t_i| prefix, N_total, t_HF, N_ex, n_sel, cluster
//      amplitudes; full non-composite visits (death and estimator of every
//      list entry, Sec. IV.B)
//  a2-a5 k_sample  : cluster selection, collapse with sign, death, estimator,
//      one spawning attempt inline or the cluster queued for multi-spawn
//  a4/a6 k_attempts: expanded multi-spawn attempts (Sec. IV.C)
//  a7-a10 k_annihilate: LSD radix sort of spawned records by rank key, sum of
//      each run of equal keys, merge into the list with the occupation
//      threshold and compaction, projected-energy numerator and record
//  batch k_sample_plan / k_sample_flat: the sampler as one persistent launch
//      over many replicas, with a work plan written on the device each step
#pragma once

#include "ccmc_state.cuh"

namespace ccmc {

#define FULLMASK 0xFFFFFFFFu

// ---------------------------------------------------------------------------
// Block and warp helpers
// ---------------------------------------------------------------------------

template <typename T>
__device__ __forceinline__ T warp_incl_scan(T v)
{
    const int lane = threadIdx.x & 31;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        T t = __shfl_up_sync(FULLMASK, v, o);
        if (lane >= o) v += t;
    }
    return v;
}

template <typename T>
__device__ __forceinline__ T warp_sum(T v)
{
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(FULLMASK, v, o);
    return v;
}

// inclusive scan of one value per thread; sm must hold 32 elements
template <typename T>
__device__ __forceinline__ T block_incl_scan(T v, T *sm, T &total)
{
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, nw = blockDim.x >> 5;
    T incl = warp_incl_scan(v);
    if (lane == 31) sm[wid] = incl;
    __syncthreads();
    if (wid == 0) {
        T w = lane < nw ? sm[lane] : T(0);
        T wi = warp_incl_scan(w);
        if (lane < nw) sm[lane] = wi;
    }
    __syncthreads();
    T off = wid > 0 ? sm[wid - 1] : T(0);
    total = sm[nw - 1];
    __syncthreads();
    return incl + off;
}

// Exclusive prefixes, in place, of four rows of blockDim.x values each (row by
// row), and their total: two barriers for the four rows.  sm holds 128.
__device__ __forceinline__ i64 block_scan4(i64 (&x)[4], i64 *sm)
{
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, nw = blockDim.x >> 5;
    i64 in[4];
    __syncthreads();   // an earlier call's reads of sm are done
#pragma unroll
    for (int r = 0; r < 4; r++) {
        in[r] = warp_incl_scan(x[r]);
        if (lane == 31) sm[r * nw + wid] = in[r];
    }
    __syncthreads();
    if (wid == 0) {
        i64 carry = 0;
        for (int q = 0; q < 4 * nw; q += 32) {
            const i64 v = q + lane < 4 * nw ? sm[q + lane] : 0, i = warp_incl_scan(v);
            if (q + lane < 4 * nw) sm[q + lane] = carry + i - v;
            carry += __shfl_sync(FULLMASK, i, 31);
        }
        if (lane == 0) sm[127] = carry;
    }
    __syncthreads();
#pragma unroll
    for (int r = 0; r < 4; r++) x[r] = sm[r * nw + wid] + in[r] - x[r];
    return sm[127];
}

template <typename T>
__device__ __forceinline__ T block_sum(T v, T *sm)
{
    T tot;
    block_incl_scan(v, sm, tot);
    return tot;
}

__device__ __forceinline__ Fix128 warp_fix(Fix128 v)
{
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        Fix128 t;
        t.lo = __shfl_xor_sync(FULLMASK, v.lo, o);
        t.hi = __shfl_xor_sync(FULLMASK, v.hi, o);
        v.add(t);
    }
    return v;
}

// integer block sum of Fix128 values; sm holds 64 u64; the result is valid in thread 0
__device__ __forceinline__ Fix128 block_fix(Fix128 v, u64 *sm)
{
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, nw = blockDim.x >> 5;
    v = warp_fix(v);
    if (lane == 0) {
        sm[2 * wid] = v.lo;
        sm[2 * wid + 1] = v.hi;
    }
    __syncthreads();
    Fix128 r = {0, 0};
    if (wid == 0) {
        if (lane < nw) {
            r.lo = sm[2 * lane];
            r.hi = sm[2 * lane + 1];
        }
        r = warp_fix(r);
    }
    __syncthreads();
    return r;
}

// ---------------------------------------------------------------------------
// Teams: the blocks of one replica that work on a phase together.  A kernel's
// team size follows the step's sizes, so that a short list or few records
// are handled by one block (its barriers are the block's own) and a long list
// by all of them, without a launch per phase: 12 to 24 launches of a step,
// most with nothing to do on small systems, became two (a step of the
// 38-orbital gas, 289 excitors: 85 -> 44 us; of the 114-orbital gas with 90,000:
// 318 -> 307 us; of the 1.1e7-excitor molecule: the same).  A barrier costs 2 to
// 4 us with tens to hundreds of blocks, less than a launch and its ramp.  The blocks of a team
// wait for each other, so a launch with more than one block per replica is
// cooperative (all resident), and every wait has a limit.
//
// A wait that runs out ends the step and every later one: the block sets
// ERRB_TIMEOUT and returns, and a kernel that finds the bit set at its start
// returns too, because the barrier words and the step's tables are then
// unfinished.  Within the launch no barrier opens too soon: a block gives up
// only after it has arrived, so the barrier it left still counts it, and the
// next one lacks it and never opens.  The next list (ccmc_set_list) clears the
// bit and the barrier words.
// ---------------------------------------------------------------------------

struct Team {
    int id, n;   // this block, blocks in the team
};

// contiguous share [lo, hi) of n elements for this block
__device__ __forceinline__ void chunk_of(Team t, i64 n, i64 &lo, i64 &hi)
{
    const i64 c = (n + t.n - 1) / t.n;
    lo = t.id * c < n ? t.id * c : n;
    hi = lo + c < n ? lo + c : n;
}

constexpr unsigned TEAM_SPINS = 1u << 24;   // polls of a wait: some ten seconds

// All threads of the team's blocks call.  bar[0] counts arrivals, bar[1] the
// barrier's generation; both are left as found plus one generation.  False if
// the wait ran out (or another block's did, which will not come to the next
// barrier): the bit is set, the caller returns.
__device__ __forceinline__ bool team_sync(unsigned *bar, Team t, DevStep *st)
{
    __shared__ int s_ok;
    __syncthreads();
    if (t.n <= 1) return true;
    if (threadIdx.x == 0) {
        // release on arrival, acquire on leaving; the block's other threads
        // are ordered with this one by the block barriers
        unsigned *gen = bar + 1, g, got;
        int ok = 1;
        asm volatile("ld.relaxed.gpu.global.u32 %0, [%1];" : "=r"(g) : "l"(gen) : "memory");   // cannot advance before this block arrives
        asm volatile("atom.add.acq_rel.gpu.global.u32 %0, [%1], 1;" : "=r"(got) : "l"(bar) : "memory");
        if (got == (unsigned)t.n - 1u) {
            asm volatile("st.relaxed.gpu.global.u32 [%0], 0;" ::"l"(bar) : "memory");
            asm volatile("red.release.gpu.global.add.u32 [%0], 1;" ::"l"(gen) : "memory");
        } else {
            const unsigned limit = st->wait_limit ? st->wait_limit : TEAM_SPINS;
            for (unsigned spins = 1;; spins++) {
                unsigned now;
                asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(now) : "l"(gen) : "memory");
                if (now != g) break;
                if (spins >= limit || ((spins & 1023u) == 0 && (__ldcg(&st->err) & ERRB_TIMEOUT))) {
                    atomicOr(&st->err, (unsigned)ERRB_TIMEOUT);
                    ok = 0;
                    break;
                }
            }
        }
        s_ok = ok;
    }
    __syncthreads();
    return s_ok != 0;
}

// sum of the partials v[stride b] of the blocks before this one, and of all
__device__ __forceinline__ void team_prefix(const i64 *v, int stride, Team t, i64 *sm, i64 &before, i64 &total)
{
    if (t.n == 1) {
        before = 0;
        total = __ldcg(v);
        return;
    }
    i64 a = 0, b = 0;
    for (int q = threadIdx.x; q < t.n; q += blockDim.x) {
        const i64 x = __ldcg(&v[(size_t)stride * q]);
        b += x;
        if (q < t.id) a += x;
    }
    a = warp_sum(a);
    b = warp_sum(b);
    const int wid = threadIdx.x >> 5, nw = blockDim.x >> 5;
    __syncthreads();
    if ((threadIdx.x & 31) == 0) {
        sm[2 * wid] = a;
        sm[2 * wid + 1] = b;
    }
    __syncthreads();
    before = total = 0;
    for (int w = 0; w < nw; w++) {
        before += sm[2 * w];
        total += sm[2 * w + 1];
    }
}

__device__ __forceinline__ u64 warp_reserve_u64(u64 *counter, u64 count)
{
    const int lane = threadIdx.x & 31;
    u64 incl = warp_incl_scan(count);
    u64 total = __shfl_sync(FULLMASK, incl, 31);
    u64 base = 0;
    if (lane == 31 && total) base = atomicAdd((unsigned long long *)counter, (unsigned long long)total);
    base = __shfl_sync(FULLMASK, base, 31);
    return base + incl - count;
}

// divisions that a step does once or seldom, out of line: each is some
// hundred instructions
static __device__ __noinline__ double div_rn(double a, double b) { return a / b; }

// n_attempts = max(1, floor(|A| / A_thresh)) with multi-spawn, else 1
static __device__ __noinline__ i64 attempts_of_thresh(double amp_abs, double a_thresh)
{
    double q = floor(amp_abs / a_thresh);
    return q < 1.0 ? 1 : (i64)q;
}

__device__ __forceinline__ i64 attempts_of(double amp_abs, const RunParams &p)
{
    if (!p.multispawn) return 1;
    if (p.a_thresh_one) {
        // floor(|A|) from the bit pattern (A / 1.0 == A exactly)
        u64 M;
        int E;
        split_double((u64)__double_as_longlong(amp_abs) & 0x7FFFFFFFFFFFFFFFULL, M, E);
        u64 q = E >= 0 ? (E >= 10 ? (1ULL << 62) : (M << E)) : (E <= -64 ? 0 : (M >> -E));
        return q < 1 ? 1 : (i64)q;
    }
    return attempts_of_thresh(amp_abs, p.a_thresh);
}

// rounding with a cutoff that is no power of two (FP64 decisions)
static __device__ __noinline__ bool round_value_fp(double x, u64 r, double cutoff, i64 *out)
{
    return stoch_round(x, unif(r), cutoff, *out);
}

// stochastic rounding of a spawned (with cutoff) or death (without) value
__device__ __forceinline__ bool round_value(double x, u64 r, const RunParams &p, bool spawn, i64 &out)
{
    if (p.int_round) return stoch_round_bits((u64)__double_as_longlong(x), r, spawn ? p.spawn_rs : p.death_rs, out);
    return round_value_fp(x, r, spawn ? p.spawn_cutoff : 0.0, &out);
}

// smallest i in [1, n-1] with prefix[i] > x (excitor owning position x); the
// bucket of x brackets the answer between the owners of its first position
// and of the next bucket's first position
__device__ __forceinline__ void pick_bracket(const int *bucket, int shift, int nbuckets, int n, u64 x, int &lo, int &hi)
{
    const int b = (int)(x >> shift);
    lo = __ldg(&bucket[b]);
    hi = b + 1 < nbuckets ? __ldg(&bucket[b + 1]) : n - 1;
}

__device__ __forceinline__ int pick_index(const PickEntry *pk, const int *bucket, int shift, int nbuckets, int n, u64 x)
{
    int lo, hi;
    pick_bracket(bucket, shift, nbuckets, n, x, lo, hi);
    while (lo < hi) {
        const int mid = lo + (hi - lo) / 2;
        if ((u64)__ldg(&pk[mid].prefix) > x) hi = mid;
        else lo = mid + 1;
    }
    return lo;
}

// two picks of one sample, their searches in step so that both loads of a
// round are in flight together
__device__ __forceinline__ void pick_two(const PickEntry *pk, const int *bucket, int shift, int nbuckets, int n, u64 x0,
                                         u64 x1, bool two, int &i0, int &i1)
{
    int lo0, hi0, lo1 = 1, hi1 = 1;
    pick_bracket(bucket, shift, nbuckets, n, x0, lo0, hi0);
    if (two) pick_bracket(bucket, shift, nbuckets, n, x1, lo1, hi1);
    while (lo0 < hi0 || lo1 < hi1) {
        const int m0 = lo0 + (hi0 - lo0) / 2, m1 = lo1 + (hi1 - lo1) / 2;
        const u64 p0 = lo0 < hi0 ? (u64)__ldg(&pk[m0].prefix) : 0;
        const u64 p1 = lo1 < hi1 ? (u64)__ldg(&pk[m1].prefix) : 0;
        if (lo0 < hi0) {
            if (p0 > x0) hi0 = m0;
            else lo0 = m0 + 1;
        }
        if (lo1 < hi1) {
            if (p1 > x1) hi1 = m1;
            else lo1 = m1 + 1;
        }
    }
    i0 = lo0;
    i1 = lo1;
}

// the excitor of a pick row
__device__ __forceinline__ Exc row_exc(const PickEntry *pk, i64 id, u64 &flags)
{
    const u64 h = __ldg(&pk[id].h), p = __ldg(&pk[id].p);
    flags = p;
    return exc_of(h, p);
}

// Simulated distribution (Sec. III): the excitor of processor q holding
// position x in [0, N_q) of that processor's entries in list order -- the
// chunk whose processor-q prefix brackets x, then a walk over the chunk;
// -1 only if the tables were inconsistent
__device__ __forceinline__ i64 local_pick(const WorkArrays &wa, const i64 *pop, i64 n, int lcs, i64 nlc, u64 q,
                                          u64 x)
{
    const i64 *row = wa.lcp + (i64)q * nlc;
    i64 lo = 0, hi = nlc - 1;   // last chunk c with row[c] <= x
    while (lo < hi) {
        const i64 mid = (lo + hi + 1) >> 1;
        if ((u64)__ldg(&row[mid]) <= x) lo = mid;
        else hi = mid - 1;
    }
    u64 acc = (u64)__ldg(&row[lo]);
    const i64 b = lo << lcs, e = b + (1LL << lcs) < n ? b + (1LL << lcs) : n;
    for (i64 i = b > 1 ? b : 1; i < e; i++) {
        if (__ldg(&wa.owner[i]) != q) continue;
        const i64 v = __ldg(&pop[i]);
        acc += (u64)(v < 0 ? -v : v);
        if (acc > x) return i;
    }
    return -1;
}

// smallest i in [lo, hi] with end[i] > t (the answer is known to lie there)
__device__ __forceinline__ i64 owner_in(const i64 *end, i64 lo, i64 hi, i64 t)
{
    while (lo < hi) {
        i64 mid = lo + (hi - lo) / 2;
        if (__ldg(&end[mid]) > t) hi = mid;
        else lo = mid + 1;
    }
    return lo;
}

// Attempt ranges: entry e owns attempts [end[e-1], end[e]) with end strictly
// increasing (every entry has at least one attempt), so 32 consecutive
// entries always cover 32 consecutive attempts.  A warp walks a contiguous
// chunk of attempts with a sliding window of 32 entry ends (one coalesced
// load per 32 attempts) and finds each lane's owner by a 5-step search over
// the window held in registers.
struct AttemptWindow {
    i64 cur;      // owner of the first attempt of the current 32
    i64 prev;     // end[cur - 1] (0 when cur == 0)
};

__device__ __forceinline__ AttemptWindow window_start(const i64 *end, i64 n, i64 t0)
{
    const int lane = threadIdx.x & 31;
    AttemptWindow w;
    i64 c = lane == 0 ? owner_in(end, 0, n - 1, t0) : 0;
    w.cur = __shfl_sync(FULLMASK, c, 0);
    i64 pv = (lane == 0 && w.cur > 0) ? end[w.cur - 1] : 0;
    w.prev = __shfl_sync(FULLMASK, pv, 0);
    return w;
}

// owner and attempt number of t = t0 + lane; advances the window past t0 + 31
__device__ __forceinline__ void window_step(const i64 *end, i64 n, i64 t0, AttemptWindow &w, i64 &owner, i64 &m)
{
    const int lane = threadIdx.x & 31;
    const i64 t = t0 + lane;
    const i64 e = w.cur + lane;
    const i64 ev = e < n ? __ldg(&end[e]) : 0x7FFFFFFFFFFFFFFFLL;
    int L = 0;
#pragma unroll
    for (int st = 16; st >= 1; st >>= 1) {
        i64 v = __shfl_sync(FULLMASK, ev, L + st - 1);
        if (v <= t) L += st;
    }
    i64 before = __shfl_sync(FULLMASK, ev, L > 0 ? L - 1 : 0);
    owner = w.cur + L;
    m = t - (L > 0 ? before : w.prev);
    // entries whose attempts all lie before t0 + 32 are finished; the next
    // window starts at the owner of attempt t0 + 32
    unsigned done = __ballot_sync(FULLMASK, ev <= t0 + 32);
    int adv = __popc(done);
    if (adv > 0) w.prev = __shfl_sync(FULLMASK, ev, adv - 1);
    w.cur += adv;
}

// One spawning attempt from dj carrying coefficient c_att (Sec. II):
// value -dtau H_ij c_att s_D(i) / p_gen, stochastically rounded, in two
// halves.  excite() runs the excitation generator and the truncation check
// (about nine draws in ten end there for the gas); attempt_finish computes the
// matrix element, the value, its stochastic rounding and the rank key.  The
// surviving draws are queued per warp and finished 32 at a time, so the second
// half runs on full warps.
template <typename R, bool GAS>
__device__ __forceinline__ bool attempt_finish(const SysDev &s, const RunParams &p, const Exc &dj, double c_att,
                                               u64 r3, u64 code, u64 &key, i64 &val, unsigned &err)
{
    const int i = (int)code & 1023, j = (int)(code >> 10) & 1023, a = (int)(code >> 20) & 1023,
              b = (int)(code >> 30) & 1023, gc = (int)(code >> 40) & 7;
    const bool dbl = GAS || gc == 0 || gc >= 3;
    int par;
    const Exc di = excited(s, dj, dbl, i, j, a, b, par);
    // matrix element and 1/p_gen in the precision R; the value itself in FP64
    double h = h_offdiag<R, GAS>(s, dj, dbl, i, j, a, b, par);
    double x = ((p.tau * h) * inv_pgen_of<R>(s, gc)) * c_att;
    if (!sign_parity(s, di)) x = -x;
    i64 v;
    if (!round_value(x, r3, p, true, v)) {
        err |= ERRB_NUMERIC;
        return false;
    }
    if (v == 0) return false;
    key = rank_key(s, di);
    val = v;
    return true;
}

// Per-warp queue of drawn attempts waiting for attempt_finish.
struct AttQueue {
    u64 h[64], p[64];
    double c[64];
    u64 r[64];
    u64 code[64];
};

// All 32 lanes call; lanes with ok append their attempt (qn < 32 on entry).
__device__ __forceinline__ void q_push(AttQueue &q, int &qn, bool ok, const Exc &dj, double c, u64 r3, u64 code)
{
    const int lane = threadIdx.x & 31;
    const unsigned m = __ballot_sync(FULLMASK, ok);
    if (ok) {
        const int e = qn + __popc(m & ((1u << lane) - 1u));
        q.h[e] = pack_h(dj);
        q.p[e] = dj.p;
        q.c[e] = c;
        q.r[e] = r3;
        q.code[e] = code;
    }
    qn += __popc(m);
    __syncwarp();
}

// Per-warp staging of spawned records: appended by ballot, written to the
// spawn buffer 32 at a time (one atomic per 32 records, 256-byte runs).
struct RecStage {
    u64 key[64];
    i64 val[64];
};

// All 32 lanes call; lanes with has append their record (rn < 32 on entry).
__device__ __forceinline__ void rec_push(RecStage &rs, int &rn, bool has, u64 k, i64 v)
{
    const int lane = threadIdx.x & 31;
    const unsigned m = __ballot_sync(FULLMASK, has);
    if (has) {
        const int e = rn + __popc(m & ((1u << lane) - 1u));
        rs.key[e] = k;
        rs.val[e] = v;
    }
    rn += __popc(m);
    __syncwarp();
}

// Direct accumulation (annihilation fast path): a spawned record whose key
// is already in the sorted excip list is added to that entry's matched-spawn
// sum with an integer atomic instead of going through the sort; only keys new
// to the list are appended to the spawn buffer.  Integer sums make the merged
// list identical either way.  The key buckets (entries whose key >> kshift
// equals b start at kbucket[b]) narrow each search to a few entries.
struct DirectView {
    const u64 *key;      // the list's keys, ascending
    const int *kb;       // key buckets
    i64 *acc;            // matched-spawn sums per entry
    unsigned char *hit;  // entries that received a direct record
    i64 n, nkb;          // list size, buckets in use (0: off)
    int ks;              // key-bucket shift
};

__device__ __forceinline__ DirectView direct_view(const ListView &L, const WorkArrays &wa, const DevStep *st)
{
    DirectView d;
    d.key = L.key;
    d.kb = wa.kbucket;
    d.acc = wa.acc;
    d.hit = wa.hit;
    d.n = st->n_occ;
    d.nkb = st->nkb;
    d.ks = st->kshift;
    return d;
}

// index of key k in the list, or -1
__device__ __forceinline__ i64 find_key(const DirectView &d, u64 k)
{
    const u64 b = k >> d.ks;
    if (b >= (u64)d.nkb) return -1;
    i64 lo = __ldg(&d.kb[b]);
    i64 hi = b + 1 < (u64)d.nkb ? (i64)__ldg(&d.kb[b + 1]) : d.n;
    while (lo < hi) {
        const i64 mid = lo + (hi - lo) / 2;
        if (__ldg(&d.key[mid]) < k) lo = mid + 1;
        else hi = mid;
    }
    return (lo < d.n && __ldg(&d.key[lo]) == k) ? lo : -1;
}

// All 32 lanes call: takes the newest (at most 32) staged records; records
// onto listed determinants are added to them directly, the others appended to
// the spawn buffer with one atomic per warp.
__device__ __forceinline__ void rec_flush_once(RecStage &rs, int &rn, DevStep *st, const SpawnBuf &sp,
                                               const DirectView &dv, unsigned &ndirect, unsigned &err)
{
    const int lane = threadIdx.x & 31;
    const int take = rn >= 32 ? 32 : rn;
    bool app = lane < take;
    u64 k = 0;
    i64 v = 0;
    if (app) {
        const int e = rn - take + lane;
        k = rs.key[e];
        v = rs.val[e];
    }
    __syncwarp();   // the stage is read before later pushes reuse it
    rn -= take;
    if (app && dv.nkb > 0) {
        const i64 pos = find_key(dv, k);
        if (pos >= 0) {
            atomicAdd((unsigned long long *)&dv.acc[pos], (unsigned long long)v);
            dv.hit[pos] = 1;
            ndirect++;
            app = false;
        }
    }
    const unsigned m = __ballot_sync(FULLMASK, app);
    if (m == 0) return;
    i64 base = 0;
    if (lane == 0) base = (i64)atomicAdd((unsigned long long *)&st->n_sp, (unsigned long long)__popc(m));
    base = __shfl_sync(FULLMASK, base, 0);
    if (app) {
        const i64 off = base + __popc(m & ((1u << lane) - 1u));
        if (off < sp.cap) {
            sp.key[0][off] = k;
            sp.pop[0][off] = v;
        } else {
            err |= ERRB_SPAWN_OVERFLOW;
        }
    }
}

// All 32 lanes call: finishes the newest (at most 32) queued attempts into
// the record stage (rn < 32 on entry).
template <typename R, bool GAS>
__device__ __forceinline__ void q_finish(AttQueue &q, int &qn, RecStage &rs, int &rn, const SysDev &s,
                                         const RunParams &p, unsigned &err)
{
    const int lane = threadIdx.x & 31;
    const int take = qn >= 32 ? 32 : qn;
    bool has = false;
    u64 k = 0;
    i64 v = 0;
    if (lane < take) {
        const int e = qn - take + lane;
        has = attempt_finish<R, GAS>(s, p, exc_of(q.h[e], q.p[e]), q.c[e], q.r[e], q.code[e], k, v, err);
    }
    __syncwarp();   // the entries are read before later pushes reuse them
    qn -= take;
    rec_push(rs, rn, has, k, v);
}

// occupation threshold: 0 < |v| < 1 becomes +-1 with probability |v|, else 0
__device__ __forceinline__ i64 threshold(const RunParams &p, u64 it, u64 key, i64 v)
{
    i64 av = v < 0 ? -v : v;
    if (av > 0 && av < (i64)FIX_ONE) {
        R4 r = draw(p.seed, p.replica, it, TAG_THRESH, key, 0);
        bool keep = (r.v[0] >> 11) < ((u64)av << 37);
        return keep ? (v < 0 ? -(i64)FIX_ONE : (i64)FIX_ONE) : 0;
    }
    return v;
}

// ---------------------------------------------------------------------------
// a1: scans over the list
// ---------------------------------------------------------------------------

// Blocks of the list scan: one per 512 entries (one row of 32 per warp).
__device__ __forceinline__ i64 scan_blocks(i64 n)
{
    const i64 b = (n + SCAN_THREADS - 1) / SCAN_THREADS;
    return b < 1 ? 1 : b;
}

// this warp's entries of the list: warp-granular chunks need no block barrier
__device__ __forceinline__ void warp_chunk_of(Team t, i64 n, i64 &lo, i64 &hi)
{
    const i64 W = (i64)t.n * (SCAN_THREADS / 32), q = (i64)t.id * (SCAN_THREADS / 32) + (threadIdx.x >> 5);
    const i64 c = (n + W - 1) / W;
    lo = q * c < n ? q * c : n;
    hi = lo + c < n ? lo + c : n;
}

// |t_i| and attempts of this warp's entries, and the block's sums in part[4 id]
__device__ __forceinline__ void d_scan_partial(const ListView &L, const DevStep *st, const RunParams &p,
                                               const WorkArrays &wa, Team t, i64 &sw, i64 &sa, i64 *sm)
{
    i64 lo, hi;
    warp_chunk_of(t, st->n_occ, lo, hi);
    sw = sa = 0;
    for (i64 i = lo + (threadIdx.x & 31); i < hi; i += 32) {
        i64 v = L.pop[i], av = v < 0 ? -v : v;
        if (i > 0) sw += av;
        if (p.fnc) sa += attempts_of(fabs((double)v / FIX_ONE), p);
    }
    sw = warp_sum(sw);
    sa = warp_sum(sa);
    const int wid = threadIdx.x >> 5;
    if ((threadIdx.x & 31) == 0) {
        sm[2 * wid] = sw;
        sm[2 * wid + 1] = sa;
    }
    __syncthreads();
    i64 bw = 0, ba = 0, tw = 0, ta = 0;   // before this warp, and the block's
    for (int w = 0; w < SCAN_THREADS / 32; w++) {
        if (w == wid) {
            bw = tw;
            ba = ta;
        }
        tw += sm[2 * w];
        ta += sm[2 * w + 1];
    }
    sw = bw;
    sa = ba;
    if (threadIdx.x == 0) {
        wa.part[4 * t.id] = tw;
        wa.part[4 * t.id + 1] = ta;
    }
}

// What the final pass needs of the step's scalars; every block computes them.
struct ScanScalars {
    int bshift, kshift;
    i64 nkb;
};

// The step's scalars from the totals tw = N_ex and ta (full non-composite
// attempts).  Every block calls; the first one stores them.
__device__ __forceinline__ ScanScalars d_scan_top(const ListView &L, DevStep *st, const RunParams &p, const WorkArrays &wa,
                                                  i64 tw, i64 ta, int lmax, Team team)
{
    const i64 n_occ = st->n_occ;
    const i64 n0 = n_occ > 0 ? L.pop[0] : 0;
    const i64 an0 = n0 < 0 ? -n0 : n0;
    const i64 ntot = an0 + tw;
    i64 n_sel = (ntot + 32768) >> 16;
    // a runaway population: abandon the step instead of sampling it
    const bool runaway = n_sel > p.work_cap || (p.fnc && ta > p.work_cap);
    if (runaway) {
        n_sel = 0;
        ta = 0;
    }
    ScanScalars r;
    // selection buckets: the smallest power of two 2^k with N_ex <= 2^(k + bucket_bits),
    // about two buckets per list entry (bounded by the bucket array), and for
    // a short list sampled often up to one per 32 samples: its populations
    // span decades, so that equal ranges of positions hold from none to
    // hundreds of its entries
    i64 nb_want = n_sel >> 5 < (1LL << 18) ? n_sel >> 5 : (1LL << 18);
    if (nb_want < 2 * n_occ) nb_want = 2 * n_occ;
    int bb = nb_want > 16 ? 64 - __clzll(nb_want - 1) : 4;   // smallest with 2^bb >= nb_want
    bb = bb < wa.bucket_bits ? bb : wa.bucket_bits;
    r.bshift = max(0, 64 - __clzll(tw) - bb);                 // smallest with tw < 2^(bshift + bb)
    // key buckets for direct accumulation: about two per list entry over the
    // list's key range (up to eight for a short list: the keys cluster),
    // within the table's capacity.  Direct accumulation pays once the step
    // spawns more than about one record per ten list entries (the buckets
    // cost a pass over the list, a sorted record several); the choice follows
    // the previous step and does not change any result
    r.kshift = 0;
    r.nkb = 0;
    if (p.direct && n_occ > 0 && 10 * st->prev_spawned > n_occ) {
        const u64 kmax = L.key[n_occ - 1];
        i64 want = 8 * n_occ < (1LL << 18) ? 8 * n_occ : (1LL << 18);
        if (want < 2 * n_occ) want = 2 * n_occ;
        if (want > (1LL << wa.kbucket_bits)) want = 1LL << wa.kbucket_bits;
        r.kshift = max(0, __clzll(want) - __clzll((i64)kmax) - 1);   // at most two below the smallest that fits
        while (r.kshift < 63 && (i64)(kmax >> r.kshift) + 1 > want) r.kshift++;
        r.nkb = (i64)(kmax >> r.kshift) + 1;
    }
    if (team.id != 0) return r;
    if (threadIdx.x < 8) {
        // |A_s| = N_ex^s / (|t_HF|^(s-1) n_sel p(s) s!), fixed operation order; one size per thread
        const int s = threadIdx.x, smax = lmax + 2;
        double mag = 0.0, mden = 0.0;
        if (s <= smax && n_sel > 0 && !(p.fnc && s < 2)) {
            const double nex_d = (double)tw / FIX_ONE, n0_d = (double)an0 / FIX_ONE;
            double pr;
            const int k = p.fnc ? (s < smax ? s - 1 : lmax) : (s < smax ? s + 1 : lmax + 2);   // p(s) = 2^-k
            pr = __longlong_as_double((i64)(1023 - k) << 52);
            if (s == 0) {
                mag = div_rn(n0_d, (double)n_sel * pr);
            } else {
                double num = 1.0, den = 1.0, fact = 1.0;
                for (int e = 0; e < s; e++) num = num * nex_d;
                for (int e = 0; e < s - 1; e++) den = den * n0_d;
                for (int e = 2; e <= s; e++) fact = fact * (double)e;
                den = den * (double)n_sel;
                den = den * pr;
                den = den * fact;
                mag = div_rn(num, den);
                mden = den;
            }
        }
        st->mag[s] = mag;
        st->mden[s] = mden;
        if (s == 0) {
            // every reference cluster has this coefficient and death value
            // (the reference's sign s_D is +1): its rounding once per step
            const double coef = n0 < 0 ? -mag : mag;
            const double x = -((p.tau * (0.0 - st->shift)) * coef);
            RoundCut cut = {0, 0, 0};
            st->hf_ok = !p.int_round || round_cut((u64)__double_as_longlong(x), p.death_rs, cut);
            st->hf_coef = coef;
            st->hf_death = x;
            st->hf_cut = cut;
        }
        // every cluster of size s has |A| = mag[s]: its attempt count and
        // the magnitude of one attempt's coefficient, once per step
        const i64 na = attempts_of(mag, p);
        st->natt_s[s] = na;
        st->cmag[s] = na > 1 ? div_rn(mag, (double)na) : mag;
    }
    if (threadIdx.x == 32) {
        if (runaway) atomicOr(&st->err, (unsigned)ERRB_RUNAWAY);
        st->n0 = n0;
        st->ntot = ntot;
        st->nex = tw;
        st->bucket_shift = r.bshift;
        st->nbuckets = tw > 0 ? (i64)(((u64)tw + (1ULL << r.bshift) - 1) >> r.bshift) : 0;
        st->n_sel = n_sel;
        st->fnc_attempts = p.fnc ? ta : 0;
        st->scan_blocks = team.n;
        st->n_step = n_occ;
        st->n_direct = 0;
        st->n_hit = 0;
        st->kshift = r.kshift;
        st->nkb = r.nkb;
        // simulated distribution: chunks of 2^lcs entries, as fine as the
        // per-processor position table allows
        if (p.nranks > 1) {
            int c = 5;
            while (c < 40 && (i64)p.nranks * ((n_occ + (1LL << c) - 1) >> c) > wa.lcp_cap) c++;
            st->lcs = c;
            st->nlc = (n_occ + (1LL << c) - 1) >> c;
        }
        st->n_sp = 0;
        st->cl_packed = 0;
        st->cl_att = 0.0;
        st->n_attempts = 0;
        st->n_keys = 0;
        st->kept_list = 0;
        st->kept_new = 0;
        st->ntot_after = 0;
    }
    return r;
}

// All 32 lanes call: each lane's run [b0, b1) of t (empty if b1 <= b0) is set
// to v.  Runs of up to 8 are written by their lane; longer ones (an excitor
// holding many particles, a gap in the keys) by the whole warp, one after
// another.
__device__ __forceinline__ void fill_run(int *t, i64 b0, i64 b1, int v)
{
    const int lane = threadIdx.x & 31;
    const bool lng = b1 - b0 > 8;
    if (!lng)
#pragma unroll 1
        for (i64 b = b0; b < b1; b++) t[b] = v;
    unsigned m = __ballot_sync(FULLMASK, lng);
#pragma unroll 1
    while (m) {
        const int src = __ffs(m) - 1;
        m &= m - 1;
        const i64 s0 = __shfl_sync(FULLMASK, b0, src), s1 = __shfl_sync(FULLMASK, b1, src);
        const int sv = __shfl_sync(FULLMASK, v, src);
        for (i64 b = s0 + lane; b < s1; b += 32) t[b] = sv;
    }
}

// prefix arrays; with full non-composite sampling also every visit's death,
// estimator contribution and attempt coefficient (Sec. IV.B)
template <typename R, bool GAS>
__device__ __forceinline__ void d_scan_final(const SysDev &s, const ListView &L, DevStep *st, const RunParams &p,
                                             const WorkArrays &wa, Team t, i64 cw, i64 ca, const ScanScalars &sc)
{
    __shared__ u64 smf[64];
    i64 lo, hi;
    warp_chunk_of(t, st->n_occ, lo, hi);
    const u64 it = st->iter;
    const double S = st->shift;
    Fix128 es = {0, 0};
    unsigned err = 0;
    const bool kb = sc.nkb > 0;
    const int bsh = sc.bshift, ksh = sc.kshift;
    // each warp scans its own chunk 32 entries at a time (no block barrier)
#pragma unroll 1
    for (i64 base = lo; base < hi; base += 32) {
        i64 i = base + (threadIdx.x & 31);
        bool ok = i < hi;
        // every read of the entry is issued before the warp scans, so that
        // one memory latency per tile is exposed instead of two
        i64 v = ok ? L.pop[i] : 0, av = v < 0 ? -v : v;
        const u64 key_i = ok && kb ? L.key[i] : 0, key_p = ok && kb && i > 0 ? L.key[i - 1] : 0;
        const double diag_i = ok && i > 0 ? L.diag[i] : 0.0;
        const Exc d = ok ? exc_of(L.h[i], L.p[i]) : Exc{0, 0, 0};
        i64 w = (ok && i > 0) ? av : 0;
        double amp = (double)v / FIX_ONE;
        i64 na = (ok && p.fnc) ? attempts_of(fabs(amp), p) : 0;
        i64 ta = 0, ia = 0;
        const i64 iw = warp_incl_scan(w);
        const i64 tw = __shfl_sync(FULLMASK, iw, 31);
        if (p.fnc) {   // attempt prefix: full non-composite visits only
            ia = warp_incl_scan(na);
            ta = __shfl_sync(FULLMASK, ia, 31);
        }
        {
            // buckets whose first position falls in [prefix[i-1], prefix[i]) start at entry i
            const u64 p0 = (u64)(cw + iw - w), p1 = (u64)(cw + iw), half = (1ULL << bsh) - 1;
            fill_run(wa.bucket, (i64)((p0 + half) >> bsh), w > 0 ? (i64)((p1 + half) >> bsh) : 0, (int)i);
            // buckets whose first key falls in (key[i-1], key[i]] start at entry i
            if (kb) fill_run(wa.kbucket, i == 0 ? 0 : (i64)(key_p >> ksh) + 1, ok ? (i64)(key_i >> ksh) + 1 : 0, (int)i);
        }
        if (ok) {
            PickEntry pe;
            pe.prefix = cw + iw;
            wa.acc[i] = 0;
            wa.before[i] = 0;
            if (kb) {
                wa.hit[i] = 0;
            }
            const double td = p.tau * ((i == 0 ? 0.0 : diag_i) - S);
            const int odd = sign_parity(s, d);
            pe.tdeath = td;
            pe.h = pack_h(d);
            pe.p = d.p | (odd ? PICK_ODD : 0) | (v < 0 ? PICK_NEG : 0);
            i64 dv = 0;
            if (p.fnc) {
                wa.att_end[i] = ca + ia;
                double coef = odd ? -amp : amp;
                if (d.n == 1 || d.n == 2) es.add(to_fix(h_ref<R, GAS>(s, d) * coef));
                R4 r = draw(p.seed, p.replica, it, TAG_VISIT, (u64)i, 0);
                double x = td * coef;
                if (!odd) x = -x;
                if (!round_value(x, r.v[0], p, false, dv)) err |= ERRB_NUMERIC;
                wa.catt[i] = na > 1 ? div_rn(coef, (double)na) : coef;
            } else {
                // <HF|H|D_i> for the single-excitor clusters of the sampler (read at these levels only)
                if (d.n == 1 || d.n == 2) wa.href[i] = h_ref<R, GAS>(s, d);
            }
            wa.picks[i] = pe;
            wa.death[i] = dv;
        }
        cw += tw;
        ca += ta;
    }
    es = block_fix(es, smf);
    if (threadIdx.x == 0) {
        wa.enum_part[2 * t.id] = es.lo;
        wa.enum_part[2 * t.id + 1] = es.hi;
    }
    if (err) atomicOr(&st->err, err);   // every thread reports its own bits
}

// Simulated distribution (Sec. III): the owner of every excitor at this
// iteration (Eq. ccmc_dist) and, per chunk of 2^lcs list entries, the |pop|
// each processor holds in it; one warp per chunk, which clears its column of
// the table first (integer sums: the table does not depend on the order)
template <int K>
__device__ __forceinline__ void d_local_table(const SysDev &s, const ListView &L, const DevStep *st, const RunParams &p, const WorkArrays &wa)
{
    if (p.nranks <= 1) return;
    const i64 n = st->n_occ, nlc = st->nlc;
    const int lcs = st->lcs, lane = threadIdx.x & 31;
    const u64 it = st->iter;
    if (st->err & ERRB_TIMEOUT) return;
    const i64 nw = (i64)gridDim.x * (blockDim.x / 32);
    for (i64 c = (i64)blockIdx.x * (blockDim.x / 32) + (threadIdx.x >> 5); c < nlc; c += nw) {
        for (i64 q = lane; q < p.nranks; q += 32) wa.lcp[q * nlc + c] = 0;
        __syncwarp();
        const i64 b = c << lcs, e = b + (1LL << lcs) < n ? b + (1LL << lcs) : n;
        for (i64 i = b + lane; i < e; i += 32) {
            if (i == 0) continue;   // the reference is not an excitor
            const Det<K> d = words_from_exc<K>(s, exc_of(L.h[i], L.p[i]));
            const u64 q = words_owner(d.w, K, it, p.nu_move, (u64)p.nranks);
            wa.owner[i] = (unsigned short)q;
            const i64 v = L.pop[i];
            atomicAdd((unsigned long long *)&wa.lcp[(i64)q * nlc + c], (unsigned long long)(v < 0 ? -v : v));
        }
        __syncwarp();
    }
}

// each processor's row of the table turned into exclusive prefixes over the
// chunks; its total is N_q
__device__ __forceinline__ void d_local_scan(const DevStep *st, const RunParams &p, const WorkArrays &wa)
{
    __shared__ i64 sm[32];
    if (p.nranks <= 1) return;
    const i64 nlc = st->nlc;
    if (st->err & ERRB_TIMEOUT) return;
    for (i64 q = blockIdx.x; q < p.nranks; q += gridDim.x) {
        i64 *row = wa.lcp + q * nlc;
        i64 carry = 0;
        for (i64 base = 0; base < nlc; base += blockDim.x) {
            const i64 c = base + threadIdx.x;
            const i64 v = c < nlc ? row[c] : 0;
            i64 tot;
            const i64 incl = block_incl_scan(v, sm, tot);
            if (c < nlc) row[c] = carry + incl - v;
            carry += tot;
        }
        if (threadIdx.x == 0) wa.nq[q] = carry;
    }
}

// ---------------------------------------------------------------------------
// a2-a5: cluster sampling (Sec. II; composites only with FNC, Sec. IV.B)
// ---------------------------------------------------------------------------

// Per-warp shared memory of the sampler: samples waiting for their picks,
// samples of the bare reference, drawn attempts and spawned records.
struct SampWarp {
    u64 g[64], v1[64], v2[64], v3[64];   // sample index and the selection draw's words 1-3
    u64 hg[64];                          // sample indices of reference clusters
    unsigned char sz[64];                // cluster sizes of the waiting samples
    AttQueue q;
    RecStage rs;
};

// Each warp runs its samples in two stages on full warps.  Stage 1 draws 32
// samples' selection words and sorts them by cost into two queues: the bare
// reference (half of the original sampler's samples: no picks, a constant
// amplitude and death value) and the clusters that need picks; sizes that
// cannot stay within l + 2 end there.  Whenever a queue holds 32, stage 2 takes
// them: picks, collapse, death and estimator for the clusters, then one
// spawning attempt each (or the append to the multi-spawn buffer).  Both
// kinds share the attempt's code, so that it is fetched once.
//
// What bounds it: instruction issue on the gas (57 % of the slots, 25 of 32
// lanes; the two Philox draws of a sample are a third of it), instruction
// fetch on the molecule.  With every size handled where it was drawn and
// bit-string determinants, 15.7 (gas) and 8.7 (molecule) lanes of 32 were
// active, with 320 bytes of local memory per thread.  1.5e8 samples of the
// 162-orbital FP32 gas: 18.7 -> 6.8 ms; 2e7 of the molecule: 5.5 ms (with the
// attempts of its clusters, which then went through a buffer) -> 3.2 ms; 64 gas
// replicas: 3.2 -> 1.45 ms.
// DIST: the simulated distribution's restricted composite draw is compiled
// in (a separate instantiation keeps it out of the plain sampler's loop)
template <typename R, bool GAS, bool DIST>
__device__ __forceinline__ void d_sample(const SysDev &s, const ListView &L, DevStep *st, const RunParams &p, const WorkArrays &wa,
                                                         const SpawnBuf &sp, const ClusterBuf &cl, int enum_base,
                                                         int vb, int vg, SampWarp &sw)
{
    __shared__ double smag[8], scmag[8], smden[8];
    __shared__ i64 snatt[8];
    __shared__ u64 smf[64];
    __shared__ i64 sm[32];
    __shared__ PhiloxStep ps;
    // what the loop needs of the step: in shared memory, because the registers
    // it leaves free decide the loop's speed (and the shift stands in the cache
    // line of the record counter: 10 steps of 2e7 molecule samples with it read
    // there 44.96 ms, 44.57 from here)
    __shared__ struct {
        DirectView dv;
        i64 n_sel;
        u64 nex;
        double coef_hf, death_x, shift;
        RoundCut hf_cut;
        int n, nbk, bshift;
        bool n0_neg, n0_zero, hf_ok, timed_out;
    } ss;
    if (threadIdx.x < 8) {
        smag[threadIdx.x] = st->mag[threadIdx.x];
        scmag[threadIdx.x] = st->cmag[threadIdx.x];
        snatt[threadIdx.x] = st->natt_s[threadIdx.x];
        smden[threadIdx.x] = st->mden[threadIdx.x];
    }
    philox_step_init(ps, st->iter, p.seed, p.replica);
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const PickEntry *pk = wa.picks;
    if (threadIdx.x == 32) {
        const i64 n0 = st->n0;
        ss.dv = direct_view(L, wa, st);
        ss.n_sel = st->n_sel;
        ss.nex = (u64)st->nex;
        ss.n = (int)st->n_occ;
        ss.nbk = (int)st->nbuckets;
        ss.bshift = st->bucket_shift;
        ss.n0_neg = n0 < 0;
        ss.n0_zero = n0 == 0;
        ss.coef_hf = st->hf_coef;
        ss.shift = st->shift;
        ss.death_x = st->hf_death;
        ss.hf_cut = st->hf_cut;
        ss.hf_ok = st->hf_ok != 0;
        ss.timed_out = (st->err & ERRB_TIMEOUT) != 0;
    }
    __syncthreads();
    if (ss.timed_out) return;
    AttQueue &q = sw.q;
    RecStage &rb = sw.rs;
    int wn = 0, hn = 0, qn = 0, rn = 0;   // warp-uniform queue fills
    Fix128 es = {0, 0};
    unsigned err = 0;
    unsigned n_valid = 0, ndirect = 0;   // valid clusters, records added directly (of this thread)
    double cl_att = 0.0;   // attempts of the clusters this thread buffers (exact below 2^53)
    i64 death_hf = 0;      // reference-cluster deaths, summed per block at the end
    const DirectView &dv = ss.dv;
    i64 g0 = (i64)vb * blockDim.x + 32 * wid;
    const i64 stride = (i64)vg * blockDim.x;
    for (;;) {
        // one action per pass, so that each piece of code is fetched from one
        // place (the loop is bound by instruction fetch when it grows):
        // finish what is waiting 32 at a time, else take 32 queued samples,
        // else draw 32 new ones; at the end whatever is left
        const bool more = g0 < ss.n_sel;
        const bool last = !more && wn + hn == 0;
        if (rn >= 32 || (last && qn == 0 && rn > 0)) {
            rec_flush_once(rb, rn, st, sp, dv, ndirect, err);
            continue;
        }
        if (qn >= 32 || (last && qn > 0)) {
            q_finish<R, GAS>(q, qn, rb, rn, s, p, err);
            continue;
        }
        if (last) break;
        int tw = 0, th = 0;   // samples taken from either queue
        if (wn >= 32) {
            tw = 32;
        } else if (hn >= 32) {
            th = 32;
        } else if (!more) {
            tw = wn;
            th = min(hn, 32 - tw);
        }
        const bool sel = tw + th == 0;   // draw new samples
        u64 g = (u64)g0 + lane;
        bool valid = true;
        Exc dj = {0, 0, 0};
        double coef = ss.coef_hf;
        if (!sel) {
            const bool is_w = lane < tw;
            valid = is_w || lane < tw + th;
            int sz = 0;
            i64 natt = 1;
            bool local = false;
            if (valid) g = is_w ? sw.g[wn - tw + lane] : sw.hg[hn - th + lane - tw];
            if (tw > 0) {
                // stage 2: picks, collapse, estimator and death of the clusters
                bool rec = false;   // a composite death record
                u64 rk = 0;
                i64 rv = 0;
                if (is_w) {
                    const int we = wn - tw + lane;
                    const u64 v1 = sw.v1[we], v2 = sw.v2[we], v3 = sw.v3[we];
                    sz = sw.sz[we];
                    local = DIST && p.nranks > 1 && sz >= 2;
                    i64 nq = 0;
                    u64 lq = 0, xa = v2, xb = v3, xc = 0, xd = 0;
                    int i0 = 0, neg = 0, par = 0;
                    // two picks a round: the selection draw's words 2-3, then its second block
#pragma unroll 1
                    for (int e = 0; e < sz && valid; e += 2) {
                        if (e == 2) {
                            const R4 r1 = step_draw_at(ps, TAG_SAMPLE, g, 0, 0xCA5A826395121157ULL);
                            xa = r1.v[0];
                            xb = r1.v[1];
                            xc = r1.v[2];
                            xd = r1.v[3];
                        } else if (e == 4) {
                            xa = xc;
                            xb = xd;
                        }
                        const bool two = e + 1 < sz;
                        int ia, ib = 0;
                        if (!local) {
                            pick_two(pk, wa.bucket, ss.bshift, ss.nbk, ss.n, below(xa, ss.nex), below(xb, ss.nex), two, ia, ib);
                        } else {
                            // simulated distribution: a composite's later
                            // excitors come from the first one's processor
                            if (e == 0) {
                                ia = pick_index(pk, wa.bucket, ss.bshift, ss.nbk, ss.n, below(xa, ss.nex));
                                lq = __ldg(&wa.owner[ia]);
                                nq = __ldg(&wa.nq[lq]);
                            } else {
                                ia = (int)local_pick(wa, L.pop, ss.n, st->lcs, st->nlc, lq, below(xa, (u64)nq));
                            }
                            if (two) ib = (int)local_pick(wa, L.pop, ss.n, st->lcs, st->nlc, lq, below(xb, (u64)nq));
                            if (ia < 0 || ib < 0) {   // tables inconsistent (cannot happen): a sticky error, not a guess
                                valid = false;
                                err |= ERRB_NUMERIC;
                                break;
                            }
                        }
                        if (e == 0) i0 = ia;
#pragma unroll 1
                        for (int k = 0; k <= (two ? 1 : 0) && valid; k++) {
                            u64 f;
                            const Exc x = row_exc(pk, k ? ib : ia, f);
                            if (f & PICK_NEG) neg ^= 1;
                            if (e + k == 0) {
                                dj = x;
                                par = (f & PICK_ODD) ? 1 : 0;
                            } else {
                                // within l + 2 (the levels add up) and
                                // sharing no orbital, else the product vanishes
                                valid = dj.n + x.n <= s.lmax + 2 && apply_excitor(s, x, dj, par);
                            }
                        }
                    }
                    if (dj.n > s.lmax + 2) valid = false;
                    if (valid) {
                        if (ss.n0_neg && ((sz - 1) & 1)) neg ^= 1;
                        double a = smag[sz];
                        if (local) {
                            // |A| = N_ex (N_q N_p)^(s-1) / (|t_HF|^(s-1) n_sel p(s) s!):
                            // selection within q times co-location N_p^-(s-1)
                            const double f = ((double)nq / FIX_ONE) * (double)p.nranks;
                            double num = (double)(i64)ss.nex / FIX_ONE;
    #pragma unroll 1
                            for (int e = 1; e < sz; e++) num = num * f;
                            a = div_rn(num, smden[sz]);
                        }
                        const double amp = neg ? -a : a;
                        coef = (par & 1) ? -amp : amp;
                        const int lev = dj.n;
                        // one excitor: its own determinant with s_D = its collapse sign, <HF|H|D> and death factor per entry
                        if (lev == 1 || lev == 2) {
                            if (sz == 1) es.add(to_fix(__ldg(&wa.href[i0]) * coef));
                            else if (!GAS) es.add(to_fix(h_ref<R, GAS>(s, dj) * coef));   // a gas composite has level 4 or more
                        }
                        // death: tau (Delta E - S) C, of a composite within the truncation only
                        if (sz == 1 || lev <= s.lmax) {
                            double x = (sz == 1 ? __ldg(&pk[i0].tdeath) : p.tau * (diag_rel<R, GAS>(s, dj) - ss.shift)) * coef;
                            if (!(sz == 1 ? (par & 1) : sign_parity(s, dj))) x = -x;
                            i64 d;
                            if (!round_value(x, v1, p, false, d)) err |= ERRB_NUMERIC;
                            if (d != 0) {
                                if (sz == 1) {
                                    atomicAdd((unsigned long long *)&wa.death[i0], (unsigned long long)d);
                                } else {
                                    rk = rank_key(s, dj);
                                    rv = d;
                                    rec = true;
                                }
                            }
                        }
                        // = attempts_of(|amp|): |amp| = mag[sz] for every cluster of
                        // size sz, unless its processor's population sets it
                        if (p.multispawn) natt = local ? attempts_of(fabs(amp), p) : snatt[sz];
                    }
                }
                rec_push(rb, rn, rec, rk, rv);
            }
            if (p.multispawn && !is_w) natt = snatt[0];
            __syncwarp();   // the entries are read before later pushes reuse them
            wn -= tw;
            hn -= th;
            n_valid += valid ? 1u : 0u;
            if (p.multispawn) {
                // queued for the attempts kernel: one counter packs
                // (clusters << CL_SHIFT | attempts)
                double catt = coef;
                if (valid) {
                    // coef / natt: the same division, done once per size
                    if (natt > 1) catt = local ? div_rn(coef, (double)natt) : (coef < 0.0 ? -scmag[sz] : scmag[sz]);
                    if (natt > p.work_cap) {   // runaway: the attempts kernel will not run them
                        err |= ERRB_RUNAWAY;
                        natt = p.work_cap + 1;
                    }
                    cl_att += (double)natt;
                }
                const u64 o = warp_reserve_u64(&st->cl_packed, valid ? ((1ULL << CL_SHIFT) | (u64)natt) : 0ULL);
                if (valid) {
                    const i64 c = (i64)(o >> CL_SHIFT);
                    if (c < cl.cap) {
                        cl.h[c] = pack_h(dj);
                        cl.p[c] = dj.p;
                        cl.catt[c] = catt;
                        cl.index[c] = g;
                        cl.end[c] = (i64)(o & CL_MASK) + natt;
                    } else {
                        err |= ERRB_CLUSTER_OVERFLOW;
                    }
                }
                continue;
            }
        }
        // the selection draw of new samples, or one attempt per valid cluster
        const R4 r = step_draw_at(ps, sel ? TAG_SAMPLE : TAG_SAMPLE_ATT, g, 0, 0);
        if (sel) {
            // the cluster size
            g0 += stride;
            valid = (i64)g < ss.n_sel;
            const u64 nr = ~r.v[0];
            const int lz = nr ? __clzll((long long)nr) : 64;
            const int sz = p.fnc ? 2 + min(lz, s.lmax) : min(lz, s.lmax + 2);
            const bool hf = valid && sz == 0;
            // a valid cluster's level is the sum of its excitors' levels: a
            // size beyond (l + 2) / (smallest level) contributes nothing
            const bool work = valid && sz > 0 && ss.nex != 0 && (sz < 2 || !ss.n0_zero) && sz * s.lmin_exc <= s.lmax + 2;
            const unsigned mh = __ballot_sync(FULLMASK, hf), mw = __ballot_sync(FULLMASK, work);
            if (hf) {
                sw.hg[hn + __popc(mh & ((1u << lane) - 1u))] = g;
                i64 d = ss.hf_cut.base + ((r.v[1] >> 11) < ss.hf_cut.thr ? ss.hf_cut.inc : 0);
                bool in_range = ss.hf_ok;
                if (!p.int_round) in_range = round_value_fp(fabs(ss.death_x), r.v[1], 0.0, &d);
                if (!in_range) err |= ERRB_NUMERIC;
                death_hf += ss.death_x < 0.0 ? -d : d;
            }
            if (work) {
                const int e = wn + __popc(mw & ((1u << lane) - 1u));
                sw.g[e] = g;
                sw.v1[e] = r.v[1];
                sw.v2[e] = r.v[2];
                sw.v3[e] = r.v[3];
                sw.sz[e] = (unsigned char)sz;
            }
            hn += __popc(mh);
            wn += __popc(mw);
            __syncwarp();
        } else {
            // the draws that survive the generator and the truncation are finished 32 at a time
            u64 code = 0;
            const bool ok = valid && excite<GAS>(s, dj, r, code);
            q_push(q, qn, ok, dj, coef, r.v[3], code);
        }
    }
    // the block's sums: E_num, reference deaths, valid clusters, direct records, attempts
    es = warp_fix(es);
    death_hf = warp_sum(death_hf);
    const unsigned nv = __reduce_add_sync(FULLMASK, n_valid), nd = __reduce_add_sync(FULLMASK, ndirect);
    if (p.multispawn) cl_att = warp_sum(cl_att);
    if (lane == 0) {
        smf[2 * wid] = es.lo;
        smf[2 * wid + 1] = es.hi;
        sm[2 * wid] = death_hf;
        sm[2 * wid + 1] = (i64)nv | ((i64)nd << 32);
        if (p.multispawn && cl_att != 0.0) atomicAdd(&st->cl_att, cl_att);
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        Fix128 e = {0, 0};
        i64 d = 0, v = 0, dr = 0;
        for (int w = 0; w < WORK_THREADS / 32; w++) {
            e.add(Fix128{smf[2 * w], smf[2 * w + 1]});
            d += sm[2 * w];
            v += sm[2 * w + 1] & 0xFFFFFFFFLL;
            dr += sm[2 * w + 1] >> 32;
        }
        if (d) atomicAdd((unsigned long long *)&wa.death[0], (unsigned long long)d);
        wa.enum_part[2 * (enum_base + vb)] = e.lo;
        wa.enum_part[2 * (enum_base + vb) + 1] = e.hi;
        if (v && !p.multispawn) {
            atomicAdd((unsigned long long *)&st->n_attempts, (unsigned long long)v);
            if (p.count_clusters) atomicAdd((unsigned long long *)&st->cl_packed, (unsigned long long)v);
        }
        if (dr) atomicAdd((unsigned long long *)&st->n_direct, (unsigned long long)dr);
    }
    if (err) atomicOr(&st->err, err);   // every thread reports its own bits
}

// ---------------------------------------------------------------------------
// a4/a6: expanded spawning attempts -- full non-composite visits first, then
// buffered composite clusters (Sec. IV.B-C)
// ---------------------------------------------------------------------------

template <typename R, bool GAS>
__device__ __forceinline__ void d_attempts(const SysDev &s, const ListView &L, DevStep *st, const RunParams &p,
                                                              const WorkArrays &wa, const SpawnBuf &sp, const ClusterBuf &cl)
{
    // the cluster attempts of a runaway population are not run (their
    // packed count may have wrapped); the step reports the error instead
    const unsigned before = st->err;
    if (before & ERRB_TIMEOUT) return;
    if ((before & ERRB_RUNAWAY) || st->cl_att > (double)p.work_cap) {
        if (threadIdx.x == 0 && blockIdx.x == 0) atomicOr(&st->err, (unsigned)ERRB_RUNAWAY);
        return;
    }
    const i64 n = st->n_occ, tf = st->fnc_attempts;
    i64 ncl = p.multispawn ? (i64)(st->cl_packed >> CL_SHIFT) : 0;
    if (ncl > cl.cap) ncl = cl.cap;
    const i64 tc = ncl > 0 ? cl.end[ncl - 1] : 0;
    const int lane = threadIdx.x & 31;
    const i64 nwarps = (i64)gridDim.x * blockDim.x / 32;
    const i64 wglob = ((i64)blockIdx.x * blockDim.x + threadIdx.x) / 32;
    unsigned err = 0;
    __shared__ AttQueue aq[WORK_THREADS / 32];
    __shared__ RecStage rsb[WORK_THREADS / 32];
    __shared__ i64 sm[32];
    __shared__ PhiloxStep ps;
    philox_step_init(ps, st->iter, p.seed, p.replica);
    __syncthreads();
    AttQueue &q = aq[threadIdx.x >> 5];
    RecStage &rb = rsb[threadIdx.x >> 5];
    int qn = 0, rn = 0;   // drawn attempts and staged records of this warp (warp-uniform)
    unsigned ndirect = 0;
    const DirectView dv = direct_view(L, wa, st);
    // part 0: full non-composite attempts (owners: list entries); part 1:
    // attempts of the composite clusters queued by k_sample; part 2: what is
    // still queued.  One action per pass, as in the sampler.
    int part = -1;
    const i64 *end = nullptr;
    i64 nown = 0, t0 = 0, a1 = 0;
    AttemptWindow w = {0, 0};
    for (;;) {
        if (rn >= 32 || (part == 2 && qn == 0 && rn > 0)) {
            rec_flush_once(rb, rn, st, sp, dv, ndirect, err);
            continue;
        }
        if (qn >= 32 || (part == 2 && qn > 0)) {
            q_finish<R, GAS>(q, qn, rb, rn, s, p, err);
            continue;
        }
        if (part == 2) break;
        if (t0 >= a1) {
            if (++part == 2) continue;
            const i64 total = part == 0 ? tf : tc;
            end = part == 0 ? wa.att_end : cl.end;
            nown = part == 0 ? n : ncl;
            const i64 per = ((total + nwarps - 1) / nwarps + 31) & ~31LL;
            t0 = wglob * per;
            a1 = t0 + per < total ? t0 + per : total;
            if (t0 < a1) w = window_start(end, nown, t0);
            continue;
        }
        i64 o, m;
        window_step(end, nown, t0, w, o, m);
        bool ok = false;
        Exc dj = {0, 0, 0};
        double ca = 0.0;
        u64 r3 = 0, code = 0;
        if (t0 + lane < a1) {
            u64 tag = TAG_VISIT_ATT, idx = (u64)o;
            if (part == 0) {
                dj = exc_of(L.h[o], L.p[o]);
                ca = wa.catt[o];
            } else {
                dj = exc_of(cl.h[o], cl.p[o]);
                ca = cl.catt[o];
                tag = TAG_SAMPLE_ATT;
                idx = cl.index[o];
            }
            const R4 r = step_draw(ps, tag, idx, (u64)m);
            ok = excite<GAS>(s, dj, r, code);
            r3 = r.v[3];
        }
        q_push(q, qn, ok, dj, ca, r3, code);
        t0 += 32;
    }
    const i64 direct = block_sum((i64)ndirect, sm);
    if (threadIdx.x == 0 && direct) atomicAdd((unsigned long long *)&st->n_direct, (unsigned long long)direct);
    if (err) atomicOr(&st->err, err);
}

// ---------------------------------------------------------------------------
// a7: LSD radix sort by rank key (stable)
// ---------------------------------------------------------------------------


constexpr int SORT_TINY = 256;   // records that are ranked by counting

// Shared memory of a sorting block: a tile in digit order, so that each
// digit's run is written out by consecutive threads to consecutive addresses,
// and the digit counts per warp.
struct SortSmem {
    u64 tk[SORT_TILE];
    i64 tv[SORT_TILE];
    unsigned w[SORT_THREADS / 32][1 << SORT_DIGIT_BITS];
    unsigned off[1 << SORT_DIGIT_BITS], tot[1 << SORT_DIGIT_BITS], tpre[1 << SORT_DIGIT_BITS], all[1 << SORT_DIGIT_BITS];
    unsigned sc[32];
};

// Sorts a tile's items (ipt per thread; item j of lane l of warp w is number
// 32 (ipt w + j) + l) by one digit into S.tk / S.tv, stably: digit, then warp, item, lane.  Leaves
// the digits' counts in S.tot and their exclusive prefix in S.tpre.
__device__ __forceinline__ void sort_tile(SortSmem &S, const u64 (&kk)[SORT_ITEMS], const i64 (&vv)[SORT_ITEMS],
                                          const bool (&ok)[SORT_ITEMS], int ipt, int shift, int bits)
{
    constexpr int NW = SORT_THREADS / 32;
    const int nd = 1 << bits;
    const unsigned mask = (unsigned)nd - 1u;
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const unsigned lt = (1u << lane) - 1u;
    __syncthreads();   // the previous tile is written out
    for (int d = lane; d < nd; d += 32) S.w[wid][d] = 0;
    __syncwarp();
    unsigned rk[SORT_ITEMS];
#pragma unroll
    for (int j = 0; j < SORT_ITEMS; j++) {
        if (j >= ipt) break;
        const unsigned d = (unsigned)(kk[j] >> shift) & mask;
        unsigned peers = __ballot_sync(FULLMASK, ok[j]);
#pragma unroll
        for (int b = 0; b < SORT_DIGIT_BITS; b++) {   // (bits past the digit's are zero)
            const unsigned bb = __ballot_sync(FULLMASK, (d >> b) & 1u);
            peers &= ((d >> b) & 1u) ? bb : ~bb;
        }
        unsigned base = 0;
        if (ok[j]) base = S.w[wid][d];
        __syncwarp();
        if (ok[j] && (peers & lt) == 0) S.w[wid][d] = base + __popc(peers);
        __syncwarp();
        rk[j] = base + __popc(peers & lt);
    }
    __syncthreads();
    const int d = threadIdx.x;   // one digit per thread
    unsigned run = 0;
    if (d < nd) {
#pragma unroll
        for (int w = 0; w < NW; w++) {
            const unsigned t = S.w[w][d];
            S.w[w][d] = run;
            run += t;
        }
        S.tot[d] = run;
    }
    unsigned all;
    const unsigned incl = block_incl_scan(d < nd ? run : 0u, S.sc, all);
    if (d < nd) S.tpre[d] = incl - run;
    __syncthreads();
#pragma unroll
    for (int j = 0; j < SORT_ITEMS; j++) {
        if (j >= ipt) break;
        const unsigned d2 = (unsigned)(kk[j] >> shift) & mask;
        if (ok[j]) {
            const unsigned tp = S.tpre[d2] + S.w[wid][d2] + rk[j];
            S.tk[tp] = kk[j];
            S.tv[tp] = vv[j];
        }
    }
    __syncthreads();
}

// Sorts the n records (k0, v0) by their lowest key_bits through the pairs
// (key[q], pop[q]); the result is in pair passes & 1, passes =
// ceil(key_bits / digit).  (k0, v0) may be pair 0.
// Up to a tile one block sorts in shared memory, nine bits a pass (about 4 us
// each; three launches per eight-bit digit took 15).  More records take a histogram, a barrier, a scatter and a barrier per
// digit; every block derives its offsets from all blocks' histograms itself.
__device__ __forceinline__ bool team_sort(const u64 *k0, const i64 *v0, u64 *const *key, i64 *const *pop, i64 n, int key_bits, int digit, unsigned *hist,
                                          unsigned *bar, Team t, DevStep *st, SortSmem &S)
{
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    u64 kk[SORT_ITEMS];
    i64 vv[SORT_ITEMS];
    bool ok[SORT_ITEMS];
    const int passes = (key_bits + digit - 1) / digit;
    if (n <= SORT_TINY) {
        // every record counts those that go before it
        if (t.id != 0) return true;
        const int i = threadIdx.x;
        const u64 k = i < n ? k0[i] : 0;
        const i64 v = i < n ? v0[i] : 0;
        if (i < n) S.tk[i] = k;
        __syncthreads();
        if (i < n) {
            int r = 0;
            for (int j = 0; j < n; j++) r += S.tk[j] < k || (S.tk[j] == k && j < i) ? 1 : 0;
            key[passes & 1][r] = k;
            pop[passes & 1][r] = v;
        }
        __syncthreads();
        return true;
    }
    if (n <= SORT_TILE) {
        if (t.id != 0) return true;
        const int lp = (key_bits + SORT_DIGIT_BITS - 1) / SORT_DIGIT_BITS, lb = (key_bits + lp - 1) / lp;
        const int ipt = (int)((n + SORT_THREADS - 1) / SORT_THREADS);
        for (int q = 0; q < lp; q++) {
#pragma unroll
            for (int j = 0; j < SORT_ITEMS; j++) {
                const int i = (wid * ipt + j) * 32 + lane;
                ok[j] = j < ipt && i < n;
                kk[j] = !ok[j] ? 0 : (q == 0 ? k0[i] : S.tk[i]);
                vv[j] = !ok[j] ? 0 : (q == 0 ? v0[i] : S.tv[i]);
            }
            sort_tile(S, kk, vv, ok, ipt, q * lb, min(lb, key_bits - q * lb));
        }
        for (int i = threadIdx.x; i < n; i += SORT_THREADS) {
            key[passes & 1][i] = S.tk[i];
            pop[passes & 1][i] = S.tv[i];
        }
        __syncthreads();
        return true;
    }
    i64 lo, hi;
    chunk_of(t, n, lo, hi);
    const i64 share = (n + t.n - 1) / t.n;
    const bool one_tile = share <= SORT_TILE;   // of every block
    const int ipt = one_tile ? (int)((share + SORT_THREADS - 1) / SORT_THREADS) : SORT_ITEMS;
    auto load_tile = [&](const u64 *kin, const i64 *vin, i64 tb) {
#pragma unroll
        for (int j = 0; j < SORT_ITEMS; j++) {
            const i64 i = tb + (wid * ipt + j) * 32 + lane;
            ok[j] = j < ipt && i < hi;
            kk[j] = ok[j] ? kin[i] : 0;
            vv[j] = ok[j] ? vin[i] : 0;
        }
    };
    int src = 0;
    for (int shift = 0; shift < key_bits; shift += digit, src ^= 1) {
        const int bits = min(digit, key_bits - shift), nd = 1 << bits;
        const u64 mask = (u64)nd - 1;
        const u64 *kin = shift == 0 ? k0 : key[src];
        const i64 *vin = shift == 0 ? v0 : pop[src];
        // the block's digit counts: of its one tile, sorted first, or from a
        // pass over its records
        if (one_tile) {
            load_tile(kin, vin, lo);
            sort_tile(S, kk, vv, ok, ipt, shift, bits);
            for (int d = threadIdx.x; d < nd; d += SORT_THREADS) hist[(size_t)t.id * nd + d] = S.tot[d];
        } else {
            for (int d = threadIdx.x; d < nd; d += SORT_THREADS) S.off[d] = 0;
            __syncthreads();
#pragma unroll 4
            for (i64 i = lo + threadIdx.x; i < hi; i += SORT_THREADS) atomicAdd(&S.off[(kin[i] >> shift) & mask], 1u);
            __syncthreads();
            for (int d = threadIdx.x; d < nd; d += SORT_THREADS) hist[(size_t)t.id * nd + d] = S.off[d];
        }
        if (!team_sync(bar, t, st)) return false;
        {
            // offset of this block's run of each digit: the digits before, and
            // the same digit's runs of the blocks before.  Every block reads
            // all counts: of many blocks four digits a load (304 blocks' rows
            // were 38 rounds of latency a pass: 9e5 records 148 -> 104 us), of
            // a few one digit a load (ten blocks: 33 us, 38 with four; scanning
            // the columns by blocks first was slower for all)
            for (int q = threadIdx.x; q < nd; q += SORT_THREADS) S.off[q] = S.all[q] = 0;
            __syncthreads();
            const bool four = nd >= 4 && t.n > 32;
            const int per = four ? nd / 4 : nd, parts = SORT_THREADS / per, part = threadIdx.x / per;
            const int d = (threadIdx.x - part * per) * (four ? 4 : 1);
            if (four) {
                uint4 before = make_uint4(0, 0, 0, 0), all = before;
#pragma unroll 8
                for (int b = part; b < t.n; b += parts) {
                    const uint4 h = __ldcg((const uint4 *)&hist[(size_t)b * nd + d]);
                    all.x += h.x;
                    all.y += h.y;
                    all.z += h.z;
                    all.w += h.w;
                    if (b < t.id) {
                        before.x += h.x;
                        before.y += h.y;
                        before.z += h.z;
                        before.w += h.w;
                    }
                }
                atomicAdd(&S.off[d], before.x);
                atomicAdd(&S.off[d + 1], before.y);
                atomicAdd(&S.off[d + 2], before.z);
                atomicAdd(&S.off[d + 3], before.w);
                atomicAdd(&S.all[d], all.x);
                atomicAdd(&S.all[d + 1], all.y);
                atomicAdd(&S.all[d + 2], all.z);
                atomicAdd(&S.all[d + 3], all.w);
            } else {
                unsigned before = 0, all = 0;
#pragma unroll 8
                for (int b = part; b < t.n; b += parts) {
                    const unsigned h = __ldcg(&hist[(size_t)b * nd + d]);
                    all += h;
                    if (b < t.id) before += h;
                }
                atomicAdd(&S.off[d], before);
                atomicAdd(&S.all[d], all);
            }
            __syncthreads();
            const unsigned v = threadIdx.x < nd ? S.all[threadIdx.x] : 0u;
            unsigned sum;
            const unsigned incl = block_incl_scan(v, S.sc, sum);
            if (threadIdx.x < nd) S.off[threadIdx.x] += incl - v;
            __syncthreads();
        }
        for (i64 tb = lo; tb < hi; tb += SORT_TILE) {
            if (!one_tile) {
                load_tile(kin, vin, tb);
                sort_tile(S, kk, vv, ok, ipt, shift, bits);
            }
            const int tn = (int)(hi - tb < (i64)SORT_TILE ? hi - tb : (i64)SORT_TILE);
            for (int q = threadIdx.x; q < tn; q += SORT_THREADS) {
                const u64 k = S.tk[q];
                const unsigned d = (unsigned)((k >> shift) & mask);
                const unsigned pos = S.off[d] + (unsigned)q - S.tpre[d];
                key[src ^ 1][pos] = k;
                pop[src ^ 1][pos] = S.tv[q];
            }
            __syncthreads();
            for (int d = threadIdx.x; d < nd; d += SORT_THREADS) S.off[d] += S.tot[d];
        }
        if (!team_sync(bar, t, st)) return false;
    }
    return true;
}

// ---------------------------------------------------------------------------
// a8: one record per distinct key with the summed weight
// ---------------------------------------------------------------------------

// Every block of the team calls; returns the number of distinct keys, or -1
// if a wait ran out.
__device__ __forceinline__ i64 team_reduce(const u64 *keys, const i64 *pops, i64 n, u64 *outkey, i64 *outpop, i64 *part,
                                           unsigned *bar, Team t, DevStep *st, i64 *sm)
{
    // warp-granular chunks: run heads are counted by ballots, without block
    // barriers in the loops
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    constexpr int NW = SORT_THREADS / 32;
    i64 lo, hi;
    chunk_of(t, n, lo, hi);
    const i64 wc = ((hi - lo + NW - 1) / NW + 31) & ~31LL;
    const i64 w0 = lo + wid * wc < hi ? lo + wid * wc : hi, w1 = w0 + wc < hi ? w0 + wc : hi;
    i64 heads = 0;
#pragma unroll 4
    for (i64 base = w0; base < w1; base += 32) {
        const i64 i = base + lane;
        heads += __popc(__ballot_sync(FULLMASK, i < w1 && (i == 0 || keys[i] != keys[i - 1])));
        if (i < w1) outpop[i] = 0;
    }
    if (lane == 0) sm[wid] = heads;
    __syncthreads();
    i64 carry = 0, c = 0;
    for (int w = 0; w < NW; w++) {
        if (w == wid) carry = c;
        c += sm[w];
    }
    if (threadIdx.x == 0) part[4 * t.id] = c;
    if (!team_sync(bar, t, st)) return -1;
    i64 before, total;
    team_prefix(part, 4, t, sm, before, total);
    carry += before;
#pragma unroll 2
    for (i64 base = w0; base < w1; base += 32) {
        const i64 i = base + lane;
        const bool ok = i < w1;
        const u64 k = ok ? keys[i] : 0;
        i64 v = ok ? pops[i] : 0;
        const bool head = ok && (i == 0 || keys[i - 1] != k);
        const unsigned m = __ballot_sync(FULLMASK, head);
        const int seg = __popc(m & (0xFFFFFFFFu >> (31 - lane)));   // run within the row, 0: begun before it
        if (head) outkey[carry + seg - 1] = k;
        // segmented warp sum; the last lane of each run adds it
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const i64 tv = __shfl_up_sync(FULLMASK, v, o);
            const int ts = __shfl_up_sync(FULLMASK, seg, o);
            if (lane >= o && ts == seg) v += tv;
        }
        const int nxt = __shfl_down_sync(FULLMASK, seg, 1);
        const bool last = lane == 31 || i + 1 >= w1 || nxt != seg;
        if (ok && last && v != 0) atomicAdd((unsigned long long *)&outpop[carry + seg - 1], (unsigned long long)v);
        carry += __popc(m);
    }
    return total;
}

// ---------------------------------------------------------------------------
// a9: merge into the list with the occupation threshold
// ---------------------------------------------------------------------------

// each reduced key: add to its list entry, or mark it new (thresholded)
__device__ __forceinline__ void d_merge_match(const ListView &L, const DevStep *st, const RunParams &p, const WorkArrays &wa,
                                              const u64 *rkey, i64 *rpop, i64 m, Team t)
{
    const i64 n = st->n_occ, nkb = st->nkb;
    const int ks = st->kshift;
    const u64 it = st->iter;
    for (i64 j = (i64)t.id * blockDim.x + threadIdx.x; j < m; j += (i64)t.n * blockDim.x) {
        const u64 k = __ldcg(&rkey[j]);
        const i64 v0 = __ldcg(&rpop[j]);
        // first entry with a key of at least k: within the key's bucket where the step has them
        i64 lo = 0, hi = n;
        if (nkb > 0) {
            const u64 b = k >> ks;
            lo = b < (u64)nkb ? (i64)__ldg(&wa.kbucket[b]) : n;
            if (b + 1 < (u64)nkb) hi = __ldg(&wa.kbucket[b + 1]);
        }
        while (lo < hi) {
            const i64 mid = lo + (hi - lo) / 2;
            if (__ldg(&L.key[mid]) < k) lo = mid + 1;
            else hi = mid;
        }
        const i64 pos = lo;
        if (pos < n && __ldg(&L.key[pos]) == k) {
            wa.acc[pos] += v0;
            wa.ins[j] = -1;
            wa.keep_s[j] = 0;
        } else {
            const i64 v = threshold(p, it, k, v0);
            rpop[j] = v;
            wa.ins[j] = pos;
            wa.keep_s[j] = v != 0 ? 1 : 0;
            // a kept new key lands right before list entry pos
            if (v != 0 && pos < n) atomicAdd(&wa.before[pos], 1);
        }
    }
}

// New populations of the block's list entries (old + death + matched spawns,
// then the occupation threshold) with their keep flags packed with the kept
// new keys inserted before them, and the keep counts of its new keys; the
// block's sums go to part[4 id] and part[4 id + 1].
__device__ __forceinline__ void d_merge_count(const ListView &L, DevStep *st, const RunParams &p, const WorkArrays &wa,
                                              i64 m, Team t, i64 *sm)
{
    i64 lo, hi, sum = 0, ksum = 0;
    chunk_of(t, m, lo, hi);
    for (i64 i = lo + threadIdx.x; i < hi; i += blockDim.x) ksum += __ldcg(&wa.keep_s[i]);
    chunk_of(t, st->n_occ, lo, hi);
    const u64 it = st->iter;
    const bool direct = st->nkb > 0;
    i64 hits = 0;   // entries that received directly added spawns: distinct keys of the step
    constexpr int ROWS = 4;
    for (i64 base = lo + threadIdx.x; base < hi; base += ROWS * (i64)blockDim.x) {
        i64 v[ROWS];
        int bf[ROWS];
#pragma unroll
        for (int r = 0; r < ROWS; r++) {
            const i64 i = base + r * (i64)blockDim.x;
            const bool ok = i < hi;
            v[r] = ok ? L.pop[i] + wa.death[i] + __ldcg(&wa.acc[i]) : 0;
            bf[r] = ok ? __ldcg(&wa.before[i]) : 0;
            if (ok && direct) hits += wa.hit[i];
        }
#pragma unroll
        for (int r = 0; r < ROWS; r++) {
            const i64 i = base + r * (i64)blockDim.x;
            if (i >= hi) break;
            // the key is read only for the few entries the threshold decides
            const i64 av = v[r] < 0 ? -v[r] : v[r];
            if (i > 0 && av > 0 && av < (i64)FIX_ONE) v[r] = threshold(p, it, L.key[i], v[r]);
            wa.newpop[i] = v[r];
            // two counts in one word (each below 2^31): the entry's keep flag
            // and the kept new keys that go before it; one prefix gives both
            const i64 w = ((i == 0 || v[r] != 0) ? 1 : 0) | ((i64)bf[r] << 32);
            wa.keep_l[i] = w;
            sum += w;
        }
    }
    // the three sums in one pass through shared memory
    sum = warp_sum(sum);
    ksum = warp_sum(ksum);
    hits = warp_sum(hits);
    const int wid = threadIdx.x >> 5;
    __syncthreads();
    if ((threadIdx.x & 31) == 0) {
        sm[3 * wid] = sum;
        sm[3 * wid + 1] = ksum;
        sm[3 * wid + 2] = hits;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        sum = ksum = hits = 0;
        for (int w = 0; w < SCAN_THREADS / 32; w++) {
            sum += sm[3 * w];
            ksum += sm[3 * w + 1];
            hits += sm[3 * w + 2];
        }
        wa.part[4 * t.id] = sum;
        wa.part[4 * t.id + 1] = ksum;
        if (hits) atomicAdd((unsigned long long *)&st->n_hit, (unsigned long long)hits);
    }
}

// The keep prefixes and the list's scatter in one pass.  The new keys' keep
// flags become their exclusive prefix in place.  Over the block's list entries:
// the exclusive prefix e of the packed words (kept entries | kept new keys
// before the entry << 32), four rows of counts read before their scans; each
// kept entry goes to e_lo + e_hi + (new keys right before it), and e is stored
// only where kept new keys are inserted (the new-key scatter reads it there).
// Returns the list's kept entries.
__device__ __forceinline__ i64 d_keep_scatter(const ListView &L, const ListView &O, DevStep *st, const WorkArrays &wa,
                                              i64 m, Team t, i64 *sm)
{
    i64 lo, hi, carry, kcarry, tot_l, tot_s;
    team_prefix(wa.part, 4, t, sm, carry, tot_l);
    __syncthreads();
    team_prefix(wa.part + 1, 4, t, sm, kcarry, tot_s);
    __syncthreads();
    const i64 kept = tot_l & 0xFFFFFFFFLL;   // the low count of the packed list flags
    if (t.id == 0 && threadIdx.x == 0) {
        st->kept_list = kept;
        st->kept_new = tot_s;
    }
    chunk_of(t, m, lo, hi);
    constexpr int ROWS = 4;
    for (i64 base = lo; base < hi; base += ROWS * (i64)blockDim.x) {
        i64 e[ROWS];
#pragma unroll
        for (int r = 0; r < ROWS; r++) {
            const i64 i = base + r * (i64)blockDim.x + threadIdx.x;
            e[r] = i < hi ? wa.keep_s[i] : 0;
        }
        const i64 tot = block_scan4(e, sm);
#pragma unroll
        for (int r = 0; r < ROWS; r++) {
            const i64 i = base + r * (i64)blockDim.x + threadIdx.x;
            if (i < hi) wa.keep_s[i] = kcarry + e[r];
        }
        kcarry += tot;
    }
    chunk_of(t, st->n_occ, lo, hi);
    i64 asum = 0;
    unsigned err = 0;
    for (i64 base = lo; base < hi; base += ROWS * (i64)blockDim.x) {
        i64 w[ROWS], v[ROWS], e[ROWS];
#pragma unroll
        for (int r = 0; r < ROWS; r++) {
            const i64 i = base + r * (i64)blockDim.x + threadIdx.x;
            w[r] = i < hi ? wa.keep_l[i] : 0;
            v[r] = i < hi ? wa.newpop[i] : 0;
        }
#pragma unroll
        for (int r = 0; r < ROWS; r++) e[r] = w[r];
        const i64 tot = block_scan4(e, sm);
#pragma unroll
        for (int r = 0; r < ROWS; r++) e[r] += carry;
        carry += tot;
#pragma unroll
        for (int r = 0; r < ROWS; r++) {
            const i64 i = base + r * (i64)blockDim.x + threadIdx.x;
            if (i >= hi) continue;
            const i64 nb = w[r] >> 32;   // kept new keys inserted right before entry i
            if (nb) wa.keep_l[i] = e[r];
            if (!(i == 0 || v[r] != 0)) continue;
            const i64 out = (e[r] & 0xFFFFFFFFLL) + (e[r] >> 32) + nb;
            if (out >= O.cap) {
                err |= ERRB_LIST_OVERFLOW;
                continue;
            }
            const u64 eh = L.h[i], ep = L.p[i], ek = L.key[i];
            const double ed = L.diag[i];
            O.h[out] = eh;
            O.p[out] = ep;
            O.key[out] = ek;
            O.pop[out] = v[r];
            O.diag[out] = ed;
            asum += v[r] < 0 ? -v[r] : v[r];
        }
    }
    asum = warp_sum(asum);
    if ((threadIdx.x & 31) == 0 && asum) atomicAdd((unsigned long long *)&st->ntot_after, (unsigned long long)asum);
    if (err) atomicOr(&st->err, err);   // every thread reports its own bits
    return kept;
}

template <typename R, bool GAS>
__device__ __forceinline__ void d_scatter_new(const SysDev &s, const ListView &O, DevStep *st, const WorkArrays &wa,
                                              const u64 *rkey, const i64 *rpop, i64 m, i64 kl, Team t, u64 *tab)
{
    const i64 n = st->n_occ;
    // the rank table in shared memory: unranking is a chain of dependent reads of it
    for (int q = threadIdx.x; q < (s.lmax + 1) * RANK_STRIDE; q += blockDim.x) tab[q] = __ldg(&s.rank_tab[q]);
    __syncthreads();
    i64 asum = 0;
    unsigned err = 0;
    for (i64 j = (i64)t.id * blockDim.x + threadIdx.x; j < m; j += (i64)t.n * blockDim.x) {
        const i64 il = __ldcg(&wa.ins[j]);
        const i64 v = __ldcg(&rpop[j]);
        if (il < 0 || v == 0) continue;
        const i64 out = __ldcg(&wa.keep_s[j]) + (il < n ? (__ldcg(&wa.keep_l[il]) & 0xFFFFFFFFLL) : kl);
        if (out >= O.cap) {
            err |= ERRB_LIST_OVERFLOW;
            continue;
        }
        const u64 k = __ldcg(&rkey[j]);
        const Exc d = unrank_key(s, tab, k);
        O.h[out] = pack_h(d);
        O.p[out] = d.p;
        O.key[out] = k;
        O.pop[out] = v;
        O.diag[out] = diag_rel<R, GAS>(s, d);
        asum += v < 0 ? -v : v;
    }
    asum = warp_sum(asum);
    if ((threadIdx.x & 31) == 0 && asum) atomicAdd((unsigned long long *)&st->ntot_after, (unsigned long long)asum);
    if (err) atomicOr(&st->err, err);   // every thread reports its own bits
}

// ---------------------------------------------------------------------------
// a10: estimator reduction and the per-step record
// ---------------------------------------------------------------------------

__device__ __forceinline__ void d_finalize(DevStep *st, const RunParams &p, const WorkArrays &wa, const ClusterBuf &cl,
                                           int enum_base, int slots, i64 list_cap, u64 *smf)
{
    // E_num partials: the scan's blocks, then the sampler's slots
    Fix128 k = {0, 0};
    const int ns = st->scan_blocks;
    for (int q = threadIdx.x; q < ns + slots; q += blockDim.x) {
        const int e = q < ns ? q : enum_base + q - ns;
        Fix128 t = {wa.enum_part[2 * e], wa.enum_part[2 * e + 1]};
        k.add(t);
    }
    k = block_fix(k, smf);
    if (threadIdx.x == 0) {
        i64 ncl = p.multispawn ? (i64)(st->cl_packed >> CL_SHIFT) : (i64)st->cl_packed;
        if (ncl > cl.cap) {
            // the generic original sampler's clusters are bounded like multi-spawn's buffer
            if (!p.multispawn) st->err |= ERRB_CLUSTER_OVERFLOW;
            ncl = cl.cap;
        }
        i64 tc = p.multispawn && ncl > 0 ? cl.end[ncl - 1] : 0;
        Record r;
        r.iter = st->iter;
        r.shift = st->shift;
        r.n0 = st->n0;
        r.ntot = st->ntot;
        r.n_sel = st->n_sel;
        r.n_visit = p.fnc ? st->n_occ : 0;
        r.n_attempts = st->fnc_attempts + tc + st->n_attempts;
        r.n_spawned = st->n_sp + st->n_direct;
        r.e_num = fix_to_double(k);
        // (sums of this kernel's blocks: past the first-level cache)
        r.ntot_after = __ldcg(&st->ntot_after);
        r.nocc_after = __ldcg(&st->kept_list) + __ldcg(&st->kept_new);
        r.n_keys = __ldcg(&st->n_keys) + __ldcg(&st->n_hit);
        r.n_clusters = ncl;
        r.n_direct = st->n_direct;
        st->prev_spawned = r.n_spawned;
        wa.ring[st->iter % RING] = r;
        st->n_start = st->n_occ;
        st->n_occ = r.nocc_after < list_cap ? r.nocc_after : list_cap;
        st->cur ^= 1;   // the merged list becomes the current one
        st->iter = st->iter + 1;
    }
}

// ---------------------------------------------------------------------------
// Kernels: each block serves replica blockIdx.y (the list kernels: the
// replicas of its shares) of an array of per-replica
// arguments (one entry for a single context, many for a batch).
// ---------------------------------------------------------------------------

// Every kernel returns if a team's wait ran out, in this step or an earlier one.
// Only the launches with teams can set the bit meanwhile: there one thread reads
// it for its block (RETURN_IF_TIMED_OUT).  The bit is read along with what the
// kernel reads first anyway; read ahead of it, it cost each kernel a memory
// latency (50 steps of the 38-orbital gas between restore and read: 2.57 ms,
// 2.63 with the bit read ahead).
#define REPLICA                               \
    const StepArgs &a = A[blockIdx.y];        \
    const int cur_ = a.st->cur

// the replica's arguments copied to shared memory (hot kernels)
#define REPLICA_SMEM                                                              \
    __shared__ StepArgs a_sm;                                                     \
    {                                                                             \
        const u64 *src_ = (const u64 *)&A[blockIdx.y];                            \
        u64 *dst_ = (u64 *)&a_sm;                                                 \
        for (int q_ = threadIdx.x; q_ < (int)(sizeof(StepArgs) / 8); q_ += blockDim.x) dst_[q_] = src_[q_]; \
    }                                                                             \
    __syncthreads();                                                              \
    const StepArgs &a = a_sm;                                                     \
    const int cur_ = a.st->cur

#define RETURN_IF_TIMED_OUT                                                       \
    __shared__ unsigned err_sm;                                                   \
    if (threadIdx.x == 0) err_sm = a.st->err;                                     \
    __syncthreads();                                                              \
    if (err_sm & ERRB_TIMEOUT) return

// Kernels that depend on neither kind nor precision (defined in ccmc_step.cu).
__global__ void __launch_bounds__(1024) k_sample_plan(const StepArgs *__restrict__ A, int nrep, FlatPlan fp,
                                                       int enum_base);
__global__ void __launch_bounds__(SCAN_THREADS) k_local_scan(const StepArgs *__restrict__ A);
// owners and position table of the simulated distribution, for K words
void launch_local_table(const StepArgs *A, int K, dim3 grid, cudaStream_t sm);

// The blocks of a batch's launch shared out between its replicas, in
// proportion to the blocks that each would use alone (units_of(r), which must
// not change during the launch).  Every block works the same shares out: a
// replica's team is a run of blocks if its share is two or more.  The blocks
// left over take the other replicas, one block each, round after round; the
// last, partly filled round has as many blocks for each as there are.  A block
// takes its replicas in this order and only later ones wait for it, so every
// wait ends.
//
// Equal shares (two blocks per SM over the replicas) left a list of 4.8e6
// entries among 200 small ones to one block: 32.5 ms a step, now 1.06 (one of
// 95,000 entries: 1.27 and 0.42 ms).  Where equal shares were right it costs
// the working out, some 3 us a launch: 64 replicas of 18,000 entries 0.951 and
// 0.956 ms a step, 700 of 280 entries 0.65 and 0.685 ms.
//
// (All that is kept between replicas is in shared memory: in registers it
// would spill in the loops of the replica's own work.)
struct Shares {
    static constexpr int KEPT = 2 * SCAN_THREADS;   // replicas whose units are read once
    i64 sm[32], want, give;       // units of the replicas that want several blocks, blocks for them
    int smi[32], kept[KEPT], list[SCAN_THREADS];
    int first, hands, full, per;  // blocks before those left over, these, rounds of these, blocks each in the last round
    int stage, base, rank, q, count;   // (stage 2: no replica wants several blocks)
    int rep, tail;                // the replica to do, the one of the last round
    Team team, tail_team;
};

template <typename U>
__device__ __forceinline__ i64 units_at(const Shares &S, int r, U units_of)
{
    return r < Shares::KEPT ? S.kept[r] : units_of(r);
}

// blocks of replica r's team, 0: done by the blocks left over
__device__ __forceinline__ int share_at(i64 u, i64 want, i64 give, int most)
{
    const i64 n = u < 2 ? 0 : u * give / want;
    return n < 2 ? 0 : (int)(n < most ? n : most);
}

template <typename U>
__device__ __forceinline__ void shares_init(Shares &S, int nrep, int most, U units_of)
{
    const int B = (int)gridDim.x, id = (int)blockIdx.x, tid = threadIdx.x;
    i64 v = 0;   // units of the replicas that want several blocks, and the other replicas
#pragma unroll
    for (int r = tid; r < Shares::KEPT; r += SCAN_THREADS) {
        const i64 u = r < nrep ? units_of(r) : 0;
        S.kept[r] = (int)u;
        v += u > 1 ? u << 24 : u;
    }
    for (int r = Shares::KEPT + tid; r < nrep; r += SCAN_THREADS) {
        const i64 u = units_of(r);
        v += u > 1 ? u << 24 : 1;
    }
    v = block_sum(v, S.sm);
    const i64 want = v >> 24, ones = v & ((1 << 24) - 1), give = want + ones <= B ? want : B * want / (want + ones);
    if (tid == 0) {
        S.stage = want ? 0 : 2;
        S.base = S.rank = S.q = S.count = 0;
        S.tail = -1;
        S.want = want;
        S.give = give;
    }
    if (want == 0) return;
    int taken = 0, teams = 0;
    for (int base = 0; base < nrep; base += SCAN_THREADS) {
        const int r = base + tid, n = r < nrep ? share_at(units_at(S, r, units_of), want, give, most) : 0;
        int tot;   // blocks, teams << 16
        const int at = taken + (block_incl_scan(n ? n | (1 << 16) : 0, S.smi, tot) & 0xFFFF) - n;
        if (id >= at && id < at + n) {
            S.rep = r;
            S.team = Team{id - at, n};
            S.count = 1;
        }
        taken += tot & 0xFFFF;
        teams += tot >> 16;
    }
    if (tid == 0) {
        const int first = taken < B ? taken : 0, hands = B - first, left = nrep - teams;
        S.first = first;
        S.hands = hands;
        S.full = left / hands;
        S.per = left % hands ? hands / (left % hands) : 0;
    }
}

// The next replica of this block in S.rep, with S.team; false if there is none.
template <typename U>
__device__ __forceinline__ bool next_share(Shares &S, int nrep, int most, U units_of)
{
    const int id = (int)blockIdx.x, tid = threadIdx.x;
    __syncthreads();
    if (S.stage == 2) {
        const int r = S.q + id;
        __syncthreads();
        if (tid == 0) {
            S.rep = r;
            S.team = Team{0, 1};
            S.q += (int)gridDim.x;
        }
        __syncthreads();
        return r < nrep;
    }
    if (S.stage == 0) {
        const int have = S.count;
        __syncthreads();
        if (tid == 0) {
            S.stage = 1;
            S.count = 0;
        }
        if (have) return true;
        __syncthreads();
    }
    if (id < S.first) return false;
    for (;;) {
        const int q = S.q, count = S.count, base = S.base, rank = S.rank;
        __syncthreads();
        if (q < count) {
            if (tid == 0) {
                S.rep = S.list[q];
                S.team = Team{0, 1};
                S.q = q + 1;
            }
            __syncthreads();
            return true;
        }
        if (base >= nrep) break;
        const int r = base + tid, hands = S.hands;
        const i64 u = r < nrep ? units_at(S, r, units_of) : 0;
        const bool one = r < nrep && share_at(u, S.want, S.give, most) == 0;
        if (tid == 0) {
            S.base = base + SCAN_THREADS;
            S.q = S.count = 0;
        }
        int tot;
        const int at = rank + block_incl_scan(one ? 1 : 0, S.smi, tot) - 1, late = at - S.full * hands;
        if (one && late < 0) {
            if (at % hands == id - S.first) S.list[atomicAdd(&S.count, 1)] = r;
        } else if (one) {
            const i64 m = u < most ? u : most;
            const int per = S.per, n = (int)(m < per ? m : per), b = id - S.first - late * per;
            if (b >= 0 && b < n) {
                S.tail = r;
                S.tail_team = Team{b, n};
            }
        }
        if (tid == 0) S.rank = rank + tot;
        __syncthreads();
    }
    const int tail = S.tail;
    __syncthreads();
    if (tail < 0) return false;
    if (tid == 0) {
        S.rep = tail;
        S.team = S.tail_team;
        S.tail = -1;
    }
    __syncthreads();
    return true;
}

// a replica's arguments copied to shared memory; false if a team's wait ran
// out for it.  All threads of the block call.
__device__ __forceinline__ bool load_replica(StepArgs &a, const StepArgs &from, unsigned &err)
{
    __syncthreads();   // the replica before is done
    const u64 *src = (const u64 *)&from;
    u64 *dst = (u64 *)&a;
    for (int q = threadIdx.x; q < (int)(sizeof(StepArgs) / 8); q += blockDim.x) dst[q] = src[q];
    __syncthreads();
    if (threadIdx.x == 0) err = a.st->err;
    __syncthreads();
    return !(err & ERRB_TIMEOUT);
}

// a1 in one launch: block sums, a barrier, then every block derives the
// totals and its prefix itself and writes its entries' rows.
template <typename R, bool GAS>
__device__ __forceinline__ void d_scan(const StepArgs &a, Team t, i64 *sm)
{
    const ListView &L = a.list[a.st->cur];
    i64 bw, ba, cw, ca, tw, ta = 0;
    d_scan_partial(L, a.st, a.p, a.wa, t, bw, ba, sm);
    if (!team_sync(a.wa.bar, t, a.st)) return;
    team_prefix(a.wa.part, 4, t, sm, cw, tw);
    ca = 0;
    if (a.p.fnc) {
        __syncthreads();
        team_prefix(a.wa.part + 1, 4, t, sm, ca, ta);
    }
    const ScanScalars sc = d_scan_top(L, a.st, a.p, a.wa, tw, ta, a.s.lmax, t);
    d_scan_final<R, GAS>(a.s, L, a.st, a.p, a.wa, t, cw + bw, ca + ba, sc);
}

// MANY: nrep replicas share the launch's blocks, teams of most blocks at most
template <typename R, bool GAS, bool MANY>
__global__ void __launch_bounds__(SCAN_THREADS, 2) k_scan(const StepArgs *__restrict__ A, int nrep, int most)
{
    __shared__ i64 sm[64];
    if constexpr (MANY) {
        __shared__ Shares S;
        __shared__ StepArgs a;
        __shared__ unsigned err;
        const auto units = [&](int r) { return scan_blocks(A[r].st->n_occ); };
        shares_init(S, nrep, most, units);
        while (next_share(S, nrep, most, units))
            if (load_replica(a, A[S.rep], err)) d_scan<R, GAS>(a, S.team, sm);
    } else {
        REPLICA_SMEM;
        const i64 b = scan_blocks(a.st->n_occ);
        RETURN_IF_TIMED_OUT;
        const Team t = {(int)blockIdx.x, (int)(b < most ? b : most)};
        if (t.id < t.n) d_scan<R, GAS>(a, t, sm);
    }
}

extern __shared__ __align__(16) unsigned char dyn_smem[];

template <typename R, bool GAS, bool DIST>
__global__ void __launch_bounds__(WORK_THREADS, SAMPLE_BLOCKS_PER_SM) k_sample(const StepArgs *__restrict__ A, int enum_base)
{
    REPLICA_SMEM;
    d_sample<R, GAS, DIST>(a.s, a.list[cur_], a.st, a.p, a.wa, a.sp, a.cl, enum_base, blockIdx.x, gridDim.x,
                           ((SampWarp *)dyn_smem)[threadIdx.x >> 5]);
}

// Persistent batch sampler: each block takes the next virtual block of the
// plan, finds its replica and runs that share of the replica's samples.
template <typename R, bool GAS, bool DIST>
__global__ void __launch_bounds__(WORK_THREADS, SAMPLE_BLOCKS_PER_SM) k_sample_flat(const StepArgs *__restrict__ A, int nrep, FlatPlan fp,
                                                                 int enum_base)
{
    __shared__ StepArgs a_sm;
    __shared__ int s_v, s_r;
    const int total = fp.vstart[nrep];
    int have = -1;
    for (;;) {
        __syncthreads();   // the previous share is finished with a_sm and s_v
        if (threadIdx.x == 0) {
            const int v = (int)atomicAdd(fp.counter, 1u);
            int r = 0;
            if (v < total) {
                int lo = 0, hi = nrep - 1;   // last r with vstart[r] <= v
                while (lo < hi) {
                    const int mid = (lo + hi + 1) >> 1;
                    if (fp.vstart[mid] <= v) lo = mid;
                    else hi = mid - 1;
                }
                r = lo;
            }
            s_v = v;
            s_r = r;
        }
        __syncthreads();
        const int v = s_v;
        if (v >= total) break;
        const int r = s_r;
        if (r != have) {
            const u64 *src = (const u64 *)&A[r];
            u64 *dst = (u64 *)&a_sm;
            for (int q = threadIdx.x; q < (int)(sizeof(StepArgs) / 8); q += blockDim.x) dst[q] = src[q];
            __syncthreads();
            have = r;
        }
        const StepArgs &a = a_sm;
        const int v0 = fp.vstart[r];
        d_sample<R, GAS, DIST>(a.s, a.list[a.st->cur], a.st, a.p, a.wa, a.sp, a.cl, enum_base, v - v0,
                               fp.vstart[r + 1] - v0, ((SampWarp *)dyn_smem)[threadIdx.x >> 5]);
    }
}

template <typename R, bool GAS>
__global__ void __launch_bounds__(WORK_THREADS, SAMPLE_BLOCKS_PER_SM) k_attempts(const StepArgs *__restrict__ A)
{
    REPLICA_SMEM;
    d_attempts<R, GAS>(a.s, a.list[cur_], a.st, a.p, a.wa, a.sp, a.cl);
}

// a7-a10: sort, reduction, merge and record in one launch.  With the phase
// timers on, what selects one phase per launch.
enum { DO_SORT = 1, DO_REDUCE = 2, DO_MERGE = 4, DO_FINALIZE = 8, DO_ALL = 15 };

struct AnnihilateShape {
    int key_bits, digit_bits;
    int enum_base, enum_slots;   // the sampler's E_num partials
};

// records in the spawn buffer
__device__ __forceinline__ i64 spawned_of(const StepArgs &a) { return a.st->n_sp < a.sp.cap ? a.st->n_sp : a.sp.cap; }

// Blocks of the annihilation of nsp records: up to a tile one block, else one
// per 1,024; one per 1,024 list entries.  (n_step, not n_occ: a block that
// starts after the last one has finished the step must see the same team.)
__device__ __forceinline__ i64 annihilate_blocks(const DevStep *st, i64 nsp)
{
    const i64 bs = sort_blocks(nsp), bm = (st->n_step + 2 * SCAN_THREADS - 1) / (2 * SCAN_THREADS);
    return bs > bm ? bs : (bm < 1 ? 1 : bm);
}

template <typename R, bool GAS>
__device__ __forceinline__ void d_annihilate(const StepArgs &a, Team team, const AnnihilateShape &as, int what, SortSmem &S, i64 *sm,
                                             bool &s_last)
{
    DevStep *st = a.st;
    const int cur_ = st->cur;
    const WorkArrays &wa = a.wa;
    const ListView &L = a.list[cur_], &O = a.list[cur_ ^ 1];
    const i64 nsp = spawned_of(a);
    const i64 bs = sort_blocks(nsp);
    const Team sort_team = {team.id, (int)(bs < team.n ? bs : team.n)};
    const int src = ((as.key_bits + as.digit_bits - 1) / as.digit_bits) & 1;   // the sorted pair
    if (nsp > 0 && sort_team.id < sort_team.n) {
        if (what & DO_SORT)
            if (!team_sort(a.sp.key[0], a.sp.pop[0], a.sp.key, a.sp.pop, nsp, as.key_bits, as.digit_bits, wa.hist, wa.bar + 32, sort_team, st, S)) return;
        if (what & DO_REDUCE) {
            const i64 keys = team_reduce(a.sp.key[src], a.sp.pop[src], nsp, a.sp.key[src ^ 1], a.sp.pop[src ^ 1], wa.part,
                                         wa.bar + 32, sort_team, st, sm);
            if (keys < 0) return;
            if (sort_team.id == 0 && threadIdx.x == 0) st->n_keys = keys;
        }
    }
    if (what & DO_MERGE) {
        if (nsp > 0 && !team_sync(wa.bar, team, st)) return;
        const i64 m = __ldcg(&st->n_keys);
        const u64 *rkey = a.sp.key[src ^ 1];
        i64 *rpop = a.sp.pop[src ^ 1];
        if (m > 0) {
            d_merge_match(L, st, a.p, wa, rkey, rpop, m, team);
            if (!team_sync(wa.bar, team, st)) return;
        }
        d_merge_count(L, st, a.p, wa, m, team, sm);
        if (!team_sync(wa.bar, team, st)) return;
        const i64 kept = d_keep_scatter(L, O, st, wa, m, team, sm);
        if (m > 0) {
            if (!team_sync(wa.bar, team, st)) return;
            d_scatter_new<R, GAS>(a.s, O, st, wa, rkey, rpop, m, kept, team, S.tk);
        }
    }
    if (what & DO_FINALIZE) {
        // the last block to come here writes the record (alone: the first)
        __syncthreads();   // the block's sums are issued
        if (threadIdx.x == 0) {
            bool last = team.id == 0;
            if ((what & DO_MERGE) && team.n > 1) {
                __threadfence();
                last = atomicAdd(wa.bar + 16, 1u) == (unsigned)team.n - 1u;
                if (last) atomicExch(wa.bar + 16, 0u);
                __threadfence();
            }
            s_last = last;
        }
        __syncthreads();
        if (s_last) d_finalize(st, a.p, wa, a.cl, as.enum_base, as.enum_slots, O.cap, (u64 *)sm);
    }
}

template <typename R, bool GAS, bool MANY>
__global__ void __launch_bounds__(SCAN_THREADS, 2) k_annihilate(const StepArgs *__restrict__ A, int nrep, int most, AnnihilateShape as,
                                                                int what)
{
    __shared__ i64 sm[128];
    __shared__ bool s_last;
    SortSmem &S = *(SortSmem *)dyn_smem;
    if constexpr (MANY) {
        __shared__ Shares W;
        __shared__ StepArgs a;
        __shared__ unsigned err;
        // (records past the buffer's capacity included: one read less)
        const auto units = [&](int r) { return annihilate_blocks(A[r].st, A[r].st->n_sp); };
        shares_init(W, nrep, most, units);
        while (next_share(W, nrep, most, units))
            if (load_replica(a, A[W.rep], err)) d_annihilate<R, GAS>(a, W.team, as, what, S, sm, s_last);
    } else {
        REPLICA_SMEM;
        const i64 b = annihilate_blocks(a.st, spawned_of(a));
        RETURN_IF_TIMED_OUT;
        const Team t = {(int)blockIdx.x, (int)(b < most ? b : most)};
        if (t.id < t.n) d_annihilate<R, GAS>(a, t, as, what, S, sm, s_last);
    }
}

// Launches a grid, cooperatively (all blocks resident) if its blocks wait for
// one another.
template <typename... P, typename... Q>
cudaError_t launch_blocks(void (*k)(P...), dim3 grid, bool cooperative, int threads, size_t smem, cudaStream_t sm, Q... args)
{
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = dim3(threads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = sm;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeCooperative;
    at[0].val.cooperative = 1;
    cfg.attrs = at;
    cfg.numAttrs = cooperative ? 1 : 0;
    return cudaLaunchKernelEx(&cfg, k, static_cast<P>(args)...);
}

// Launches a kernel whose blocks wait for their replica's other blocks, teams
// of most blocks at most: as many blocks as fit on the GPU, of a single
// replica's at most those.
template <typename... P, typename... Q>
cudaError_t launch_team(void (*k)(P...), const StepArgs *A, int nrep, int most, int threads, size_t smem, cudaStream_t sm, Q... args)
{
    int dev = 0, sms = 0, per = 0;
    if (cudaError_t e = cudaGetDevice(&dev)) return e;
    if (cudaError_t e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev)) return e;
    if (smem)
        if (cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem)) return e;
    if (cudaError_t e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, k, threads, smem)) return e;
    int g = per * sms;
    if (most > g) most = g;
    if (most < 1) most = 1;
    if (nrep == 1) g = most;
    return launch_blocks(k, dim3(g), g > 1, threads, smem, sm, A, nrep, most, args...);
}

// ---------------------------------------------------------------------------
// The whole step for nrep replicas (grid dimension y), the same sequence
// every step, so it can be captured once in a CUDA graph.
// ---------------------------------------------------------------------------

template <typename R, bool GAS>
cudaError_t launch_phases(const StepArgs *A, int nrep, int K, const Shapes &sh, bool multi_att, cudaStream_t sm,
                          i64 *launches, const cudaEvent_t *ev, const FlatPlan *plan)
{
    auto mark = [&](int phase) {
        if (ev) cudaEventRecord(ev[phase], sm);
    };
    const dim3 gwork(sh.work_grid, nrep);
    const int team = min(sh.scan_grid, sh.sort_grid);
    mark(0);
    auto *scan = nrep > 1 ? k_scan<R, GAS, true> : k_scan<R, GAS, false>;
    if (cudaError_t e = launch_team(scan, A, nrep, team, SCAN_THREADS, 0, sm)) return e;
    launches[0] += 1;
    if (sh.nranks > 1) {
        // simulated distribution: owners and per-processor position tables
        launch_local_table(A, K, gwork, sm);
        k_local_scan<<<dim3(sh.nranks < 1024 ? sh.nranks : 1024, nrep), SCAN_THREADS, 0, sm>>>(A);
        launches[0] += 2;
    }
    mark(1);
    const size_t smem = (WORK_THREADS / 32) * sizeof(SampWarp);
    const bool dist = sh.nranks > 1;
    if (plan) {
        auto *k = dist ? k_sample_flat<R, GAS, true> : k_sample_flat<R, GAS, false>;
        if (cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem)) return e;
        k_sample_plan<<<1, 1024, 0, sm>>>(A, nrep, *plan, sh.scan_grid);
        k<<<plan->grid, WORK_THREADS, smem, sm>>>(A, nrep, *plan, sh.scan_grid);
        launches[1] += 2;
    } else {
        auto *k = dist ? k_sample<R, GAS, true> : k_sample<R, GAS, false>;
        if (cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem)) return e;
        k<<<gwork, WORK_THREADS, smem, sm>>>(A, sh.scan_grid);
        launches[1] += 1;
    }
    mark(2);
    if (multi_att) {
        k_attempts<R, GAS><<<gwork, WORK_THREADS, 0, sm>>>(A);
        launches[2] += 1;
    }
    const AnnihilateShape as = {sh.key_bits, sh.digit_bits, sh.scan_grid, plan ? plan->wmax : sh.work_grid};
    auto *annihilate = nrep > 1 ? k_annihilate<R, GAS, true> : k_annihilate<R, GAS, false>;
    // one launch, or with the phase timers one per phase (a7, a8, a9, a10)
    for (int ph = 0; ph < 4; ph++) {
        mark(3 + ph);
        if (!ev && ph > 0) continue;
        if (cudaError_t e = launch_team(annihilate, A, nrep, team, SCAN_THREADS, sizeof(SortSmem), sm, as, ev ? 1 << ph : (int)DO_ALL))
            return e;
        launches[3 + ph] += 1;
    }
    mark(7);
    return cudaGetLastError();
}

}  // namespace ccmc
