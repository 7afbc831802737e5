// ccmc_device.cuh -- device building blocks of the CCMC time step.
//
// Conventions (shared with the rest of the library, see include/ccmc.h):
// spin-orbital p is bit (p & 63) of word (p >> 6); 2q = alpha, 2q+1 = beta;
// the Hartree-Fock (HF) determinant is the lowest N bits; populations are
// int64 multiples of 2^-16.  Floating point is FP64 without fused
// multiply-add (the library is compiled with -fmad=false) and every
// expression below keeps the operation order documented beside it, so that
// decisions taken from FP64 values (stochastic rounding) are reproducible.
#pragma once

#include <cstdint>
#include <cstring>
#include <cuda_runtime.h>

namespace ccmc {

typedef unsigned long long u64;
typedef long long i64;

constexpr int MAXK = 6;            // words per determinant (M <= 384)
constexpr int RANK_STRIDE = 384;   // row stride of the rank tables (positions < M)
constexpr int MAX_EXC = 6;         // largest excitation level of a collapsed cluster (lmax + 2)
constexpr double FIX_ONE = 65536.0;

// Philox counter tags (bits 56..63 of counter word 1).
enum : u64 {
    TAG_SAMPLE = 1,      // cluster selection of sample g
    TAG_SAMPLE_ATT = 2,  // spawning attempt m of sample g
    TAG_VISIT = 3,       // full non-composite death draw of list entry i
    TAG_VISIT_ATT = 4,   // full non-composite attempt m of list entry i
    TAG_THRESH = 5       // occupation threshold of the excitor with a given key
};

// Device error bits (sticky status word).
enum : unsigned {
    ERRB_SPAWN_OVERFLOW = 1u,
    ERRB_NUMERIC = 2u,
    ERRB_LIST_OVERFLOW = 4u,
    ERRB_CLUSTER_OVERFLOW = 8u,
    ERRB_RUNAWAY = 16u,
    ERRB_TIMEOUT = 32u
};

// Hamiltonian and generator tables as seen by the kernels (passed by value).
struct SysDev {
    int kind;            // 0 UEG, 1 generic
    int nel, nso, lmax;
    int nw;
    u64 hf[MAXK];
    u64 valid[MAXK];     // bits < nso
    u64 virt[MAXK];      // bits in [nel, nso)
    // UEG
    int nmax;
    // k_i + k_j - k_a has components within 3 nmax, so a cube of side
    // 6 nmax + 1 holds every sum: lin[] is a wave's linear offset in it and
    // grid[mid + lin_i + lin_j - lin_a] the spatial orbital there, or -1
    int mid;
    const short *lin;    // per spatial orbital
    const short *grid;
    const int *kv;       // 3 ints per spatial orbital
    const int *kv4;      // the same packed as signed bytes (x, y, z, 0)
    const double *vtab;  // Coulomb by integer |n|^2
    double inv_pgen_ueg;
    u64 npairs, nvirt;
    const unsigned *pairs;   // pair index -> x | y << 16 (x < y, index = y (y - 1) / 2 + x)
    // generic integrals
    int norb;
    const double *h1;
    const double *eri;
    int nv[2];
    u64 ns_nd, ns;
    u64 ndcase[3];
    double inv_pgen_single[2];
    double inv_pgen_double[3];
    // rank key: tab[c * RANK_STRIDE + q] = sum_{j=0}^{l-c} C(q, j)
    const u64 *rank_tab;
    u64 cocc;
    int lmin_exc;        // smallest excitation level of any non-reference list entry
    const double *fock;  // reference Fock diagonal per spin-orbital
    // FP32 form: tables rounded from the FP64 ones
    const float *vtab_f, *h1_f, *eri_f;
    const float *fock_f;
    float inv_pgen_ueg_f;
    float inv_pgen_single_f[2];
    float inv_pgen_double_f[3];
};

// table selection by real type
template <typename R> struct Tab;
template <> struct Tab<double> {
    static __device__ __forceinline__ const double *vtab(const SysDev &s) { return s.vtab; }
    static __device__ __forceinline__ const double *h1(const SysDev &s) { return s.h1; }
    static __device__ __forceinline__ const double *eri(const SysDev &s) { return s.eri; }
    static __device__ __forceinline__ const double *fock(const SysDev &s) { return s.fock; }
};
template <> struct Tab<float> {
    static __device__ __forceinline__ const float *vtab(const SysDev &s) { return s.vtab_f; }
    static __device__ __forceinline__ const float *h1(const SysDev &s) { return s.h1_f; }
    static __device__ __forceinline__ const float *eri(const SysDev &s) { return s.eri_f; }
    static __device__ __forceinline__ const float *fock(const SysDev &s) { return s.fock_f; }
};

template <int K>
struct Det {
    u64 w[K];
};

// ---------------------------------------------------------------------------
// Philox-4x64-10 (Salmon, Moraes, Dror & Shaw, SC'11)
// ---------------------------------------------------------------------------

struct R4 {
    u64 v[4];
};

// 64x64 -> 128-bit product (host builds: four 32x32 -> 64 multiply-adds):
// x*m = p0 + 2^32 (xL mH + xH mL) + 2^64 xH mH; with t = xL mH + hi32(p0) and
// u = xH mL + lo32(t) (neither overflows), lo = lo32(p0) | lo32(u) << 32 and
// hi = xH mH + hi32(t) + hi32(u).
__host__ __device__ __forceinline__ void mulhilo64(u64 x, u64 m, u64 &hi, u64 &lo)
{
#ifdef __CUDA_ARCH__
    hi = __umul64hi(x, m);   // measured faster on sm_103a than the limb form below
    lo = x * m;
    return;
#endif
    const u64 xl = x & 0xFFFFFFFFULL, xh = x >> 32, ml = m & 0xFFFFFFFFULL, mh = m >> 32;
    const u64 p0 = xl * ml;
    const u64 t = xl * mh + (p0 >> 32);
    const u64 u = xh * ml + (t & 0xFFFFFFFFULL);
    hi = xh * mh + (t >> 32) + (u >> 32);
    lo = (p0 & 0xFFFFFFFFULL) | (u << 32);
}

__host__ __device__ __forceinline__ R4 philox(u64 c0, u64 c1, u64 c2, u64 c3, u64 k0, u64 k1)
{
    // two rounds per loop iteration: the sampler inlines several draws, and
    // fully unrolled rounds made its loop overflow the instruction cache
#pragma unroll 2
    for (int r = 0; r < 10; r++) {
        const u64 m0 = 0xD2E7470EE14C6C93ULL, m1 = 0xCA5A826395121157ULL;
        u64 hi0, lo0, hi1, lo1;
        mulhilo64(c0, m0, hi0, lo0);
        mulhilo64(c2, m1, hi1, lo1);
        u64 n0 = hi1 ^ c1 ^ k0;
        u64 n2 = hi0 ^ c3 ^ k1;
        c0 = n0;
        c1 = lo1;
        c2 = n2;
        c3 = lo0;
        k0 += 0x9E3779B97F4A7C15ULL;
        k1 += 0xBB67AE8584CAA73BULL;
    }
    R4 o;
    o.v[0] = c0;
    o.v[1] = c1;
    o.v[2] = c2;
    o.v[3] = c3;
    return o;
}

__host__ __device__ __forceinline__ R4 draw(u64 k0, u64 k1, u64 it, u64 tag, u64 index, u64 block)
{
    return philox(it, (tag << 56) | index, block, 0, k0, k1);
}

// The draws of one step: the counter's first word (the iteration), its last
// (zero) and the key are the same for every draw, so the products of the first
// round, one product of the second and all round keys are computed once per
// block and kept in shared memory.  A draw is then one product plus eight full
// rounds.  Bound by the integer multiplier (a 64 x 64 -> 128-bit product is
// four 32-bit wide multiplies of about four issue slots each): 371 issue slots
// per draw at full warps against 504 of the plain loop (148 M draws, 367 and
// 498 us on one GB300; limb and carry-chain forms of the product were slower).
struct PhiloxStep {
    u64 k0;          // key word 0
    u64 u_hi, u_lo;  // second round's product of the third word, key xor-ed into its high half
    u64 v;           // second round: low half of the iteration's product xor key
    ulonglong2 rk[8];   // round keys of rounds 3-10
};

// every thread of the block calls; the caller synchronises
__device__ __forceinline__ void philox_step_init(PhiloxStep &ps, u64 it, u64 k0, u64 k1)
{
    const u64 m0 = 0xD2E7470EE14C6C93ULL, m1 = 0xCA5A826395121157ULL;
    const u64 w0 = 0x9E3779B97F4A7C15ULL, w1 = 0xBB67AE8584CAA73BULL;
    const int t = threadIdx.x;
    if (t < 8) ps.rk[t] = make_ulonglong2(k0 + (u64)(t + 2) * w0, k1 + (u64)(t + 2) * w1);
    if (t == 8) {
        const u64 n2 = __umul64hi(it, m0) ^ k1;   // third word after the first round
        ps.k0 = k0;
        ps.u_hi = __umul64hi(n2, m1) ^ (k0 + w0);
        ps.u_lo = n2 * m1;
        ps.v = (it * m0) ^ (k1 + w1);
    }
}

// draw(k0, k1, it, tag, index, block) with the block's first-round product
// (hi1, lo1) = block * m1 given
__device__ __forceinline__ R4 step_draw_at(const PhiloxStep &ps, u64 tag, u64 index, u64 hi1, u64 lo1)
{
    const u64 m0 = 0xD2E7470EE14C6C93ULL, m1 = 0xCA5A826395121157ULL;
    u64 hi, lo;
    mulhilo64(((tag << 56) | index) ^ ps.k0 ^ hi1, m0, hi, lo);
    u64 c0 = ps.u_hi ^ lo1, c1 = ps.u_lo, c2 = hi ^ ps.v, c3 = lo;
#pragma unroll
    for (int r = 0; r < 8; r++) {
        const ulonglong2 k = ps.rk[r];
        u64 hi0, lo0, hi1r, lo1r;
        mulhilo64(c0, m0, hi0, lo0);
        mulhilo64(c2, m1, hi1r, lo1r);
        c0 = hi1r ^ c1 ^ k.x;
        c2 = hi0 ^ c3 ^ k.y;
        c1 = lo1r;
        c3 = lo0;
    }
    R4 o;
    o.v[0] = c0;
    o.v[1] = c1;
    o.v[2] = c2;
    o.v[3] = c3;
    return o;
}

__device__ __forceinline__ R4 step_draw(const PhiloxStep &ps, u64 tag, u64 index, u64 block)
{
    u64 hi1, lo1;
    mulhilo64(block, 0xCA5A826395121157ULL, hi1, lo1);
    return step_draw_at(ps, tag, index, hi1, lo1);
}

// ---------------------------------------------------------------------------
// The paper's distribution of excitors over N_p processors (Sec. III, Eq.
// ccmc_dist), simulated on one GPU: a determinant hash (Philox-4x64-10 under
// a fixed key as a mixing function over the bit string, three words per
// call, each call taking the previous result as its fourth counter word)
// and the owner o = (hash(D) + i) >> nu_move, p = hash(D xor o) mod N_p,
// with o xor-ed into the first word; nu_move >= 64 never moves an excitor.
// ---------------------------------------------------------------------------

constexpr u64 HASH_K0 = 0x243F6A8885A308D3ULL, HASH_K1 = 0x13198A2E03707344ULL;

__host__ __device__ __forceinline__ u64 words_hash(const u64 *w, int nw)
{
    u64 h = 0;
    for (int g = 0; g < nw; g += 3)
        h = philox(w[g], g + 1 < nw ? w[g + 1] : 0, g + 2 < nw ? w[g + 2] : 0, h, HASH_K0, HASH_K1).v[0];
    return h;
}

__host__ __device__ __forceinline__ u64 words_owner(const u64 *w, int nw, u64 it, int nu_move, u64 n_ranks)
{
    const u64 h = words_hash(w, nw);
    const u64 o = nu_move >= 64 ? 0 : (h + it) >> nu_move;
    u64 x[6];
    for (int i = 0; i < nw; i++) x[i] = w[i];
    x[0] ^= o;
    return words_hash(x, nw) % n_ranks;
}

// uniform in [0,1) from the top 53 bits
__device__ __forceinline__ double unif(u64 r) { return (double)(r >> 11) * 0x1p-53; }

// integer in [0, n): high word of r*n
__device__ __forceinline__ u64 below(u64 r, u64 n) { return __umul64hi(r, n); }

// ---------------------------------------------------------------------------
// Determinants as excitation lists
//
// The kernels hold a determinant as its difference from HF: the holes (empty
// spin-orbitals below N) and the particles (occupied ones from N), each an
// ascending list of 10-bit fields in one 64-bit word (positions < 384, at
// most six of each); unused fields are zero, and bits 60-63 of the hole word
// are the level n, the number of fields in either list.  Everything the step
// asks of a determinant -- the k-th occupied or empty orbital, parities,
// levels, rank keys, matrix elements -- costs a few integer operations per
// hole and particle in registers.  The bit-string form needs population
// counts (8 issue slots each on sm_103a; an attempt used about 40) and
// indexes its words by position, which put them in local memory.  The lists
// also make every kernel independent of the number of words.  Their loops are
// short and kept rolled: the sampler's loop is bound by instruction fetch
// when it is unrolled.
// ---------------------------------------------------------------------------

constexpr int FB = 10;                            // bits per field
constexpr u64 FIELDS = (1ULL << 60) - 1ULL;       // the six fields of a word
constexpr u64 FIELD_LSB = 0x0004010040100401ULL;  // lowest bit of every field

struct Exc {
    u64 h, p;   // fields only
    int n;
};

__host__ __device__ __forceinline__ int field(u64 x, int m) { return (int)(x >> (FB * m)) & 1023; }

// number of the first cnt fields below v
__device__ __forceinline__ int fields_below(u64 x, int cnt, int v)
{
    int c = 0;
#pragma unroll 1
    for (int m = 0; m < cnt; m++, x >>= FB) c += ((int)x & 1023) < v ? 1 : 0;
    return c;
}

__device__ __forceinline__ bool has_field(u64 x, int cnt, int v)
{
    bool e = false;
#pragma unroll 1
    for (int m = 0; m < cnt; m++, x >>= FB) e = e || ((int)x & 1023) == v;
    return e;
}

// v inserted before field c
__device__ __forceinline__ u64 insert_at(u64 x, int c, int v)
{
    const u64 low = (1ULL << (FB * c)) - 1ULL;
    return (x & low) | ((u64)v << (FB * c)) | ((x & ~low) << FB);
}

// field c taken out
__device__ __forceinline__ u64 remove_at(u64 x, int c)
{
    const u64 low = (1ULL << (FB * c)) - 1ULL;
    return (x & low) | ((x >> FB) & ~low);
}

// parity of the sum of the fields
__device__ __forceinline__ int sum_parity(u64 x)
{
    u64 y = x & FIELD_LSB;
    unsigned z = (unsigned)(y ^ (y >> 30));   // fields 3-5 onto 0-2
    z ^= (z >> FB) ^ (z >> (2 * FB));
    return (int)(z & 1u);
}

__device__ __forceinline__ u64 pack_h(const Exc &e) { return e.h | ((u64)e.n << 60); }

__device__ __forceinline__ Exc exc_of(u64 hn, u64 p)
{
    Exc e;
    e.h = hn & FIELDS;
    e.p = p & FIELDS;
    e.n = (int)(hn >> 60);
    return e;
}

// bit string -> lists (level at most MAX_EXC; fields beyond are dropped)
template <int K>
__device__ __forceinline__ Exc exc_from_words(const SysDev &s, const Det<K> &d)
{
    Exc e = {0, 0, 0};
    int np = 0;
#pragma unroll
    for (int w = 0; w < K; w++) {
        for (u64 m = s.hf[w] & ~d.w[w]; m; m &= m - 1) {
            if (e.n < MAX_EXC) e.h |= (u64)(64 * w + __ffsll((long long)m) - 1) << (FB * e.n);
            e.n++;
        }
        for (u64 m = d.w[w] & s.virt[w]; m; m &= m - 1) {
            if (np < MAX_EXC) e.p |= (u64)(64 * w + __ffsll((long long)m) - 1) << (FB * np);
            np++;
        }
    }
    return e;
}

template <int K>
__device__ __forceinline__ Det<K> words_from_exc(const SysDev &s, const Exc &e)
{
    Det<K> d;
#pragma unroll
    for (int w = 0; w < K; w++) d.w[w] = s.hf[w];
    u64 h = e.h, p = e.p;
    for (int m = 0; m < e.n; m++, h >>= FB, p >>= FB) {
        const int a = (int)h & 1023, b = (int)p & 1023;
#pragma unroll
        for (int w = 0; w < K; w++) {
            if ((a >> 6) == w) d.w[w] &= ~(1ULL << (a & 63));
            if ((b >> 6) == w) d.w[w] |= 1ULL << (b & 63);
        }
    }
    return d;
}

// s_D = <D|c_D|HF>: annihilating the holes h_1 < ... < h_n of HF in ascending
// order meets h_m - (m-1) occupied orbitals below h_m; creating the particles
// in descending order meets the N - n remaining electrons each time.  The sign
// is therefore (-1)^(sum h_m - n(n-1)/2 + n(N-n)); this is its parity bit.
__device__ __forceinline__ int sign_parity(const SysDev &s, int hsum_parity, int n)
{
    return (hsum_parity + n * (n - 1) / 2 + n * (s.nel - n)) & 1;
}

__device__ __forceinline__ int sign_parity(const SysDev &s, const Exc &e)
{
    return sign_parity(s, sum_parity(e.h), e.n);
}

// Applies excitor e to cur: annihilators of its holes in ascending order,
// then creators of its particles in descending order, accumulating the parity
// of the occupied orbitals passed.  Returns false if the product vanishes (an
// orbital emptied or filled twice; so does a repeated excitor).
__device__ __forceinline__ bool apply_excitor(const SysDev &s, const Exc &e, Exc &cur, int &parity)
{
    // one pass over cur counts, for each orbital of e (at most four of each),
    // the fields below it
    // (the counts packed four bits each: registers decide the sampler's speed)
    bool ok = true;
    unsigned ch = 0, cp = 0;
    u64 th = cur.h, tp = cur.p;
#pragma unroll 1
    for (int q = cur.n; q > 0; q--, th >>= FB, tp >>= FB) {
        const int h = (int)th & 1023, p = (int)tp & 1023;
#pragma unroll
        for (int m = 0; m < 4; m++) {
            if (m >= e.n) break;
            const int x = field(e.h, m), y = field(e.p, m);
            ok = ok && h != x && p != y;
            if (h < x) ch += 1u << (4 * m);
            if (p < y) cp += 1u << (4 * m);
        }
    }
    // x - c core orbitals lie below a hole x with c holes below it (e's
    // smaller ones among them); N - n + c orbitals below a particle with c
    // particles below it (n: all holes of the product; e's larger ones are
    // created first)
    const int ntot = cur.n + e.n;
#pragma unroll 1
    for (int m = 0; m < e.n; m++, ch >>= 4, cp >>= 4) {
        const int x = field(e.h, m), y = field(e.p, m), cx = (int)(ch & 15u) + m, cy = (int)(cp & 15u);
        cur.h = insert_at(cur.h, cx, x);
        cur.p = insert_at(cur.p, cy + m, y);
        parity += x + cx + s.nel - ntot + cy;
    }
    cur.n = ntot;
    return ok;
}

// ---------------------------------------------------------------------------
// Rank key: key = rank_V * C_O - rank_H (order-preserving on level <= l)
// ---------------------------------------------------------------------------

__device__ __forceinline__ u64 rank_key(const SysDev &s, const Exc &e)
{
    u64 rv = 0, rh = 0;
#pragma unroll 1
    for (int c = 0; c < e.n; c++) {
        const int m = e.n - 1 - c;   // digits from the top
        rv += __ldg(&s.rank_tab[c * RANK_STRIDE + (field(e.p, m) - s.nel)]);
        rh += __ldg(&s.rank_tab[c * RANK_STRIDE + field(e.h, m)]);
    }
    return rv * s.cocc - rh;
}

__device__ __forceinline__ Exc unrank_key(const SysDev &s, const u64 *tab, u64 key)
{
    Exc e = {0, 0, 0};
    u64 rv = (key + s.cocc - 1) / s.cocc;
    u64 rh = rv * s.cocc - key;
    // digit c of a rank: the largest position q below the previous digit with
    // tab[c][q] <= rank (tab[c][q] grows with q; tab[c][0] = 1, so a zero
    // rank has no further digits) -- a binary search per digit
    int top = s.nso - s.nel;
    for (int c = 0; c <= s.lmax && rv > 0 && top > 0; c++) {
        const u64 *t = tab + c * RANK_STRIDE;
        int lo = 0, hi = top - 1;   // tab[c][0] = 1 <= rv
        while (lo < hi) {
            const int mid = (lo + hi + 1) >> 1;
            if (t[mid] <= rv) lo = mid;
            else hi = mid - 1;
        }
        rv -= t[lo];
        e.p = (e.p << FB) | (u64)(lo + s.nel);   // the digits descend
        e.n++;
        top = lo;
    }
    top = s.nel;
    for (int c = 0; c <= s.lmax && rh > 0 && top > 0; c++) {
        const u64 *t = tab + c * RANK_STRIDE;
        int lo = 0, hi = top - 1;
        while (lo < hi) {
            const int mid = (lo + hi + 1) >> 1;
            if (t[mid] <= rh) lo = mid;
            else hi = mid - 1;
        }
        rh -= t[lo];
        e.h = (e.h << FB) | (u64)lo;
        top = lo;
    }
    return e;
}

// ---------------------------------------------------------------------------
// Matrix elements (Slater-Condon rules).  GAS selects the Hamiltonian kind at
// compile time: the two kinds' element and generator code is never both in
// one kernel's loop.
// ---------------------------------------------------------------------------

// |k_p - k_q|^2 of two spin-orbitals' plane waves
__device__ __forceinline__ int ueg_n2(const SysDev &s, int p, int q)
{
    const int a = __ldg(&s.kv4[p >> 1]), b = __ldg(&s.kv4[q >> 1]);
    const int d = (int)__vsub4((unsigned)a, (unsigned)b);   // each |component| <= 2 nmax < 128
    return __dp4a(d, d, 0);
}

template <typename R>
__device__ __forceinline__ R eri_at(const SysDev &s, int p, int q, int r, int t)
{
    size_t n = (size_t)s.norb;
    return __ldg(&Tab<R>::eri(s)[((p * n + q) * n + r) * n + t]);
}

// physicists' <pq|rs> for a momentum-conserving (UEG) or any (generic) quadruple
template <typename R, bool GAS>
__device__ __forceinline__ R g2(const SysDev &s, int p, int q, int r, int t)
{
    if (((p ^ r) & 1) || ((q ^ t) & 1)) return R(0);
    if (GAS) return __ldg(&Tab<R>::vtab(s)[ueg_n2(s, p, r)]);
    return eri_at<R>(s, p >> 1, r >> 1, q >> 1, t >> 1);
}

// <pq||pq> for p != q in the precision R: gas, minus the exchange Coulomb
// term (callers skip opposite spins, whose pair term is the omitted q = 0
// Coulomb term); molecule, (pp|qq) minus (pq|qp) for equal spins.
template <typename R, bool GAS>
__device__ __forceinline__ R pair_ex(const SysDev &s, int p, int q)
{
    if (GAS) return -__ldg(&Tab<R>::vtab(s)[ueg_n2(s, p, q)]);
    const int P = p >> 1, Q = q >> 1;
    R t = eri_at<R>(s, P, P, Q, Q);
    if (((p ^ q) & 1) == 0) t = t - eri_at<R>(s, P, Q, Q, P);
    return t;
}

template <bool GAS>
__device__ __forceinline__ bool pair_zero(int p, int q)
{
    return GAS && ((p ^ q) & 1);
}

// H_DD - E_HF from the excitation of D relative to HF: holes H and particles
// P ascending, sum_P F_a - sum_H F_i + sum_{i<j in H} <ij||ij>
// + sum_{a<b in P} <ab||ab> - sum_{a in P, i in H} <ai||ai>, in this order,
// in the precision R and promoted to double.
template <typename R, bool GAS>
__device__ __noinline__ double diag_rel(const SysDev &s, const Exc d)
{
    const R *f = Tab<R>::fock(s);
    const int n = d.n;   // <= 4
    R e = R(0);
    if constexpr (GAS) {
#pragma unroll 1
        for (int x = 0; x < 2 * n; x++) {
            const R t = __ldg(&f[x < n ? field(d.p, x) : field(d.h, x - n)]);
            e = x < n ? e + t : e - t;
        }
    } else {
        // the integrals are in the second-level cache at best: the reads of a
        // row of pairs are issued together, the sum keeps its order (1.1e7
        // molecule excitors with 9e5 new ones a step: 164 -> 140 us; the gas's
        // small tables are faster read one by one)
        R t[8];
#pragma unroll
        for (int x = 0; x < 4; x++) {
            t[x] = x < n ? __ldg(&f[field(d.p, x)]) : R(0);
            t[4 + x] = x < n ? __ldg(&f[field(d.h, x)]) : R(0);
        }
#pragma unroll
        for (int x = 0; x < 4; x++)
            if (x < n) e = e + t[x];
#pragma unroll
        for (int x = 0; x < 4; x++)
            if (x < n) e = e - t[4 + x];
    }
    // pairs of holes, pairs of particles, particle-hole pairs
#pragma unroll 1
    for (int k = 0; k < 3; k++) {
        const u64 u = k == 0 ? d.h : d.p, v = k == 1 ? d.p : d.h;
#pragma unroll 1
        for (int x = 0; x < n; x++) {
            const int a = field(u, x), y0 = k == 2 ? 0 : x + 1;
            if constexpr (GAS) {
#pragma unroll 1
                for (int y = y0; y < n; y++) {
                    const int b = field(v, y);
                    if (pair_zero<GAS>(a, b)) continue;
                    const R t = pair_ex<R, GAS>(s, a, b);
                    e = k == 2 ? e - t : e + t;
                }
            } else {
                R t[4];
#pragma unroll
                for (int q = 0; q < 4; q++)
                    if (y0 + q < n) t[q] = pair_ex<R, GAS>(s, a, field(v, y0 + q));
#pragma unroll
                for (int q = 0; q < 4; q++)
                    if (y0 + q < n) e = k == 2 ? e - t[q] : e + t[q];
            }
        }
    }
    return (double)e;
}

// <bra|H|ket> for determinants differing by one or two spin-orbitals.
// holes i<j are in ket only, particles a<b in bra only; par is the parity of
// a+_a a+_b a_j a_i |ket>.  Computed in R, returned as double.
template <typename R, bool GAS>
__device__ __forceinline__ double h_offdiag(const SysDev &s, const Exc &ket, bool dbl, int i, int j, int a, int b, int par)
{
    if (GAS || dbl) {
        R v1 = g2<R, GAS>(s, a, b, i, j);
        R v2 = g2<R, GAS>(s, a, b, j, i);
        R d = v1 - v2;
        return (double)(par ? -d : d);
    }
    if ((i ^ a) & 1) return 0.0;
    const int A = a >> 1, I = i >> 1;
    R acc = __ldg(&Tab<R>::h1(s)[A * s.norb + I]);
    // the other occupied spin-orbitals, ascending: the core without the holes, then the particles
    u64 holes = ket.h, parts = ket.p;
    int left = ket.n;
#pragma unroll 1
    for (int k = 0; k < s.nel + ket.n; k++) {
        int o = k;
        if (k >= s.nel) {
            o = (int)parts & 1023;
            parts >>= FB;
        } else if (left > 0 && ((int)holes & 1023) == k) {
            holes >>= FB;
            left--;
            continue;
        }
        if (o == i) continue;
        const int Kk = o >> 1;
        R t = eri_at<R>(s, A, I, Kk, Kk);
        if (((a ^ o) & 1) == 0) t = t - eri_at<R>(s, A, Kk, Kk, I);
        acc = acc + t;
    }
    return (double)(par ? -acc : acc);
}

// <HF|H|D> for D at level 1 or 2 (the gas has no level 1): i < j the
// particles, a < b the holes.  Below a hole lie x - c core orbitals, below a
// particle N - n + c; every hole lies below every particle.
template <typename R, bool GAS>
__device__ __forceinline__ double h_ref(const SysDev &s, const Exc &d)
{
    const int i = field(d.p, 0), j = field(d.p, 1), a = field(d.h, 0), b = field(d.h, 1);
    // one hole and particle: N - 1 + a; two: N - 2 + (N - 1 - 1) + a + (b - 1)
    const int par = GAS || d.n == 2 ? (a + b + 1) & 1 : (s.nel - 1 + a) & 1;
    return h_offdiag<R, GAS>(s, d, d.n == 2, i, j, a, b, par);
}

// ---------------------------------------------------------------------------
// Excitation generators
// ---------------------------------------------------------------------------

// pair index -> (x < y) with index = y(y-1)/2 + x, from a table: two square
// roots' worth of arithmetic per draw otherwise
__device__ __forceinline__ void pair_of(const SysDev &s, u64 idx, int &x, int &y)
{
    const unsigned v = __ldg(&s.pairs[idx]);
    x = (int)(v & 0xFFFFu);
    y = (int)(v >> 16);
}

// 1/p_gen of a generator case (0: gas double; 1, 2: molecule single of spin
// 0, 1; 3, 4, 5: molecule double of spin case 0, 1, mixed) in the precision
// R, promoted to double.
template <typename R>
__device__ __forceinline__ double inv_pgen_of(const SysDev &s, int gc)
{
    if (sizeof(R) == 4) {
        float f = gc == 0 ? s.inv_pgen_ueg_f : (gc < 3 ? s.inv_pgen_single_f[gc - 1] : s.inv_pgen_double_f[gc - 3]);
        return (double)f;
    }
    return gc == 0 ? s.inv_pgen_ueg : (gc < 3 ? s.inv_pgen_single[gc - 1] : s.inv_pgen_double[gc - 3]);
}

// k-th occupied spin-orbital (ascending): the core without the holes, then
// the particles
__device__ __forceinline__ int kth_occupied(const SysDev &s, const Exc &e, int k)
{
    const int core = s.nel - e.n;
    if (k >= core) return field(e.p, k - core);
    u64 t = e.h;
#pragma unroll 1
    for (int m = 0; m < e.n; m++, t >>= FB)
        if (((int)t & 1023) <= k) k++;
    return k;
}

// k-th empty spin-orbital (ascending): the holes, then the virtuals without
// the particles
__device__ __forceinline__ int kth_empty(const SysDev &s, const Exc &e, int k)
{
    if (k < e.n) return field(e.h, k);
    int q = s.nel + k - e.n;
    u64 t = e.p;
#pragma unroll 1
    for (int m = 0; m < e.n; m++, t >>= FB)
        if (((int)t & 1023) <= q) q++;
    return q;
}

// k-th empty spin-orbital of one spin (ascending), -1 if there are fewer
__device__ __forceinline__ int kth_empty_spin(const SysDev &s, const Exc &e, int k, int spin)
{
    u64 t = e.h;
    int c = 0, q = -1;
#pragma unroll 1
    for (int m = 0; m < e.n; m++, t >>= FB) {
        const int x = (int)t & 1023;
        if ((x & 1) != spin) continue;
        if (c == k) q = x;
        c++;
    }
    if (k < c) return q;
    q = s.nel + ((s.nel ^ spin) & 1) + 2 * (k - c);
    t = e.p;
#pragma unroll 1
    for (int m = 0; m < e.n; m++, t >>= FB) {
        const int x = (int)t & 1023;
        if ((x & 1) == spin && x <= q) q += 2;
    }
    return q < s.nso ? q : -1;
}

// One draw of the excitation generator from dj.  Returns false for a null
// draw or one that leaves the truncation; otherwise code = i | j << 10 |
// a << 20 | b << 30 | gc << 40 with the holes i<j and particles a<b relative
// to dj (j = b = 0 for a single) and the generator case gc (see inv_pgen_of).
template <bool GAS>
__device__ __forceinline__ bool excite(const SysDev &s, const Exc &dj, const R4 &r, u64 &code)
{
    int i, j = 0, a, b = 0, gc;
    if (GAS) {
        int x, y;
        pair_of(s, below(r.v[1], s.npairs), x, y);
        const int aa = kth_empty(s, dj, (int)below(r.v[2], s.nvirt));
        i = kth_occupied(s, dj, x);
        j = kth_occupied(s, dj, y);
        const int sb = (i & 1) + (j & 1) - (aa & 1);
        if (sb < 0 || sb > 1) return false;
        const int bs = __ldg(&s.grid[s.mid + __ldg(&s.lin[i >> 1]) + __ldg(&s.lin[j >> 1]) - __ldg(&s.lin[aa >> 1])]);
        const int bb = 2 * bs + sb;
        if (bs < 0 || bb == aa) return false;
        // occupied already?
        if (bb < s.nel ? !has_field(dj.h, dj.n, bb) : has_field(dj.p, dj.n, bb)) return false;
        a = min(aa, bb);
        b = max(aa, bb);
        gc = 0;
    } else {
        const bool dbl = !(below(r.v[0], s.ns_nd) < s.ns);
        int x, y = 0;
        if (dbl) pair_of(s, below(r.v[1], s.npairs), x, y);
        else x = (int)below(r.v[1], (u64)s.nel);
        i = kth_occupied(s, dj, x);
        if (dbl) j = kth_occupied(s, dj, y);
        // the empty orbitals: one of i's spin; or two of the pair's spin, or one of each
        const int c = dbl && ((i ^ j) & 1) ? 2 : (i & 1);
        const u64 many = dbl ? s.ndcase[c] : (u64)s.nv[c];
        if (many == 0) return false;
        const u64 q = below(r.v[2], many);
        int ka = (int)q, kb = 0;
        if (dbl && c < 2) pair_of(s, q, ka, kb);
        if (c == 2) {
            ka = (int)((unsigned)q / (unsigned)s.nv[1]);
            kb = (int)((unsigned)q - (unsigned)ka * (unsigned)s.nv[1]);
        }
        a = kth_empty_spin(s, dj, ka, c == 2 ? 0 : c);
        if (a < 0) return false;
        if (dbl) {
            const int bb = kth_empty_spin(s, dj, kb, c == 2 ? 1 : c);
            if (bb < 0) return false;
            b = max(a, bb);
            a = min(a, bb);
        }
        gc = (dbl ? 3 : 1) + c;
    }
    // the level changes by the core orbitals emptied and filled
    const int N = s.nel;
    int lev = dj.n + (i < N ? 1 : 0) - (a < N ? 1 : 0);
    if (GAS || gc >= 3) lev += (j < N ? 1 : 0) - (b < N ? 1 : 0);
    if (lev > s.lmax) return false;
    code = (u64)i | ((u64)j << 10) | ((u64)a << 20) | ((u64)b << 30) | ((u64)gc << 40);
    return true;
}

// dj with the drawn excitation i j -> a b applied (its level is within the
// truncation) and the parity of a+_a a+_b a_j a_i on dj.  Each orbital is
// counted once in the list it belongs to, which gives both its parity and its
// place in the new list; the orbitals that leave a list are taken out first,
// so that no list ever grows past six fields.
__device__ __forceinline__ Exc excited(const SysDev &s, const Exc &dj, bool dbl, int i, int j, int a, int b, int &parity)
{
    const int N = s.nel;
    const bool ih = i < N, jh = dbl && j < N, ah = a < N, bh = dbl && b < N;   // the core's
    int ci = 0, cj = 0, ca = 0, cb = 0;
    u64 th = dj.h, tp = dj.p;
#pragma unroll 1
    for (int m = dj.n; m > 0; m--, th >>= FB, tp >>= FB) {
        const int h = (int)th & 1023, p = (int)tp & 1023;
        ci += (ih ? h : p) < i ? 1 : 0;
        cj += (jh ? h : p) < j ? 1 : 0;
        ca += (ah ? h : p) < a ? 1 : 0;
        cb += (bh ? h : p) < b ? 1 : 0;
    }
    // occupied below x: x - c in the core, N - n + c above it; i and j are
    // removed below what follows them, b added above a
    int par = (ih ? i : N + dj.n) + ci + (ah ? a : N + dj.n) + ca + (i < a ? 1 : 0);
    if (dbl)
        par += (jh ? j : N + dj.n) + cj + (bh ? b : N + dj.n) + cb + 1 + (j < a ? 1 : 0) + (i < b ? 1 : 0) + (j < b ? 1 : 0);
    parity = par & 1;
    Exc e = dj;
    // holes: a and b filled, i and j emptied
    if (ah) e.h = remove_at(e.h, ca);
    if (bh) e.h = remove_at(e.h, cb - (ah ? 1 : 0));
    if (ih) e.h = insert_at(e.h, ci - (ah && a < i ? 1 : 0) - (bh && b < i ? 1 : 0), i);
    if (jh) e.h = insert_at(e.h, cj - (ah && a < j ? 1 : 0) - (bh && b < j ? 1 : 0) + (ih ? 1 : 0), j);
    // particles: i and j removed, a and b added
    const bool ip = !ih, jp = dbl && !jh, ap = !ah, bp = dbl && !bh;
    if (ip) e.p = remove_at(e.p, ci);
    if (jp) e.p = remove_at(e.p, cj - (ip ? 1 : 0));
    if (ap) e.p = insert_at(e.p, ca - (ip && i < a ? 1 : 0) - (jp && j < a ? 1 : 0), a);
    if (bp) e.p = insert_at(e.p, cb - (ip && i < b ? 1 : 0) - (jp && j < b ? 1 : 0) + (ap ? 1 : 0), b);
    e.n = dj.n + (ih ? 1 : 0) + (jh ? 1 : 0) - (ah ? 1 : 0) - (bh ? 1 : 0);
    return e;
}

// ---------------------------------------------------------------------------
// Stochastic rounding onto the 2^-16 grid (below cutoff: +-cutoff with
// probability |x|/cutoff).  Returns false on overflow of the fixed-point range.
// ---------------------------------------------------------------------------

__device__ __forceinline__ bool stoch_round(double x, double u, double cutoff, i64 &out)
{
    double ax = fabs(x);
    if (!(ax < 0x1p46)) {
        out = 0;
        return false;
    }
    i64 n;
    if (ax < cutoff) {
        n = (u * cutoff < ax) ? (i64)(cutoff * FIX_ONE) : 0;
    } else {
        double q = ax * FIX_ONE;
        double f = floor(q);
        n = (i64)f + ((u < q - f) ? 1 : 0);
    }
    out = x < 0.0 ? -n : n;
    return true;
}

// The same decision taken with integer arithmetic on the FP64 bit pattern.
// Every FP64 operation of stoch_round is exact -- scaling by 2^16, floor, the
// subtraction q - f, the 53-bit uniform u and, for a power-of-two cutoff,
// u * cutoff -- so comparing the exact values as scaled integers reproduces
// it bit for bit without using the (narrow) FP64 pipe.

// m < v 2^d for an integer m < 2^53 is m < this threshold (the ceiling of v 2^d;
// v 2^d is below 2^53 where d > 0)
__host__ __device__ __forceinline__ u64 scaled_threshold(u64 v, int d)
{
    if (d >= 0) return v << (d & 63);
    if (d <= -64) return v != 0 ? 1 : 0;
    return (v >> -d) + ((v & ((1ULL << -d) - 1ULL)) != 0 ? 1 : 0);
}

// |x| = M * 2^E exactly (M < 2^53)
__host__ __device__ __forceinline__ void split_double(u64 abits, u64 &M, int &E)
{
    u64 ex = abits >> 52, fr = abits & ((1ULL << 52) - 1ULL);
    if (ex == 0) {
        M = fr;
        E = -1074;
    } else {
        M = fr | (1ULL << 52);
        E = (int)ex - 1075;
    }
}

// Rounding parameters: cutoff must be 0 or a power of two (checked on the host).
struct RoundSpec {
    u64 cutoff_bits;   // bit pattern of the cutoff (0 = no cutoff)
    int cutoff_e;      // u * cutoff = m_u * 2^cutoff_e
    i64 cutoff_fixed;  // cutoff in fixed point
};

// |x| -> base, or base + inc when the uniform's integer mu = r >> 11 (u = mu 2^-53)
// is below thr; false when |x| leaves the fixed-point range
struct RoundCut {
    u64 thr;
    i64 base, inc;
};

__host__ __device__ __forceinline__ bool round_cut(u64 xbits, const RoundSpec &rs, RoundCut &c)
{
    const u64 ab = xbits & 0x7FFFFFFFFFFFFFFFULL;
    c.thr = 0;
    c.base = c.inc = 0;
    if (!(ab < 0x42D0000000000000ULL)) return false;   // |x| < 2^46 (also rejects inf and NaN)
    u64 M;
    int E;
    split_double(ab, M, E);
    u64 v = M;
    int d = E - rs.cutoff_e;               // |x| < cutoff: u cutoff < |x|
    c.inc = rs.cutoff_fixed;
    if (ab >= rs.cutoff_bits) {
        const int e = E + 16;              // q = |x| 2^16 = M 2^e; u < q - floor(q)
        c.inc = 1;
        d = 53 + e;
        if (e >= 0) {
            c.base = (i64)(M << e);
            v = 0;
            d = 0;
        } else if (e > -64) {
            c.base = (i64)(M >> -e);
            v = M & ((1ULL << -e) - 1ULL);
        }
    }
    c.thr = scaled_threshold(v, d);
    return true;
}

__host__ __device__ __forceinline__ bool stoch_round_bits(u64 xbits, u64 r, const RoundSpec &rs, i64 &out)
{
    RoundCut c;
    const bool ok = round_cut(xbits, rs, c);
    const i64 n = c.base + ((r >> 11) < c.thr ? c.inc : 0);
    out = (xbits >> 63) ? -n : n;
    return ok;
}

// ---------------------------------------------------------------------------
// Exact fixed-point accumulation of FP64 terms: each term is truncated to a
// multiple of 2^-64 and summed as a 128-bit two's-complement integer, so the
// sum is independent of the order of the terms and uses no FP64 operations.
// ---------------------------------------------------------------------------

struct Fix128 {
    u64 lo, hi;
    __host__ __device__ __forceinline__ void add(const Fix128 &b)
    {
        u64 l = lo + b.lo;
        hi = hi + b.hi + (l < lo ? 1ULL : 0ULL);
        lo = l;
    }
};

__host__ __device__ __forceinline__ Fix128 to_fix(double x)
{
    u64 bits;
    memcpy(&bits, &x, 8);
    Fix128 r = {0, 0};
    u64 ab = bits & 0x7FFFFFFFFFFFFFFFULL;
    if (ab >= 0x43E0000000000000ULL) return r;   // |x| >= 2^63: out of range (not produced by the step)
    u64 M;
    int E;
    split_double(ab, M, E);
    int sft = E + 64;                            // value * 2^64 = M * 2^sft
    if (sft >= 64) {
        r.hi = M << (sft - 64);
    } else if (sft > 0) {
        r.lo = M << sft;
        r.hi = M >> (64 - sft);
    } else if (sft > -64) {
        r.lo = M >> (-sft);
    }
    if (bits >> 63) {                            // negate
        r.lo = ~r.lo;
        r.hi = ~r.hi;
        u64 l = r.lo + 1;
        r.hi += (l == 0) ? 1ULL : 0ULL;
        r.lo = l;
    }
    return r;
}

__host__ __device__ __forceinline__ double fix_to_double(Fix128 v)
{
    bool neg = (v.hi >> 63) != 0;
    if (neg) {
        v.lo = ~v.lo;
        v.hi = ~v.hi;
        u64 l = v.lo + 1;
        v.hi += (l == 0) ? 1ULL : 0ULL;
        v.lo = l;
    }
    double d = (double)v.hi + (double)v.lo * 0x1p-64;
    return neg ? -d : d;
}

}  // namespace ccmc
