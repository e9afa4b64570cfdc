// Streaming pass over the two logit rows of an instance, as CTA-level device code, by one CTA or one cluster per row.
//
// In a single read of the rows it produces
//   - the log-sum-exp of the target row at temp_target and, per 1024-element chunk,
//     the (max, sum exp2) pair the resample draw later uses as a two-level CDF
//     (distributions from logits: App. A, first paragraph);
//   - the draft support: the `ksel` largest draft logits, equal logits resolved in
//     favour of the smaller id (top-k reduction of the problem, App. N), together
//     with the target logits at those ids.
//
// One warp takes a chunk, in batches of U 128-bit vectors of each row per lane, all of them loaded before the first is used;
// differences and scalings as packed pairs.
//
// Selection without a second pass: a threshold tau that is provably not above the ksel-th largest draft logit is derived
// from running maxima of disjoint groups of elements (each of the ksel largest group maxima is a distinct element, so the
// ksel-th largest of them bounds the answer from below), refined whenever the part read has grown fourfold; vectors with an
// element >= tau are appended to a shared candidate list and the exact answer is taken from the list at the end.  Where the
// list would not hold what is still to come, a refined threshold cuts it (keep_listed).  If it overflows all the same
// (adversarially ordered rows) an exact multi-pass radix selection over the row replaces it.
#pragma once
#include "gr_common.cuh"

namespace gr {

constexpr int kMaxChunks = 2049;     // V <= 2^21
constexpr int kMaxCluster = 8;
constexpr int kRankAll = 128;        // listed vectors that are taken apart as they are; more go through a last threshold first
constexpr int kRankKeys = 256;       // and elements of them where no threshold has been met yet (rows that are listed whole)

// Arguments common to every row.
struct ScanArgs {
    const void* q; const void* p;    // logits
    int V, ksel;
    float sc_t, sc_d;                // log2(e) / temperature
    double temp_t, temp_d;
    char* ws; char* params;          // workspace records; params block or nullptr (the caller wants the records only)
    int pstride, kcap;
};

// Shared memory.  NTHR threads, VCAP listed vectors, CAP candidates, CH chunk entries.
template <int NTHR, int VCAP, int CAP, int CH>
struct __align__(16) ScanShared {
    static constexpr int kThr = NTHR, kList = VCAP, kCap = CAP, kCh = CH;
    static_assert(20 * VCAP >= 8 * CAP && VCAP % 2 == 0, "the candidates take the list's place");
    GR_ARRAY(unsigned long long, keys, 5 * VCAP / 2);   // listed 16-byte vectors, then their first ids; in their place later composite keys
    GR_ARRAY(float2, chunk, CH);
    double lse[1], part[NTHR / 32], top;
    unsigned long long prefix;
    GR_ARRAY(unsigned int, gkey, NTHR);
    GR_ARRAY(int, hist, 256);
    int need, cnt, bad, kept;
    float tau;
    // cluster-split rows (used in the leading CTA): what the others found; bit 1 of part_bad: one of their accesses was skipped
    GR_ARRAY(int, part_cnt, kMaxCluster);
    GR_ARRAY(int, part_bad, kMaxCluster);
    // bounds-checked build: whether an access to one of the arrays was skipped
    __device__ void reset_checks() {
        GR_ARRAY_RESET(keys); GR_ARRAY_RESET(chunk); GR_ARRAY_RESET(gkey); GR_ARRAY_RESET(hist); GR_ARRAY_RESET(part_cnt); GR_ARRAY_RESET(part_bad);
    }
    __device__ int checks() {
        return GR_ARRAY_BAD(keys) | GR_ARRAY_BAD(chunk) | GR_ARRAY_BAD(gkey) | GR_ARRAY_BAD(hist) | GR_ARRAY_BAD(part_cnt) | GR_ARRAY_BAD(part_bad);
    }
};

template <typename T> struct VecTraits;
template <> struct VecTraits<float> {
    static constexpr int N = 4;
    static constexpr unsigned long long kBad = 0x7fc000007fc00000ull, kNone = 0xff800000ff800000ull;        // elements that are -infinity
    __device__ static float largest(const ulonglong2& v) { return fmaxf(fmaxf(f_lo(v.x), f_hi(v.x)), fmaxf(f_lo(v.y), f_hi(v.y))); }
    // sums of 0 * logit: zero until a NaN or an infinity makes them NaN, whatever the size of the finite ones (masks down to
    // the type's lowest value)
    typedef unsigned long long Check;
    __device__ static void check(Check& c, const ulonglong2& v) { c = fma2(v.x, 0ull, c); c = fma2(v.y, 0ull, c); }
    __device__ static bool bad(Check c) { return !(f_lo(c) == 0.f) || !(f_hi(c) == 0.f); }
    __device__ static ulonglong2 alone(float x) { ulonglong2 v; v.x = (kNone & ~0xffffffffull) | __float_as_uint(x); v.y = kNone; return v; }
    __device__ static float element(const ulonglong2& v, int i) { const unsigned long long w = i < 2 ? v.x : v.y; return i & 1 ? f_hi(w) : f_lo(w); }
    // the two packed pairs of a 16-byte vector, i = 0, 1
    __device__ static unsigned long long pair(const ulonglong2& v, int i) { return i == 0 ? v.x : v.y; }
    static constexpr int kPairs = 2;
};
template <> struct VecTraits<__nv_bfloat16> {
    static constexpr int N = 8;
    static constexpr unsigned int kBad = 0x7fc07fc0u;
    static constexpr unsigned long long kNone = 0xff80ff80ff80ff80ull;
    __device__ static __nv_bfloat162 two(unsigned int w) { return *reinterpret_cast<const __nv_bfloat162*>(&w); }
    // (on the packed elements: a third of the instructions of unpacking them first)
    __device__ static float largest(const ulonglong2& v) {
        const __nv_bfloat162 m = __hmax2(__hmax2(two((unsigned int)v.x), two((unsigned int)(v.x >> 32))), __hmax2(two((unsigned int)v.y), two((unsigned int)(v.y >> 32))));
        const unsigned int w = *reinterpret_cast<const unsigned int*>(&m);
        return fmaxf(__uint_as_float(w << 16), __uint_as_float(w & 0xffff0000u));
    }
    typedef unsigned int Check;
    __device__ static void check(Check& c, const ulonglong2& v) {
        const unsigned int w[4] = {(unsigned int)v.x, (unsigned int)(v.x >> 32), (unsigned int)v.y, (unsigned int)(v.y >> 32)};
#pragma unroll
        for (int i = 0; i < 4; i++) asm("fma.rn.bf16x2 %0, %1, %2, %0;" : "+r"(c) : "r"(w[i]), "r"(0u));
    }
    __device__ static bool bad(Check c) { return !(__uint_as_float(c << 16) == 0.f) || !(__uint_as_float(c & 0xffff0000u) == 0.f); }
    __device__ static ulonglong2 alone(float x) { ulonglong2 v; v.x = (kNone & ~0xffffull) | (__float_as_uint(x) >> 16); v.y = kNone; return v; }
    __device__ static float element(const ulonglong2& v, int i) {
        const unsigned long long w = i < 4 ? v.x : v.y;
        return __uint_as_float((unsigned int)((w >> (16 * (i & 3))) & 0xffffull) << 16);
    }
    __device__ static unsigned long long pair(const ulonglong2& v, int i) {
        const unsigned int w = (unsigned int)((i < 2 ? v.x : v.y) >> (32 * (i & 1)));
        return ((unsigned long long)(w & 0xffff0000u) << 32) | (unsigned long long)(w << 16);
    }
    static constexpr int kPairs = 4;
};
__device__ __forceinline__ float ex2(float x) {
    float y;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}
__device__ __forceinline__ float warp_max(float x) { return fkey_inv(__reduce_max_sync(0xffffffffu, fkey(x))); }
// (max, sum) of two parts of a sum of exp2((x - max) sc); an empty part is (-inf, 0)
__device__ __forceinline__ void osm_merge(float& m, float& s, float mo, float so, float sc) {
    const float mn = fmaxf(m, mo);
    const float a = (m == mn) ? s : s * ex2((m - mn) * sc);
    const float b = (mo == mn) ? so : so * ex2((mo - mn) * sc);
    s = a + b; m = mn;
}
__device__ __forceinline__ ulonglong2 ldg_stream(const void* p) {
    ulonglong2 v;
    asm volatile("ld.global.cs.v2.u64 {%0, %1}, [%2];" : "=l"(v.x), "=l"(v.y) : "l"(p));
    return v;
}

// Address of a shared-memory object in the CTA of rank `rank` of this cluster.
__device__ __forceinline__ unsigned int cluster_addr(const void* p, unsigned int rank) {
    unsigned int r;
    asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"((unsigned int)__cvta_generic_to_shared(p)), "r"(rank));
    return r;
}
__device__ __forceinline__ void st_cluster(unsigned int addr, unsigned int v) {
    asm volatile("st.shared::cluster.u32 [%0], %1;" ::"r"(addr), "r"(v) : "memory");
}
__device__ __forceinline__ void st_cluster(unsigned int addr, unsigned long long v) {
    asm volatile("st.shared::cluster.u64 [%0], %1;" ::"r"(addr), "l"(v) : "memory");
}
__device__ __forceinline__ void cluster_barrier() {
    asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
    asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
}

// The `need`-th largest of the threads' running maxima (16 leading key bits, rounded down); never below the old threshold.
// A bit of it per counting barrier (140 to 200 cycles each; one warp searching 512 values in shared memory took three times as long, four bits a round by
// ballots and shared counts half as long again).  Where there is a threshold the new one is mostly less than 128 steps above it, a factor of two:
// eight barriers then, for sixteen (one headline row 60.2 -> 58.7 us a call with the merge of parts below, 512 rows of 50257 92.5 -> 91.3 fused, 4096 bf16 rows 1438 -> 1430).
// Returns the length of the list, the same for every thread (nobody appends between the first of the barriers and the last).
template <class SS>
__device__ __forceinline__ int refine_tau(SS& sh, float mx, int need)
{
    const unsigned int key = fkey(mx);
    const float old = sh.tau;
    unsigned int res = 0, bit = 1u << 31;
    if (old > -INFINITY) {
        const unsigned int from = fkey(old) & 0xffff0000u;
        if (!(__syncthreads_count(key >= from + (128u << 16)) >= need)) { res = from; bit = 64u << 16; }
    }
#pragma unroll 1
    for (; bit >= 1u << 16; bit >>= 1) {
        const unsigned int t = res + bit;
        if (__syncthreads_count(key >= t) >= need) res = t;
    }
    const int listed = sh.cnt;
    if (threadIdx.x == 0) sh.tau = fmaxf(old, fkey_inv(res));
    __syncthreads();
    return listed;
}

// A vector that holds a candidate goes into the list as it is (with the elements beside it: eight tests and appends of their
// own were a third of the pass's instructions in bf16, where nearly every warp's vector of a wide support holds one).
template <class SS>
__device__ __forceinline__ void push_vector(SS& sh, const ulonglong2& v, int id) {
    const int slot = atomicAdd(&sh.cnt, 1);
    if (slot < SS::kList) {
        GR_ARRAY_AS(ulonglong2, sh.keys, slot) = v;
        GR_ARRAY_AS(int, sh.keys, 4 * SS::kList + slot) = id;
    }
}

// Cuts the list of `listed` vectors to those that hold an element >= tau, in place: a round's vectors are read before any of
// them is written, and what is kept of them goes to places at or before their own.
template <typename T, class SS>
__device__ __forceinline__ void keep_listed(SS& sh, int listed)
{
    const float tau = sh.tau;
    if (threadIdx.x == 0) sh.kept = 0;
#pragma unroll 1
    for (int e0 = 0; e0 < listed; e0 += SS::kThr) {
        const int e = e0 + (int)threadIdx.x;
        ulonglong2 v = VecTraits<T>::alone(-INFINITY);
        int id = 0;
        if (e < listed) { v = GR_ARRAY_AS(ulonglong2, sh.keys, e); id = GR_ARRAY_AS(int, sh.keys, 4 * SS::kList + e); }
        __syncthreads();
        if (e < listed && VecTraits<T>::largest(v) >= tau) {
            const int slot = atomicAdd(&sh.kept, 1);
            GR_ARRAY_AS(ulonglong2, sh.keys, slot) = v;
            GR_ARRAY_AS(int, sh.keys, 4 * SS::kList + slot) = id;
        }
    }
    __syncthreads();
    if (threadIdx.x == 0) sh.cnt = sh.kept;
    __syncthreads();
}

// Exact selection of the ksel largest composite keys among this CTA's chunks by eight 8-bit radix passes over them (slow
// path, taken only when the candidate list overflowed); they are left in sh.keys, their number in sh.cnt.
template <typename T, class SS>
__device__ __noinline__ void exact_select_slow(SS& sh, const T* prow, int V, int head, int nch, int first, int stride, int ksel)
{
    constexpr int kAhead = 8;                // loads in flight per thread
    const int tid = threadIdx.x;
    if (tid == 0) { sh.prefix = 0ull; sh.need = ksel; }
    __syncthreads();
#pragma unroll 1
    for (int pass = 0; pass < 9; pass++) {
        // (the ninth pass collects)
        const int shift = 56 - 8 * pass;
        if (pass < 8) for (int i = tid; i < 256; i += SS::kThr) sh.hist[i] = 0;
        if (pass == 8 && tid == 0) sh.cnt = 0;
        __syncthreads();
        const unsigned long long prefix = sh.prefix;
        // (a round's chunks are neighbours; all threads take part, also where the row has fewer chunks than the CTA warps)
        for (int c = first; c < nch; c += stride) {
            const int e1 = chunk_end(min(c + SS::kThr / 32, nch) - 1, head, nch, V);
            for (int i0 = chunk_begin(c, head) + tid; i0 < e1; i0 += kAhead * SS::kThr) {
                float v[kAhead];
#pragma unroll
                for (int u = 0; u < kAhead; u++) v[u] = i0 + u * SS::kThr < e1 ? load_logit<T>(prow, i0 + u * SS::kThr) : 0.f;
#pragma unroll
                for (int u = 0; u < kAhead; u++) {
                    const int i = i0 + u * SS::kThr;
                    if (i >= e1) break;
                    const unsigned long long key = ckey(v[u], i);
                    if (pass == 8) {
                        if (key >= prefix) {
                            const int slot = atomicAdd(&sh.cnt, 1);
                            if (slot < SS::kCap) sh.keys[slot] = key;
                        }
                    } else if (pass == 0 || (key >> (shift + 8)) == (prefix >> (shift + 8))) {
                        atomicAdd(&sh.hist[(int)((key >> shift) & 255ull)], 1);
                    }
                }
            }
        }
        __syncthreads();
        if (pass < 8 && tid == 0) {
            int need = sh.need, acc = 0, bin = 255;
            for (; bin > 0; bin--) {
                if (acc + sh.hist[bin] >= need) break;
                acc += sh.hist[bin];
            }
            sh.need = need - acc;
            sh.prefix = prefix | ((unsigned long long)bin << shift);
        }
        __syncthreads();
    }
}

// The nsel largest of the M composite keys in sh.keys, handed to `take(rank, key)`.  (Four threads to a key where there are
// enough of them.)
template <class SS, class F>
__device__ __forceinline__ void rank_select(SS& sh, int M, int nsel, F take)
{
    if (4 * M <= SS::kThr) {
        const int e = threadIdx.x >> 2, part = threadIdx.x & 3;
        const unsigned long long me = e < M ? sh.keys[e] : ~0ull;
        int rank = 0;
#pragma unroll 4
        for (int j = part; j < M; j += 4) rank += (sh.keys[j] > me) ? 1 : 0;
        __syncwarp();
        rank += __shfl_xor_sync(0xffffffffu, rank, 1);
        rank += __shfl_xor_sync(0xffffffffu, rank, 2);
        if (part == 0 && e < M && rank < nsel) take(rank, me);
        return;
    }
#pragma unroll 1
    for (int e = threadIdx.x; e < M; e += SS::kThr) {
        const unsigned long long me = sh.keys[e];
        int rank = 0;
#pragma unroll 4
        for (int j = 0; j < M; j++) rank += (sh.keys[j] > me) ? 1 : 0;
        if (rank < nsel) take(rank, me);
    }
}

// The nsel largest of the keys of `cn` parts, part p in descending order at sh.keys[p kMaxSupport ...]: a key's rank is its place in its own
// part and the numbers of larger keys in the others, by bisection in all of them at once.  (Put together and counted, 400 keys took 4 k cycles.)
template <class SS, class F>
__device__ __forceinline__ void rank_parts(SS& sh, int cn, int nsel, F take)
{
#pragma unroll 1
    for (int e = threadIdx.x; e < cn * kMaxSupport; e += SS::kThr) {
        const int part = e / kMaxSupport, at = e % kMaxSupport;
        if (at >= sh.part_cnt[part]) continue;
        const unsigned long long me = sh.keys[e];
        int pos[kMaxCluster];
#pragma unroll
        for (int p = 0; p < kMaxCluster; p++) pos[p] = 0;
#pragma unroll 1
        for (int s = kMaxSupport; s > 0; s >>= 1) {
#pragma unroll
            for (int p = 0; p < kMaxCluster; p++) {
                if (p < cn && pos[p] + s <= sh.part_cnt[p] && sh.keys[p * kMaxSupport + pos[p] + s - 1] > me) pos[p] += s;
            }
        }
        int rank = 0;
#pragma unroll
        for (int p = 0; p < kMaxCluster; p++) rank += pos[p];            // (in its own part: its place)
        if (rank < nsel) take(rank, me);
    }
}

// Terms of the row's log-sum-exp, in fp64 from the chunk table (so that the chunk masses sum to one): a chunk per thread.
template <class SS>
__device__ __forceinline__ void lse_terms(SS& sh, int nch, double temp_t)
{
    const int tid = threadIdx.x, lane = tid & 31;
    float mf = -INFINITY;
    for (int c = lane; c < nch; c += 32) mf = fmaxf(mf, sh.chunk[c].x);
    const double top = (double)warp_max(mf);
    double acc = 0.0;
#pragma unroll 1
    for (int c = tid; c < nch; c += SS::kThr) acc += (double)sh.chunk[c].y * exp_neg((top - (double)sh.chunk[c].x) / temp_t);
    if ((tid & ~31) < nch) {
#pragma unroll 1
        for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
    }
    if (lane == 0) sh.part[tid >> 5] = acc;
    if (tid == 0) sh.top = top;
}

// Row b, by this CTA (cn == 1) or by the cn CTAs of its cluster, of which this is number cr and number 0 writes the results.
// kFull: the support is the whole vocabulary and exceeds kMaxSupport; no support is selected (the draft row is read for
// unusable logits only).
template <typename T, bool kFull, int kInFlight, class SS>
__device__ __forceinline__ void scan_row(const ScanArgs& A, SS& sh, long long b, int cr, int cn, int* check)
{
    using VT = VecTraits<T>;
    constexpr int N = VT::N;
    constexpr int S = kChunk / (32 * N);   // vectors per lane and chunk
    constexpr int U = kInFlight < S ? kInFlight : S, NB = S / U;   // vectors of each row in flight, batches
    constexpr int W = SS::kThr / 32;
    static_assert(S % U == 0, "a chunk is a whole number of batches");
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int V = A.V, ksel = A.ksel;
    const T* qrow = (const T*)A.q + (size_t)b * V;
    const T* prow = (const T*)A.p + (size_t)b * V;
    const int head = row_head(A.q, b, V, (int)sizeof(T));
    const int nch = num_chunks(V, head);
    const int first = cr * W, stride = cn * W;           // this CTA's chunks: first + warp, + stride, ...
    const bool take_all = !kFull && V <= SS::kCap;       // every element is a candidate
    const bool use_tau = !kFull && !take_all;
    if (tid == 0) { sh.cnt = 0; sh.bad = 0; sh.tau = -INFINITY; sh.reset_checks(); }
    if (kFull && tid < 3) sh.hist[tid] = 0;
    if (cn > 1) cluster_barrier(); else __syncthreads();

    float g0 = -INFINITY;                  // running maximum of this thread's draft logits
    typename VT::Check chk = 0;
    const float sc_t = A.sc_t;
    const unsigned long long sc2 = f_pack(sc_t, sc_t);
    float kmax = -INFINITY, kmin = INFINITY;                // range of the log-ratios draft / target (kFull)
    // (with the rounding error of the target's product added back: ids masked by one huge value in both rows at one
    // temperature get the key 0, and not a rounding error as large as the range of all the others; a key that overflows is
    // left out, its id belongs to the first or the last bucket in any case)
    auto ratio_range = [&](unsigned long long x, unsigned long long v) {
        const unsigned long long down = f_pack(-sc_t, -sc_t), m = mul2(x, down);
        const unsigned long long err = fma2(x, down, m ^ 0x8000000080000000ull);
        const unsigned long long key = add2(fma2(v, f_pack(A.sc_d, A.sc_d), m), err);
        kmax = fmaxf(kmax, fmaxf(f_lo(key), f_hi(key))); kmin = fminf(kmin, fminf(f_lo(key), f_hi(key)));
    };
    const int rounds = (nch + stride - 1) / stride;
    float m0 = -INFINITY, s0 = 0.f, m1 = m0, s1 = s0, m2 = m0, s2 = s0, m3, s3;     // sums of the last four chunks
    const int vec_end = head + ((V - head) / N) * N, tail = V - vec_end;

    int r = 0, part = use_tau ? 1 : rounds;                 // rounds up to the next threshold
#pragma unroll 1
    while (true) {
#pragma unroll 1
        for (; r < min(part, rounds); r++) {
            const int c = first + r * stride + warp;
            const bool cvalid = c < nch;
            const bool whole = cvalid && head + (c + 1) * kChunk <= vec_end;
            // target: this lane's (max, sum exp2) of the chunk, vector by vector; the elements before the first and behind the
            // last vector come first.  (The order of these fp32 sums is part of the results: it decides the last bit of the
            // chunk masses, and with 10^5 ids a resampled token can hang on that.)
            float cm = -INFINITY, cs = 0.f;
#pragma unroll 1
            for (int nb = 0; nb < NB; nb++) {
                const int base = head + c * kChunk + (nb * U * 32 + lane) * N;
                const bool sample = use_tau && r == 0 && nb == 0;
                const float tau = sample ? INFINITY : (use_tau ? *((volatile float*)&sh.tau) : -INFINITY);
                ulonglong2 qv[U], pv[U];
                // One batch; `all`: every vector of it lies within the row, as in all chunks but the last (the tests of each vector, at its load and at
                // each use, were a third of the instructions).
                auto batch = [&](auto all) {
                    auto in = [&](int i0) { return decltype(all)::value || i0 + N <= vec_end; };
#pragma unroll
                    for (int u = 0; u < U; u++) {
                        const int i0 = base + u * 32 * N;
                        bool ok = in(i0);
#ifdef GR_CHECK
                        if (ok && (i0 < 0 || i0 + N > V || ((size_t)(qrow + i0) & 15) || ((size_t)(prow + i0) & 15))) { if (check) *check = 1; ok = false; }
#endif
                        if (ok) { qv[u] = ldg_stream(qrow + i0); pv[u] = ldg_stream(prow + i0); }
                    }
                    auto scalar = [&](int i) {
                        const float x = load_logit<T>(qrow, i), v = load_logit<T>(prow, i);
                        const float mn = fmaxf(cm, x);
                        cs = fmaf(cs, ex2((cm - mn) * sc_t), ex2((x - mn) * sc_t));
                        cm = mn;
                        chk = x - x == 0.f && v - v == 0.f ? chk : VT::kBad;
                        g0 = fmaxf(g0, v);
                        if (kFull) ratio_range(f_pack(x, x), f_pack(v, v));
                        if (!kFull && v >= tau) push_vector(sh, VT::alone(v), i);
                    };
                    if (nb == 0) {
                        if (c == 0 && lane < head) scalar(lane);
                        if (c == nch - 1 && lane < tail) scalar(vec_end + lane);
                    }
#pragma unroll
                    for (int u = 0; u < U; u++) {
                        if (in(base + u * 32 * N)) {
                            unsigned long long x[VT::kPairs];
#pragma unroll
                            for (int i = 0; i < VT::kPairs; i++) x[i] = VT::pair(qv[u], i);
                            VT::check(chk, qv[u]);
                            const float mn = fmaxf(cm, VT::largest(qv[u]));
                            // (exactly one where the maximum stands)
                            const float keep = ex2((cm - mn) * sc_t);
                            const unsigned long long nm = f_pack(-mn, -mn);
#pragma unroll
                            for (int i = 0; i < VT::kPairs; i++) {
                                const unsigned long long y = mul2(add2(x[i], nm), sc2);
                                const float e0 = ex2(f_lo(y)), e1 = ex2(f_hi(y));
                                cs = i == 0 ? fmaf(cs, keep, e0) : cs + e0;
                                cs += e1;
                            }
                            cm = mn;
                        }
                    }
                    // draft
#pragma unroll
                    for (int u = 0; u < U; u++) {
                        if (in(base + u * 32 * N)) {
                            const float vm = VT::largest(pv[u]);
                            VT::check(chk, pv[u]);
                            g0 = fmaxf(g0, vm);
                            if (kFull) {
#pragma unroll
                                for (int i = 0; i < VT::kPairs; i++) ratio_range(VT::pair(qv[u], i), VT::pair(pv[u], i));
                            }
                            if (!kFull && vm >= tau) push_vector(sh, pv[u], base + u * 32 * N);
                        }
                    }
                };
                if (whole) batch(std::true_type());
                else if (cvalid) batch(std::false_type());
                if (sample) {
                    // the first batch had no threshold: it gives one, and its draft logits, still in registers, are tested now
                    refine_tau(sh, g0, ksel);
                    if (cvalid) {
                        const float t1 = *((volatile float*)&sh.tau);
#pragma unroll
                        for (int u = 0; u < U; u++) {
                            if ((whole || base + u * 32 * N + N <= vec_end) && VT::largest(pv[u]) >= t1) push_vector(sh, pv[u], base + u * 32 * N);
                        }
                        auto scalar = [&](int i) {
                            const float v = load_logit<T>(prow, i);
                            if (v >= t1) push_vector(sh, VT::alone(v), i);
                        };
                        if (c == 0 && lane < head) scalar(lane);
                        if (c == nch - 1 && lane < tail) scalar(vec_end + lane);
                    }
                }
            }
            // the chunk's lanes put together (a butterfly from 16 lanes down), four chunks at a time: two lanes that meet each go on
            // with one of two chunks, so that four take six steps of a lane and not twenty
            m3 = m2; s3 = s2; m2 = m1; s2 = s1; m1 = m0; s1 = s0; m0 = cm; s0 = cs;
            if ((r & 3) == 3 || r == rounds - 1) {
                auto meet = [&](float& ma, float& sa, float mb, float sb, int o) {
                    const bool up = (lane & o) != 0;
                    const float ms = up ? ma : mb, ss = up ? sa : sb;
                    ma = up ? mb : ma; sa = up ? sb : sa;
                    const float mo = __shfl_xor_sync(0xffffffffu, ms, o), so = __shfl_xor_sync(0xffffffffu, ss, o);
                    osm_merge(ma, sa, mo, so, sc_t);
                };
                __syncwarp();
                float ma = m0, sa = s0, mb = m2, sb = s2;
                meet(ma, sa, m1, s1, 16);
                meet(mb, sb, m3, s3, 16);
                meet(ma, sa, mb, sb, 8);
#pragma unroll
                for (int o = 4; o > 0; o >>= 1) {
                    const float mo = __shfl_xor_sync(0xffffffffu, ma, o), so = __shfl_xor_sync(0xffffffffu, sa, o);
                    osm_merge(ma, sa, mo, so, sc_t);
                }
                const int age = (lane >> 4) + ((lane >> 3) & 1) * 2, at = c - age * stride;
                if ((lane & 7) == 0 && age <= (r & 3) && at >= 0 && at < nch) sh.chunk[at] = make_float2(ma, sa);
            }
        }
        if (r >= rounds) break;
        // A better threshold whenever the part read has grown fourfold.  With N groups (threads) about A = N ln(1 / (1 - k / N)) of
        // the elements read so far reach a fresh threshold (k = 50: 53 at 512 threads, 56 at 256; k = 100: 111, 127; k = 128: 147,
        // 177), so A elements come with the first part and 3 A more per fourfold.  Where the list does not hold what is expected
        // until the next threshold, and a quarter more (A <= k + k^2 / N), it is cut by this one: it then fits random rows of any
        // length at any support.  (Uncut, k = 128 at 256 threads lists 1370 vectors of 128256 fp32 logits, and most rows took the
        // exact selection: 1024 rows, acceptance alone, 1450 us; now 215, and 209 at k = 100, where nothing is cut.  A call or the
        // cut inside the loop over the rounds cost calls that need no cut 1 to 2 %.)
        const int listed = refine_tau(sh, g0, ksel);
        const int more = (ksel + ksel * ksel / SS::kThr) * min(3 * r, rounds - r);           // times r
        if (listed <= SS::kList && 5 * more > 4 * (SS::kList - listed) * r) keep_listed<T>(sh, listed);
        part *= 4;
    }
    // non-finite inputs
    {
        const bool badl = VT::bad(chk);
        if (__any_sync(0xffffffffu, badl) && lane == 0) atomicOr(&sh.bad, 1);
    }
    // ---- candidates: a last threshold from the list itself, then composite keys of those that pass it
    __syncthreads();
    if (cn == 1) lse_terms(sh, nch, A.temp_t);
    int M = 0, nsel = 0;
    if (!kFull) {
        nsel = ksel < V ? ksel : V;
        M = min(sh.cnt, SS::kList);
        bool over = sh.cnt > SS::kList;
        if (!over) {
            constexpr int kPer = (SS::kList + SS::kThr - 1) / SS::kThr;
            ulonglong2 vv[kPer];
            int id[kPer];
            float own = -INFINITY;
#pragma unroll
            for (int u = 0; u < kPer; u++) {
                const int e = tid + u * SS::kThr;
                vv[u].x = VT::kNone; vv[u].y = VT::kNone; id[u] = 0;
                if (e < M) { vv[u] = GR_ARRAY_AS(ulonglong2, sh.keys, e); id[u] = GR_ARRAY_AS(int, sh.keys, 4 * SS::kList + e); }
                own = fmaxf(own, VT::largest(vv[u]));
            }
            // (the threads' shares of the list are the groups: in a short row the threads' maxima are too few to tell anything, and
            // ranking 1500 elements among themselves took 60 us)
            if (M > kRankAll) refine_tau(sh, own, nsel);
            else if (sh.tau == -INFINITY && M * N > kRankKeys) {
                // Up to 1024 elements in few vectors, all of them candidates: halves of a vector are the groups, quarters up to
                // 64 vectors, so that there are as many as a support has tokens.  (400 rows, k = 8: 1000 bf16 logits 115 -> 31 us,
                // 600 64 -> 31, 500 fp32 ones 51 -> 31.)
                static_assert(2 * kRankAll <= SS::kThr && 2 * (kRankKeys / 4) >= kMaxSupport && 4 * (kRankKeys / 8) >= kMaxSupport, "groups");
                const int lg = M > kRankAll / 2 ? 1 : 2, e = tid >> lg, n0 = (tid & ((1 << lg) - 1)) * (N >> lg);
                float most = -INFINITY;
                if (e < M) {
                    const ulonglong2 v = GR_ARRAY_AS(ulonglong2, sh.keys, e);
                    for (int i = 0; i < N >> lg; i++) most = fmaxf(most, VT::element(v, n0 + i));
                }
                refine_tau(sh, most, nsel);
            }
            const float tau = sh.tau;
            if (tid == 0) sh.kept = 0;
            __syncthreads();
            if (own >= tau) {
#pragma unroll
                for (int u = 0; u < kPer; u++) {
                    if (VT::largest(vv[u]) >= tau) {
#pragma unroll
                        for (int i = 0; i < N; i++) {
                            const float v = VT::element(vv[u], i);
                            if (v >= tau && v > -INFINITY) {
                                const int slot = atomicAdd(&sh.kept, 1);
                                if (slot < SS::kCap) sh.keys[slot] = ckey(v, id[u] + i);
                            }
                        }
                    }
                }
            }
            __syncthreads();
            M = sh.kept;
            over = M > SS::kCap;
        }
        if (over) {
            __syncthreads();
            exact_select_slow<T>(sh, prow, V, head, nch, first, stride, nsel);
            M = min(sh.cnt, SS::kCap);
        }
    }
    if (cn > 1) {
        // ---- the other CTAs' parts to the first one: chunk entries, status, and each one's own nsel largest keys
        const unsigned int lead_chunk = cluster_addr(&sh.chunk[0], 0), lead_keys = cluster_addr(&sh.keys[0], 0);
        if (cr > 0) {
            for (int c = first + warp; c < nch; c += stride) {
                if (lane == 0) {
                    const float2 t = sh.chunk[c];
#ifdef GR_CHECK
                    if (c >= SS::kCh) { *check = 1; continue; }
#endif
                    st_cluster(lead_chunk + 8u * (unsigned)c, f_pack(t.x, t.y));
                }
            }
        }
        const int keep = min(M, nsel);
        // (the leader's list is overwritten only after it has taken its own largest: a barrier on both sides)
        unsigned long long own = 0ull;
        int own_rank = -1;
        // keep <= kMaxSupport <= kThr candidates survive in one CTA; a thread may hold several of the M, so survivors go
        // through the upper half of the key array
        constexpr int stage = SS::kCap - kMaxSupport;
        const bool overlap = M > SS::kCap - kMaxSupport;
        if (!overlap) rank_select(sh, M, keep, [&](int rank, unsigned long long key) { sh.keys[stage + rank] = key; });
        __syncthreads();
        if (!overlap && tid < keep) { own = sh.keys[stage + tid]; own_rank = tid; }
        if (overlap) {
            // (a list this full comes from rows of ties only: one thread per key, ranks counted from global order)
            for (int e = tid; e < M; e += SS::kThr) {
                const unsigned long long me = sh.keys[e];
                int rank = 0;
                for (int j = 0; j < M; j++) rank += (sh.keys[j] > me) ? 1 : 0;
                if (rank < keep) sh.gkey[rank] = (unsigned int)e;
            }
            __syncthreads();
            if (tid < keep) { own = sh.keys[sh.gkey[tid]]; own_rank = tid; }
        }
#ifdef GR_CHECK
        if (own_rank >= kMaxSupport || (cr + 1) * kMaxSupport > SS::kCap) { *check = 1; own_rank = -1; }
#endif
        cluster_barrier();
        if (tid == 0) {
            st_cluster(cluster_addr(&sh.part_cnt[cr], 0), (unsigned int)keep);
            st_cluster(cluster_addr(&sh.part_bad[cr], 0), (unsigned int)(sh.bad | ((sh.checks() | (check ? *check : 0)) ? 2 : 0)));
        }
        if (own_rank >= 0) st_cluster(lead_keys + 8u * (unsigned)(cr * kMaxSupport + own_rank), own);
        cluster_barrier();
        if (cr > 0) return;
        M = 0;
        for (int i = 0; i < cn; i++) M += sh.part_cnt[i];
        if (tid == 0) {
            for (int i = 1; i < cn; i++) {
                sh.bad |= sh.part_bad[i] & 1;
                if (check && (sh.part_bad[i] & 2)) *check = 1;
            }
        }
    }

    if (kFull) {
        // (sh.hist is zero)
        const unsigned a = __reduce_max_sync(0xffffffffu, fkey(g0)), k1 = __reduce_max_sync(0xffffffffu, fkey(kmax));
        const unsigned k0 = __reduce_max_sync(0xffffffffu, fkey(-kmin));
        if (lane == 0) {
            atomicMax(&GR_ARRAY_AS(unsigned, sh.hist, 0), a); atomicMax(&GR_ARRAY_AS(unsigned, sh.hist, 1), k1);
            atomicMax(&GR_ARRAY_AS(unsigned, sh.hist, 2), k0);
        }
    }
    // ---- row totals (the terms are in shared memory since a barrier at least)
    if (cn > 1) lse_terms(sh, nch, A.temp_t);
    if (cn > 1 || kFull) __syncthreads();
    if (tid == SS::kThr - 1) {
        double acc = sh.part[0];
#pragma unroll
        for (int w = 1; w < W; w++) acc += sh.part[w];
        sh.lse[0] = sh.top / A.temp_t + m_log(acc);
        if (!isfinite(sh.lse[0])) sh.bad = 1;
    }
    // ---- exact support out of the candidates
    char* wsb = A.ws + (size_t)b * ws_stride();
    if (!kFull) {
        int* w_id_raw = reinterpret_cast<int*>(wsb + sizeof(WsHeader));
        float* w_dl_raw = reinterpret_cast<float*>(w_id_raw + kMaxSupport);
        GR_PTR(int) w_id = GR_MKPTR(int, w_id_raw, kMaxSupport, check);
        GR_PTR(float) w_dl = GR_MKPTR(float, w_dl_raw, kMaxSupport, check);
        GR_PTR(float) w_tl = GR_MKPTR(float, w_dl_raw + kMaxSupport, kMaxSupport, check);
        if (M < nsel) nsel = M;   // cannot happen for finite rows; keeps the writes in range
        auto take = [&](int rank, unsigned long long key) {
            int id = (int)(0xffffffffu - (unsigned int)key);
#ifdef GR_CHECK
            if (id < 0 || id >= V) { if (check) *check = 1; id = 0; }
#endif
            w_id[rank] = id;
            w_dl[rank] = fkey_inv((unsigned int)(key >> 32));
            w_tl[rank] = load_logit<T>(qrow, id);
        };
        if (cn > 1) rank_parts(sh, cn, nsel, take);
        else rank_select(sh, M, nsel, take);
    }
    __syncthreads();
    // ---- outputs: workspace header, chunk table and the header fields owned by this pass
    if (tid == 0) {
        WsHeader* wh = reinterpret_cast<WsHeader*>(wsb);
        wh->lse_t = sh.lse[0];
        wh->flagged = 0; wh->taken = 0;
        wh->count = nsel;
        wh->bad = sh.bad;
        wh->check = sh.checks() | (check ? *check : 0);
        if (kFull) {
            FullRow fr;
            fr.pmax = fkey_inv(GR_ARRAY_AS(unsigned, sh.hist, 0)); fr.kmax = fkey_inv(GR_ARRAY_AS(unsigned, sh.hist, 1));
            fr.kmin = -fkey_inv(GR_ARRAY_AS(unsigned, sh.hist, 2)); fr.qmax = (float)sh.top;
            *reinterpret_cast<FullRow*>(wsb + sizeof(WsHeader)) = fr;
        }
    }
    if (A.params == nullptr) return;
    char* pb = A.params + (size_t)b * A.pstride;
    ParamView pv = view_params(pb, A.kcap, V, check);
    for (int c = tid; c < nch; c += SS::kThr) pv.chunk[c] = sh.chunk[c];
    if (tid == 0) {
        Header* h = pv.h;
        h->magic = 0;            // completed by the solve
        h->V = V; h->nch = nch; h->head = head;
        h->q_row = qrow;
        h->dtype = sizeof(T) == 2 ? GR_BF16 : GR_F32;
        h->lse_t = sh.lse[0];
        h->temp_target = (float)A.temp_t;
        h->kcap = A.kcap; h->stride = A.pstride;
    }
}

}  // namespace gr
