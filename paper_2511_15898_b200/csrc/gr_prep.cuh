// Steps shared by the two solve kernels (one CTA per instance, any block size that is a multiple of 32
// and at least the support size): distributions on the support, ratio order, subset selection,
// outer residuals and blocks; writing the rule into the params block.
#pragma once
#include "gr_common.cuh"

namespace gr {

constexpr int kNeedFallback = 100;   // internal status: the fast kernel asks the general kernel to redo the instance

// CTA-wide reductions; `scratch` needs one double per warp.  Every thread gets the result.  (Out of line where they are used
// once per instance; the general kernel's iteration takes the inline forms.)
__device__ __forceinline__ double reduce_max(double v, GR_PTR(double) scratch) {
    __syncwarp();
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v = fmax(v, __shfl_xor_sync(0xffffffffu, v, o));
    const int nw = blockDim.x >> 5;
    __syncthreads();
    if ((threadIdx.x & 31) == 0) scratch[threadIdx.x >> 5] = v;
    __syncthreads();
    double r = scratch[0];
#pragma unroll 1
    for (int i = 1; i < nw; i++) r = fmax(r, scratch[i]);
    return r;
}
__device__ __forceinline__ double reduce_sum(double v, GR_PTR(double) scratch) {
    __syncwarp();
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    const int nw = blockDim.x >> 5;
    __syncthreads();
    if ((threadIdx.x & 31) == 0) scratch[threadIdx.x >> 5] = v;
    __syncthreads();
    double r = 0.0;
#pragma unroll 1
    for (int i = 0; i < nw; i++) r += scratch[i];
    return r;
}
static __device__ __noinline__ double block_reduce_max(double v, GR_PTR(double) scratch) { return reduce_max(v, scratch); }
static __device__ __noinline__ double block_reduce_sum(double v, GR_PTR(double) scratch) { return reduce_sum(v, scratch); }

// order-preserving map double -> uint64 (larger double, larger key; the two zeros have one key)
__device__ __forceinline__ unsigned long long order_key(double x) {
    const unsigned long long u = (unsigned long long)__double_as_longlong(x + 0.0);
    return (u >> 63) ? ~u : (u | 0x8000000000000000ull);
}
// How many of keys[lo .. hi) are above `key`.  Integers, strict comparisons and several loads ahead: 50 fp64 keys with the
// tie rule in the comparison took 5.8 k cycles, a warp's ballots 5.4 k, this with what surrounds it 1.3 k.
__device__ __forceinline__ int count_above(GR_PTR(const unsigned long long) keys, int lo, int hi, unsigned long long key)
{
    int n0 = 0, n1 = 0;
#pragma unroll 8
    for (int j = lo; j < hi; j += 2) {
        const unsigned long long a = keys[j], b = keys[min(j + 1, hi - 1)];
        n0 += a > key ? 1 : 0;
        n1 += (b > key && j + 1 < hi) ? 1 : 0;
    }
    return n0 + n1;
}

// The same over keys[0 .. k), 16-byte aligned, with zeros (no key) up to the next multiple of four.
__device__ __forceinline__ int count_above_all(GR_PTR(const unsigned long long) keys, int k, unsigned long long key)
{
    int n0 = 0, n1 = 0;
#pragma unroll 4
    for (int j = 0; j < k; j += 4) {
        const ulonglong2 a = ld_ull2(keys + j), b = ld_ull2(keys + j + 2);
        n0 += (a.x > key ? 1 : 0) + (b.x > key ? 1 : 0);
        n1 += (a.y > key ? 1 : 0) + (b.y > key ? 1 : 0);
    }
    return n0 + n1;
}

// Position of this thread's token among those of [lo, hi): larger keys first, equal keys by smaller id.  keys and ids are visible to all;
// `scratch` is overwritten.  Every thread of the CTA calls it (as many threads as tokens at least; lo == hi: no token), a group's threads with one range.
// kAll: one range from 0 on, padded for count_above_all.
template <bool kAll>
__device__ __forceinline__ int ratio_rank(GR_PTR(const unsigned long long) keys, GR_PTR(const int) ids, GR_PTR(int) scratch, int lo, int hi,
                                          unsigned long long key, int my_id)
{
    const int tid = threadIdx.x;
    const bool on = lo < hi;
    int rank = !on ? 0 : kAll ? count_above_all(keys, hi, key) : lo + count_above(keys, lo, hi, key);
    // equal keys have met at one rank: whoever does not find himself there has company
    if (on) scratch[rank] = tid;
    __syncthreads();
    if (__syncthreads_or(on && scratch[rank] != tid)) {
        if (on) {
            int before = 0;
            for (int j = lo; j < hi; j++) before += (keys[j] == key && ids[j] < my_id) ? 1 : 0;
            rank += before;
        }
    }
    return rank;
}
// Prefix sums of two arrays (dst[j] = src[0] + ... + src[j - 1], dst[0] = 0), each summed in order, one after the other, by a thread of
// its own (threads 0 and 32, which own what they wrote until the next barrier), eight loads ahead of the additions.
__device__ __forceinline__ void prefix_sums(GR_PTR(const double) src0, GR_PTR(double) dst0, GR_PTR(const double) src1, GR_PTR(double) dst1, int k)
{
    if (threadIdx.x == 0 || threadIdx.x == 32) {
        GR_PTR(const double) src = src0;
        GR_PTR(double) dst = dst0;
        if (threadIdx.x == 32) { src = src1; dst = dst1; }
        double acc = 0.0;
        dst[0] = 0.0;
#pragma unroll 1
        for (int j0 = 0; j0 < k; j0 += 8) {
            double v[8];
#pragma unroll
            for (int u = 0; u < 8; u++) v[u] = src[min(j0 + u, k - 1)];
#pragma unroll
            for (int u = 0; u < 8; u++) {
                acc += v[u];
                if (j0 + u < k) dst[j0 + u + 1] = acc;
            }
        }
    }
}

// shared-memory arrays of the preparation (KP entries each; psi and Dr: KP + 4)
struct PrepSm {
    GR_PTR(double) d, tg, p, r, key, psi, Dr;
    GR_PTR(int) id, blk, itmp;
    GR_PTR(double) red;     // two doubles per warp of reduction scratch
    GR_PTR(double) out3;    // 3 doubles: jstar, nblocks, alpha*
};
struct PrepResult { int k, jstar, nblocks; double alpha_star, lse_t; };

struct WsView { const WsHeader* h; GR_PTR(const int) id; GR_PTR(const float) dl; GR_PTR(const float) tl; };
__device__ inline WsView view_ws(const char* ws, long long b, int* flag = nullptr) {
    WsView v;
    v.h = reinterpret_cast<const WsHeader*>(ws + (size_t)b * ws_stride());
    const int* ids = reinterpret_cast<const int*>((const char*)v.h + sizeof(WsHeader));
    const float* dls = reinterpret_cast<const float*>(ids + kMaxSupport);
    v.id = GR_MKPTR(const int, ids, kMaxSupport, flag);
    v.dl = GR_MKPTR(const float, dls, kMaxSupport, flag);
    v.tl = GR_MKPTR(const float, dls + kMaxSupport, kMaxSupport, flag);
    (void)flag;
    return v;
}

// Header of an instance for which no rule exists (support beyond the capacity, or unusable logits).
__device__ inline void write_no_rule(Header* h, int n, bool bad, float* alpha_out, int* status_out, long long b) {
    h->n = n; h->k = 0; h->jstar = 0; h->nblocks = 0;
    h->status = bad ? GR_BAD_LOGITS : GR_SUPPORT_TOO_LARGE;
    h->alpha_star = __longlong_as_double(0x7ff8000000000000ll);
    h->resid_total = 1.0; h->gnorm = 0.0; h->iters = 0;
    h->magic = kMagic;
    alpha_out[b] = __int_as_float(0x7fc00000);
    status_out[b] = h->status;
}

// Everything before the convex minimisation.  Every thread of the CTA calls it; the block has at least as many threads
// as the support has tokens.  Bound by latency (a chain of short steps on at most 128 numbers), so every step but the
// in-order prefix sums is one position per thread with warp scans and ballots.
__device__ inline PrepResult prep_instance(const PrepSm& sm, const WsView& wv, Header* hdr, int V, int n, int topk,
                                           double temp_t, double temp_d)
{
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, nw = blockDim.x >> 5;
    const int kfull = (topk <= 0 || topk >= V) ? V : topk;
    const int k = wv.h->count;
    const int kw = (k + 31) >> 5;                 // warps that hold tokens
    const bool on = tid < k;
    double lse_t = wv.h->lse_t;
    // ---- distributions on the support (App. A; App. N): fp64 from the fp32 / bf16 logits
    double a_i = 0.0, b_i = 0.0, bmax = 0.0;
    unsigned long long key = 0ull;
    int my_id = 0;
    if (on) {
        my_id = wv.id[tid];
        a_i = m_div((double)wv.tl[tid], temp_t);
        const double2 b2 = m_div2((double)wv.dl[tid], (double)wv.dl[0], temp_d);
        // (the streaming pass leaves the support in descending order: the first entry is the largest)
        b_i = b2.x; bmax = b2.y;
        key = order_key(b_i - a_i);
        sm.itmp[tid] = my_id;
    }
    if (tid < ((k + 3) & ~3)) GR_PCAST(unsigned long long, sm.key)[tid] = key;
    const double eb = on ? m_exp(b_i - bmax) : 0.0;
    const double bsum = block_reduce_sum(eb, sm.red);
    double tg_i;
    if (kfull == V) {
        // the support is the whole vocabulary: normalise the target in fp64 over these same entries, so that
        // it sums to one to rounding (the streaming kernel's fp32 sum is only good to ~1e-7, which would
        // leave the outermost block's flows inconsistent with the mass of the tuples that feed them)
        const double amax = block_reduce_max(on ? a_i : -1.0e300, sm.red);
        const double ea = on ? m_exp(a_i - amax) : 0.0;
        const double asum = block_reduce_sum(ea, sm.red);
        lse_t = amax + m_log(asum);
        tg_i = m_div(ea, asum);
        if (tid == 0) hdr->lse_t = lse_t;
    } else {
        tg_i = on ? m_exp(a_i - lse_t) : 0.0;
    }
    // ---- ratio order: decreasing log-ratio key, equal keys by smaller id (Sec. 5.1)
    // (the reductions above made the keys visible)
    const int rank = ratio_rank<true>(GR_PCAST(const unsigned long long, sm.key), sm.itmp, sm.blk, 0, on ? k : 0, key, my_id);
    if (on) {
        sm.id[rank] = my_id;
        sm.tg[rank] = tg_i;
        sm.d[rank] = m_div(eb, bsum);
    }
    __syncthreads();
    // ---- prefix sums in order, psi along the chain, H* and alpha* (Eq. "subset-select")
    prefix_sums(sm.tg, sm.psi, sm.d, sm.Dr, k);
    // both distributions are normalised
    if (tid == 0 && kfull == V) sm.psi[k] = 1.0;
    if (tid == 32) sm.Dr[k] = 1.0;
    __syncthreads();
    // thread `pos` owns psi[pos + 1]
    double v = 1.0e300;
    if (on) {
        double pw = 1.0, sq = sm.Dr[tid + 1];
#pragma unroll 1
        for (int e = n; e > 0; e >>= 1) { if (e & 1) pw *= sq; sq *= sq; }
        v = sm.psi[tid + 1] - pw;
        sm.psi[tid + 1] = v;
    }
    // minimum of psi over the positions from this one up (inclusive of psi[pos + 1]): a suffix scan, exact in any order
    double suf = v;
#pragma unroll 1
    for (int o = 1; o < 32; o <<= 1) {
        const double t = __shfl_down_sync(0xffffffffu, suf, o);
        if (lane + o < 32) suf = fmin(suf, t);
    }
    __syncthreads();
    if (lane == 0) sm.red[warp] = suf;
    __syncthreads();
    double best = 0.0;                            // psi of the empty prefix
#pragma unroll 1
    for (int w2 = 0; w2 < kw; w2++) {
        const double t = sm.red[w2];
        best = fmin(best, t);
        if (w2 > warp) suf = fmin(suf, t);
    }
    // first strict minimum of psi (H* = the prefix up to it)
    __syncthreads();
    {
        const unsigned hit = __ballot_sync(0xffffffffu, on && best < 0.0 && v == best);
        if (lane == 0) sm.red[warp] = hit ? (double)(warp * 32 + __ffs(hit)) : 0.0;
    }
    __syncthreads();
    int jstar = 0;
#pragma unroll 1
    for (int w2 = kw - 1; w2 >= 0; w2--) { const double t = sm.red[w2]; if (t > 0.0) jstar = (int)t; }
    // ---- outer residuals by cumulative minima along the increasing-ratio chain; blocks end at
    //      every new strict minimum (Sec. 6.1, Thm "polymatroid", Lemma "q-convex").  `suf` is the running minimum
    //      that reaches this position; its block number counts the strict minima above it.
    const bool outer = on && tid >= jstar;
    const double c = on ? sm.psi[tid] : 0.0;
    const unsigned recs = __ballot_sync(0xffffffffu, outer && c < suf);
    if (lane == 0) sm.red[nw + warp] = (double)__popc(recs);
    __syncthreads();
    if (on) {
        if (!outer) {
            sm.p[tid] = sm.tg[tid]; sm.r[tid] = 0.0; sm.blk[tid] = -1;
        } else {
            int blk = __popc(recs & ~((2u << lane) - 1u));
#pragma unroll 1
            for (int w2 = warp + 1; w2 < kw; w2++) blk += (int)sm.red[nw + w2];
            const double rr = c < suf ? suf - c : 0.0;
            sm.r[tid] = rr;
            sm.p[tid] = sm.tg[tid] - rr;
            sm.blk[tid] = blk;
            // the lowest position of the chain closes the last block: it is open unless this position is a record
            if (tid == jstar) sm.out3[1] = (double)(blk + 1);
        }
    }
    if (tid == 0) {
        sm.out3[0] = (double)jstar;
        if (jstar >= k) sm.out3[1] = 0.0;
        sm.out3[2] = 1.0 + best;
    }
    __syncthreads();
    PrepResult pr;
    pr.k = k; pr.jstar = jstar; pr.nblocks = (int)sm.out3[1]; pr.alpha_star = 1.0 + best; pr.lse_t = lse_t;
    return pr;
}

// Truncation sets of the truncated variant (Sec. 6.2 "tunable errors", Sec. 6.3, Algorithm 1): the fewest tokens with
//   inner:  T in H*,       gamma_T   = drf(H*)^n - drf(T)^n      <= tau,
//   outer:  T in V \ H*,   epsilon_T = 1 - (drf(H*) + drf(T))^n  <= tau,
// i.e. tokens in decreasing drf (equal drf: smaller id first) until the bound holds.  in_T[pos] = 1 / 0 for the
// k support positions (ratio order); scratch: k ints.  sm.key and sm.psi are overwritten.  Every thread of the CTA calls it (blockDim.x >= k,
// two warps at least).  The bounds of both groups' prefixes fall with their length (sums and powers of numbers that grow are monotone in floating
// point too), so a token is in the set if and only if the bound of those before it does not hold yet: one token per thread, and only the sums are a chain.
// (One thread walking both groups, a power per token, took 23 k cycles of 50 tokens and n = 8: 512 rows of 128256, tau = 1e-3, solve 180 us, so 171.)
__device__ inline void truncation_sets(const PrepSm& sm, GR_PTR(int) in_T, GR_PTR(int) scratch, int k, int jstar, int n,
                                       double tau)
{
    const int tid = threadIdx.x;
    // rank inside the own group (H* or the outer support) by (drf descending, id ascending)
    const bool on = tid < k, inner = tid < jstar;
    const int lo = inner ? 0 : jstar, hi = inner ? jstar : k;
    const double dv = on ? sm.d[tid] : 0.0;
    GR_PTR(unsigned long long) keys = GR_PCAST(unsigned long long, sm.key);
    if (on) keys[tid] = order_key(dv);
    __syncthreads();
    const int rank = ratio_rank<false>(keys, sm.id, scratch, lo, on ? hi : lo, order_key(dv), on ? sm.id[tid] : 0);
    __syncthreads();
    if (on) { scratch[rank] = tid; sm.key[rank] = dv; }
    __syncthreads();
    // sums before a token, in order: a thread for each group (the outer one's begin with the mass of H*), eight loads ahead of the additions
    if (tid == 0 || tid == 32) {
        const int b0 = tid == 0 ? 0 : jstar, b1 = tid == 0 ? jstar : k;
        double acc = tid == 0 ? 0.0 : sm.Dr[jstar];
#pragma unroll 1
        for (int j0 = b0; j0 < b1; j0 += 8) {
            double v[8];
#pragma unroll
            for (int u = 0; u < 8; u++) v[u] = sm.key[min(j0 + u, b1 - 1)];
#pragma unroll
            for (int u = 0; u < 8; u++) {
                if (j0 + u < b1) sm.psi[j0 + u] = acc;
                acc += v[u];
            }
        }
    }
    __syncthreads();
    if (on) {
        auto powi = [](double x, int e) {
            double r = 1.0;
#pragma unroll 1
            for (; e > 0; e >>= 1) { if (e & 1) r *= x; x *= x; }
            return r;
        };
        // (this thread's rank in the order of masses, whichever token it is)
        const double before = powi(sm.psi[tid], n), all = powi(sm.Dr[jstar], n);
        in_T[scratch[tid]] = (inner ? all - before : 1.0 - before) > tau ? 1 : 0;
    }
    __syncthreads();
}

// The T-part of positions lo .. hi-1 gathered into contiguous arrays (draft masses, right-hand sides, positions);
// returns how many.  Every thread of the CTA calls it; `count` is one int of shared memory.
__device__ inline int gather_truncated(GR_PTR(const int) in_T, int lo, int hi, GR_PTR(const double) d,
                                       GR_PTR(const double) rhs, GR_PTR(double) dT, GR_PTR(double) rT, GR_PTR(int) map,
                                       int* count)
{
    __syncthreads();
    if (threadIdx.x == 0) {
        int m = 0;
        for (int j = lo; j < hi; j++)
            if (in_T[j]) { dT[m] = d[j]; rT[m] = rhs[j]; map[m] = j; m++; }
        *count = m;
    }
    __syncthreads();
    return *count;
}

// The header of a solved instance and the per-instance outputs, by thread 0, after the CTA has written the rule's arrays.
// `check_flag` / `check_before`: the bounds-checked build's per-CTA flag and what the streaming kernel reported for
// the row (nullptr / 0 otherwise): a skipped access turns the status into GR_CHECK_FAILED.
__device__ inline void write_rule_header(const ParamView& pv, const PrepResult& pr, int n, int status, double gnorm,
                                         int iters, float* alpha_out, int* status_out, long long b,
                                         const int* check_flag, int check_before)
{
    if (threadIdx.x == 0) {
        if (check_before || (check_flag && *check_flag)) status = GR_CHECK_FAILED;
        Header* h = pv.h;
        h->n = n; h->k = pr.k; h->jstar = pr.jstar; h->nblocks = pr.nblocks; h->status = status;
        h->alpha_star = pr.alpha_star;
        h->resid_total = 1.0 - pr.alpha_star;
        h->gnorm = gnorm; h->iters = iters;
        h->magic = kMagic;
        alpha_out[b] = (float)pr.alpha_star;
        status_out[b] = status == kNeedFallback ? GR_NOT_CONVERGED : status;
    }
}

// Rule arrays (except w, which the solvers write as they go) and the header.
__device__ inline void write_rule(const PrepSm& sm, const ParamView& pv, int KP, const PrepResult& pr, int n,
                                  int status, double gnorm, int iters, float* alpha_out, int* status_out, long long b,
                                  const int* check_flag = nullptr, int check_before = 0)
{
    const int tid = threadIdx.x;
    for (int j = tid; j < KP; j += blockDim.x) {
        const bool in = j < pr.k;
        pv.id[j] = in ? sm.id[j] : -1;
        pv.blk[j] = in ? sm.blk[j] : -2;
        pv.r[j] = in ? sm.r[j] : 0.0;
        pv.p[j] = in ? sm.p[j] : 0.0;
        if (!in) pv.w[j] = 0.0;
    }
    __syncthreads();
    write_rule_header(pv, pr, n, status, gnorm, iters, alpha_out, status_out, b, check_flag, check_before);
}

}  // namespace gr
