// Slice of the transport for the drafted tuple and the accept / resample draw
// (Eq. "cases", Eq. "approx-c", "normalized" in Algorithm 1; App. A steps 3-4), as CTA-level
// device code: one CTA serves one instance.  Used by the stand-alone verify kernel and by the
// solve kernels when they are given the drafted tokens (fused solve + verify).
#pragma once
#include "gr_common.cuh"

namespace gr {

// What a solve kernel needs to finish an instance with its draw; draft == nullptr: not fused.
struct FusedArgs {
    const int* draft;          // [batch, n]
    const float* uni;          // [batch, 2]
    int* out_token;            // [batch]
    unsigned char* out_acc;    // [batch]
    int* vstatus;              // [batch]
};

// Shared-memory scratch of one verifying CTA.
struct VerifyScratch {
    GR_PTR(double) res;        // residuals of one chunk of the target row, in id order
    GR_PTR(double) p;          // support: flow,
    GR_PTR(double) red;        // one double per warp; [32]: mass before the selected chunk
    GR_PTR(int) id;            // id,
    GR_PTR(int) chunk;         // chunk of the target row that holds it
    GR_PTR(int) tok;           // drafted tokens and their positions in the ratio order
    GR_PTR(int) pos;
    GR_PTR(int) dec;           // token, accepted, status, whether to resample; two search results
    int* flag;                 // bounds-checked build: where skipped accesses are reported
};
constexpr int kChunkSpan = kChunk + 8;           // longest chunk: the first one also holds the row's unaligned head
constexpr int kVerifyScratchBytes = (kChunkSpan + kMaxSupport + 34) * 8 + (2 * kMaxSupport + 2 * kMaxDrafts + 8) * 4;
// base: 8-byte aligned, kVerifyScratchBytes long
__device__ inline VerifyScratch verify_scratch(void* base, int* flag = nullptr) {
    VerifyScratch v;
    double* d = reinterpret_cast<double*>(base);
    v.res = GR_MKPTR(double, d, kChunkSpan, flag); d += kChunkSpan;
    v.p = GR_MKPTR(double, d, kMaxSupport, flag); d += kMaxSupport;
    v.red = GR_MKPTR(double, d, 34, flag); d += 34;
    int* t = reinterpret_cast<int*>(d);
    v.id = GR_MKPTR(int, t, kMaxSupport, flag); t += kMaxSupport;
    v.chunk = GR_MKPTR(int, t, kMaxSupport, flag); t += kMaxSupport;
    v.tok = GR_MKPTR(int, t, kMaxDrafts, flag); t += kMaxDrafts;
    v.pos = GR_MKPTR(int, t, kMaxDrafts, flag); t += kMaxDrafts;
    v.dec = GR_MKPTR(int, t, 8, flag);
    v.flag = flag;
    return v;
}

__device__ __forceinline__ double warp_sum(double v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}
__device__ __forceinline__ double warp_incl_scan(double v, int lane) {
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        double t = __shfl_up_sync(0xffffffffu, v, o);
        if (lane >= o) v += t;
    }
    return v;
}
// Inclusive prefix over the CTA's threads, *total gets the sum.  (One barrier before the slots may be reused.)
static __device__ __noinline__ double block_incl_scan(double v, GR_PTR(double) red, double* total)
{
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
    v = warp_incl_scan(v, lane);
    __syncthreads();
    if (lane == 31) red[warp] = v;
    __syncthreads();
    double off = 0.0, tot = 0.0;
#pragma unroll 1
    for (int w = 0; w < nw; w++) { const double t = red[w]; if (w < warp) off += t; tot += t; }
    *total = tot;
    return v + off;
}

// Inverse CDF of the resample distribution in ascending id order at `frac` of its total, by the whole CTA.
// Residual of id i: the outer residual r_i on support ids (0 on H*), tgt_i elsewhere.
// Two levels: per-chunk masses from the scan kernel's table minus the flow p_i of the support ids in the chunk (one
// chunk per thread), then an exact fp64 pass over the one chunk selected (its residuals in shared memory, a run of
// consecutive ids per thread).  Bound by the latency of three dependent reads; with one warp per instance the two
// passes took 25 us.
// Only an id of positive residual is ever returned.  A chunk's mass comes from fp32 sums: where all its ids are in H* or
// masked, a rounding error of theirs can be left and select it; the nearest chunk that does hold some residual then stands
// in for it (the next one up, at its first id; if there is none, the next one down, at its last).
__device__ inline int resample_draw(const Header* h, const ParamView& pv, int k, double frac, const VerifyScratch& vs)
{
    const int tid = threadIdx.x, bd = blockDim.x;
    const int nch = h->nch, head = h->head, V = h->V, dtype = h->dtype;
    const double rT = m_div(1.0, (double)h->temp_target), lse = h->lse_t;
    const void* row = h->q_row;
    // the total residual mass is known in closed form (1 - alpha*, or 1 when the target itself is sampled)
    double thr = frac * (k > 0 ? h->resid_total : 1.0);
    int lo = 0, hi = nch, origin = -1;          // chunks looked at; the one that was selected in vain
#pragma unroll 1
    while (true) {
        if (tid == 0) { vs.dec[4] = 0x7fffffff; vs.dec[5] = -1; }
        double run = 0.0;
        int sel = 0x7fffffff;
#pragma unroll 1
        for (int c0 = 0; c0 < hi; c0 += bd) {
            const int c = c0 + tid;
            const bool in = c >= lo && c < hi;
            // flows of the support ids per chunk, as integers (2^-62 units: the sums do not depend on the order of the atomics)
            GR_PTR(unsigned long long) sub = GR_PCAST(unsigned long long, vs.res);
            sub[tid] = 0ull;
            __syncthreads();
            for (int j = tid; j < k; j += bd) {
                const int at = vs.chunk[j] - c0;
                if (at >= 0 && at < bd) atomicAdd(&sub[at], (unsigned long long)__double2ll_rn(vs.p[j] * 4611686018427387904.0));
            }
            double R = 0.0;
            if (in) {
                const float2 ms = pv.chunk[c];
                R = (double)ms.y * m_exp((double)ms.x * rT - lse);
            }
            __syncthreads();
            if (in) R = fmax(R - (double)(long long)sub[tid] * (1.0 / 4611686018427387904.0), 0.0);
            double tot;
            const double inc = block_incl_scan(R, vs.red, &tot) + run;
            if (R > 0.0 && inc > thr) atomicMin(&vs.dec[4], c);
            if (R > 0.0) atomicMax(&vs.dec[5], c);
            __syncthreads();
            sel = vs.dec[4];
            if (sel == c) vs.red[32] = inc - R;
            run += tot;
            if (sel != 0x7fffffff) break;
        }
        __syncthreads();
        double want = 1.0e300;                      // (rounding left the threshold above the total: the last id of positive mass)
        if (sel != 0x7fffffff) want = thr - vs.red[32];
        else sel = vs.dec[5];
        int found = 0x7fffffff, last = -1, cb = 0;
        if (sel >= 0) {
            // ---- exact pass over the chunk in id order
            cb = chunk_begin(sel, head);
            const int len = chunk_end(sel, head, nch, V) - cb;
            // (four loads in flight: they come from HBM)
#pragma unroll 1
            for (int e0 = tid; e0 < len; e0 += 4 * bd) {
                float x[4];
#pragma unroll
                for (int u = 0; u < 4; u++) {
                    const int e = min(e0 + u * bd, len - 1);
                    x[u] = dtype == GR_BF16 ? __bfloat162float(((const __nv_bfloat16*)row)[cb + e]) : __ldg((const float*)row + cb + e);
                }
#pragma unroll
                for (int u = 0; u < 4; u++) {
                    if (e0 + u * bd >= len) break;
                    vs.res[e0 + u * bd] = exp_neg(lse - (double)x[u] * rT);
                }
            }
            __syncthreads();
            for (int j = tid; j < k; j += bd) if (vs.chunk[j] == sel) vs.res[vs.id[j] - cb] = pv.r[j];
            if (tid == 0) { vs.dec[4] = 0x7fffffff; vs.dec[5] = -1; }
            __syncthreads();
            const int per = ((len + bd - 1) / bd) | 1;              // (odd: no bank conflicts)
            const int e0 = min(tid * per, len), e1 = min(e0 + per, len);
            double sum = 0.0;
            int lastp = -1;
#pragma unroll 4
            for (int e = e0; e < e1; e++) { const double r = vs.res[e]; sum += r; if (r > 0.0) lastp = e; }
            double tot;
            const double inc = block_incl_scan(sum, vs.red, &tot);
            double acc = inc - sum;
            int hit = -1;
            if (lastp >= 0 && inc > want) {
                hit = lastp;                        // (the run's sum and its walk round differently)
#pragma unroll 4
                for (int e = e0; e < lastp; e++) { const double r = vs.res[e]; acc += r; if (hit == lastp && r > 0.0 && acc > want) hit = e; }
            }
            if (hit >= 0) atomicMin(&vs.dec[4], hit);
            if (lastp >= 0) atomicMax(&vs.dec[5], lastp);
            __syncthreads();
            found = vs.dec[4]; last = vs.dec[5];
        }
        if (found != 0x7fffffff) return cb + found;
        if (last >= 0) return cb + last;
        // nothing there: the chunks above the one selected, then those below
        if (thr > 1.0e299) { if (sel < 0) return -1; hi = sel; }
        else {
            if (origin < 0) origin = sel < 0 ? 0 : sel;
            lo = sel + 1; thr = 0.0;
            if (sel < 0 || lo >= nch) { lo = 0; hi = origin; thr = 1.0e300; }
        }
        __syncthreads();
    }
}

// One lane's share of the slice pi(.|omega) (Eq. "cases", Eq. "approx-c", "normalized" in Algorithm 1): lane s < n
// holds drafted token s.  uniq: first occurrence of its token; pi: its probability (0 for repeats and for tokens
// outside the serving system); inner: every drafted token lies in H*; rho: mass of the resample segment.
struct SliceLane { bool uniq, inner; double pi, rho; };

// Slice of a solved instance (k > 0) for the drafted tuple, one warp; `pos` is the position of this lane's drafted token in
// the ratio order (lanes >= n: any).  Returns GR_OK, or GR_DRAFT_OUT_OF_SUPPORT when a drafted token is not in the support.
__device__ inline int slice_instance(const Header* h, const ParamView& pv, int pos, int lane, SliceLane& sl)
{
    const int n = h->n, jstar = h->jstar;
    sl.uniq = false; sl.inner = false; sl.pi = 0.0; sl.rho = 0.0;
    const bool missing = __any_sync(0xffffffffu, lane < n && pos < 0);
    if (missing) return GR_DRAFT_OUT_OF_SUPPORT;
    // distinct tokens in order of first occurrence; the lowest-ratio position met
    const unsigned same = __match_any_sync(0xffffffffu, lane < n ? pos : -1 - lane);
    const bool uniq = lane < n && __ffs(same) - 1 == lane;
    const int maxpos = __reduce_max_sync(0xffffffffu, lane < n ? pos : -1);
    const bool inner = maxpos < jstar;
    double wv = 0.0;
    bool served = false;
    if (uniq) {
        served = inner || pv.blk[pos] == pv.blk[maxpos];
        if (served) wv = pv.w[pos];
    }
    const double W = warp_sum(wv) + (inner ? 1.0 : 0.0);
    sl.uniq = uniq; sl.inner = inner;
    if (W > 0.0) {
        sl.pi = wv / W;
    } else {
        // (truncated variant) every served token carries weight 0: they share the tuple equally
        const int cnt = __popc(__ballot_sync(0xffffffffu, served));
        sl.pi = served ? 1.0 / (double)cnt : 0.0;
    }
    sl.rho = inner ? 1.0 / W : 0.0;
    return GR_OK;
}

// Support and drafted tokens into the scratch, and where each drafted token sits in the ratio order (-1: nowhere).
__device__ inline void locate_drafts(const Header* h, const ParamView& pv, const int* draft_row, const VerifyScratch& vs)
{
    const int tid = threadIdx.x, bd = blockDim.x, k = h->k, n = h->n, nch = h->nch, head = h->head;
    if (tid < kMaxDrafts) { vs.tok[tid] = tid < n ? draft_row[tid] : -1; vs.pos[tid] = -1; }
    for (int j = tid; j < k; j += bd) {
        const int id = pv.id[j];
        vs.id[j] = id; vs.p[j] = pv.p[j]; vs.chunk[j] = chunk_of(id, head, nch);
    }
    __syncthreads();
    for (int j = tid; j < k; j += bd) {
        const int id = vs.id[j];
#pragma unroll 4
        for (int s = 0; s < n; s++) if (vs.tok[s] == id) vs.pos[s] = j;
    }
    __syncthreads();
}

// The whole verification of one instance by one CTA (at least two warps).  `h` is the instance's header (already checked
// to carry the magic number); a rule marked partial is accepted only from the kernel that solved it for these drafts.
// Every thread gets the result.
__device__ inline void verify_instance(const Header* h, const int* draft_row, const float* uni_row, const VerifyScratch& vs,
                                       bool allow_partial, int& token, int& accepted, int& status)
{
    const int lane = threadIdx.x & 31;
    token = -1; accepted = 0;
    status = h->status;
    if (status == GR_BAD_LOGITS) return;
    if (status == GR_PARTIAL_RULE) {
        if (!allow_partial) return;
        status = GR_OK;
    }
    ParamView pv = view_params((void*)h, h->kcap, h->V, vs.flag);
    const int k = h->k;
    const double u0 = (double)uni_row[0], u1 = (double)uni_row[1];
    locate_drafts(h, pv, draft_row, vs);
    if (k == 0) {
        // no rule was solved: emit a sample of the target distribution itself
        token = resample_draw(h, pv, 0, u1, vs);
        if (token >= 0) {
            for (int s = 0; s < h->n; s++) if (vs.tok[s] == token) accepted = 1;
        }
        return;
    }
    if (threadIdx.x < 32) {
        const int tok = vs.tok[lane];
        SliceLane sl;
        int tk = -1, ac = 0, again = 0;
        const int st = slice_instance(h, pv, vs.pos[lane], lane, sl);
        if (st == GR_OK) {
            const double cum = warp_incl_scan(sl.pi, lane);
            const unsigned hit = __ballot_sync(0xffffffffu, sl.uniq && sl.pi > 0.0 && cum > u0);
            const unsigned posm = __ballot_sync(0xffffffffu, sl.uniq && sl.pi > 0.0);
            if (hit || !sl.inner) {
                tk = __shfl_sync(0xffffffffu, tok, hit ? __ffs(hit) - 1 : 31 - __clz(posm));
                ac = 1;
            } else {
                again = 1;
            }
        }
        if (lane == 0) { vs.dec[0] = tk; vs.dec[1] = ac; vs.dec[2] = st; vs.dec[3] = again; }
    }
    __syncthreads();
    if (vs.dec[2] != GR_OK) { status = vs.dec[2]; return; }
    token = vs.dec[0]; accepted = vs.dec[1];
    if (vs.dec[3]) token = resample_draw(h, pv, k, u1, vs);
}

// Which system the drafted tuple selects (Eq. "cases"): -1 the inner system (every drafted token in H*), b >= 0 the
// outer block b (the lowest-ratio block met), -2 when a drafted token is outside the support (then every system is
// solved and the draw reports the error).  Every thread of the CTA calls it; id / blk are in ratio order.
__device__ inline int selected_system(const int* draft_row, int n, int k, int jstar, GR_PTR(const int) sid,
                                      GR_PTR(const int) sblk, int* s_sel)
{
    const int tid = threadIdx.x;
    if (tid == 0) *s_sel = -1;
    __syncthreads();
    int missing = 0;
    if (tid < n) {
        const int t = draft_row[tid];
        int pos = -1;
        for (int j = 0; j < k; j++) if (sid[j] == t) pos = j;
        if (pos < 0) missing = 1; else atomicMax(s_sel, pos);
    }
    missing = __syncthreads_or(missing);
    const int maxpos = *s_sel;
    __syncthreads();
    if (missing || maxpos < 0) return -2;
    return maxpos < jstar ? -1 : sblk[maxpos];
}

// Draw of instance b by a solve kernel's CTA, after the rule (or the no-rule header) was written and the CTA synchronised.
static __device__ __noinline__ void fused_draw(const FusedArgs& fa, const Header* h, long long b, int n, void* scratch,
                                               int* check_flag = nullptr)
{
    int token, accepted, status;
    verify_instance(h, fa.draft + (size_t)b * n, fa.uni + 2 * (size_t)b, verify_scratch(scratch, check_flag), true, token,
                    accepted, status);
    if (check_flag && *check_flag) status = GR_CHECK_FAILED;
    if (threadIdx.x == 0) {
        fa.out_token[b] = token;
        fa.out_acc[b] = (unsigned char)accepted;
        fa.vstatus[b] = status;
    }
}

}  // namespace gr
