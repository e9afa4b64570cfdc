// Optimal acceptance for an untruncated draft on a large vocabulary (support = V > GR_MAX_SUPPORT).
//
// The rule itself is not solved there (status GR_SUPPORT_TOO_LARGE), but alpha* = 1 + min_H psi(H) only needs
// the ratio order of the whole vocabulary and a prefix scan (Eq. "subset-select", Sec. 5.1):
// psi_j = Tg_j - Dr_j^n over the prefixes of the order by descending draft / target ratio.
//
// bucket_alpha_kernel finds that minimum without sorting the row: the log-ratio keys are binned into 4096 equal
// buckets (a monotone map, so the bucket order is the ratio order), the bucket masses give psi exactly at every
// bucket boundary, and a lower bound on psi inside a bucket (the ratios inside it span one bucket width) leaves
// only the few buckets next to the minimum to be ordered exactly, in shared memory.  One pass over the row (its maxima and
// the range of the keys come from the streaming pass) and one over the 2-byte bucket numbers it leaves behind.
// A row whose candidate buckets do not fit is handed to fullsort_alpha_kernel: one CTA per instance sorts (key, id)
// pairs of the row in global scratch with a bitonic network, then scans tgt and drf along the order.
// The network's passes with a compare distance below the tile size (4096 pairs, 48 KB) run on tiles staged in
// shared memory: 15 trips through global memory for a 65536-entry row instead of 136.
#include "gr_prep.cuh"

namespace gr {

constexpr int kFsThreads = 1024;
constexpr int kFsTile = 4096;          // pairs per shared-memory tile
constexpr int kFsSmemBytes = kFsTile * 12;

__host__ __device__ inline int next_pow2(int v) { int p = 1; while (p < v) p <<= 1; return p; }
__host__ size_t fullsort_scratch_bytes(int V) { return (size_t)next_pow2(V) * 12; }

// order-preserving map double -> uint64 (larger double, larger key)
__device__ inline unsigned long long dkey(double x) {
    unsigned long long u = (unsigned long long)__double_as_longlong(x);
    return (u >> 63) ? ~u : (u | 0x8000000000000000ull);
}
// true when (ka, ia) comes before (kb, ib): larger key first, equal keys by smaller id
__device__ inline bool before(unsigned long long ka, int ia, unsigned long long kb, int ib) {
    return ka > kb || (ka == kb && ia < ib);
}

constexpr int kBkThreads = 1024;
constexpr int kBkBuckets = 4096;
constexpr int kBkPer = kBkBuckets / kBkThreads;   // buckets per thread in the scan over buckets
constexpr int kBkMaxCand = 4096;                  // elements of candidate buckets held in shared memory
constexpr int kBkFew = 128;                       // up to so many are taken without ordering them
constexpr int kBkTab = 128, kBkCopies = 16;       // 2^(42 + j / 128), a copy for every lane of a half-warp
constexpr int kBkSmemBytes = kBkBuckets * (4 * 4 + 4 + 4) + kBkMaxCand * (8 + 4 + 4 + 4 + 4) + kBkTab * kBkCopies * 8;

// exp(-y) in units of 2^-42, rounded to an integer (masses are summed as integers: exact, order-free).  y >= 0, up to infinity.
// 2^(k/128) from a table times a degree-4 Taylor polynomial on |r| <= ln2/256 (1.2e-15 relative, a hundredth of the unit; degree 5 and 32
// entries took two operations more), scaled and rounded by one multiplication and addition: nine fp64 operations.
__device__ __forceinline__ unsigned long long mass_fixed(double y, GR_PTR(const double) tab)
{
    constexpr double ln2 = 0.6931471805599453, magic = 6755399441055744.0;         // 1.5 * 2^52
    y = __hiloint2double(min(__double2hiint(y), 0x40468000), __double2loint(y));   // (at 45 and beyond it rounds to nothing)
    const double m = fma(y, -kBkTab / ln2, magic);
    const int k = __double2loint(m);
    const double r = fma(magic - m, ln2 / kBkTab, -y);
    double p = fma(r, 4.1666666666666664e-02, 1.6666666666666666e-01);
    p = fma(r, p, 0.5);
    p = fma(r, p, 1.0);
    p = fma(r, p, 1.0);
    const double s = tab[(k & (kBkTab - 1)) * kBkCopies];                      // (tab: this lane's copy)
    const double u = fma(p, __hiloint2double(__double2hiint(s) + (k & ~(kBkTab - 1)) * ((1 << 20) / kBkTab), __double2loint(s)), 4503599627370496.0);   // 2^52
    return (unsigned long long)__double_as_longlong(u) - 0x4330000000000000ull;
}

// 64-bit sum in shared memory out of native 32-bit atomics: the carry out of the low word is rare
__device__ __forceinline__ void add_mass(GR_PTR(unsigned) lo, GR_PTR(unsigned) hi, int c, unsigned long long v)
{
    const unsigned l = (unsigned)v, old = atomicAdd(&lo[c], l);
    const unsigned h = (unsigned)(v >> 32) + (old + l < l ? 1u : 0u);
    if (h != 0u) atomicAdd(&hi[c], h);
}

// Draft counts of one call: everything but the last step is common to them.
struct NList { int count; int n[GR_MAX_ALPHA_N]; };

// x^n by squaring
__device__ __forceinline__ double power(double x, int n)
{
    double r = 1.0;
    for (; n > 0; n >>= 1) { if (n & 1) r *= x; x *= x; }
    return r;
}

// Exclusive prefixes over the CTA of two 64-bit integers per thread, in place; total gets the sums.  s_w: two slots per warp (32 of them).
__device__ inline void block_exscan_u64(unsigned long long* v, unsigned long long* s_w, unsigned long long* total)
{
    static_assert(kBkThreads == 1024, "one slot per lane");
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    auto warp_scan = [&](unsigned long long* x) {
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const unsigned long long t0 = __shfl_up_sync(0xffffffffu, x[0], o), t1 = __shfl_up_sync(0xffffffffu, x[1], o);
            if (lane >= o) { x[0] += t0; x[1] += t1; }
        }
    };
    unsigned long long inc[2] = {v[0], v[1]};
    warp_scan(inc);
    if (lane == 31) { s_w[2 * warp] = inc[0]; s_w[2 * warp + 1] = inc[1]; }
    __syncthreads();
    unsigned long long all[2] = {s_w[2 * lane], s_w[2 * lane + 1]};
    warp_scan(all);
#pragma unroll
    for (int k = 0; k < 2; k++) {
        const unsigned long long off = __shfl_sync(0xffffffffu, all[k], (warp + 31) & 31);
        total[k] = __shfl_sync(0xffffffffu, all[k], 31);
        v[k] = (warp > 0 ? off : 0ull) + inc[k] - v[k];
    }
}
// Minimum over the CTA, for every thread (s_r: a slot per warp; a barrier before its next use is the caller's).
__device__ inline double block_min(double v, double* s_r)
{
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v = fmin(v, __shfl_xor_sync(0xffffffffu, v, o));
    if ((threadIdx.x & 31) == 0) s_r[threadIdx.x >> 5] = v;
    __syncthreads();
    v = s_r[threadIdx.x & 31];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v = fmin(v, __shfl_xor_sync(0xffffffffu, v, o));
    return v;
}

// flag[0] of the instance's scratch region: bit j set when fullsort_alpha_kernel has to do the row for the j-th draft count.
// With a params block and `rule_status` it also writes the header of a row without a rule (nl.n[0] drafts).
// 512 rows of 50257 in fp32: the call 202 us, 222 before (bucket numbers and masses out of scaled logits formed first, a polynomial of degree 5, every thread
// its own quotients and exponentials, candidates ordered in three rounds); 201 with exponents out of products rounded first, which fail for logits of 1e17 and more.  A row takes 71 k cycles, one to an SM: 46 k its masses (instruction
// issue: 116 instructions per 32 ids in all, fp64 25 of them), 4 k sums, 5 k bounds, 6 k numbers read back, 6 k candidates; the 206 MB it reads are a fifth of the time.
template <typename T>
__global__ void __launch_bounds__(kBkThreads)
bucket_alpha_kernel(const T* __restrict__ q, const T* __restrict__ p, int V, const __grid_constant__ NList nl, double rt, double rd,
                    const char* __restrict__ ws, char* __restrict__ scratch, size_t scratch_stride,
                    char* __restrict__ params, int pstride, int force_sort, float* __restrict__ alpha_out,
                    int* __restrict__ status_out, int* __restrict__ rule_status)
{
    extern __shared__ __align__(16) unsigned char bk_smem[];
    pdl_wait();
    GR_CHECK_FLAG_DECL;
    GR_CHECK_FLAG_INIT;
    double* const ckey_raw = reinterpret_cast<double*>(bk_smem);
    double* const tab_raw = ckey_raw + kBkMaxCand;
    unsigned* const w_raw = reinterpret_cast<unsigned*>(tab_raw + kBkTab * kBkCopies);
    int* const i_raw = reinterpret_cast<int*>(w_raw + 4 * kBkBuckets);
    GR_PTR(double) ckey = GR_MKPTR(double, ckey_raw, kBkMaxCand, GR_CHECK_FLAG);    // candidate elements: key,
    GR_PTR(double) tab_all = GR_MKPTR(double, tab_raw, kBkTab * kBkCopies, GR_CHECK_FLAG);
    GR_PTR(const double) tab = tab_all + (threadIdx.x & (kBkCopies - 1));
    // target and draft mass of a bucket, then the exclusive prefix (low and high words)
    GR_PTR(unsigned) tl = GR_MKPTR(unsigned, w_raw, kBkBuckets, GR_CHECK_FLAG), th = GR_MKPTR(unsigned, w_raw + kBkBuckets, kBkBuckets, GR_CHECK_FLAG);
    GR_PTR(unsigned) dl = GR_MKPTR(unsigned, w_raw + 2 * kBkBuckets, kBkBuckets, GR_CHECK_FLAG), dh = GR_MKPTR(unsigned, w_raw + 3 * kBkBuckets, kBkBuckets, GR_CHECK_FLAG);
    GR_PTR(int) cnt = GR_MKPTR(int, i_raw, kBkBuckets, GR_CHECK_FLAG);              // elements of a candidate bucket / fill cursor
    GR_PTR(int) seg = GR_MKPTR(int, i_raw + kBkBuckets, kBkBuckets, GR_CHECK_FLAG); // start of a candidate's segment; -1: none
    GR_PTR(int) cid = GR_MKPTR(int, i_raw + 2 * kBkBuckets, kBkMaxCand, GR_CHECK_FLAG);                      // id,
    GR_PTR(int) sid = GR_MKPTR(int, i_raw + 2 * kBkBuckets + kBkMaxCand, kBkMaxCand, GR_CHECK_FLAG);         // ids in order,
    GR_PTR(int) lid = GR_MKPTR(int, i_raw + 2 * kBkBuckets + 2 * kBkMaxCand, kBkMaxCand, GR_CHECK_FLAG);     // ids and
    GR_PTR(int) lbk = GR_MKPTR(int, i_raw + 2 * kBkBuckets + 3 * kBkMaxCand, kBkMaxCand, GR_CHECK_FLAG);     // buckets as found
    __shared__ double s_r[kBkThreads / 32], s_c[6], s_up[32], s_at[32];      // s_c: bucket width, scales; s_at[warp] s_up[lane]: bounds on the ratios
    __shared__ unsigned long long s_w[2 * kBkThreads / 32];
    __shared__ int s_nelem, s_found, s_fallback, s_lo, s_hi;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const long long b = blockIdx.x;
    const char* const rec = ws + (size_t)b * ws_stride();
    const WsHeader* wh = reinterpret_cast<const WsHeader*>(rec);
    // (no params block and a status array when called for the optimal acceptance alone)
    Header* hdr = params ? reinterpret_cast<Header*>(params + (size_t)b * pstride) : nullptr;
    char* const scr = scratch + (size_t)b * scratch_stride;
    int* flag = reinterpret_cast<int*>(scr);
    if (tid == 0 && status_out) status_out[b] = wh->bad != 0 ? GR_BAD_LOGITS : GR_OK;
    if (tid == 0 && rule_status) write_no_rule(hdr, nl.n[0], wh->bad != 0, alpha_out, rule_status, b);
    if (wh->bad != 0 || force_sort) {
        if (tid == 0) {
            flag[0] = (1 << nl.count) - 1;          // (a bad row returns at once there too)
            if (wh->bad != 0 && status_out)
                for (int j = 0; j < nl.count; j++) alpha_out[(size_t)b * nl.count + j] = nanf("");
        }
        return;
    }
    const T* qrow = q + (size_t)b * V;
    const T* prow = p + (size_t)b * V;
    const FullRow fr = *reinterpret_cast<const FullRow*>(rec + sizeof(WsHeader));
    // Exponents: a logit's distance from its row's maximum, times the reciprocal temperature (a rounding or two from the quotients the sort
    // uses, which moves alpha* by ~1e-16).  The subtraction comes first: zero for the maximum and never negative, however large the logits are.
    // (One operation less as m - a rt with m rounded, but what m loses, 2^-53 of it, is then every exponent's error: from logits of 1e17
    // on the maximum itself had no mass.)
    const double qm = (double)fr.qmax, pm = (double)fr.pmax;
    auto exp_t = [&](float x) { return __dmul_rn(qm - (double)x, rt); };
    auto exp_d = [&](float v) { return __dmul_rn(pm - (double)v, rd); };
    // The keys here are the log-ratios draft / target less those of the rows' maxima, exp_t - exp_d: nothing of them is lost to what a row's
    // logits have in common.  Bucket of a key: floor((kmax - key) * invw), clamped, one fused operation on the key and so a non-increasing function of
    // it in floating point too.  The streaming pass's kmax and kmin are fp32 values, and keys that overflow fp32 are not among
    // them: a key may lie outside (in the first or the last bucket; the bounds below hold for any kmax and width), and without a usable range there
    // is one bucket.
    const double ln2 = 0.6931471805599453;
    const double span = ((double)fr.kmax - (double)fr.kmin) * ln2;
    const bool ranged = span > 0.0 && span < INFINITY;
    const double kmax = ranged ? (double)fr.kmax * ln2 - (pm * rd - qm * rt) : 0.0;
    // (what every thread needs the same is formed by one: a quotient by 1024 threads keeps the fp64 units busy for 700 cycles)
    if (tid == 0) s_c[0] = ranged ? (double)kBkBuckets / (span * (1.0 + 1e-9)) : 0.0;
    // (masses and counts lie behind one another)
    static_assert(5 * kBkBuckets % (4 * kBkThreads) == 0 && kBkBuckets == 4 * kBkThreads && kBkTab <= kBkThreads, "a vector per thread");
#pragma unroll
    for (int u = 0; u < 5 * kBkBuckets / (4 * kBkThreads); u++) reinterpret_cast<uint4*>(w_raw)[tid + u * kBkThreads] = make_uint4(0u, 0u, 0u, 0u);
    reinterpret_cast<int4*>(i_raw + kBkBuckets)[tid] = make_int4(-1, -1, -1, -1);
    if (tid < kBkTab) {
        const double v = exp2(42.0 + (double)tid / kBkTab);
#pragma unroll
        for (int c = 0; c < kBkCopies; c++) tab_all[tid * kBkCopies + ((c + tid) & (kBkCopies - 1))] = v;
    }
    if (tid == 0) { s_nelem = 0; s_found = 0; s_fallback = 0; s_lo = kBkBuckets; s_hi = -1; }
    __syncthreads();
    const double invw = s_c[0];
    // ---- the row: bucket masses (integers: the sums do not depend on the order of the atomics), bucket numbers to scratch
    // (number of id i at code[i + shift], so that a vector of logits has its numbers in one aligned store)
    constexpr int N = 16 / (int)sizeof(T);
    const int head = row_head(q, b, V, (int)sizeof(T)), shift = (N - head % N) % N;
    unsigned short* const code_raw = reinterpret_cast<unsigned short*>(scr + 16);
    GR_PTR(unsigned short) code = GR_MKPTR(unsigned short, code_raw, V + 16, GR_CHECK_FLAG);
    auto key_of = [&](float x, float v) { return exp_t(x) - exp_d(v); };
    const double c0 = kmax * invw;
    auto element = [&](float x, float v) {
        const double yt = exp_t(x), yd = exp_d(v), t = fma(yt - yd, -invw, c0);
        // (clamped by the leading word, to [0, 4096): the trailing one of a number that the magic constant does not hold says nothing)
        static_assert(kBkBuckets == 4096, "0x40affffe: the last numbers below it");
        const double u = __hiloint2double(min(max(__double2hiint(t), 0), 0x40affffe), __double2loint(t));
        const int c = __double2loint(__dadd_rd(u, 6755399441055744.0));
        add_mass(tl, th, c, mass_fixed(yt, tab));
        add_mass(dl, dh, c, mass_fixed(yd, tab));
        return c;
    };
    const int nvec = (V - head) / N, tail0 = head + nvec * N;
    if (tid < head) code[tid + shift] = (unsigned short)element(load_logit<T>(qrow, tid), load_logit<T>(prow, tid));
    if (tid < V - tail0) code[tail0 + tid + shift] = (unsigned short)element(load_logit<T>(qrow, tail0 + tid), load_logit<T>(prow, tail0 + tid));
    const uint4* const qv = reinterpret_cast<const uint4*>(qrow + head);
    const uint4* const pv = reinterpret_cast<const uint4*>(prow + head);
    uint4 xq = make_uint4(0u, 0u, 0u, 0u), xp = xq;
    if (tid < nvec) { xq = __ldg(qv + tid); xp = __ldg(pv + tid); }
#pragma unroll 1
    for (int e = tid; e < nvec; e += kBkThreads) {
        const uint4 cq = xq, cp = xp;
        if (e + kBkThreads < nvec) { xq = __ldg(qv + e + kBkThreads); xp = __ldg(pv + e + kBkThreads); }
        const unsigned wq[4] = {cq.x, cq.y, cq.z, cq.w}, wp[4] = {cp.x, cp.y, cp.z, cp.w};
        unsigned out[N / 2];
#pragma unroll
        for (int z = 0; z < N; z += 2) {
            float x0, x1, v0, v1;
            if (N == 4) {
                x0 = __uint_as_float(wq[z & 3]); x1 = __uint_as_float(wq[(z + 1) & 3]);
                v0 = __uint_as_float(wp[z & 3]); v1 = __uint_as_float(wp[(z + 1) & 3]);
            } else {
                x0 = __uint_as_float(wq[z / 2] << 16); x1 = __uint_as_float(wq[z / 2] & 0xffff0000u);
                v0 = __uint_as_float(wp[z / 2] << 16); v1 = __uint_as_float(wp[z / 2] & 0xffff0000u);
            }
            const int c0 = element(x0, v0), c1 = element(x1, v1);
            out[z / 2] = (unsigned)c0 | ((unsigned)c1 << 16);
        }
        const int at = head + e * N + shift;                       // a multiple of N; at + N <= V + N
#ifdef GR_CHECK
        if (at < 0 || at + N > V + 16) { s_check_flag = 1; continue; }
#endif
        if (N == 4) *reinterpret_cast<uint2*>(code_raw + at) = make_uint2(out[0], out[1]);
        else *reinterpret_cast<uint4*>(code_raw + at) = make_uint4(out[0], out[1], out[N / 2 - 2], out[N / 2 - 1]);
    }
    __syncthreads();
    // ---- prefixes over the buckets, psi at every boundary, lower bound inside every bucket
    // (a thread's four buckets lie in one vector of each table)
    static_assert(kBkPer == 4, "a vector per thread");
    auto join = [](unsigned l, unsigned h) { return ((unsigned long long)h << 32) | l; };
    unsigned long long totT, totD;
    {
        const uint4 tv = ld_u4(tl + 4 * tid), tw = ld_u4(th + 4 * tid), dv = ld_u4(dl + 4 * tid), dw = ld_u4(dh + 4 * tid);
        const unsigned long long mT[4] = {join(tv.x, tw.x), join(tv.y, tw.y), join(tv.z, tw.z), join(tv.w, tw.w)};
        const unsigned long long mD[4] = {join(dv.x, dw.x), join(dv.y, dw.y), join(dv.z, dw.z), join(dv.w, dw.w)};
        unsigned long long s[2] = {(mT[0] + mT[1]) + (mT[2] + mT[3]), (mD[0] + mD[1]) + (mD[2] + mD[3])}, tot[2];
        block_exscan_u64(s, s_w, tot);
        totT = tot[0]; totD = tot[1];
        auto put = [&](GR_PTR(unsigned) l, GR_PTR(unsigned) h, unsigned long long x, const unsigned long long* m) {
            const unsigned long long y = x + m[0], z = y + m[1], w = z + m[2];
            st_u4(l + 4 * tid, make_uint4((unsigned)x, (unsigned)y, (unsigned)z, (unsigned)w));
            st_u4(h + 4 * tid, make_uint4((unsigned)(x >> 32), (unsigned)(y >> 32), (unsigned)(z >> 32), (unsigned)(w >> 32)));
        };
        put(tl, th, s[0], mT);
        put(dl, dh, s[1], mD);
    }
    // tgt_i / drf_i = exp(-key_i) * rscale.  Every ratio of bucket c is at least rho: its keys are at most kmax - c w (rho of a thread's first bucket
    // as a product of two numbers, of the others one from the other; where the factors are far from overflowing).  The number of an id is rounded: its
    // key lies at most 2^-53 |kmax| above  kmax - c w (1 - 2^-53).  The 1e-12 taken off the width and the 1e-9 off rho cover that for kmax up to 1e7;
    // beyond, rho is zero unless c w is nearly kmax, which the 1e-12 covers.  (The draft's likeliest id has a key of at least zero: a kmax below, by fp32
    // rounding, leaves every id with draft mass in the first bucket.)
    const double wide = invw > 0.0 ? (1.0 - 1e-12) / invw : 0.0;
    if (warp == 0) s_up[lane] = exp((double)(lane * kBkPer) * fmin(wide, 1.0));
    else if (warp == 1) s_at[lane] = exp((double)(32 * lane * kBkPer) * wide - kmax);
    else if (tid == 64) { s_c[1] = 1.0 / (double)totT; s_c[4] = (double)(V + 1) * s_c[1] + 1e-14; }
    else if (tid == 96) s_c[2] = 1.0 / (double)totD;
    else if (tid == 128) s_c[3] = (double)totD / (double)totT * (1.0 - 1e-9);
    else if (tid == 160) s_c[5] = exp(fmin(wide, 1.0));
    __syncthreads();
    const double iT = s_c[1], iD = s_c[2], rscale = s_c[3], slack = s_c[4], grow = s_c[5];
    const double rho_first = wide <= 1.0 ? s_at[warp] * s_up[lane] * rscale : exp((double)(tid * kBkPer) * wide - kmax) * rscale;
    int todo = 0;                                           // draft counts left to the sort
#pragma unroll 1
    for (int ni = 0; ni < nl.count; ni++) {
    const int n = nl.n[ni];
    double lb[kBkPer], best = 0.0;                          // psi of the empty prefix
    // (the masses are read back as prefixes: holding them in registers across this loop spilled, 10 % of the kernel)
    unsigned long long pT[kBkPer + 1], pD[kBkPer + 1];
    {
        const uint4 tv = ld_u4(tl + 4 * tid), tw = ld_u4(th + 4 * tid), dv = ld_u4(dl + 4 * tid), dw = ld_u4(dh + 4 * tid);
        const bool last = tid == kBkThreads - 1;
        pT[0] = join(tv.x, tw.x); pT[1] = join(tv.y, tw.y); pT[2] = join(tv.z, tw.z); pT[3] = join(tv.w, tw.w);
        pD[0] = join(dv.x, dw.x); pD[1] = join(dv.y, dw.y); pD[2] = join(dv.z, dw.z); pD[3] = join(dv.w, dw.w);
        pT[4] = last ? totT : join(tl[last ? 0 : 4 * tid + 4], th[last ? 0 : 4 * tid + 4]);
        pD[4] = last ? totD : join(dl[last ? 0 : 4 * tid + 4], dh[last ? 0 : 4 * tid + 4]);
    }
    double rho_next = rho_first, T0 = (double)pT[0] * iT, D0 = (double)pD[0] * iD;
    double D1[kBkPer], dn[kBkPer];
    {
        double x[kBkPer];
#pragma unroll
        for (int u = 0; u < kBkPer; u++) { x[u] = D1[u] = (double)pD[u + 1] * iD; dn[u] = 1.0; }
#pragma unroll 1
        for (int e = n; e > 0; e >>= 1) {
#pragma unroll
            for (int u = 0; u < kBkPer; u++) { if (e & 1) dn[u] *= x[u]; x[u] *= x[u]; }
        }
    }
#pragma unroll
    for (int u = 0; u < kBkPer; u++) {
        const int c = tid * kBkPer + u;
        const double T1 = (double)pT[u + 1] * iT;
        const bool empty = pT[u + 1] == pT[u] && pD[u + 1] == pD[u];
        best = fmin(best, T1 - dn[u]);
        // Inside the bucket every ratio tgt / drf is at least rho (its keys are at most kmax - c w; the first bucket has no
        // such limit), so a prefix that ends inside it has  psi >= T0 + rho (D - D0) - D^n,  concave in D: its minimum
        // over [D0, D1] is at an end.  At D0 that is the previous boundary's psi; at D1 it is the bound below.  The slack
        // covers the rounding of the target's masses to integers (one unit per id).  That of the draft's is not in it: it is
        // of the size by which rounding moves psi itself, n half units per id (at most n V 2^-43, 1.8e-7 for 50257 ids and 32
        // drafts).
        const double rho = c == 0 ? 0.0 : rho_next;
        rho_next = wide <= 1.0 ? rho_next * grow : exp((double)(c + 1) * wide - kmax) * rscale;
        lb[u] = empty ? 1.0 : T0 + rho * (D1[u] - D0) - dn[u] - slack;
        T0 = T1; D0 = D1[u];
    }
    best = block_min(best, s_r);
    // ---- candidate buckets: those whose interior could hold a smaller psi
#pragma unroll
    for (int u = 0; u < kBkPer; u++) {
        const int c = tid * kBkPer + u;
        if (lb[u] < best) { seg[c] = 0; atomicMin(&s_lo, c); atomicMax(&s_hi, c); }
    }
    __syncthreads();
    const int lo = s_lo, hi = s_hi;
    // ---- their elements, found by the bucket numbers
    if (hi >= lo) {
        const int ncode = V + shift;
        // (numbers less the first candidate's, two at a time: below `cap` is a candidate's range)
        const unsigned cap = (unsigned)(hi - lo + 1) * 0x10001u, down = ((unsigned)(-lo) & 0xffffu) * 0x10001u;
#pragma unroll 4
        for (int e = tid; e < (ncode + 7) / 8; e += kBkThreads) {
            const uint4 w = *reinterpret_cast<const uint4*>(code_raw + 8 * e);     // (16-byte aligned; within the region)
            const unsigned ww[4] = {w.x, w.y, w.z, w.w};
            const unsigned least = __vminu2(__vminu2(__viaddmin_u16x2(w.x, down, cap), __viaddmin_u16x2(w.y, down, cap)),
                                                 __vminu2(__viaddmin_u16x2(w.z, down, cap), __viaddmin_u16x2(w.w, down, cap)));
            if (least == cap) continue;
#pragma unroll
            for (int z = 0; z < 8; z++) {
                const int c = (int)((ww[z / 2] >> (16 * (z & 1))) & 0xffffu), i = 8 * e + z - shift;
                if (c >= lo && c <= hi && i >= 0 && i < V && seg[c] >= 0) {
                    const int at = atomicAdd(&s_found, 1);
                    if (at < kBkMaxCand) { lid[at] = i; lbk[at] = c; }
                    atomicAdd(&cnt[c], 1);
                }
            }
        }
    }
    __syncthreads();
    const int found = s_found;
    // ---- A few elements (nearly every row: 32 on average of N(0, 3) logits): each one's prefix is summed by a warp, over the elements
    // of its bucket that come before it.  (Segments, ranks and walk, below, are three more rounds to memory: 10 k cycles of 77 k.)
    bool crowded = false;
    if (found <= kBkFew) {
        if (found > 0) {
            GR_PTR(unsigned long long) mt_f = GR_PCAST(unsigned long long, cid), md_f = GR_PCAST(unsigned long long, sid);
            if (tid < found) {
                const int i = lid[tid];
                const float x = load_logit<T>(qrow, i), v = load_logit<T>(prow, i);
                ckey[tid] = key_of(x, v);
                mt_f[tid] = mass_fixed(exp_t(x), tab); md_f[tid] = mass_fixed(exp_d(v), tab);
            }
            __syncthreads();
            for (int e = warp; e < found; e += kBkThreads / 32) {
                const int c = lbk[e], i = lid[e];
                const double ke = ckey[e];
                unsigned long long cT = 0, cD = 0;
                for (int j = lane; j < found; j += 32) {
                    const double kj = ckey[j];
                    if (lbk[j] == c && (kj > ke || (kj == ke && lid[j] <= i))) { cT += mt_f[j]; cD += md_f[j]; }
                }
                __syncwarp();
#pragma unroll
                for (int o = 16; o > 0; o >>= 1) { cT += __shfl_xor_sync(0xffffffffu, cT, o); cD += __shfl_xor_sync(0xffffffffu, cD, o); }
                cT += join(tl[c], th[c]); cD += join(dl[c], dh[c]);
                best = fmin(best, (double)cT * iT - power((double)cD * iD, n));
            }
            // (block_min's slots have been read by all)
            best = block_min(best, s_r);
        }
    } else {
#pragma unroll
        for (int u = 0; u < kBkPer; u++) {
            const int c = tid * kBkPer + u;
            if (seg[c] >= 0) {
                const int L = cnt[c];
                if (found > kBkMaxCand) s_fallback = 1;
                else if (L >= 2) { seg[c] = atomicAdd(&s_nelem, L); cnt[c] = 0; }
                else seg[c] = -1;
            }
        }
        __syncthreads();
        crowded = s_fallback != 0;
        // ---- each bucket into its own segment, ordered by (key descending, id ascending) by counting
        if (!crowded && s_nelem > 0) {
            constexpr int kOwn = kBkMaxCand / kBkThreads;
            int pos[kOwn];
#pragma unroll
            for (int u = 0; u < kOwn; u++) {
                const int e = tid + u * kBkThreads;
                pos[u] = -1;
                if (e < found) {
                    const int c = lbk[e], i = lid[e];
                    if (seg[c] >= 0) {
                        pos[u] = seg[c] + atomicAdd(&cnt[c], 1);
                        ckey[pos[u]] = key_of(load_logit<T>(qrow, i), load_logit<T>(prow, i)); cid[pos[u]] = i;
                    }
                }
            }
            __syncthreads();
#pragma unroll
            for (int u = 0; u < kOwn; u++) {
                if (pos[u] >= 0) {
                    const int c = lbk[tid + u * kBkThreads], off = seg[c], L = cnt[c];
                    const double ke = ckey[pos[u]];
                    const int ie = cid[pos[u]];
                    int rank = 0;
                    for (int j = off; j < off + L; j++) {
                        const double kj = ckey[j];
                        rank += (kj > ke || (kj == ke && cid[j] < ie)) ? 1 : 0;
                    }
                    sid[off + rank] = ie;
                }
            }
            __syncthreads();
        }
        // ---- one warp per candidate bucket walks the prefixes
        if (!crowded && s_nelem > 0) {
            for (int c = lo + warp; c <= hi; c += kBkThreads / 32) {
                const int off = seg[c];
                if (off < 0) continue;
                const int L = cnt[c];
                unsigned long long cT = ((unsigned long long)th[c] << 32) | tl[c], cD = ((unsigned long long)dh[c] << 32) | dl[c];
                for (int base = 0; base < L; base += 32) {
                    unsigned long long tf = 0, df = 0;
                    if (base + lane < L) {
                        const int id = sid[off + base + lane];
                        tf = mass_fixed(exp_t(load_logit<T>(qrow, id)), tab);
                        df = mass_fixed(exp_d(load_logit<T>(prow, id)), tab);
                    }
                    for (int o = 1; o < 32; o <<= 1) {
                        const unsigned long long t2 = __shfl_up_sync(0xffffffffu, tf, o), d2 = __shfl_up_sync(0xffffffffu, df, o);
                        if (lane >= o) { tf += t2; df += d2; }
                    }
                    if (base + lane < L)
                        best = fmin(best, (double)(cT + tf) * iT - power((double)(cD + df) * iD, n));
                    cT += __shfl_sync(0xffffffffu, tf, 31); cD += __shfl_sync(0xffffffffu, df, 31);
                }
            }
            best = block_min(best, s_r);
        }
    }
    if (crowded) todo |= 1 << ni;
    else if (tid == 0) {
        if (hdr) { hdr->alpha_star = 1.0 + best; hdr->resid_total = -best; }
        alpha_out[(size_t)b * nl.count + ni] = (float)(1.0 + best);
    }
    if (ni + 1 < nl.count) {
        __syncthreads();
        for (int c = tid; c < kBkBuckets; c += kBkThreads) { cnt[c] = 0; seg[c] = -1; }
        if (tid == 0) { s_nelem = 0; s_found = 0; s_fallback = 0; s_lo = kBkBuckets; s_hi = -1; }
        __syncthreads();
    }
    }
    if (tid == 0) {
        flag[0] = todo;
        if (GR_CHECK_VALUE || wh->check) {          // (bounds-checked build: an access was out of range)
            if (hdr) hdr->status = GR_CHECK_FAILED;
            if (status_out) status_out[b] = GR_CHECK_FAILED;
            if (rule_status) rule_status[b] = GR_CHECK_FAILED;
            for (int j = 0; j < nl.count; j++) alpha_out[(size_t)b * nl.count + j] = nanf("");
        }
    }
}

template <typename T>
__global__ void __launch_bounds__(kFsThreads)
fullsort_alpha_kernel(const T* __restrict__ q, const T* __restrict__ p, int V, const __grid_constant__ NList nl, double temp_t, double temp_d,
                      const char* __restrict__ ws, char* __restrict__ scratch, char* __restrict__ params, int pstride,
                      int batch, float* __restrict__ alpha_out)
{
    __shared__ double s_a[kFsThreads / 32], s_b[kFsThreads / 32];
    __shared__ double s_carry[2];
    __shared__ double s_min[kFsThreads / 32];
    pdl_wait();
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    // (normally no row is left to it: a grid of one wave looks, all its rows' flags at once)
    {
        int any = 0;
        for (long long b = blockIdx.x + (long long)tid * gridDim.x; b < batch; b += (long long)kFsThreads * gridDim.x)
            any |= *reinterpret_cast<const int*>(scratch + (size_t)b * next_pow2(V) * 12);
        if (!__syncthreads_or(any)) return;
    }
#pragma unroll 1
    for (long long b = blockIdx.x; b < batch; b += gridDim.x) {
    const WsHeader* wh = reinterpret_cast<const WsHeader*>(ws + (size_t)b * ws_stride());
    Header* hdr = params ? reinterpret_cast<Header*>(params + (size_t)b * pstride) : nullptr;
    if (wh->bad != 0) continue;                     // header / status already say GR_BAD_LOGITS
    const T* qrow = q + (size_t)b * V;
    const T* prow = p + (size_t)b * V;
    const int VP = next_pow2(V);
    unsigned long long* key = reinterpret_cast<unsigned long long*>(scratch + (size_t)b * VP * 12);
    // the first word of the region says whether bucket_alpha_kernel left this row to the sort
    const int todo = reinterpret_cast<const int*>(key)[0];
    __syncthreads();
    if (todo == 0) continue;
    int* idx = reinterpret_cast<int*>(key + VP);
    for (int i = tid; i < VP; i += kFsThreads) {
        if (i < V) {
            const double a = (double)load_logit<T>(qrow, i) / temp_t;
            const double d = (double)load_logit<T>(prow, i) / temp_d;
            key[i] = dkey(d - a); idx[i] = i;
        } else {
            key[i] = 0ull; idx[i] = 0x7fffffff;     // padding sorts last
        }
    }
    __syncthreads();
    // bitonic network over the VP pairs ("before" order ascending in position).  Compare-exchange of positions
    // i < l in the stage of block size k: ascending when (i & k) == 0.
    extern __shared__ __align__(16) unsigned char fs_smem[];
    unsigned long long* tk = reinterpret_cast<unsigned long long*>(fs_smem);
    int* ti = reinterpret_cast<int*>(tk + kFsTile);
    const int TL = VP < kFsTile ? VP : kFsTile;
    // the passes of distance j0, j0/2, ..., 1 of stage k on every tile, in shared memory; with whole = true all
    // stages 2 .. TL of the tile (the network's first log2 TL stages)
    auto tile_passes = [&](int k, int j0, bool whole) {
        for (int t0 = 0; t0 < VP; t0 += TL) {
            for (int e = tid; e < TL; e += kFsThreads) { tk[e] = key[t0 + e]; ti[e] = idx[t0 + e]; }
            __syncthreads();
            for (int kk = whole ? 2 : k; kk <= (whole ? TL : k); kk <<= 1) {
                for (int j2 = whole ? (kk >> 1) : j0; j2 > 0; j2 >>= 1) {
                    for (int pr = tid; pr < TL / 2; pr += kFsThreads) {
                        const int i = 2 * pr - (pr & (j2 - 1)), l = i + j2;
                        const unsigned long long ki = tk[i], kl = tk[l];
                        const int ii = ti[i], il = ti[l];
                        const bool up = ((t0 + i) & kk) == 0;
                        const bool wrong = up ? before(kl, il, ki, ii) : before(ki, ii, kl, il);
                        if (wrong) { tk[i] = kl; tk[l] = ki; ti[i] = il; ti[l] = ii; }
                    }
                    __syncthreads();
                }
            }
            for (int e = tid; e < TL; e += kFsThreads) { key[t0 + e] = tk[e]; idx[t0 + e] = ti[e]; }
            __syncthreads();
        }
    };
    tile_passes(0, 0, true);
    for (int k = 2 * TL; k <= VP; k <<= 1) {
        for (int j2 = k >> 1; j2 >= TL; j2 >>= 1) {
            for (int pr = tid; pr < VP / 2; pr += kFsThreads) {
                const int i = 2 * pr - (pr & (j2 - 1)), l = i + j2;
                const unsigned long long ki = key[i], kl = key[l];
                const int ii = idx[i], il = idx[l];
                const bool up = (i & k) == 0;
                const bool wrong = up ? before(kl, il, ki, ii) : before(ki, ii, kl, il);
                if (wrong) { key[i] = kl; key[l] = ki; idx[i] = il; idx[l] = ii; }
            }
            __syncthreads();
        }
        tile_passes(k, TL >> 1, false);
    }
    // log-sum-exp of both rows in fp64 (the streaming kernel's fp32 sums are good to ~1e-7 only, and the draft's
    // error enters alpha* multiplied by n through Dr^n)
    double mt = -1.0e300, md = -1.0e300;
    for (int i = tid; i < V; i += kFsThreads) {
        mt = fmax(mt, (double)load_logit<T>(qrow, i) / temp_t);
        md = fmax(md, (double)load_logit<T>(prow, i) / temp_d);
    }
    for (int o = 16; o > 0; o >>= 1) {
        mt = fmax(mt, __shfl_xor_sync(0xffffffffu, mt, o));
        md = fmax(md, __shfl_xor_sync(0xffffffffu, md, o));
    }
    if (lane == 0) { s_a[warp] = mt; s_b[warp] = md; }
    __syncthreads();
    mt = s_a[0]; md = s_b[0];
    for (int w2 = 1; w2 < kFsThreads / 32; w2++) { mt = fmax(mt, s_a[w2]); md = fmax(md, s_b[w2]); }
    __syncthreads();
    double st0 = 0.0, sd0 = 0.0;
    for (int i = tid; i < V; i += kFsThreads) {
        st0 += exp((double)load_logit<T>(qrow, i) / temp_t - mt);
        sd0 += exp((double)load_logit<T>(prow, i) / temp_d - md);
    }
    for (int o = 16; o > 0; o >>= 1) {
        st0 += __shfl_xor_sync(0xffffffffu, st0, o);
        sd0 += __shfl_xor_sync(0xffffffffu, sd0, o);
    }
    if (lane == 0) { s_a[warp] = st0; s_b[warp] = sd0; }
    __syncthreads();
    st0 = 0.0; sd0 = 0.0;
    for (int w2 = 0; w2 < kFsThreads / 32; w2++) { st0 += s_a[w2]; sd0 += s_b[w2]; }
    __syncthreads();
    const double lse_t = mt + log(st0), lse_d = md + log(sd0);
    // prefix sums of tgt and drf along the order, psi_j = Tg_j - Dr_j^n, running minimum
#pragma unroll 1
    for (int ni = 0; ni < nl.count; ni++) {
    if (((todo >> ni) & 1) == 0) continue;
    const int n = nl.n[ni];
    if (tid == 0) { s_carry[0] = 0.0; s_carry[1] = 0.0; }
    __syncthreads();
    double best = 0.0;                              // psi of the empty prefix
    constexpr int kPer = 4;
    for (int base = 0; base < V; base += kFsThreads * kPer) {
        double ta[kPer], da[kPer];
        double st = 0.0, sd = 0.0;
#pragma unroll
        for (int u = 0; u < kPer; u++) {
            const int j = base + tid * kPer + u;
            double tv = 0.0, dv = 0.0;
            if (j < V) {
                const int id = idx[j];
                tv = exp((double)load_logit<T>(qrow, id) / temp_t - lse_t);
                dv = exp((double)load_logit<T>(prow, id) / temp_d - lse_d);
            }
            st += tv; sd += dv; ta[u] = st; da[u] = sd;
        }
        // exclusive offsets of this thread: warp scan, then across warps
        double wt = st, wd = sd;
        for (int o = 1; o < 32; o <<= 1) {
            const double t2 = __shfl_up_sync(0xffffffffu, wt, o), d2 = __shfl_up_sync(0xffffffffu, wd, o);
            if (lane >= o) { wt += t2; wd += d2; }
        }
        if (lane == 31) { s_a[warp] = wt; s_b[warp] = wd; }
        __syncthreads();
        double ot = s_carry[0], od = s_carry[1];
        for (int w2 = 0; w2 < warp; w2++) { ot += s_a[w2]; od += s_b[w2]; }
        ot += wt - st; od += wd - sd;
#pragma unroll
        for (int u = 0; u < kPer; u++) {
            const int j = base + tid * kPer + u;
            if (j < V) {
                double Tg = ot + ta[u], Dr = od + da[u];
                if (j == V - 1) { Tg = 1.0; Dr = 1.0; }     // both distributions are normalised
                const double psi = Tg - pow(Dr, (double)n);
                best = fmin(best, psi);
            }
        }
        __syncthreads();
        if (tid == kFsThreads - 1) { s_carry[0] = ot + st; s_carry[1] = od + sd; }
        __syncthreads();
    }
    for (int o = 16; o > 0; o >>= 1) best = fmin(best, __shfl_xor_sync(0xffffffffu, best, o));
    if (lane == 0) s_min[warp] = best;
    __syncthreads();
    if (tid == 0) {
        for (int w2 = 1; w2 < kFsThreads / 32; w2++) best = fmin(best, s_min[w2]);
        if (hdr) { hdr->alpha_star = 1.0 + best; hdr->resid_total = -best; }
        alpha_out[(size_t)b * nl.count + ni] = (float)(1.0 + best);
    }
    __syncthreads();
    }
    }
}

void launch_fullsort(const void* q, const void* p, int dtype, int V, const int* n_list, int n_count, double temp_t,
                     double temp_d, int batch, const char* ws, char* scratch, char* params, int pstride, int force_sort, float* alpha_out,
                     int* status_out, int* rule_status, cudaStream_t st)
{
    NList nl;
    nl.count = n_count;
    for (int j = 0; j < n_count; j++) nl.n[j] = n_list[j];
    // function attributes belong to the device: set once per device (a failure shows up as a launch error)
    static bool configured[kMaxDevices] = {false};
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kMaxDevices) dev = -1;
    if (dev < 0 || !configured[dev]) {
        const bool ok = cudaFuncSetAttribute(fullsort_alpha_kernel<float>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                             kFsSmemBytes) == cudaSuccess &&
                        cudaFuncSetAttribute(fullsort_alpha_kernel<__nv_bfloat16>,
                                             cudaFuncAttributeMaxDynamicSharedMemorySize, kFsSmemBytes) == cudaSuccess &&
                        cudaFuncSetAttribute(bucket_alpha_kernel<float>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                             kBkSmemBytes) == cudaSuccess &&
                        cudaFuncSetAttribute(bucket_alpha_kernel<__nv_bfloat16>,
                                             cudaFuncAttributeMaxDynamicSharedMemorySize, kBkSmemBytes) == cudaSuccess;
        if (dev >= 0 && ok) configured[dev] = true;
    }
    const size_t sstride = (size_t)next_pow2(V) * 12;       // (room for V + 16 bucket numbers behind the flag: V > GR_MAX_SUPPORT)
    const int sort_grid = batch < kSms ? batch : kSms;
    if (dtype == GR_F32) {
        launch_pdl(bucket_alpha_kernel<float>, batch, kBkThreads, kBkSmemBytes, st, (const float*)q, (const float*)p, V, nl,
                   1.0 / temp_t, 1.0 / temp_d, ws, scratch, sstride, params, pstride, force_sort, alpha_out, status_out, rule_status);
        launch_pdl(fullsort_alpha_kernel<float>, sort_grid, kFsThreads, kFsSmemBytes, st, (const float*)q, (const float*)p, V,
                   nl, temp_t, temp_d, ws, scratch, params, pstride, batch, alpha_out);
    } else {
        launch_pdl(bucket_alpha_kernel<__nv_bfloat16>, batch, kBkThreads, kBkSmemBytes, st, (const __nv_bfloat16*)q,
                   (const __nv_bfloat16*)p, V, nl, 1.0 / temp_t, 1.0 / temp_d, ws, scratch, sstride, params, pstride, force_sort,
                   alpha_out, status_out, rule_status);
        launch_pdl(fullsort_alpha_kernel<__nv_bfloat16>, sort_grid, kFsThreads, kFsSmemBytes, st, (const __nv_bfloat16*)q,
                   (const __nv_bfloat16*)p, V, nl, temp_t, temp_d, ws, scratch, params, pstride, batch, alpha_out);
    }
}

}  // namespace gr
