// Optimal acceptance alpha* = 1 + min_H psi(H) alone, for several draft counts n at once
// (Eq. "subset-select"; the prefix sums along the ratio order do not depend on n, only
// psi_j = Tg_j - Dr_j^n does).  One CTA per instance, after the streaming kernel.
#include "gr_prep.cuh"

namespace gr {

constexpr int kAlphaThreads = 128;
struct NList { int n[GR_MAX_ALPHA_N]; int count; };

__global__ void __launch_bounds__(kAlphaThreads)
alpha_kernel(const char* __restrict__ ws, int V, int topk, double temp_t, double temp_d, NList nl,
             float* __restrict__ alpha_out, int* __restrict__ status_out)
{
    __shared__ __align__(16) unsigned long long s_key[kMaxSupport];
    __shared__ double s_tg[kMaxSupport], s_d[kMaxSupport], s_Tg[kMaxSupport + 1], s_Dr[kMaxSupport + 1];
    __shared__ int s_id[kMaxSupport], s_at[kMaxSupport];
    __shared__ double s_red[32];
    pdl_wait();
    const int tid = threadIdx.x;
    const long long b = blockIdx.x;
    const WsView wv = view_ws(ws, b);
    const int k = wv.h->count;
    if (wv.h->bad != 0 || k <= 0) {
        if (tid < nl.count) alpha_out[(size_t)b * nl.count + tid] = __int_as_float(0x7fc00000);
        if (tid == 0) status_out[b] = wv.h->bad != 0 ? GR_BAD_LOGITS : GR_SUPPORT_TOO_LARGE;
        return;
    }
    const int kfull = (topk <= 0 || topk >= V) ? V : topk;
    double lse_t = wv.h->lse_t;
    // distributions on the support in fp64 (App. A; App. N), as in the solve kernels
    double a_i = 0.0, b_i = 0.0;
    int my_id = 0;
    if (tid < k) {
        my_id = wv.id[tid];
        a_i = (double)wv.tl[tid] / temp_t;
        b_i = (double)wv.dl[tid] / temp_d;
    }
    // (the streaming pass leaves the support in descending order: the first entry is the largest)
    const double bmax = (double)wv.dl[0] / temp_d;
    const double bsum = block_reduce_sum(tid < k ? exp(b_i - bmax) : 0.0, GR_MKPTR(double, s_red, 32, nullptr));
    const double lse_d = bmax + log(bsum);
    if (kfull == V) {
        const double amax = block_reduce_max(tid < k ? a_i : -1.0e300, GR_MKPTR(double, s_red, 32, nullptr));
        const double asum = block_reduce_sum(tid < k ? exp(a_i - amax) : 0.0, GR_MKPTR(double, s_red, 32, nullptr));
        lse_t = amax + log(asum);
    }
    // ratio order: decreasing log-ratio, equal keys by smaller id (Sec. 5.1)
    const unsigned long long key = tid < k ? order_key(b_i - a_i) : 0ull;
    if (tid < ((k + 3) & ~3)) { s_key[tid] = key; s_id[tid] = my_id; }
    __syncthreads();
    const int rank = ratio_rank<true>(GR_MKPTR(const unsigned long long, s_key, kMaxSupport, nullptr), GR_MKPTR(const int, s_id, kMaxSupport, nullptr),
                                GR_MKPTR(int, s_at, kMaxSupport, nullptr), 0, tid < k ? k : 0, key, my_id);
    if (tid < k) {
        s_tg[rank] = exp(a_i - lse_t);
        s_d[rank] = exp(b_i - lse_d);
    }
    __syncthreads();
    prefix_sums(GR_MKPTR(const double, s_tg, kMaxSupport, nullptr), GR_MKPTR(double, s_Tg, kMaxSupport + 1, nullptr),
                GR_MKPTR(const double, s_d, kMaxSupport, nullptr), GR_MKPTR(double, s_Dr, kMaxSupport + 1, nullptr), k);
    // both distributions are normalised
    if (tid == 0 && kfull == V) s_Tg[k] = 1.0;
    if (tid == 32) s_Dr[k] = 1.0;
    __syncthreads();
    // one warp per draft count: min over the prefixes of Tg_j - Dr_j^n
    const int warp = tid >> 5, lane = tid & 31;
    for (int e = warp; e < nl.count; e += kAlphaThreads / 32) {
        const int n = nl.n[e];
        double best = 0.0;                       // psi of the empty prefix
        for (int j = 1 + lane; j <= k; j += 32) {
            double pw = 1.0, sq = s_Dr[j];
            for (int m = n; m > 0; m >>= 1) { if (m & 1) pw *= sq; sq *= sq; }
            best = fmin(best, s_Tg[j] - pw);
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) best = fmin(best, __shfl_xor_sync(0xffffffffu, best, o));
        if (lane == 0) alpha_out[(size_t)b * nl.count + e] = (float)(1.0 + best);
    }
    if (tid == 0) status_out[b] = wv.h->check ? GR_CHECK_FAILED : GR_OK;    // (never set but in the bounds-checked build)
}

void launch_alpha(const char* ws, int V, int topk, double temp_t, double temp_d, const int* n_list, int n_count,
                  int batch, float* alpha_out, int* status_out, cudaStream_t st)
{
    NList nl;
    nl.count = n_count;
    for (int i = 0; i < GR_MAX_ALPHA_N; i++) nl.n[i] = i < n_count ? n_list[i] : 1;
    launch_pdl(alpha_kernel, batch, kAlphaThreads, 0, st, ws, V, topk, temp_t, temp_d, nl, alpha_out, status_out);
}

}  // namespace gr
