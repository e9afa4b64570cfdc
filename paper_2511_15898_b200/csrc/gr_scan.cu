// The streaming pass as a kernel of its own (gr_scan.cuh): one CTA per row, or a cluster of CTAs per row where there are
// too few rows to fill the chip.
#include "gr_scan.cuh"

namespace gr {

constexpr int kScanThreads = 512;

// (1280 listed vectors hold what random rows bring between two cuts of the list at any support up to 128, and 2048 candidates what
// the last threshold leaves of it; with them four CTAs fit an SM.)
template <int NTHR> using ScanSm = ScanShared<NTHR, 1280, 2048, kMaxChunks>;

template <typename T, bool kFull, int kInFlight, int NTHR, int CTAS>
__global__ void __launch_bounds__(NTHR, CTAS)
scan_kernel(const __grid_constant__ ScanArgs A, int cn)
{
    __shared__ ScanSm<NTHR> sh;
    pdl_wait();
    GR_CHECK_FLAG_DECL;
    GR_CHECK_FLAG_INIT;
    scan_row<T, kFull, kInFlight>(A, sh, (long long)(blockIdx.x / cn), (int)(blockIdx.x % cn), cn, GR_CHECK_FLAG);
}

template <typename T>
static void launch_scan_t(const ScanArgs& A, bool full_large, int batch, cudaStream_t st)
{
    // Rows beyond one wave of two CTAs per SM: four CTAs of 256 threads per SM, half a chunk in flight per warp.  A row's rounds,
    // its thresholds and its selection at the end leave gaps that three other rows fill better than one (alpha* alone, 512 rows
    // of 50257 in fp32 54 -> 47 us, 4096 of 152064 in bf16 556 -> 505, 1024 of 128256 194 -> 189).  Up to one such wave, and
    // where a second wave of the small CTAs would be a quarter full, CTAs of 512 threads, two per SM: a row takes less time
    // (296 rows of 50257 44 -> 50 us with the small ones, 700 rows of 128256 153 -> 166).
    constexpr int kWave = 2 * kSms;
    const bool small = batch > kWave && !(batch > 2 * kWave && batch <= 5 * kWave / 2);
    if (full_large) {
        if (small) launch_pdl(scan_kernel<T, true, 4, kScanThreads / 2, 4>, batch, kScanThreads / 2, 0, st, A, 1);
        else launch_pdl(scan_kernel<T, true, 4, kScanThreads, 2>, batch, kScanThreads, 0, st, A, 1);
        return;
    }
    // Few rows are latency instead (a row on one CTA: 37 us, eight rounds to memory): a cluster of CTAs per row then, one CTA per
    // SM, a whole chunk in flight per warp, as long as every warp keeps a chunk (1 row 17 us, 32 rows 22).
    // The numbers of rows are those up to which the clusters ran in one wave: the 148 SMs do not come in groups of 8, and a
    // cluster of 8 beyond the 14th, or of 4 beyond the 32nd, cost 12 us.  Up to 148 long rows go in pairs of CTAs, two per SM
    // (80 rows of 128256 50 -> 44 us, 140 rows 52 -> 50; of 50257 no gain).
    int cn = 1;
    const int want = batch <= 14 ? 8 : batch <= 32 ? 4 : batch <= kSms / 2 ? 2 : 1;
    while (cn < want && A.V >= 2 * cn * (kScanThreads / 32) * kChunk) cn *= 2;
    if (cn > 1) launch_pdl_cluster(cn, scan_kernel<T, false, 8, kScanThreads, 1>, batch * cn, kScanThreads, 0, st, A, cn);
    else if (want == 1 && batch <= kSms && A.V >= 64 * kChunk)
        launch_pdl_cluster(2, scan_kernel<T, false, 4, kScanThreads, 2>, batch * 2, kScanThreads, 0, st, A, 2);
    else if (small) launch_pdl(scan_kernel<T, false, 4, kScanThreads / 2, 4>, batch, kScanThreads / 2, 0, st, A, 1);
    else launch_pdl(scan_kernel<T, false, 4, kScanThreads, 2>, batch, kScanThreads, 0, st, A, 1);
}

void launch_scan(const void* q, const void* p, int dtype, int V, int ksel, bool full_large, double temp_t,
                 double temp_d, int batch, char* ws, char* params, int pstride, int kcap, cudaStream_t st)
{
    const double log2e = 1.4426950408889634;
    ScanArgs A;
    A.q = q; A.p = p; A.V = V; A.ksel = ksel;
    A.sc_t = (float)(log2e / temp_t); A.sc_d = (float)(log2e / temp_d);
    A.temp_t = temp_t; A.temp_d = temp_d; A.ws = ws; A.params = params; A.pstride = pstride; A.kcap = kcap;
    if (dtype == GR_F32) launch_scan_t<float>(A, full_large, batch, st);
    else launch_scan_t<__nv_bfloat16>(A, full_large, batch, st);
}

}  // namespace gr
