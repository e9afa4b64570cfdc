// The streaming pass as a kernel of its own (gr_scan.cuh): one CTA per row, or a cluster of CTAs per row where there are
// too few rows to fill the chip.
#include "gr_scan.cuh"

namespace gr {

constexpr int kScanThreads = 512;

typedef ScanShared<kScanThreads, 2048, kMaxChunks> ScanSm;

template <typename T, bool kFull, int kInFlight, int CTAS>
__global__ void __launch_bounds__(kScanThreads, CTAS)
scan_kernel(const __grid_constant__ ScanArgs A, int cn)
{
    __shared__ ScanSm sh;
    pdl_wait();
    GR_CHECK_FLAG_DECL;
    GR_CHECK_FLAG_INIT;
    scan_row<T, kFull, kInFlight>(A, sh, (long long)(blockIdx.x / cn), (int)(blockIdx.x % cn), cn, GR_CHECK_FLAG);
}

template <typename T>
static void launch_scan_t(const ScanArgs& A, bool full_large, int batch, cudaStream_t st)
{
    // One CTA per row, two CTAs per SM, half a chunk in flight per warp: 1024 fp32 rows of 128256 at 5.4 TB/s, what is
    // missing to the copy rate being the last of four waves.  Few rows are latency instead (a row on one CTA: 37 us, eight
    // rounds to memory): a cluster of CTAs per row then, one CTA per SM, a whole chunk in flight per warp, as long as
    // every warp keeps a chunk (1 row 22 us, 32 rows 27, 64 rows 33; were 37, 39, 39).  The numbers of rows are those
    // up to which the clusters ran in one wave: the 148 SMs do not come in groups of 8, and a cluster of 8 beyond the 14th, or
    // of 4 beyond the 32nd, cost 12 us.
    int cn = 1;
    if (!full_large) {
        const int want = batch <= 14 ? 8 : batch <= 32 ? 4 : batch <= 74 ? 2 : 1;
        while (cn < want && A.V >= 2 * cn * (kScanThreads / 32) * kChunk) cn *= 2;
    }
    if (full_large) launch_pdl(scan_kernel<T, true, 4, 2>, batch, kScanThreads, 0, st, A, 1);
    else if (cn > 1) launch_pdl_cluster(cn, scan_kernel<T, false, 8, 1>, batch * cn, kScanThreads, 0, st, A, cn);
    else launch_pdl(scan_kernel<T, false, 4, 2>, batch, kScanThreads, 0, st, A, 1);
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
