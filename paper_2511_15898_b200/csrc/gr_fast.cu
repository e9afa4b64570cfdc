// Dispatch of the fast per-instance solve (kernels in gr_fast.cuh; one translation unit per series length).
#include "gr_verify.cuh"

namespace gr {

#define GR_FAST_ARGS                                                                                              \
    char *ws, char *params, int pstride, int kcap, int V, int n, int topk, double temp_t, double temp_d,   \
        double tol, int max_iters, double qstep, double tau, int batch, float *alpha_out, int *status_out,       \
        FusedArgs fa, cudaStream_t st
namespace fast {
int launch_fast_n4_m32(GR_FAST_ARGS);
int launch_fast_n4_m32w(GR_FAST_ARGS);
int launch_fast_n4_m64(GR_FAST_ARGS);
int launch_fast_n4_m64w(GR_FAST_ARGS);
int launch_fast_n8_m32(GR_FAST_ARGS);
int launch_fast_n8_m32w(GR_FAST_ARGS);
int launch_fast_n8_m64(GR_FAST_ARGS);
int launch_fast_n8_m64w(GR_FAST_ARGS);
int launch_fast_n8_m128(GR_FAST_ARGS);
int launch_fast_n8_m128w(GR_FAST_ARGS);
int launch_fast_n16_m32(GR_FAST_ARGS);
int launch_fast_n16_m32w(GR_FAST_ARGS);
int launch_fast_n16_m32h(GR_FAST_ARGS);
int launch_fast_n16_m64(GR_FAST_ARGS);
int launch_fast_n16_m64w(GR_FAST_ARGS);
int launch_fast_n16_m128(GR_FAST_ARGS);
int launch_fast_n16_m128h(GR_FAST_ARGS);
int launch_fast_n16_m128w(GR_FAST_ARGS);
int launch_fast_c24_m32(GR_FAST_ARGS);
int launch_fast_c24_m32w(GR_FAST_ARGS);
int launch_fast_c24_m64(GR_FAST_ARGS);
int launch_fast_c24_m128(GR_FAST_ARGS);
}

// Returns 1 when no fast variant covers the shape (the caller then runs the general kernel on everything);
// after a return of 0 the caller runs the general kernel on the instances this one flagged (normally none).
int launch_fast(GR_FAST_ARGS)
{
    if (kcap <= 0 || kcap > 128 || n < 2) return 1;
#define GR_FAST_PASS ws, params, pstride, kcap, V, n, topk, temp_t, temp_d, tol, max_iters, qstep, tau, batch, alpha_out, status_out, fa, st
    // Twice to four times the threads per instance, and registers without spills, where the batch leaves an SM with one
    // instance (two of the narrow supports): an instance is a chain of dependent steps then, and 1 row of the headline shape
    // takes 50.5 us a call for 59.0, 128 rows 75 for 83, 64 whole rows of 16 ids 58 for 67.  Beyond one wave the other variants' places
    // count for more (series of 16 and up to 128 tokens: from two waves on, gr_fast_n16.cu; 1024 rows of 9001, n = 8, k = 50: 253 us a call in the wide variant, 138 in the other; 512 rows, n = 16, k = 20, 92 and 71).
    const bool one = batch <= kSms, two = batch <= 2 * kSms;
    if (n > 16) {
        if (kcap <= 32) return two ? fast::launch_fast_c24_m32w(GR_FAST_PASS) : fast::launch_fast_c24_m32(GR_FAST_PASS);
        if (kcap <= 64) return fast::launch_fast_c24_m64(GR_FAST_PASS);
        return fast::launch_fast_c24_m128(GR_FAST_PASS);
    }
    if (kcap <= 32) {
        if (n <= 4) return two ? fast::launch_fast_n4_m32w(GR_FAST_PASS) : fast::launch_fast_n4_m32(GR_FAST_PASS);
        if (n <= 8) return two ? fast::launch_fast_n8_m32w(GR_FAST_PASS) : fast::launch_fast_n8_m32(GR_FAST_PASS);
        if (two) return fast::launch_fast_n16_m32w(GR_FAST_PASS);
        return batch <= 4 * kSms ? fast::launch_fast_n16_m32h(GR_FAST_PASS) : fast::launch_fast_n16_m32(GR_FAST_PASS);
    }
    if (kcap <= 64) {
        if (n <= 4) return one ? fast::launch_fast_n4_m64w(GR_FAST_PASS) : fast::launch_fast_n4_m64(GR_FAST_PASS);
        if (n <= 8) return one ? fast::launch_fast_n8_m64w(GR_FAST_PASS) : fast::launch_fast_n8_m64(GR_FAST_PASS);
        return one ? fast::launch_fast_n16_m64w(GR_FAST_PASS) : fast::launch_fast_n16_m64(GR_FAST_PASS);
    }
    if (n <= 8) return one ? fast::launch_fast_n8_m128w(GR_FAST_PASS) : fast::launch_fast_n8_m128(GR_FAST_PASS);
    if (one) return fast::launch_fast_n16_m128w(GR_FAST_PASS);
    return two ? fast::launch_fast_n16_m128h(GR_FAST_PASS) : fast::launch_fast_n16_m128(GR_FAST_PASS);
}

}  // namespace gr
