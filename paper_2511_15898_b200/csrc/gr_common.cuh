// Shared device-side definitions of the global-resolution library: the layout of
// the params block and of the workspace, and small helpers.
#pragma once
#include <cuda_runtime.h>
#include <cuda_bf16.h>
#include <cuda_fp16.h>
#include <stdint.h>
#include <type_traits>
#include "gr.h"

namespace gr {

// ---- Bounds-checked build.  Compiled with -DGR_CHECK (paper_2511_15898_b200.build.build_library(check=True), a
// separate library file) every pointer into shared memory, into the workspace records and into the params block
// carries its extent (and every array of a shared structure its own): an access outside it is SKIPPED (a read gives 0) and raises a per-CTA flag, which the kernel
// turns into the instance's status GR_CHECK_FAILED.  It stands in for a memory checker on machines where none may
// run; nothing traps or asserts.  Without the macro the same names are plain pointers and cost nothing.
#ifdef GR_CHECK
template <class T> struct CkNonConst { typedef T type; };
template <class T> struct CkNonConst<const T> { typedef T type; };
template <class T>
struct CkPtr {
    T* p; long long n; int* bad;
    mutable typename CkNonConst<T>::type sink;
    __host__ __device__ CkPtr() : p(nullptr), n(0), bad(nullptr), sink() {}
    __host__ __device__ CkPtr(T* p_, long long n_, int* bad_) : p(p_), n(n_), bad(bad_), sink() {}
    template <class U> __host__ __device__ CkPtr(const CkPtr<U>& o) : p(o.p), n(o.n), bad(o.bad), sink() {}
    __device__ T& operator[](long long i) const {
        if (i >= 0 && i < n) return p[i];
        if (bad) *bad = 1;
        sink = typename CkNonConst<T>::type();
        return sink;
    }
    __device__ T& operator*() const { return (*this)[0]; }
    __host__ __device__ CkPtr operator+(long long k) const { return CkPtr(p + k, n - k, bad); }
    __host__ __device__ CkPtr operator-(long long k) const { return CkPtr(p - k, n + k, bad); }
    template <class U> __host__ __device__ CkPtr<U> as() const {
        return CkPtr<U>(reinterpret_cast<U*>(p), n * (long long)sizeof(T) / (long long)sizeof(U), bad);
    }
};
// An array that is a member of a shared structure (whose address the accesses do not pass around): it carries the report.
template <class T, int N>
struct CkArray {
    T a[N];
    int bad;
    union { unsigned long long word[2]; } sink;
    template <class U> __device__ U& as(long long i) {
        if (i >= 0 && (i + 1) * (long long)sizeof(U) <= (long long)sizeof(a)) return reinterpret_cast<U*>(a)[i];
        bad = 1;
        sink.word[0] = sink.word[1] = 0ull;
        return *reinterpret_cast<U*>(&sink);
    }
    __device__ T& operator[](long long i) { return as<T>(i); }
};
#define GR_ARRAY(T, name, count) ::gr::CkArray<T, (count)> name
#define GR_ARRAY_AS(U, array, i) ((array).template as<U>(i))
#define GR_ARRAY_RESET(array) ((void)((array).bad = 0))
#define GR_ARRAY_BAD(array) ((array).bad)
#define GR_PTR(T) ::gr::CkPtr<T>
#define GR_MKPTR(T, ptr, count, flag) ::gr::CkPtr<T>((ptr), (count), (flag))
#define GR_PCAST(T, ptr) ((ptr).template as<T>())
#define GR_CHECK_FLAG_DECL __shared__ int s_check_flag
#define GR_CHECK_FLAG (&s_check_flag)
#define GR_CHECK_FLAG_INIT do { if (threadIdx.x == 0) s_check_flag = 0; __syncthreads(); } while (0)
#define GR_CHECK_VALUE (s_check_flag)
#else
template <class T> using RawPtr = T*;       // (an alias, so that "GR_PTR(double) a, b;" declares two pointers)
#define GR_PTR(T) ::gr::RawPtr<T>
#define GR_ARRAY(T, name, count) T name[count]
#define GR_ARRAY_AS(U, array, i) (reinterpret_cast<U*>(array)[i])
#define GR_ARRAY_RESET(array) ((void)0)
#define GR_ARRAY_BAD(array) (0)
#define GR_MKPTR(T, ptr, count, flag) (ptr)
#define GR_PCAST(T, ptr) (reinterpret_cast<T*>(ptr))
#define GR_CHECK_FLAG_DECL
#define GR_CHECK_FLAG (nullptr)
#define GR_CHECK_FLAG_INIT do { } while (0)
#define GR_CHECK_VALUE (0)
#endif

// Vector loads and stores through these pointers (the address is aligned to the vector).  The bounds-checked build takes
// the elements one by one, each checked.
#ifdef GR_CHECK
template <class P> __device__ inline float4 ld_f4(const P& p) { return make_float4(p[0], p[1], p[2], p[3]); }
template <class P> __device__ inline float2 ld_f2(const P& p) { return make_float2(p[0], p[1]); }
template <class P> __device__ inline double2 ld_d2(const P& p) { return make_double2(p[0], p[1]); }
template <class P> __device__ inline uint2 ld_u2(const P& p) { return make_uint2(p[0], p[1]); }
template <class P> __device__ inline uint4 ld_u4(const P& p) { return make_uint4(p[0], p[1], p[2], p[3]); }
template <class P> __device__ inline ulonglong2 ld_ull2(const P& p) { return make_ulonglong2(p[0], p[1]); }
template <class P> __device__ inline void st_f4(const P& p, float4 v) { p[0] = v.x; p[1] = v.y; p[2] = v.z; p[3] = v.w; }
template <class P> __device__ inline void st_u4(const P& p, uint4 v) { p[0] = v.x; p[1] = v.y; p[2] = v.z; p[3] = v.w; }
template <class P> __device__ inline void st_f2(const P& p, float2 v) { p[0] = v.x; p[1] = v.y; }
template <class P> __device__ inline void st_d2(const P& p, double2 v) { p[0] = v.x; p[1] = v.y; }
template <class P> __device__ inline uint4 ld_h8(const P& p) {
    uint32_t w[4];
    for (int z = 0; z < 4; z++) w[z] = (uint32_t)__half_as_ushort(p[2 * z]) | ((uint32_t)__half_as_ushort(p[2 * z + 1]) << 16);
    return make_uint4(w[0], w[1], w[2], w[3]);
}
template <class P> __device__ inline void st_h2(const P& p, uint32_t v) {
    p[0] = __ushort_as_half((unsigned short)(v & 0xffffu)); p[1] = __ushort_as_half((unsigned short)(v >> 16));
}
template <class P> __device__ inline void st_h8(const P& p, uint4 v) { st_h2(p, v.x); st_h2(p + 2, v.y); st_h2(p + 4, v.z); st_h2(p + 6, v.w); }
#else
__device__ __forceinline__ float4 ld_f4(const float* p) { return *reinterpret_cast<const float4*>(p); }
__device__ __forceinline__ float2 ld_f2(const float* p) { return *reinterpret_cast<const float2*>(p); }
__device__ __forceinline__ double2 ld_d2(const double* p) { return *reinterpret_cast<const double2*>(p); }
__device__ __forceinline__ uint2 ld_u2(const uint32_t* p) { return *reinterpret_cast<const uint2*>(p); }
__device__ __forceinline__ uint4 ld_u4(const uint32_t* p) { return *reinterpret_cast<const uint4*>(p); }
__device__ __forceinline__ ulonglong2 ld_ull2(const unsigned long long* p) { return *reinterpret_cast<const ulonglong2*>(p); }
__device__ __forceinline__ void st_f4(float* p, float4 v) { *reinterpret_cast<float4*>(p) = v; }
__device__ __forceinline__ void st_u4(uint32_t* p, uint4 v) { *reinterpret_cast<uint4*>(p) = v; }
__device__ __forceinline__ void st_f2(float* p, float2 v) { *reinterpret_cast<float2*>(p) = v; }
__device__ __forceinline__ void st_d2(double* p, double2 v) { *reinterpret_cast<double2*>(p) = v; }
__device__ __forceinline__ uint4 ld_h8(const __half* p) { return *reinterpret_cast<const uint4*>(p); }
__device__ __forceinline__ void st_h2(__half* p, uint32_t v) { *reinterpret_cast<uint32_t*>(p) = v; }
__device__ __forceinline__ void st_h8(__half* p, uint4 v) { *reinterpret_cast<uint4*>(p) = v; }
#endif

constexpr int kMaxSupport = GR_MAX_SUPPORT;   // largest support the convex programs are solved on
constexpr int kMaxDrafts = GR_MAX_DRAFTS;     // largest n
constexpr int kChunk = 1024;                  // elements per chunk of the target-row mass table
constexpr uint32_t kMagic = 0x47525031u;      // "GRP1"

// Header of one instance inside the params block (96 bytes).
struct __align__(16) Header {
    uint32_t magic;
    int V, n, k;              // k = support size (0 when the rule was not solved)
    int jstar, nblocks;       // |H*|, number of outer blocks
    int status, nch;          // solve status, number of chunks in the mass table
    double alpha_star;        // 1 + psi(H*)
    double lse_t;             // log sum exp of target logits / temp_target
    double resid_total;       // total residual mass the resample segment is drawn from
    double gnorm;             // L1 gradient norm at the returned weights (all systems summed)
    const void* q_row;        // this instance's target row
    int dtype, head;          // logits element type; elements before the first 16-byte boundary
    float temp_target;
    int iters;                // gradient evaluations spent (low 16 bits); bit 16: the norm of some system is a prediction
    int kcap;                 // capacity of the per-support arrays
    int stride;               // bytes from one instance's header to the next
};
static_assert(sizeof(Header) == 96, "params header layout");
// The evaluation count a system's solver returns carries, in bit 16, whether its last gradient norm was predicted
// from the final Newton step instead of evaluated; per instance the counts add up and the bits are or-ed.
constexpr int kItersMask = 0xffff;
constexpr int kItersPredicted = 1 << 16;
__host__ __device__ inline int add_iters(int total, int it) {
    return (((total & kItersMask) + (it & kItersMask)) & kItersMask) | ((total | it) & ~kItersMask);
}

// Per-instance params block: Header, then
//   int    id[kcap]     token id in ratio order (position 0 = largest drf/tgt)
//   int    blk[kcap]    -1 on H*, else block number counted from the lowest ratio
//   double w[kcap]      exp(alpha_i)
//   double r[kcap]      outer residual (0 on H*)
//   double p[kcap]      flow p_i = tgt_i - r_i
//   float2 chunk[nchcap]  (max, sum exp2) of target logits per 1024-element chunk
__host__ __device__ inline int round16(int x) { return (x + 15) & ~15; }
__host__ __device__ inline int kcap_of(int V, int topk) {
    int k = (topk <= 0 || topk >= V) ? V : topk;
    return k <= kMaxSupport ? ((k + 3) & ~3) : 0;
}
__host__ __device__ inline int nchcap_of(int V) { return (V + kChunk - 1) / kChunk + 1; }
__host__ __device__ inline int params_stride(int V, int topk) {
    return round16((int)sizeof(Header) + kcap_of(V, topk) * 32 + nchcap_of(V) * 8);
}
struct ParamView {
    Header* h; GR_PTR(int) id; GR_PTR(int) blk; GR_PTR(double) w; GR_PTR(double) r; GR_PTR(double) p; GR_PTR(float2) chunk;
};
// (V and `flag` only matter to the bounds-checked build: extent of the chunk table, where to report)
__host__ __device__ inline ParamView view_params(void* base, int kcap, int V = 1 << 21, int* flag = nullptr) {
    ParamView v;
    char* c = (char*)base;
    v.h = (Header*)c; c += sizeof(Header);
    v.w = GR_MKPTR(double, (double*)c, kcap, flag); c += (size_t)kcap * 8;
    v.r = GR_MKPTR(double, (double*)c, kcap, flag); c += (size_t)kcap * 8;
    v.p = GR_MKPTR(double, (double*)c, kcap, flag); c += (size_t)kcap * 8;
    v.id = GR_MKPTR(int, (int*)c, kcap, flag); c += (size_t)kcap * 4;
    v.blk = GR_MKPTR(int, (int*)c, kcap, flag); c += (size_t)kcap * 4;
    v.chunk = GR_MKPTR(float2, (float2*)c, nchcap_of(V), flag);
    (void)V; (void)flag;
    return v;
}

// Workspace of one instance (written by the scan kernel, read by the solve kernel).
struct __align__(16) WsHeader {
    double lse_t;        // log sum exp of target logits / temp_target
    int flagged, taken;  // record 0 only: instances the fast kernel left to the general one, and how many of them that one
                         // has begun (the streaming pass clears both)
    int count;           // entries that follow (the support, k of them)
    int bad;             // 1 when a non-finite logit was met
    int check;           // bounds-checked build: the streaming kernel skipped an out-of-range access on this row
    int flagged_id;      // record i: the i-th instance left to the general kernel
};
// then: int id[kMaxSupport]; float dl[kMaxSupport]; float tl[kMaxSupport];
// Of a whole-vocabulary row the streaming pass keeps, where the support would be: the draft row's maximum and the range of
// the log-ratio draft / target (fp32, in units of log 2; it only places buckets).
struct FullRow { float pmax, kmax, kmin, qmax; };
__host__ __device__ inline int ws_stride() { return (int)sizeof(WsHeader) + kMaxSupport * 12; }

// alignment head of row b: elements before the first 16-byte boundary
__host__ __device__ inline int row_head(const void* base, long long b, int V, int esize) {
    unsigned long long a = (unsigned long long)base + (unsigned long long)b * (unsigned long long)V * esize;
    int mis = (int)(a & 15ull);
    int head = mis ? (16 - mis) / esize : 0;
    return head < V ? head : V;
}
__host__ __device__ inline int num_chunks(int V, int head) {
    int body = V - head;
    int nch = (body + kChunk - 1) / kChunk;
    return nch < 1 ? 1 : nch;
}
// chunk that holds element i
__device__ inline int chunk_of(int i, int head, int nch) {
    if (i < head) return 0;
    int c = (i - head) / kChunk;
    return c < nch ? c : nch - 1;
}
__device__ inline int chunk_begin(int c, int head) { return c == 0 ? 0 : head + c * kChunk; }
__device__ inline int chunk_end(int c, int head, int nch, int V) {
    if (c == nch - 1) return V;
    int e = head + (c + 1) * kChunk;
    return e < V ? e : V;
}

template <typename T> __device__ inline float load_logit(const T* row, int i);
template <> __device__ inline float load_logit<float>(const float* row, int i) { return __ldg(row + i); }
template <> __device__ inline float load_logit<__nv_bfloat16>(const __nv_bfloat16* row, int i) {
    return __bfloat162float(row[i]);
}
__device__ inline float load_logit_dyn(const void* row, int dtype, int i) {
    return dtype == GR_BF16 ? load_logit<__nv_bfloat16>((const __nv_bfloat16*)row, i)
                            : load_logit<float>((const float*)row, i);
}

// order-preserving map float -> uint32 (larger float, larger key)
__device__ inline uint32_t fkey(float f) {
    uint32_t u = __float_as_uint(f + 0.f);       // (-0 + 0 = +0: the two zeros compare equal, so they get one key)
    return (u & 0x80000000u) ? ~u : (u | 0x80000000u);
}
__device__ inline float fkey_inv(uint32_t k) {
    uint32_t u = (k & 0x80000000u) ? (k & 0x7fffffffu) : ~k;
    return __uint_as_float(u);
}
// composite key: larger logit first, equal logits: smaller id first
__device__ inline unsigned long long ckey(float v, int id) {
    return ((unsigned long long)fkey(v) << 32) | (unsigned long long)(0xffffffffu - (uint32_t)id);
}

// fp64 functions kept out of line: the solve kernels call them from many places, and a small batch runs most of their code
// exactly once per SM, so what it waits for is instruction fetches.
static __device__ __noinline__ double m_exp(double x) { return exp(x); }
static __device__ __noinline__ double m_log(double x) { return log(x); }
static __device__ __noinline__ double m_div(double a, double b) { return a / b; }
static __device__ __noinline__ double2 m_div2(double a0, double a1, double b) { return make_double2(a0 / b, a1 / b); }

// exp(-y) for y >= 0 (fp64): Cody and Waite's range reduction by a two-part ln 2 and a degree-13 Taylor polynomial on
// |r| <= ln2/2 (truncation below 1e-17 relative), summed in pairs and fours (Estrin's scheme: a third of Horner's chain,
// which is what a warp alone on its scheduler waits for); results below 2^-1000 are flushed to zero.
__device__ __forceinline__ double exp_neg(double y)
{
    const double t = -y;
    const double kf = rint(t * 1.4426950408889634);
    double r = fma(-kf, 6.93147180369123816490e-01, t);
    r = fma(-kf, 1.90821492927058770002e-10, r);
    const double r2 = r * r, r4 = r2 * r2;
    const double a0 = 1.0 + r, a1 = fma(r, 1.6666666666666666e-01, 0.5);                    // 1/2!, 1/3!
    const double a2 = fma(r, 8.333333333333333e-03, 4.1666666666666664e-02);                // 1/4!, 1/5!
    const double a3 = fma(r, 1.984126984126984e-04, 1.388888888888889e-03);                 // 1/6!, 1/7!
    const double a4 = fma(r, 2.7557319223985893e-06, 2.48015873015873e-05);                 // 1/8!, 1/9!
    const double a5 = fma(r, 2.505210838544172e-08, 2.755731922398589e-07);                 // 1/10!, 1/11!
    const double a6 = fma(r, 1.6059043836821613e-10, 2.08767569878681e-09);                 // 1/12!, 1/13!
    const double b0 = fma(r2, a1, a0), b1 = fma(r2, a3, a2), b2 = fma(r2, a5, a4);
    const double p = fma(r4, fma(r4, fma(r4, a6, b2), b1), b0);
    const int k = (int)kf;
    return kf < -1000.0 ? 0.0 : __hiloint2double(__double2hiint(p) + (k << 20), __double2loint(p));
}

// Two fp32 numbers in one 64-bit register pair (sm_100's packed arithmetic: one instruction for both).
__device__ __forceinline__ float f_lo(unsigned long long v) { return __uint_as_float((unsigned int)v); }
__device__ __forceinline__ float f_hi(unsigned long long v) { return __uint_as_float((unsigned int)(v >> 32)); }
__device__ __forceinline__ unsigned long long f_pack(float lo, float hi) {
    return ((unsigned long long)__float_as_uint(hi) << 32) | __float_as_uint(lo);
}
__device__ __forceinline__ unsigned long long add2(unsigned long long a, unsigned long long b) {
    unsigned long long r;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}
__device__ __forceinline__ unsigned long long mul2(unsigned long long a, unsigned long long b) {
    unsigned long long r;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}
__device__ __forceinline__ unsigned long long fma2(unsigned long long a, unsigned long long b, unsigned long long c) {
    unsigned long long r;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
    return r;
}
// Brings `bytes` from p on into the first-level cache, a line per thread (as many threads as lines at least); nothing waits for it.
__device__ __forceinline__ void touch_lines(const void* p, int bytes)
{
    const int at = 128 * (int)threadIdx.x;
    if (at < bytes) {
        unsigned v;
        asm volatile("ld.global.u32 %0, [%1];" : "=r"(v) : "l"((const char*)p + at));
        (void)v;
    }
}
// Programmatic dependent launch.  Every kernel of a call is launched with launch_pdl and begins with this: its launch is
// prepared while the predecessor runs, but it touches no memory until the predecessor has completed (which, by the same
// rule, had waited for its own).  No kernel lets its successor's CTAs in early (griddepcontrol.launch_dependents): they
// settled on whichever SMs the last wave left free, many on a few, and stayed there when all the others were idle (128
// rows of 128256: solve and draw on 20 SMs, 150 us a call against 119).
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
template <class... P>
inline cudaError_t launch_pdl_cluster(int cluster, void (*kernel)(P...), int grid, int block, int smem, cudaStream_t st,
                                      std::remove_const_t<P>... args)
{
    cudaLaunchConfig_t cfg = {};
    cudaLaunchAttribute at[2] = {};
    at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[0].val.programmaticStreamSerializationAllowed = 1;
    at[1].id = cudaLaunchAttributeClusterDimension;
    at[1].val.clusterDim.x = (unsigned)cluster; at[1].val.clusterDim.y = 1; at[1].val.clusterDim.z = 1;
    cfg.gridDim = dim3((unsigned)grid); cfg.blockDim = dim3((unsigned)block);
    cfg.dynamicSmemBytes = (size_t)smem; cfg.stream = st; cfg.attrs = at; cfg.numAttrs = cluster > 1 ? 2 : 1;
    return cudaLaunchKernelEx(&cfg, kernel, args...);
}
template <class... P, class... A>
inline cudaError_t launch_pdl(void (*kernel)(P...), int grid, int block, int smem, cudaStream_t st, A... args)
{
    return launch_pdl_cluster<P...>(1, kernel, grid, block, smem, st, static_cast<P>(args)...);
}

constexpr int kSms = 148;                     // SMs of the chip: size of the grids that look for work
constexpr int kMaxDevices = 64;               // per-device caches of the host code (function attributes, streams)

}  // namespace gr
