// jac_sweep_noalloc: synchronous Jacobi sweeps that allocate no memory.
//
// Some callers cannot allocate device memory at the point where they need a
// solve: code running under a caching allocator or memory pool that owns
// every byte of the device, code that must not hit a device-wide
// synchronisation inside cudaMalloc/cudaFree (real-time loops, work issued
// from a callback), or plug-ins whose host application forbids allocation
// after start-up.  For them this file offers one entry point that works only
// on the caller's buffers plus a fixed scratch area that is part of the
// library image itself.
//
// The scratch is a file-scope static __device__ array (JAC_NOALLOC_SCRATCH_BYTES
// bytes, 256-byte aligned).  Every GPU that loads the library holds it until
// the process exits.  Host code cannot use the array's name as a device
// address, so the first call in each CUDA context (the device's primary
// context for runtime-API callers; again after cudaDeviceReset, which makes a
// new one) looks the address up with cudaGetSymbolAddress, with that device
// current, and caches it per context; make that first call before any stream
// capture.  Under CUDA's default lazy module loading that look-up is also
// when the library's device code is loaded into the context and the array's
// device memory is committed.  All calls share the one array and it keeps the
// last call's contents: each call clears the parts that must start at zero,
// and calls whose work overlaps on the GPU (different streams, or different
// host threads) race on it.
#include <cuda_runtime.h>

#include <cmath>
#include <cstdint>
#include <cstring>
#include <mutex>
#include <string>

#include "../../include/jacobi.h"
#include "jac_rounds.h"

// cuCtxGetCurrent / cuCtxGetId, fetched through the runtime's driver entry
// points so that the library does not link libcuda directly.
typedef struct CUctx_st* jac_cu_context;
typedef int (*jac_cu_ctx_get_current_fn)(jac_cu_context*);
typedef int (*jac_cu_ctx_get_id_fn)(jac_cu_context, unsigned long long*);

namespace jac {
void record_thread_error(const std::string& msg);   // jac_api.cu
jac_status host_exception(jac_ctx* c) noexcept;    // jac_api.cu
}

namespace {

constexpr long long kMaxRows = 4194304;                          // 2^22 rows
constexpr int kBlock = 256;
constexpr long long kMaxBlocks = (kMaxRows + kBlock - 1) / kBlock;
// layout: [ x scratch: kMaxRows doubles ][ partials: 3 x kMaxBlocks doubles ][ control: 64 bytes ]
// (partials: sum r_i^2, max |r_i| and sum b_i^2 of each block)
constexpr size_t kOffPartial = (size_t)kMaxRows * sizeof(double);
constexpr size_t kOffCtl = kOffPartial + 3 * (size_t)kMaxBlocks * sizeof(double);
constexpr size_t kScratchBytes = kOffCtl + 64;
static_assert(kScratchBytes == JAC_NOALLOC_SCRATCH_BYTES, "scratch size must match the header");

static __device__ __align__(256) unsigned char g_scratch[kScratchBytes];

struct NoallocCtl {
    unsigned int ticket;    // blocks finished in the current launch
    unsigned int pad;
    double bb;              // ||b||_2^2
    double ss;              // sum r_i^2 of the last evaluated iterate
    double mx;              // max |r_i|
};

// The larger of two magnitudes; a NaN wins.
__device__ __forceinline__ double max_nan(double v, double m)
{
    return (v > m || v != v) ? v : m;
}

// Sums over a block, valid in thread 0: warp shuffle trees, then the warps'
// sums in order.
__device__ __forceinline__ void block_sums(double& ss, double& mx, double& bb)
{
    __shared__ double s_ss[kBlock / 32], s_mx[kBlock / 32], s_bb[kBlock / 32];
    for (int o = 16; o > 0; o >>= 1) {
        ss += __shfl_down_sync(0xffffffffu, ss, o);
        bb += __shfl_down_sync(0xffffffffu, bb, o);
        mx = max_nan(__shfl_down_sync(0xffffffffu, mx, o), mx);
    }
    if ((threadIdx.x & 31) == 0) {
        s_ss[threadIdx.x >> 5] = ss;
        s_mx[threadIdx.x >> 5] = mx;
        s_bb[threadIdx.x >> 5] = bb;
    }
    __syncthreads();
    if (threadIdx.x == 0)
        for (int w = 1; w < kBlock / 32; ++w) {
            ss += s_ss[w];
            bb += s_bb[w];
            mx = max_nan(s_mx[w], mx);
        }
}

// Entries staged at a time: a block's 256 rows of up to 7 entries in one round (21.5
// KB; registers, not this, hold an SM to five blocks); longer rows take several rounds.
constexpr int kCap = 7 * kBlock;
constexpr int kGather = 7;   // x loads of a row issued together

__device__ __forceinline__ unsigned shared_addr(const void* p)
{
    return (unsigned)__cvta_generic_to_shared(p);
}

// t / d, correctly rounded, in five FP64 operations where the division takes about
// twice as many, on a chip whose FP64 pipe bounds the sweep: a single-precision
// reciprocal of d (its leading bits, moved between the formats with integer
// operations), one Newton step, and Markstein's quotient correction (Markstein, IBM
// J. Res. Dev. 34 (1990) 111): q = t r, z = q + (t - d q) r.  r is good to 2^-44 and
// the value rounded to z within 2^-33 of an ulp of t / d, so z is right unless that
// value lies as close to a midpoint.  Two tests find that out:
//   in single precision, beside the FP64 pipe: the correction c = (t - d q) r in ulps
//     of q, at most 2^9 and good to 2^-12, against the ulps that the rounding moved;
//   for the one quotient in 2,000 next to a midpoint (or past the end of q's
//     binade): t - d z, exact in one FMA for z within an ulp of t / d, is below half
//     an ulp of z times |d| exactly where z is the nearest number.
// Where neither passes, where z is a power of two (its lower neighbour is nearer),
// outside exponents that keep every step normal, and for t = 0, the division itself.
// 3,374,850 rows, us a sweep: without the tests 92.2, both 93.0, the exact one for
// every row 96.0, the first alone 96.2 (a warp in 60 divides), IEEE division 105.
//
// short_quotient: the value and whether the first test passed; checked_quotient: what
// holds where it did not.  The kernel stores the first before it knows.
__device__ __forceinline__ bool short_quotient(double t, double d, double& z)
{
    const unsigned dh = (unsigned)__double2hiint(d), dl = (unsigned)__double2loint(d);
    const unsigned th = (unsigned)__double2hiint(t);
    const unsigned de = (dh >> 20) & 0x7ffu, te = (th >> 20) & 0x7ffu;
    z = 0.0;
    if (de - 923u > 200u || te - 200u > 1600u) return false;     // |d| in 2^-100 .. 2^101, |t| in 2^-823 .. 2^778
    const float f = __uint_as_float((dh & 0x80000000u) | (((dh & 0x7fffffffu) - (896u << 20)) << 3) | (dl >> 29));
    float rf;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(rf) : "f"(f));
    const unsigned rb = __float_as_uint(rf);
    const double r0 = __hiloint2double((int)((rb & 0x80000000u) | (((rb & 0x7fffffffu) >> 3) + (896u << 20))),
                                       (int)(rb << 29));
    const double r = __fma_rn(__fma_rn(-d, r0, 1.0), r0, r0);
    const double q = __dmul_rn(t, r);
    const double rem = __fma_rn(-d, q, t);
    z = __fma_rn(rem, r, q);
    // rem r in ulps of q, in single precision, and the ulps that the rounding took
    const unsigned mh = (unsigned)__double2hiint(rem), qh = (unsigned)__double2hiint(q);
    const unsigned zh = (unsigned)__double2hiint(z), zl = (unsigned)__double2loint(z);
    const unsigned qe = (qh >> 20) & 0x7ffu;
    const unsigned mb = __funnelshift_l((unsigned)__double2loint(rem), mh & 0x7fffffffu, 3) - ((te - 179u) << 23);
    // (rem is 0, where z = q is exact and any m will do, or at least 2^-105 |t|)
    const float m = __uint_as_float(mb | ((mh ^ th) & 0x80000000u));
    const float c = __fmul_rn(m, __uint_as_float((rb & 0x7fffffffu) + ((te - qe) << 23)));
    const float off = __fsub_rn(c, (float)(int)(zl - (unsigned)__double2loint(q)));
    const bool plain = ((zh ^ qh) & 0xfff00000u) == 0 && ((zh & 0xfffffu) | zl) != 0;
    return plain && fabsf(off) < 0.4997f;
}

__device__ __forceinline__ double checked_quotient(double t, double d, double z)
{
    const unsigned dh = (unsigned)__double2hiint(d), zh = (unsigned)__double2hiint(z);
    const int back = __double2hiint(__fma_rn(-d, z, t)) & 0x7fffffff;
    // high word of |d| 2^(e - 53), e the exponent of z (at least 2^-1001)
    const int half = (int)((dh & 0x7fffffffu) + (zh & 0x7ff00000u) - (1076u << 20));
    return back < half && ((zh & 0xfffffu) | (unsigned)__double2loint(z)) ? z : t / d;   // (z = 0: the division)
}

// One sweep on a CSR matrix that stores its diagonal, one thread per row:
//   s_i = sum_{j != i} a_ij x_j (stored order),  x'_i = (b_i - s_i) / a_ii,
// and in the last sweep of a call (LAST) also
//   r_i = (b_i - s_i) - a_ii x_i
// with the residual sums and ||b||^2 reduced by the last block to finish, in
// a fixed order: the call returns those of its last sweep only, so the
// sweeps before it compute none (each takes three more FP64 operations per
// row and a reduction on a chip whose FP64 pipe is the co-bottleneck).
//
// A block copies its rows' entries into shared memory with coalesced
// asynchronous copies of one entry each (the caller's arrays have no more
// than their types' alignment), then each thread walks its row there: a
// thread reading its 56-byte row straight from memory makes every warp load
// touch 14 lines.  The copies, which read nothing that a sweep writes, start
// before griddepcontrol.wait: the launches of a call depend on one another
// programmatically, so a sweep's matrix is already arriving while the sweep
// before it drains.
//
// Bound by the FP64 pipe (six FMAs, a subtraction and the quotient's five
// operations per 7-point row) with the 104 bytes a row moves close behind: about
// 60 us each for 3,374,850 rows, which take 93 us a sweep (105 with IEEE
// division; 3,050 before rows were staged); 110,592 rows 8.2 us, 1,188 rows
// 4.0 us.  Five blocks an SM (48 registers) measured best, seven gathers
// together as good as eight; a block that copies its next tile while it sums one
// (two buffers, four blocks) took 105 us.
template <bool LAST>
__global__ void __launch_bounds__(kBlock, 5) k_noalloc_sweep(int n, const int* __restrict__ rowptr,
                                                             const int* __restrict__ col,
                                                             const double* __restrict__ val,
                                                             const double* __restrict__ b, const double* x, double* y,
                                                             unsigned char* scratch)
{
    __shared__ double s_val[kCap];
    __shared__ int s_col[kCap];
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    const int r0 = blockIdx.x * kBlock, i = r0 + threadIdx.x;
    const int p0 = rowptr[r0], p1 = rowptr[r0 + kBlock < n ? r0 + kBlock : n];
    const int kb = i < n ? rowptr[i] : 0, ke = i < n ? rowptr[i + 1] : 0;
    const double bi = i < n ? b[i] : 0.0;
    double s = 0.0, d = 0.0, xi = 0.0;
    bool waited = false;
    jac::for_each_round<kCap>(p0, p1, [&](int first, int count) {
        if (waited) __syncthreads();        // the round before has been read
#pragma unroll
        for (int q = 0; q < kCap; q += kBlock) {
            const int at = q + threadIdx.x;
            if (at < count) {
                asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"(shared_addr(s_val + at)),
                             "l"(val + first + at)
                             : "memory");
                asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(shared_addr(s_col + at)),
                             "l"(col + first + at)
                             : "memory");
            }
        }
        asm volatile("cp.async.wait_all;" ::: "memory");
        if (!waited) asm volatile("griddepcontrol.wait;" ::: "memory");
        waited = true;
        __syncthreads();
        // this thread's part of the round; the loop ends at the warp's longest
        int from;
        const int len = jac::row_part(kb, ke, first, count, from);
        const int most = (int)__reduce_max_sync(0xffffffffu, (unsigned)len);
        for (int o = 0; o < most; o += kGather) {
            double xv[kGather];
            int j[kGather];
#pragma unroll
            for (int u = 0; u < kGather; ++u) {
                j[u] = i;
                if (o + u < len) {
                    j[u] = s_col[from + o + u];
                    xv[u] = x[j[u]];
                }
            }
#pragma unroll
            for (int u = 0; u < kGather; ++u) {
                if (o + u >= most) break;
                if (o + u < len && j[u] == i) {
                    d = s_val[from + o + u];
                    xi = xv[u];
                }
                // a warp whose rows all have their diagonal here skips the FMA
                if (__any_sync(0xffffffffu, j[u] != i) && j[u] != i) s = __fma_rn(s_val[from + o + u], xv[u], s);
            }
        }
    });
    const double t = bi - s;
    if (i < n) {
        double z;
        const bool sure = short_quotient(t, d, z);
        y[i] = z;
        if (!sure) y[i] = checked_quotient(t, d, z);
    }
    if constexpr (LAST) {
        double ss = 0.0, mx = 0.0, bb = 0.0;
        if (i < n) {
            bb = bi * bi;
            const double r = __fma_rn(-d, xi, t);
            ss = r * r;
            mx = fabs(r);
            // a zero or missing diagonal, or an overflow, is reported as NaN
            if (d == 0.0 || !(mx <= 1.7976931348623157e308)) mx = __longlong_as_double(0x7ff8000000000000ll);
        }
        double* part = reinterpret_cast<double*>(scratch + kOffPartial);
        NoallocCtl* ctl = reinterpret_cast<NoallocCtl*>(scratch + kOffCtl);
        __shared__ int s_last;
        block_sums(ss, mx, bb);
        if (threadIdx.x == 0) {
            part[blockIdx.x] = ss;
            part[kMaxBlocks + blockIdx.x] = mx;
            part[2 * kMaxBlocks + blockIdx.x] = bb;
            __threadfence();
            s_last = (atomicAdd(&ctl->ticket, 1u) == gridDim.x - 1);
        }
        __syncthreads();
        if (s_last) {
            // the whole last block adds the blocks' sums, thread-strided then the
            // block's tree (one thread alone took 3 ms for 13,000 blocks)
            __threadfence();
            ss = mx = bb = 0.0;
            for (unsigned q = threadIdx.x; q < gridDim.x; q += kBlock) {
                ss += __ldcg(part + q);
                mx = max_nan(__ldcg(part + kMaxBlocks + q), mx);
                bb += __ldcg(part + 2 * kMaxBlocks + q);
            }
            block_sums(ss, mx, bb);
            if (threadIdx.x == 0) {
                ctl->ss = ss;
                ctl->mx = mx;
                ctl->bb = bb;
                ctl->ticket = 0;
            }
        }
    }
}

cudaError_t launch_sweep(bool first, bool last, int n, const int* rowptr, const int* col, const double* val,
                         const double* b, const double* x, double* y, unsigned char* scratch, cudaStream_t s)
{
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)((n + kBlock - 1) / kBlock));
    cfg.blockDim = dim3(kBlock);
    cfg.stream = s;
    // a call's first sweep waits for everything before it on the stream, the
    // others' prologues overlap the sweep before them
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = first ? 0 : 1;
    return last ? cudaLaunchKernelEx(&cfg, k_noalloc_sweep<true>, n, rowptr, col, val, b, x, y, scratch)
                : cudaLaunchKernelEx(&cfg, k_noalloc_sweep<false>, n, rowptr, col, val, b, x, y, scratch);
}

std::mutex g_mu;
// scratch address per CUDA context (its process-unique id); a small table,
// reused round-robin once full
constexpr int kCtxSlots = 64;
struct AddrSlot {
    unsigned long long ctx_id;
    unsigned char* addr;
};
AddrSlot g_slots[kCtxSlots] = {};
int g_next_slot = 0;
jac_cu_ctx_get_current_fn g_get_current = nullptr;
jac_cu_ctx_get_id_fn g_get_id = nullptr;

jac_status fail(jac_status st, const std::string& m)
{
    jac::record_thread_error(m);      // readable through jac_last_error(NULL)
    return st;
}

}  // namespace

extern "C" jac_status jac_sweep_noalloc(int64_t n, const int32_t* rowptr, const int32_t* col, const double* val,
                                        const double* b, const double* x_in, double* x_out, int32_t k,
                                        double* relres_out, void* stream)
try {
    if (n < 1) return fail(JAC_EINVAL, "jac_sweep_noalloc: n must be >= 1");
    if (n > kMaxRows)
        return fail(JAC_EINVAL, "jac_sweep_noalloc: n exceeds the fixed scratch limit of 4194304 rows");
    if (k < 0) return fail(JAC_EINVAL, "jac_sweep_noalloc: k must be >= 0");
    if (!rowptr || !col || !val || !b || !x_in || !x_out)
        return fail(JAC_EINVAL, "jac_sweep_noalloc: NULL pointer");
    if (x_in == x_out) return fail(JAC_EINVAL, "jac_sweep_noalloc: x_in and x_out must not alias");
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return fail(JAC_ECUDA, std::string("jac_sweep_noalloc: ") + cudaGetErrorString(e));
    if (dev < 0 || dev >= 256) return fail(JAC_EINVAL, "jac_sweep_noalloc: device ordinal out of range");
    unsigned char* scratch = nullptr;
    {
        // One-time set-up per CUDA context (with its device current): the
        // device address of the static scratch array.  The array lives in the
        // context's copy of the module, so a new context (cudaDeviceReset, a
        // caller's own driver-API context) gets its own look-up.
        std::lock_guard<std::mutex> lk(g_mu);
        if (!g_get_current || !g_get_id) {
            cudaDriverEntryPointQueryResult q1 = cudaDriverEntryPointSymbolNotFound, q2 = q1;
            void* f1 = nullptr;
            void* f2 = nullptr;
            e = cudaGetDriverEntryPointByVersion("cuCtxGetCurrent", &f1, 12000, cudaEnableDefault, &q1);
            if (e == cudaSuccess)
                e = cudaGetDriverEntryPointByVersion("cuCtxGetId", &f2, 12000, cudaEnableDefault, &q2);
            if (e != cudaSuccess || q1 != cudaDriverEntryPointSuccess || q2 != cudaDriverEntryPointSuccess)
                return fail(JAC_ECUDA, "jac_sweep_noalloc: the driver's cuCtxGetCurrent/cuCtxGetId are unavailable");
            g_get_current = reinterpret_cast<jac_cu_ctx_get_current_fn>(f1);
            g_get_id = reinterpret_cast<jac_cu_ctx_get_id_fn>(f2);
        }
        jac_cu_context cu = nullptr;
        if (g_get_current(&cu) != 0 || !cu) {
            // no context is current yet on this thread: make the device's
            // primary context current (cudaSetDevice initialises it)
            e = cudaSetDevice(dev);
            if (e != cudaSuccess || g_get_current(&cu) != 0 || !cu)
                return fail(JAC_ECUDA, "jac_sweep_noalloc: no CUDA context is current on this thread");
        }
        unsigned long long id = 0;
        if (g_get_id(cu, &id) != 0) return fail(JAC_ECUDA, "jac_sweep_noalloc: cuCtxGetId failed");
        for (int q = 0; q < kCtxSlots; ++q)
            if (g_slots[q].addr && g_slots[q].ctx_id == id) scratch = g_slots[q].addr;
        if (!scratch) {
            void* p = nullptr;
            // (and both kernels, which lazy loading would otherwise load at the first
            // call that launches each)
            cudaFuncAttributes fa;
            e = cudaGetSymbolAddress(&p, g_scratch);
            if (e == cudaSuccess) e = cudaFuncGetAttributes(&fa, k_noalloc_sweep<false>);
            if (e == cudaSuccess) e = cudaFuncGetAttributes(&fa, k_noalloc_sweep<true>);
            if (e != cudaSuccess)
                return fail(JAC_ECUDA, std::string("jac_sweep_noalloc: cudaGetSymbolAddress: ") + cudaGetErrorString(e));
            scratch = static_cast<unsigned char*>(p);
            g_slots[g_next_slot] = AddrSlot{id, scratch};
            g_next_slot = (g_next_slot + 1) % kCtxSlots;
        }
    }
    cudaStream_t s = (cudaStream_t)stream;
    const int nn = (int)n;
    double* xs = reinterpret_cast<double*>(scratch);
    // the ticket must start at zero: a previous call may have been interrupted
    e = cudaMemsetAsync(scratch + kOffCtl, 0, sizeof(NoallocCtl), s);
    if (e == cudaSuccess && k == 0)
        e = cudaMemcpyAsync(x_out, x_in, (size_t)n * sizeof(double), cudaMemcpyDeviceToDevice, s);
    // ping-pong between x_out and the scratch vector so that sweep k-1 writes x_out
    const double* src = x_in;
    for (int i = 0; i < k && e == cudaSuccess; ++i) {
        double* dst = ((k - 1 - i) % 2 == 0) ? x_out : xs;
        e = launch_sweep(i == 0, i == k - 1, nn, rowptr, col, val, b, src, dst, scratch, s);
        src = dst;
    }
    NoallocCtl h;
    std::memset(&h, 0, sizeof(h));
    if (e == cudaSuccess) e = cudaMemcpyAsync(&h, scratch + kOffCtl, sizeof(h), cudaMemcpyDeviceToHost, s);
    if (e == cudaSuccess) e = cudaStreamSynchronize(s);
    if (e != cudaSuccess) return fail(JAC_ECUDA, std::string("jac_sweep_noalloc: ") + cudaGetErrorString(e));
    if (k > 0) {
        if (!(h.ss <= 1.7976931348623157e308) || !(h.mx <= 1.7976931348623157e308))
            return fail(JAC_ENUMERIC, "jac_sweep_noalloc: the residual became NaN or Inf (zero diagonal or divergence)");
        if (relres_out) *relres_out = h.bb > 0.0 ? std::sqrt(h.ss) / std::sqrt(h.bb) : std::sqrt(h.ss);
    }
    return JAC_OK;
} catch (...) {
    // an error message that could not be allocated, or a failed mutex lock
    return jac::host_exception(nullptr);
}
