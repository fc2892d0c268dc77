// noalloc.cu -- vp_alloc_static: the reallocation step without any device
// allocation.
//
// Some callers cannot allocate device memory while they work: a serving
// process that reserved all device memory up front for a pool it manages
// itself, or code that must not call cudaMalloc in the middle of a step
// because cudaMalloc may synchronise the whole device.  For them this file
// offers the reallocation step (the same arithmetic as vp_adapt's: the
// fixed-order sum of d_h, n_h = max(2, floor(N_ev d_h / sum d)) or the "+2"
// form, exclusive offsets) on buffers the caller provides, with its scratch in
// a static device array instead of memory it allocates.
#include <cstdarg>
#include <cstdio>
#include <mutex>
#include <string>

#include "alloc_core.cuh"
#include "vp_internal.cuh"

namespace vp {
const char *set_error_message(vp_status s, const char *msg);  // api.cu
}

namespace {

constexpr uint64_t kStaticMaxHc = 1ull << 22;          // 4,194,304 hypercubes
constexpr int kStaticMaxBlocks = (int)(kStaticMaxHc / 1024);

// Scratch of vp_alloc_static: 4096 x 16 bytes + counters, ~64 KB per device.
struct StaticScratch {
    double part[kStaticMaxBlocks];               // fixed-order block sums of d_h
    unsigned long long bsum[kStaticMaxBlocks];   // block sums of n_h -> block offsets
    double sum_d, c;                             // c: N_ev / sum d, or 0 (see alloc_one)
    unsigned int done_sum, done_alloc;
};

static __device__ __align__(256) StaticScratch g_alloc_scratch;

// Three launches, one CTA of 256 threads per block of 1024 hypercubes, each
// waiting for the one before it in pdl_wait (its launch overlaps the other's
// end).  Bound: latency (the two serial tails, one CTA each); the streams take
// 20 B of HBM per hypercube (d_h read, n_h and the offset written; d_h and n_h
// are read again from L2).  Against one FP64 division and a floor per
// hypercube and a single thread adding the block sums one after the other --
// ~240 ns each, 397 of 430 us at 1,679,616 hypercubes -- here one FP64 product
// per hypercube (alloc_one) and a scan of 16 block sums per thread.

// The sum of d_h in the library's fixed order: thread t takes the terms t,
// t + 256, t + 512, t + 768 of its block, whose first two halving levels are
// its own, then halving through shared memory and shuffles; the last CTA adds
// the block sums in the fixed tree.
__global__ void __launch_bounds__(256) ks_sum(const double *d_h, uint64_t n_hc, double n_ev_d,
                                              StaticScratch *sc) {
    __shared__ double sh[256];
    __shared__ bool s_last;
    vp::pdl_wait();
    vp::pdl_trigger();
    const int t = threadIdx.x;
    const uint64_t h0 = (uint64_t)blockIdx.x * 1024 + t;
    double v[4];
#pragma unroll
    for (int q = 0; q < 4; ++q) v[q] = h0 + 256 * q < n_hc ? d_h[h0 + 256 * q] : 0.0;
    sh[t] = __dadd_rn(__dadd_rn(v[0], v[2]), __dadd_rn(v[1], v[3]));
    __syncthreads();
    for (int s = 128; s >= 64; s >>= 1) {
        if (t < s) sh[t] = __dadd_rn(sh[t], sh[t + s]);
        __syncthreads();
    }
    if (t < 32) {
        double r = __dadd_rn(sh[t], sh[t + 32]);
        for (int s = 16; s >= 1; s >>= 1) r = __dadd_rn(r, __shfl_down_sync(0xffffffffu, r, s));
        if (t == 0) {
            sc->part[blockIdx.x] = r;
            __threadfence();
            s_last = atomicAdd(&sc->done_sum, 1u) == gridDim.x - 1;
        }
    }
    __syncthreads();
    if (!s_last) return;
    __threadfence();
    double S[1];  // the block sums in the library's fixed tree order
    vp::block_tree_sum<1>(sc->part, gridDim.x, sh, S);
    if (t != 0) return;
    sc->done_sum = 0u;  // (for the next call, should a later launch of this one fail)
    sc->sum_d = S[0];
    // (c only where sum d and the quotient are normal numbers and no N_ev d_h
    // can overflow, so that alloc_one's product is within a few ulp of the
    // IEEE quotient)
    const double c = S[0] >= 2.2250738585072014e-308 ? n_ev_d * (1.0 / S[0]) : 0.0;
    const bool ok = c >= 2.2250738585072014e-308 && c <= 1.7976931348623157e308 &&
                    n_ev_d * S[0] <= 1.7976931348623157e308;
    sc->c = ok ? c : 0.0;
}

// The reading's quotient as written, for sums so large that N_ev d_h may
// overflow and for d_h outside [0, sum d] (a call, so that its FP64 work stays
// out of the common path).
__device__ __noinline__ uint32_t alloc_literal(double dh, double n_ev_d, double sum_d, int plus2) {
    const double q = __ddiv_rn(__dmul_rn(n_ev_d, dh), sum_d);
    double fl = floor(q);
    if (__dsub_rn(__dadd_rn(fl, 1.0), q) <= __dmul_rn(q, 8.8817841970012523e-16)) fl += 1.0;
    if (plus2) return (uint32_t)fl + 2u;
    return fl > 2.0 ? (uint32_t)fl : 2u;
}

// Exclusive scan of one 64-bit value per thread over a CTA of 256 threads (N_ev
// may lie close to 2^32 here, so a block's sum may pass it); *total: the sum.
__device__ __forceinline__ unsigned long long scan64(unsigned long long v, unsigned long long *s_w,
                                                     unsigned long long *total) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    unsigned long long inc = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const unsigned long long u = __shfl_up_sync(0xffffffffu, inc, o);
        if (lane >= o) inc += u;
    }
    if (lane == 31) s_w[warp] = inc;
    __syncthreads();
    unsigned long long base = 0ull, all = 0ull;
#pragma unroll
    for (int w = 0; w < 8; ++w) {
        const unsigned long long x = s_w[w];
        if (w < warp) base += x;
        all += x;
    }
    __syncthreads();  // s_w may be reused
    *total = all;
    return base + inc - v;
}

// (VEC: d_h, n_h and offsets start on 16-byte boundaries, so a thread's four
// consecutive hypercubes move in vector loads and stores)
template <bool VEC>
__global__ void __launch_bounds__(256) ks_alloc(const double *d_h, uint64_t n_hc, double n_ev_d,
                                                int plus2, uint32_t *n_h, uint64_t *off,
                                                StaticScratch *sc) {
    __shared__ unsigned long long s_w[8];
    __shared__ bool s_last;
    vp::pdl_wait();
    vp::pdl_trigger();
    vp::AllocK K;
    K.n_ev_d = n_ev_d;
    K.sum_d = __ldcg(&sc->sum_d);
    K.c = __ldcg(&sc->c);
    K.dmin = 4.4501477170144028e-308;  // 2^-1021: N_ev d_h is a normal number from here
    K.n_hc = n_hc;
    K.plus2 = plus2 != 0;
    if (!vp::finite_bits(K.sum_d)) return;  // allocation left unchanged
    // d_h whose bits pass `lit` take the quotient as written: all but zero where
    // N_ev d_h may overflow, else a negative one or one above the sum (outside
    // the documented range; none where sum d is not positive)
    const uint64_t sum_bits = (uint64_t)__double_as_longlong(K.sum_d);
    const uint64_t lit = (int64_t)sum_bits <= 0 ? ~0ull
                         : vp::finite_bits(n_ev_d * K.sum_d) ? sum_bits : 0ull;
    const uint64_t h0 = (uint64_t)blockIdx.x * 1024 + 4u * threadIdx.x;
    const bool full = h0 + 4 <= n_hc;
    double dh[4];
    if (VEC && full) {
        const double2 a = *(const double2 *)(d_h + h0), b = *(const double2 *)(d_h + h0 + 2);
        dh[0] = a.x; dh[1] = a.y; dh[2] = b.x; dh[3] = b.y;
    } else {
#pragma unroll
        for (int q = 0; q < 4; ++q) dh[q] = h0 + q < n_hc ? d_h[h0 + q] : 0.0;
    }
    uint32_t n[4];
    unsigned long long own = 0ull;
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        n[q] = 0u;
        if (h0 + q < n_hc)
            n[q] = (uint64_t)__double_as_longlong(dh[q]) > lit
                       ? alloc_literal(dh[q], n_ev_d, K.sum_d, plus2)
                       : vp::alloc_one(dh[q], K, 0);
        own += n[q];
    }
    if (VEC && full) {
        *(uint4 *)(n_h + h0) = make_uint4(n[0], n[1], n[2], n[3]);
    } else {
#pragma unroll
        for (int q = 0; q < 4; ++q)
            if (h0 + q < n_hc) n_h[h0 + q] = n[q];
    }
    unsigned long long tot;
    scan64(own, s_w, &tot);
    if (threadIdx.x == 0) {
        sc->bsum[blockIdx.x] = tot;
        __threadfence();
        s_last = atomicAdd(&sc->done_alloc, 1u) == gridDim.x - 1;
    }
    __syncthreads();
    if (!s_last) return;
    __threadfence();
    // the block sums' exclusive scan, 16 consecutive ones per thread (4096 in all)
    constexpr int kV = kStaticMaxBlocks / 256;
    unsigned long long v[kV], mine = 0ull;
#pragma unroll
    for (int k = 0; k < kV; ++k) {
        const unsigned q = threadIdx.x * kV + k;
        v[k] = q < gridDim.x ? __ldcg(sc->bsum + q) : 0ull;
    }
#pragma unroll
    for (int k = 0; k < kV; ++k) {
        const unsigned long long x = v[k];
        v[k] = mine;
        mine += x;
    }
    const unsigned long long ex = scan64(mine, s_w, &tot);
#pragma unroll
    for (int k = 0; k < kV; ++k) {
        const unsigned q = threadIdx.x * kV + k;
        if (q < gridDim.x) sc->bsum[q] = ex + v[k];
    }
    if (threadIdx.x == 0) {
        off[n_hc] = tot;
        sc->done_alloc = 0u;  // (see done_sum)
    }
}

template <bool VEC>
__global__ void __launch_bounds__(256) ks_offsets(const uint32_t *n_h, uint64_t n_hc,
                                                  uint64_t *off, StaticScratch *sc) {
    __shared__ unsigned long long s_w[8];
    vp::pdl_wait();
    // (whatever overlapping calls may have left: the last of their calls to get
    // here leaves zeros, every kernel of theirs that counts being done)
    if (blockIdx.x == 0 && threadIdx.x == 0) sc->done_sum = sc->done_alloc = 0u;
    if (!vp::finite_bits(__ldcg(&sc->sum_d))) return;
    const uint64_t h0 = (uint64_t)blockIdx.x * 1024 + 4u * threadIdx.x;
    const bool full = h0 + 4 <= n_hc;
    uint32_t n[4];
    if (VEC && full) {
        const uint4 v = *(const uint4 *)(n_h + h0);
        n[0] = v.x; n[1] = v.y; n[2] = v.z; n[3] = v.w;
    } else {
#pragma unroll
        for (int q = 0; q < 4; ++q) n[q] = h0 + q < n_hc ? n_h[h0 + q] : 0u;
    }
    const unsigned long long blk = __ldcg(sc->bsum + blockIdx.x);
    unsigned long long tot;
    const unsigned long long e0 =
        blk + scan64((unsigned long long)n[0] + n[1] + n[2] + n[3], s_w, &tot);
    const unsigned long long e1 = e0 + n[0], e2 = e1 + n[1], e3 = e2 + n[2];
    if (VEC && full) {
        ulonglong2 *o = (ulonglong2 *)(off + h0);
        o[0] = make_ulonglong2(e0, e1);
        o[1] = make_ulonglong2(e2, e3);
    } else {
        if (h0 < n_hc) off[h0] = e0;
        if (h0 + 1 < n_hc) off[h0 + 1] = e1;
        if (h0 + 2 < n_hc) off[h0 + 2] = e2;
        if (h0 + 3 < n_hc) off[h0 + 3] = e3;
    }
}

template <typename... KArgs, typename... Args>
cudaError_t launch256(void (*k)(KArgs...), unsigned blocks, cudaStream_t s, Args... args) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(blocks);
    cfg.blockDim = dim3(256);
    cfg.stream = s;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, k, args...);
}

// Device address of the scratch, looked up once per device.
constexpr int kMaxDevices = 64;
std::mutex g_scratch_mu;
StaticScratch *g_scratch_ptr[kMaxDevices] = {};

vp_status scratch_for_current_device(StaticScratch **out) {
    int dev = -1;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) {
        vp::set_error_message(VP_ECUDA, cudaGetErrorString(e));
        return VP_ECUDA;
    }
    if (dev < 0 || dev >= kMaxDevices) {
        vp::set_error_message(VP_EINVAL, "vp_alloc_static: device index beyond 64");
        return VP_EINVAL;
    }
    std::lock_guard<std::mutex> lock(g_scratch_mu);
    if (!g_scratch_ptr[dev]) {
        void *p = nullptr;
        e = cudaGetSymbolAddress(&p, g_alloc_scratch);
        if (e != cudaSuccess || !p) {
            vp::set_error_message(VP_ECUDA, "vp_alloc_static: cudaGetSymbolAddress of the scratch failed");
            return VP_ECUDA;
        }
        g_scratch_ptr[dev] = (StaticScratch *)p;
    }
    *out = g_scratch_ptr[dev];
    return VP_OK;
}

}  // namespace

extern "C" vp_status vp_alloc_static(const double *d_h, int64_t n_hc, int64_t n_ev, int plus2,
                                     uint32_t *n_h, uint64_t *offsets, void *stream) {
    if (!d_h || !n_h || !offsets)
        return vp::set_error_message(VP_EINVAL, "vp_alloc_static: NULL buffer"), VP_EINVAL;
    if (n_hc < 1 || (uint64_t)n_hc > kStaticMaxHc)
        return vp::set_error_message(
                   VP_EINVAL, "vp_alloc_static: n_hc must be 1..4194304 (the static scratch holds "
                              "4096 blocks of 1024 hypercubes)"),
               VP_EINVAL;
    // every n_h is at most floor(N_ev) (+ 2 with plus2) and is stored as a
    // 32-bit integer: larger N_ev would not fit (the contexts bound N_ev more
    // tightly still, through the Philox counter)
    if (n_ev < 2 || n_ev > (int64_t)0xFFFFFFFFll - 2)
        return vp::set_error_message(VP_EINVAL, "vp_alloc_static: n_ev must be 2 .. 4294967293"),
               VP_EINVAL;
    StaticScratch *sc = nullptr;
    vp_status st = scratch_for_current_device(&sc);
    if (st != VP_OK) return st;
    cudaStream_t s = (cudaStream_t)stream;
    const unsigned blocks = (unsigned)(((uint64_t)n_hc + 1023) / 1024);
    const bool vec = (((uintptr_t)d_h | (uintptr_t)n_h | (uintptr_t)offsets) & 15u) == 0;
    cudaError_t e = launch256(ks_sum, blocks, s, d_h, (uint64_t)n_hc, (double)n_ev, sc);
    if (e == cudaSuccess)
        e = launch256(vec ? ks_alloc<true> : ks_alloc<false>, blocks, s, d_h, (uint64_t)n_hc,
                      (double)n_ev, plus2 ? 1 : 0, n_h, offsets, sc);
    if (e == cudaSuccess)
        e = launch256(vec ? ks_offsets<true> : ks_offsets<false>, blocks, s,
                      (const uint32_t *)n_h, (uint64_t)n_hc, offsets, sc);
    if (e != cudaSuccess) {
        vp::set_error_message(VP_ECUDA, cudaGetErrorString(e));
        return VP_ECUDA;
    }
    return VP_OK;
}
