// convert.cu -- layout and precision conversions: the documented site-major
// exchange layout <-> the native structure-of-arrays blocks the hop streams,
// precision changes between native fields, and gauge-link packing (with the
// optional two-row compression).  The paper's Gridarray layout (Sec. 3.1)
// keeps one degree of freedom of many sites contiguous so that whole SIMD
// registers load at once; the native layout does the same for a warp.
#include <algorithm>
#include <cstring>

#include "lqcd_kernels.h"
#include "pdl.cuh"

namespace lq {

namespace {

template <int SP, typename T>
__device__ __forceinline__ void load_sm(const void* base, size_t site, cplx<T> (&s)[12]) {
    if constexpr (SP == LQ_F64) {
        const double2* q = reinterpret_cast<const double2*>(base) + site * 12;
#pragma unroll
        for (int k = 0; k < 12; ++k) {
            double2 v = q[k];
            s[k] = {(T)v.x, (T)v.y};
        }
    } else {
        const float4* q = reinterpret_cast<const float4*>(base) + site * 6;
#pragma unroll
        for (int k = 0; k < 6; ++k) {
            float4 v = q[k];
            s[2 * k] = {(T)v.x, (T)v.y};
            s[2 * k + 1] = {(T)v.z, (T)v.w};
        }
    }
}

constexpr int kBlock = 128;

// Arithmetic of a conversion: FP64 only where both sides are FP64 or one is and the other holds
// FP32 values to widen or round; FP32 otherwise (FP32 -> FP64 -> FP32 costs two conversions a real
// on the FP64 unit and changes nothing).
template <int DP, int SP>
using ConvT = typename std::conditional<DP == LQ_F64 || SP == LQ_F64, double, float>::type;

// grid.y = rhs * nparity + parity index
template <int DP, int SP>
__global__ void __launch_bounds__(kBlock) spinor_to_native_kernel(char* nat, const void* sm, Geom g, bool full,
                                                                  int parity, int nparity) {
    pdl_enter();
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= g.Vh) return;
    const int pi = blockIdx.y % nparity;
    const int rhs = blockIdx.y / nparity;
    const int p = full ? pi : parity;
    const size_t nsites_sm = full ? 2 * (size_t)g.Vh : (size_t)g.Vh;
    const size_t site = (size_t)rhs * nsites_sm + (full ? lexi_of(g, i, p) : (size_t)i);
    char* blk = nat + ((size_t)rhs * nparity + pi) * (size_t)spinor_site_bytes(DP) * g.Vh;
    cplx<ConvT<DP, SP>> s[12];
    load_sm<SP>(sm, site, s);
    store_spinor<DP>(blk, g.Vh, i, s);
}

// The site-major side is written through shared memory, so that a warp's stores cover whole
// sites (192 or 96 consecutive bytes): a thread that wrote its own site put 16 bytes into each of
// 32 lines with every store (32^4, FP64: 182 us for 403 MB, here 82 us; FP32 to FP32 88 and 41 us).
// A site's slot is 16 bytes longer than the site, which keeps both sides free of bank conflicts.
template <int NP, int SP>
__global__ void __launch_bounds__(kBlock) spinor_from_native_kernel(void* sm, const char* nat, Geom g, bool full,
                                                                    int parity, int nparity) {
    using T = ConvT<NP, SP>;
    constexpr int CH = SP == LQ_F64 ? 12 : 6;  // 16-byte chunks of a site
    constexpr int PITCH = CH + 1;
    __shared__ uint4 slots[kBlock * PITCH];
    __shared__ size_t where[kBlock];
    // No early start of the next launch (pdl_enter): a spinor_to_native_kernel that follows would find
    // L1 cut to what this kernel's shared memory leaves (16^4, FP64: 53.2 against 50.1 us).
    asm volatile("griddepcontrol.wait;" ::: "memory");
    const int t = threadIdx.x, w = t & ~31, lane = t & 31;
    const int i = blockIdx.x * kBlock + t;
    const int pi = blockIdx.y % nparity;
    const int rhs = blockIdx.y / nparity;
    const int p = full ? pi : parity;
    if (blockIdx.x * kBlock + w >= g.Vh) return;  // the warp's first site
    if (i < g.Vh) {
        const size_t nsites_sm = full ? 2 * (size_t)g.Vh : (size_t)g.Vh;
        where[t] = (size_t)rhs * nsites_sm + (full ? lexi_of(g, i, p) : (size_t)i);
        cplx<T> s[12];
        load_spinor<NP>(nat + ((size_t)rhs * nparity + pi) * (size_t)spinor_site_bytes(NP) * g.Vh, g.Vh, i, s);
        if constexpr (SP == LQ_F64) {
            double2* q = reinterpret_cast<double2*>(slots + t * PITCH);
#pragma unroll
            for (int k = 0; k < 12; ++k) q[k] = make_double2(s[k].re, s[k].im);
        } else {
            float4* q = reinterpret_cast<float4*>(slots + t * PITCH);
#pragma unroll
            for (int k = 0; k < 6; ++k)
                q[k] = make_float4((float)s[2 * k].re, (float)s[2 * k].im, (float)s[2 * k + 1].re,
                                   (float)s[2 * k + 1].im);
        }
    }
    __syncwarp();
    const int sites = min(32, g.Vh - (int)blockIdx.x * kBlock - w);
#pragma unroll
    for (int k = 0; k < CH; ++k) {
        const int c = k * 32 + lane, j = c / CH, part = c - j * CH;
        if (j < sites) reinterpret_cast<uint4*>(sm)[where[w + j] * CH + part] = slots[(w + j) * PITCH + part];
    }
}

template <int DP, int SP>
__global__ void native_convert_kernel(char* dst, const char* src, int Vh) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= Vh) return;
    const char* sb = src + (size_t)blockIdx.y * spinor_site_bytes(SP) * Vh;
    char* db = dst + (size_t)blockIdx.y * spinor_site_bytes(DP) * Vh;
    cplx<float> sf[12];
    cplx<double> sd[12];
    if constexpr (SP == LQ_F64 || DP == LQ_F64) {
        load_spinor<SP, double>(sb, Vh, i, sd);
        store_spinor<DP, double>(db, Vh, i, sd);
    } else {
        load_spinor<SP, float>(sb, Vh, i, sf);
        store_spinor<DP, float>(db, Vh, i, sf);
    }
}

// FIXED: the fixed-point records of hop_fixed.cuh (DP = LQ_F64)
template <int DP, bool R12, int SP, bool FIXED = false>
__global__ void links_kernel(char* dst, const void* src, Geom g, size_t link_block) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= g.Vh) return;
    const int p = blockIdx.y;
    const size_t site = lexi_of(g, i, p);
#pragma unroll
    for (int mu = 0; mu < 4; ++mu) {
        cplx<double> u[9];
        const size_t base = (site * 4 + mu) * 9;
#pragma unroll
        for (int k = 0; k < 9; ++k) {
            if constexpr (SP == LQ_F64) {
                double2 v = reinterpret_cast<const double2*>(src)[base + k];
                u[k] = {v.x, v.y};
            } else {
                float2 v = reinterpret_cast<const float2*>(src)[base + k];
                u[k] = {(double)v.x, (double)v.y};
            }
        }
        if constexpr (FIXED) store_link_fixed(dst + (size_t)(p * 4 + mu) * link_block, g.Vh, i, u);
        else store_link<DP, R12>(dst + (size_t)(p * 4 + mu) * link_block, g.Vh, i, u);
    }
}

// Largest deviation of a link from SU(3): max over the entries of |U^dag U - 1|
// and |det U - 1|, in FP64.  Two-row compression rebuilds row 3 as
// conj(row 1 x row 2), which is row 3 only for a special unitary matrix.
template <int SP>
__global__ void link_su3_deviation_kernel(const void* src, long nlinks, unsigned long long* out) {
    double dev = 0.0;
    for (long l = (long)blockIdx.x * blockDim.x + threadIdx.x; l < nlinks; l += (long)gridDim.x * blockDim.x) {
        cplx<double> u[9];
#pragma unroll
        for (int k = 0; k < 9; ++k) {
            if constexpr (SP == LQ_F64) {
                const double2 v = reinterpret_cast<const double2*>(src)[l * 9 + k];
                u[k] = {v.x, v.y};
            } else {
                const float2 v = reinterpret_cast<const float2*>(src)[l * 9 + k];
                u[k] = {(double)v.x, (double)v.y};
            }
        }
        // d = the largest |.| seen; fmax would drop a NaN, so NaNs are tracked in nan_seen
        double d = 0.0;
        bool nan_seen = false;
        auto take = [&](cplx<double> z) {
            const double v = sqrt(z.re * z.re + z.im * z.im);
            nan_seen = nan_seen || !(v == v);
            d = v > d ? v : d;
        };
#pragma unroll
        for (int i = 0; i < 3; ++i) {
#pragma unroll
            for (int j = 0; j < 3; ++j) {
                cplx<double> g = {i == j ? -1.0 : 0.0, 0.0};  // (U^dag U)_ij - delta_ij
#pragma unroll
                for (int k = 0; k < 3; ++k) cmac_conj(g, u[3 * k + i], u[3 * k + j]);
                take(g);
            }
        }
        // det U by the first row's cofactors
        cplx<double> m0 = {0, 0}, m1 = {0, 0}, m2 = {0, 0};
        cmac(m0, u[4], u[8]);
        cmac(m0, cneg(u[5]), u[7]);
        cmac(m1, u[5], u[6]);
        cmac(m1, cneg(u[3]), u[8]);
        cmac(m2, u[3], u[7]);
        cmac(m2, cneg(u[4]), u[6]);
        cplx<double> det = {-1.0, 0.0};
        cmac(det, u[0], m0);
        cmac(det, u[1], m1);
        cmac(det, u[2], m2);
        take(det);
        if (nan_seen) d = __longlong_as_double(0x7ff0000000000000LL);  // NaN counts as infinitely far
        dev = fmax(dev, d);
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) dev = fmax(dev, __shfl_xor_sync(0xffffffffu, dev, o));
    // non-negative doubles order like their bit patterns
    if ((threadIdx.x & 31) == 0) atomicMax(out, (unsigned long long)__double_as_longlong(dev));
}

// |v| cut to FP32 without the FP64 unit (4 for |v| >= 2, infinities and NaNs; 0 below 2^-126)
__device__ __forceinline__ float abs_f32(double v) {
    const unsigned h = (unsigned)__double2hiint(v) & 0x7fffffffu;
    if (h >= 0x40000000u) return 4.0f;
    if (h < 0x38100000u) return 0.0f;
    return __uint_as_float(((h - 0x38000000u) << 3) | ((unsigned)__double2loint(v) >> 29));
}
__device__ __forceinline__ float abs_f32(float v) { return fabsf(v) < 2.0f ? fabsf(v) : 4.0f; }

__device__ __forceinline__ bool nonzero(double v) {
    return (((unsigned)__double2hiint(v) << 1) | (unsigned)__double2loint(v)) != 0;
}
__device__ __forceinline__ bool nonzero(float v) { return v != 0.0f; }

// The links that the fixed-point FP64 hop cannot take.  Its sums are bounded for entries up to 1 and
// rows and columns of 1-norm up to 2.75 (SU(3): sqrt 6), and it keeps an entry to 2^-59, which is
// enough where every row and column holds a real of at least 1/4 (SU(3): 1/sqrt 6) and loses
// digits for links of a smaller scale.  A link that is exactly zero (an open boundary) is exact.
template <typename T>
__global__ void link_fixed_check_kernel(const T* src, long nlinks, unsigned* bad) {
    unsigned n = 0;
    for (long l = (long)blockIdx.x * blockDim.x + threadIdx.x; l < nlinks; l += (long)gridDim.x * blockDim.x) {
        float row[3] = {}, col[3] = {}, row_max[3] = {}, col_max[3] = {};
        bool ok = true, zero = true;
#pragma unroll
        for (int k = 0; k < 18; ++k) {
            const T v = src[l * 18 + k];
            const float f = abs_f32(v);
            zero = zero && !nonzero(v);
            ok = ok && f <= 1.000001f;
            row[k / 6] += f;
            col[k / 2 % 3] += f;
            row_max[k / 6] = fmaxf(row_max[k / 6], f);
            col_max[k / 2 % 3] = fmaxf(col_max[k / 2 % 3], f);
        }
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            ok = ok && row[k] <= 2.75f && col[k] <= 2.75f;
            ok = ok && row_max[k] >= 0.25f && col_max[k] >= 0.25f;
        }
        n += ok || zero ? 0 : 1;
    }
    if (n) atomicAdd(bad, n);
}

}  // namespace

#define LQ_DP_SWITCH(dp, BODY)                              \
    switch (dp) {                                           \
    case LQ_F64: { constexpr int DP = LQ_F64; BODY; } break; \
    case LQ_F32: { constexpr int DP = LQ_F32; BODY; } break; \
    case LQ_F16: { constexpr int DP = LQ_F16; BODY; } break; \
    default: { constexpr int DP = LQ_BF16; BODY; } break;    \
    }

// SMs of the current device, found once (0 where that fails)
static int sm_count() {
    static const int sms = [] {
        int dev = 0, n = 0;
        if (cudaGetDevice(&dev) != cudaSuccess ||
            cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess) {
            cudaGetLastError();
            n = 0;
        }
        return n;
    }();
    return sms;
}

// A conversion to or from site-major of up to four blocks per SM is launched as a programmatic
// dependent: what it takes there is the launch (D on FP64 site-major fields, 4^4: 20.5 -> 16.8 us,
// 8^3 x 16: 20.9 -> 18.0, 16^4: 51.6 -> 50.1).  A larger one is not: started beside the end of a hop,
// which holds most of L1 as shared memory, spinor_to_native_kernel lacks the L1 that gathers its 16-byte
// reads into lines (32^4 FP64 after an FP32 hop: 163 -> 227 us for the two).
template <typename... KArgs, typename... Args>
static cudaError_t launch_conversion(void (*kern)(KArgs...), dim3 grid, cudaStream_t st, Args... args) {
    if (grid.x * (size_t)grid.y <= 4 * (size_t)sm_count())
        return launch_pdl(kern, grid, dim3(kBlock), 0, st, args...);
    kern<<<grid, kBlock, 0, st>>>(args...);
    return cudaGetLastError();
}

cudaError_t launch_spinor_to_native(int dst_prec, void* dst, int src_prec, const void* src, const Geom& g, bool full,
                                    int parity, int nrhs, cudaStream_t st) {
    cudaError_t e = cudaSuccess;
    const int np = full ? 2 : 1;
    dim3 grid((g.Vh + kBlock - 1) / kBlock, nrhs * np);
    char* d = static_cast<char*>(dst);
    if (src_prec == LQ_F64) {
        LQ_DP_SWITCH(dst_prec, e = launch_conversion(spinor_to_native_kernel<DP, LQ_F64>, grid, st, d, src, g, full, parity, np))
    } else {
        LQ_DP_SWITCH(dst_prec, e = launch_conversion(spinor_to_native_kernel<DP, LQ_F32>, grid, st, d, src, g, full, parity, np))
    }
    return e;
}

cudaError_t launch_spinor_from_native(int dst_prec, void* dst, int src_prec, const void* src, const Geom& g,
                                      bool full, int parity, int nrhs, cudaStream_t st) {
    cudaError_t e = cudaSuccess;
    const int np = full ? 2 : 1;
    dim3 grid((g.Vh + kBlock - 1) / kBlock, nrhs * np);
    const char* n = static_cast<const char*>(src);
    if (dst_prec == LQ_F64) {
        LQ_DP_SWITCH(src_prec, e = launch_conversion(spinor_from_native_kernel<DP, LQ_F64>, grid, st, dst, n, g, full, parity, np))
    } else {
        LQ_DP_SWITCH(src_prec, e = launch_conversion(spinor_from_native_kernel<DP, LQ_F32>, grid, st, dst, n, g, full, parity, np))
    }
    return e;
}

cudaError_t launch_native_convert(int dst_prec, void* dst, int src_prec, const void* src, int Vh, int nblocks,
                                  cudaStream_t st) {
    dim3 grid((Vh + kBlock - 1) / kBlock, nblocks);
    char* d = static_cast<char*>(dst);
    const char* s = static_cast<const char*>(src);
#define LQ_SP_CASE(SPV)                                                                         \
    case SPV: {                                                                                 \
        LQ_DP_SWITCH(dst_prec, (native_convert_kernel<DP, SPV><<<grid, kBlock, 0, st>>>(d, s, Vh))) \
    } break;
    switch (src_prec) {
        LQ_SP_CASE(LQ_F64)
        LQ_SP_CASE(LQ_F32)
        LQ_SP_CASE(LQ_F16)
        LQ_SP_CASE(LQ_BF16)
    }
#undef LQ_SP_CASE
    return cudaGetLastError();
}

cudaError_t launch_links_to_native(int dst_prec, bool r12, void* dst, int src_prec, const void* src, const Geom& g,
                                   cudaStream_t st) {
    dim3 grid((g.Vh + kBlock - 1) / kBlock, 2);
    const size_t lb = (size_t)link_site_bytes(dst_prec, r12) * g.Vh;
    char* d = static_cast<char*>(dst);
    if (src_prec == LQ_F64) {
        if (r12) { LQ_DP_SWITCH(dst_prec, (links_kernel<DP, true, LQ_F64><<<grid, kBlock, 0, st>>>(d, src, g, lb))) }
        else { LQ_DP_SWITCH(dst_prec, (links_kernel<DP, false, LQ_F64><<<grid, kBlock, 0, st>>>(d, src, g, lb))) }
    } else {
        if (r12) { LQ_DP_SWITCH(dst_prec, (links_kernel<DP, true, LQ_F32><<<grid, kBlock, 0, st>>>(d, src, g, lb))) }
        else { LQ_DP_SWITCH(dst_prec, (links_kernel<DP, false, LQ_F32><<<grid, kBlock, 0, st>>>(d, src, g, lb))) }
    }
    return cudaGetLastError();
}

cudaError_t launch_links_fixed(void* dst, int src_prec, const void* src, const Geom& g, cudaStream_t st) {
    dim3 grid((g.Vh + kBlock - 1) / kBlock, 2);
    const size_t lb = (size_t)link_site_bytes(LQ_F64, false) * g.Vh;
    char* d = static_cast<char*>(dst);
    if (src_prec == LQ_F64) links_kernel<LQ_F64, false, LQ_F64, true><<<grid, kBlock, 0, st>>>(d, src, g, lb);
    else links_kernel<LQ_F64, false, LQ_F32, true><<<grid, kBlock, 0, st>>>(d, src, g, lb);
    return cudaGetLastError();
}

cudaError_t launch_links_fixed_check(int src_prec, const void* src, long nlinks, unsigned* bad, cudaStream_t st) {
    const int grid = (int)std::min<long>((nlinks + 255) / 256, 4096);
    if (src_prec == LQ_F64)
        link_fixed_check_kernel<<<grid, 256, 0, st>>>(static_cast<const double*>(src), nlinks, bad);
    else
        link_fixed_check_kernel<<<grid, 256, 0, st>>>(static_cast<const float*>(src), nlinks, bad);
    return cudaGetLastError();
}

cudaError_t link_su3_deviation(int src_prec, const void* src, long nlinks, double* dev, cudaStream_t st) {
    unsigned long long* d = nullptr;
    cudaError_t e = cudaMalloc(&d, sizeof(*d));
    if (e != cudaSuccess) return e;
    unsigned long long v = 0;
    e = cudaMemsetAsync(d, 0, sizeof(*d), st);
    const int grid = (int)std::min<long>((nlinks + 255) / 256, 4096);
    if (e == cudaSuccess && nlinks > 0) {
        if (src_prec == LQ_F64) link_su3_deviation_kernel<LQ_F64><<<grid, 256, 0, st>>>(src, nlinks, d);
        else link_su3_deviation_kernel<LQ_F32><<<grid, 256, 0, st>>>(src, nlinks, d);
        e = cudaGetLastError();
    }
    if (e == cudaSuccess) e = cudaMemcpyAsync(&v, d, sizeof(v), cudaMemcpyDeviceToHost, st);
    if (e == cudaSuccess) e = cudaStreamSynchronize(st);
    cudaFree(d);
    std::memcpy(dev, &v, sizeof(v));
    return e;
}

}  // namespace lq
