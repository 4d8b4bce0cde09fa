// su3.cu -- the lattice-wide colour-matrix product C[x] = A[x] B[x] of the
// paper's SU(3) matrix-matrix benchmark (Sec. 3.3, Fig. 4a-c).
//
// Layout: n 3x3 complex matrices [x][row][col]{re, im}, the paper's array of
// two-element structures; 144 bytes per FP64 matrix, 72 per FP32 matrix.
// A persistent block walks tiles of TS consecutive matrices:
//   * one thread moves the tile of A and the tile of B into one of two
//     shared-memory stages with bulk asynchronous copies (cp.async.bulk, the
//     one-dimensional TMA path), which complete on that stage's mbarrier;
//     the copies of the next tile are in flight while this one is multiplied;
//   * thread t multiplies matrix t of the tile.  Its shared-memory reads have
//     a stride of 72 or 144 bytes, which touches every bank once per phase;
//   * the products go to one of two output buffers (FP64: over the tile of A),
//     which one thread writes back with a bulk store.
// FP32 is bound by HBM bandwidth (216 bytes and 198 flop per matrix).  FP64
// would be bound by the FP64 units: 198 flop take longer at GB300's FP64 rate
// than its 432 bytes take to move.  Matrices of SU(3) scale are therefore
// multiplied in fixed point on the integer units, but for the few reals that
// these would give less precisely.  Every barrier wait is bounded; a wait that runs
// out is counted in g_wait_timeouts and its block stops.  Before it returns,
// the block waits (bounded again) for the copies it issued into its other
// stage, and for its bulk stores, so that no copy into its shared memory is
// left in flight.  The copies of the stage whose wait ran out are not waited
// for a second time: that wait already lasted about a second, while a tile's
// copies take microseconds.
#include <cuda_runtime.h>

#include <algorithm>
#include <cstdint>

#include "fixed.cuh"
#include "lqcd.h"
#include "lqcd_internal.cuh"
#include "trace.h"

namespace lq {

__device__ unsigned g_wait_timeouts;

namespace {

template <typename T>
struct Cx2;
template <>
struct Cx2<double> {
    using type = double2;
};
template <>
struct Cx2<float> {
    using type = float2;
};

__device__ __forceinline__ uint32_t smem_u32(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }

__device__ __forceinline__ void mbar_init(uint32_t bar, uint32_t count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(count) : "memory");
}

__device__ __forceinline__ void mbar_arrive_expect_tx(uint32_t bar, uint32_t bytes) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes) : "memory");
}

__device__ __forceinline__ uint64_t globaltimer_ns() {
    uint64_t t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}

// Poll the barrier's phase; false once about a second has passed without
// completion (the iteration cap is a second bound should the timer stall).
__device__ __forceinline__ bool mbar_wait_bounded(uint32_t bar, uint32_t parity) {
    const uint64_t t0 = globaltimer_ns();
    for (int i = 0; i < (1 << 26); ++i) {
        uint32_t done;
        asm volatile(
            "{\n\t.reg .pred p;\n\t"
            "mbarrier.test_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
            "selp.u32 %0, 1, 0, p;\n\t}"
            : "=r"(done)
            : "r"(bar), "r"(parity)
            : "memory");
        if (done) return true;
        if ((i & 255) == 255 && globaltimer_ns() - t0 > 1000000000ull) return false;
        __nanosleep(32);
    }
    return false;
}

__device__ __forceinline__ void bulk_load(uint32_t dst, const void* src, uint32_t bytes, uint32_t bar) {
    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(dst),
                 "l"(src), "r"(bytes), "r"(bar)
                 : "memory");
}

__device__ __forceinline__ void bulk_store(void* dst, uint32_t src, uint32_t bytes) {
    asm volatile("cp.async.bulk.global.shared::cta.bulk_group [%0], [%1], %2;" ::"l"(dst), "r"(src), "r"(bytes)
                 : "memory");
}

template <typename T2>
__device__ __forceinline__ void su3_product(const T2 (&a)[9], const T2 (&b)[9], T2 (&c)[9]) {
#pragma unroll
    for (int i = 0; i < 3; ++i) {
#pragma unroll
        for (int j = 0; j < 3; ++j) {
            T2 s;
            s.x = a[3 * i].x * b[j].x - a[3 * i].y * b[j].y;
            s.y = a[3 * i].x * b[j].y + a[3 * i].y * b[j].x;
#pragma unroll
            for (int k = 1; k < 3; ++k) {
                s.x = fma(a[3 * i + k].x, b[3 * k + j].x, s.x);
                s.x = fma(-a[3 * i + k].y, b[3 * k + j].y, s.x);
                s.y = fma(a[3 * i + k].x, b[3 * k + j].y, s.y);
                s.y = fma(a[3 * i + k].y, b[3 * k + j].x, s.y);
            }
            c[3 * i + j] = s;
        }
    }
}

// The FP64 product in fixed point (fixed.cuh): every real of A and B (at most 1) is cut to a
// multiple of 2^-59, and a real of C is a sum of six products, lo lo parts left out, rounded once.
// Before that rounding it is 2^-58.2 off as a standard deviation (exact-integer restatement on random and
// smooth links; worst case 12.5 2^-58, for SU(3) 9 2^-58).  An FP64 sum is some u = 2^-53 times S off,
// the sum of the six products' absolute values (worst case 6 u S).  So that no real has less precision
// than in FP64, those with S < 1/32 (there 0.87 u S, worst case 12.5) are formed with the FP64 unit, and so
// are all of a pair that holds a real above 1 or more than kSu3Few such.  Largest error over S measured,
// on random and smooth links exp(i eps H), eps 0.3 to 1e-6: 4.3 u, as with the FP64 unit alone
// (a line at 1/64: 6.5 u, at 1/16 4.3 u).
//
// 108 FP64 instructions at 77 clocks a warp and SM sub-partition compare with about 1,800 integer and FP32
// ones here.  48^4, smooth links: 991 us in FP64, 501 us here (467 where no sum is small, 421 without
// the sums S; 0.68 of the HBM time of its bytes), with three blocks an SM and in place.  Where all of every pair
// goes to the FP64 unit: 1027-1045 us; A = 1 and a smooth B 1049.  S after the fixed-point product: 483 and
// 1190-1207 us.  lo lo included, which would allow a line at 1/64: 534 us.
constexpr float kSu3Weak = 1.0f / 32;
constexpr int kSu3Few = 8;  // weak reals of a pair that are formed one at a time, not with all of it

__device__ __forceinline__ uint4 load16(const double2* p) { return *reinterpret_cast<const uint4*>(p); }

// |x| of a double below 2 in FP32, from its high word; 2^-60 for anything smaller
__device__ __forceinline__ float abs_cut(uint32_t hi) {
    return __int_as_float(max((int)(hi & 0x7fffffffu) - 0x38000000, 0x04300000) << 3);
}

// One bit for each real of A B (2 (3 i + j) + {re, im}) with S < kSu3Weak; top: the largest
// high word of the two matrices (max_hi).
__device__ __forceinline__ uint32_t su3_weak(const double2* a, const double2* b, float& top) {
    cplx<float> x[9];
    top = 0.f;
#pragma unroll
    for (int k = 0; k < 9; ++k) {
        const uint4 v = load16(a + k);
        top = max_hi(top, v.y, v.w);
        x[k] = {abs_cut(v.y), abs_cut(v.w)};
    }
    uint32_t weak = 0;
#pragma unroll
    for (int j = 0; j < 3; ++j) {
        cplx<float> y[3];
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            const uint4 v = load16(b + 3 * k + j);
            top = max_hi(top, v.y, v.w);
            y[k] = {abs_cut(v.y), abs_cut(v.w)};
        }
#pragma unroll
        for (int i = 0; i < 3; ++i) {
            cplx<float> s = {0.f, 0.f};
#pragma unroll
            for (int k = 0; k < 3; ++k) {
                fma2(s, x[3 * i + k].re, y[k]);
                fma2(s, x[3 * i + k].im, cplx<float>{y[k].im, y[k].re});
            }
            if (s.re < kSu3Weak) weak |= 1u << 2 * (3 * i + j);
            if (s.im < kSu3Weak) weak |= 2u << 2 * (3 * i + j);
        }
    }
    return weak;
}

// Those of the reals in `weak` that have a product of two nonzero factors (the others are zero).
__device__ __noinline__ uint32_t su3_nonzero(const double2* a, const double2* b, uint32_t weak) {
    uint32_t ar = 0, ai = 0, br = 0, bi = 0;  // bit 3 i + k of A, 3 j + k of B
    auto bit = [](uint32_t lo, uint32_t hi, int k) { return ((lo | hi << 1) != 0 ? 1u : 0u) << k; };
#pragma unroll
    for (int k = 0; k < 9; ++k) {
        const uint4 x = load16(a + k), y = load16(b + k);
        const int t = 3 * (k % 3) + k / 3;
        ar |= bit(x.x, x.y, k);
        ai |= bit(x.z, x.w, k);
        br |= bit(y.x, y.y, t);
        bi |= bit(y.z, y.w, t);
    }
    uint32_t some = 0;
#pragma unroll
    for (int i = 0; i < 3; ++i) {
#pragma unroll
        for (int j = 0; j < 3; ++j) {
            const uint32_t xr = ar >> 3 * i, xi = ai >> 3 * i, yr = br >> 3 * j, yi = bi >> 3 * j;
            if (((xr & yr) | (xi & yi)) & 7u) some |= 1u << 2 * (3 * i + j);
            if (((xr & yi) | (xi & yr)) & 7u) some |= 2u << 2 * (3 * i + j);
        }
    }
    return weak & some;
}

// Real e of A B with the FP64 unit.
__device__ __noinline__ double su3_real(const double2* a, const double2* b, int e) {
    const int i = e / 6, j = (e >> 1) % 3;
    const bool im = e & 1;
    double s = 0;
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        const double2 x = a[3 * i + k], y = b[3 * k + j];
        s = fma(x.x, im ? y.y : y.x, s);
        s = fma(im ? x.y : -x.y, im ? y.x : y.y, s);
    }
    return s;
}

__device__ __forceinline__ bool su3_product_fixed(const double2* a, const double2* b, double2 (&c)[9]) {
    constexpr int EB = 1022;
    constexpr uint32_t E2 = ((uint32_t)EB << 21) + 0x1fffffu + (5u << 21);
    constexpr int kOne = 0x3ff00001;
    float top;
    uint32_t weak = su3_weak(a, b, top);
    if (!(__float_as_int(top) <= kOne)) return false;
    if (__popc(weak) > kSu3Few) {
        weak = su3_nonzero(a, b, weak);
        if (__popc(weak) > kSu3Few) return false;
    }
    Fix2 fa[18];
#pragma unroll
    for (int i = 0; i < 3; ++i) {
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            fa[6 * i + k] = fix_one(words(a[3 * i + k].x), E2, 0);
            fa[6 * i + 3 + k] = fix_one(words(a[3 * i + k].y), E2, 0);
        }
    }
#pragma unroll
    for (int j = 0; j < 3; ++j) {
        Fix2 x[6], y[6];  // column j as the factors of the real and of the imaginary part
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            x[k] = y[3 + k] = fix_one(words(b[3 * k + j].x), E2, 0);
            y[k] = fix_one(words(b[3 * k + j].y), E2, 0);
            x[3 + k] = {-y[k].hi, -y[k].lo};
        }
#pragma unroll
        for (int i = 0; i < 3; ++i) {
            const Fix2 u[6] = {fa[6 * i], fa[6 * i + 1], fa[6 * i + 2], fa[6 * i + 3], fa[6 * i + 4], fa[6 * i + 5]};
            // units of 2^60 / 2^118 = 2^-58
            c[3 * i + j] = make_double2(fix_to_double(fix_dot(u, x), 1021, 0u), fix_to_double(fix_dot(u, y), 1021, 0u));
        }
    }
    while (weak) {
        const int e = __ffs((int)weak) - 1;
        weak &= weak - 1;
        const double v = su3_real(a, b, e);
#pragma unroll
        for (int k = 0; k < 9; ++k) {
            if (e == 2 * k) c[k].x = v;
            if (e == 2 * k + 1) c[k].y = v;
        }
    }
    return true;
}

// Shared memory: stage s holds the tile of A at 2*s*TB and of B at (2*s+1)*TB,
// output buffer o at (4+o)*TB, the two stage barriers after them.  FP64 has no output
// buffers: a thread writes its product over its own matrix of A, and the stage is filled
// again once the store has read it.  That leaves room for 3 blocks an SM instead of 2,
// which the integer product needs to hide its latencies (see su3_product_fixed).
template <typename T, int TS>
struct Su3Cfg {
    using T2 = typename Cx2<T>::type;
    static constexpr bool IN_PLACE = sizeof(T) == 8;
    static constexpr int MB = 9 * (int)sizeof(T2);  // bytes per matrix
    static constexpr int TB = TS * MB;              // bytes per tile
    static constexpr int BARS = (IN_PLACE ? 4 : 6) * TB;
    static constexpr int SMEM = BARS + 16;
};

// stall != 0 (testing only) arms each stage barrier for 16 more bytes than its
// copies bring, so that the bounded wait runs out.
template <typename T, int TS>
__global__ void __launch_bounds__(TS, sizeof(T) == 8 ? 3 : 1) su3_mul_kernel(const char* A, const char* B, char* C, long n, int stall) {
    using Cfg = Su3Cfg<T, TS>;
    using T2 = typename Cfg::T2;
    constexpr int MB = Cfg::MB, TB = Cfg::TB;
    extern __shared__ __align__(128) unsigned char sm[];
    __shared__ int s_ok;
    uint64_t* bars = reinterpret_cast<uint64_t*>(sm + Cfg::BARS);
    const int t = threadIdx.x;
    const long ntiles = (n + TS - 1) / TS;
    // matrices of a tile, and those moved by the bulk copies: a bulk copy moves a
    // multiple of 16 bytes, so an odd last FP32 matrix goes by plain loads and stores
    auto count = [&](long tile) { return (int)(n - tile * TS < TS ? n - tile * TS : TS); };
    auto bulk = [&](int cnt) { return (sizeof(T) == 4 && (cnt & 1)) ? cnt - 1 : cnt; };
    auto issue = [&](long tile, int s) {
        const uint32_t bytes = (uint32_t)bulk(count(tile)) * MB;
        const uint32_t bar = smem_u32(&bars[s]);
        mbar_arrive_expect_tx(bar, 2 * bytes + (stall ? 16u : 0u));
        if (bytes) {
            bulk_load(smem_u32(sm + 2 * s * TB), A + tile * TB, bytes, bar);
            bulk_load(smem_u32(sm + (2 * s + 1) * TB), B + tile * TB, bytes, bar);
        }
    };
    if (t == 0) {
        mbar_init(smem_u32(&bars[0]), 1);
        mbar_init(smem_u32(&bars[1]), 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        for (int s = 0; s < 2; ++s) {
            const long tile = blockIdx.x + (long)s * gridDim.x;
            if (tile < ntiles) issue(tile, s);
        }
    }
    int it = 0;
    for (long tile = blockIdx.x; tile < ntiles; tile += gridDim.x, ++it) {
        const int s = it & 1;
        if (t == 0) {
            const bool ok = mbar_wait_bounded(smem_u32(&bars[s]), (uint32_t)((it >> 1) & 1));
            if (!ok) atomicAdd(&g_wait_timeouts, 1u);
            s_ok = ok;
        }
        __syncthreads();  // the tile is visible to every thread (or the wait ran out)
        if (!s_ok) {
            // drain the other stage: its tile's copies were issued one iteration ago
            if (t == 0 && tile + gridDim.x < ntiles &&
                !mbar_wait_bounded(smem_u32(&bars[s ^ 1]), (uint32_t)(((it + 1) >> 1) & 1)))
                atomicAdd(&g_wait_timeouts, 1u);
            break;
        }
        const int cnt = count(tile), nb = bulk(cnt);
        unsigned char* cbuf = sm + (Cfg::IN_PLACE ? 2 * s : 4 + (it & 1)) * TB;
        if (t < cnt) {
            T2 c[9];
            const T2* pa = t < nb ? reinterpret_cast<const T2*>(sm + 2 * s * TB + t * MB)
                                  : reinterpret_cast<const T2*>(A + (tile * TS + t) * MB);
            const T2* pb = t < nb ? reinterpret_cast<const T2*>(sm + (2 * s + 1) * TB + t * MB)
                                  : reinterpret_cast<const T2*>(B + (tile * TS + t) * MB);
            bool done = false;
            if constexpr (sizeof(T) == 8) done = su3_product_fixed(pa, pb, c);
            if (!done) {
                T2 a[9], b[9];
#pragma unroll
                for (int k = 0; k < 9; ++k) {
                    a[k] = pa[k];
                    b[k] = pb[k];
                }
                su3_product(a, b, c);
            }
            T2* pc = t < nb ? reinterpret_cast<T2*>(cbuf + t * MB) : reinterpret_cast<T2*>(C + (tile * TS + t) * MB);
#pragma unroll
            for (int k = 0; k < 9; ++k) pc[k] = c[k];
        }
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");  // C buffer -> bulk-store reads
        __syncthreads();  // every thread is done with stage s and has written the C buffer
        if (t == 0) {
            if (nb) bulk_store(C + tile * TB, smem_u32(cbuf), (uint32_t)nb * MB);
            asm volatile("cp.async.bulk.commit_group;" ::: "memory");
            const long next = tile + 2L * gridDim.x;
            if (Cfg::IN_PLACE) asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory");
            if (next < ntiles) issue(next, s);
            // the store issued one iteration ago has read the buffer the next iteration fills
            if (!Cfg::IN_PLACE) asm volatile("cp.async.bulk.wait_group.read 1;" ::: "memory");
        }
    }
    if (t == 0) asm volatile("cp.async.bulk.wait_group 0;" ::: "memory");
}

template <typename T, int TS>
int launch_su3(void* C, const void* A, const void* B, long n, cudaStream_t st, int stall = 0) {
    using Cfg = Su3Cfg<T, TS>;
    auto kern = su3_mul_kernel<T, TS>;
    static int grid_max = 0;  // resident blocks on this device, found once
    if (!grid_max) {
        int dev = 0, sms = 0, per_sm = 0;
        if (cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, Cfg::SMEM) != cudaSuccess ||
            cudaGetDevice(&dev) != cudaSuccess ||
            cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess ||
            cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, TS, Cfg::SMEM) != cudaSuccess)
            return LQ_ERR_CUDA;
        grid_max = std::max(1, sms * std::max(per_sm, 1));
    }
    const long ntiles = (n + TS - 1) / TS;
    const int grid = (int)std::min<long>(ntiles, grid_max);
    kern<<<grid, TS, Cfg::SMEM, st>>>(static_cast<const char*>(A), static_cast<const char*>(B),
                                      static_cast<char*>(C), n, stall);
    return cudaGetLastError() == cudaSuccess ? LQ_OK : LQ_ERR_CUDA;
}

bool overlaps(const void* p, const void* q, size_t bytes) {
    const uintptr_t a = (uintptr_t)p, b = (uintptr_t)q;
    return a < b + bytes && b < a + bytes;
}

}  // namespace
}  // namespace lq

extern "C" {

int lq_su3_mul(void* C, const void* A, const void* B, long n, int fmt, void* stream) {
    lq::TraceRange trace_("lqcd/su3_mul");
    if (n < 0 || (fmt != LQ_F64 && fmt != LQ_F32)) return LQ_ERR_ARG;
    if (n == 0) return LQ_OK;
    if (!A || !B || !C) return LQ_ERR_ARG;
    if (((uintptr_t)A | (uintptr_t)B | (uintptr_t)C) & 15) return LQ_ERR_LAYOUT;
    const size_t bytes = (size_t)n * (fmt == LQ_F64 ? 144 : 72);
    if ((C != A && lq::overlaps(C, A, bytes)) || (C != B && lq::overlaps(C, B, bytes))) return LQ_ERR_ARG;
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    return fmt == LQ_F64 ? lq::launch_su3<double, 128>(C, A, B, n, st) : lq::launch_su3<float, 256>(C, A, B, n, st);
}

int lq_test_stalled_wait(void) {
    // one tile of zero matrices, product kernel with its barrier armed for bytes that never come
    const long n = 256;
    void* buf = nullptr;
    if (cudaMalloc(&buf, 3 * 72 * n) != cudaSuccess) {
        cudaGetLastError();
        return LQ_ERR_NOMEM;
    }
    char* p = static_cast<char*>(buf);
    int rc = cudaMemset(buf, 0, 3 * 72 * n) == cudaSuccess ? LQ_OK : LQ_ERR_CUDA;
    if (rc == LQ_OK) rc = lq::launch_su3<float, 256>(p + 2 * 72 * n, p, p + 72 * n, n, nullptr, 1);
    if (rc == LQ_OK && cudaDeviceSynchronize() != cudaSuccess) rc = LQ_ERR_CUDA;
    cudaFree(buf);
    return rc;
}

int lq_wait_timeouts(unsigned* count) {
    if (!count) return LQ_ERR_ARG;
    unsigned v = 0;
    const unsigned zero = 0;
    if (cudaDeviceSynchronize() != cudaSuccess ||
        cudaMemcpyFromSymbol(&v, lq::g_wait_timeouts, sizeof v) != cudaSuccess ||
        cudaMemcpyToSymbol(lq::g_wait_timeouts, &zero, sizeof zero) != cudaSuccess)
        return LQ_ERR_CUDA;
    *count = v;
    return v ? LQ_ERR_TIMEOUT : LQ_OK;
}

}  // extern "C"
