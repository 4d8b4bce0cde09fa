// hop_fixed.cuh -- the FP64 Wilson hop with its products and sums in 64-bit
// fixed point on the integer multipliers.
//
// What bounds the plain FP64 hop (hop.cuh) is the FP64 unit: GB300 issues 1.67
// FP64 lanes per clock and SM (measured), a site needs 864 FP64 instructions,
// so one even-odd hop on 32^4 takes 0.9 ms where its bytes take 0.12 ms.  The
// 32x32+64-bit integer multiply-add runs at 63 lanes per clock and SM
// (measured), 38 times that rate.  Here a site's arithmetic is integer:
//
//   * block floating point: of the 24 reals of a neighbour the largest exponent
//     is found, and each becomes the signed integer x 2^59 / 2^B, 2^B above all
//     neighbours so far, as two words hi * 2^30 + lo (|hi| < 2^29, lo < 2^30), whose
//     spin projection (sums of two) still fits two 32-bit words;
//   * links are packed once as u 2^58 = hi * 2^30 + lo (|lo| <= 2^29);
//   * a real product is three multiply-adds: hi*hi, and hi*lo + lo*hi into a
//     second 64-bit sum that is rounded in at the end of each dot product
//     (lo*lo, at most 2^-57 of the block, is dropped);
//   * the 24 sums over 8 directions are 64-bit integers in units of 2^(B-57).
//     A neighbour larger than 2^B moves the sums to its exponent.
//
// Precision: a sum of 48 products is 2^-56.2 of the block off (standard deviation, exact-integer
// restatement on Gaussian neighbours; worst case 190 2^-58: 96 from lo*lo, 48 from links kept to 2^-59,
// 22 from spinors cut at 2^-59, 24 from rounding 8 products and moving the sums).  The block is 1 to
// 4 times the largest neighbour component.  An FP64 sum is some u = 2^-53 times sum |U| |h| off (worst
// case 15 u).  So that no component has less precision than in FP64, a sum is kept only if its terms
// add up to 1/16 of the block (sizes are summed along with the terms), which is then 1.8 u of it (95 u in
// the worst case); a site with any other goes to slow_site, which sums in FP64 from the links the
// handle was given.  Largest error of a component over
// sum |U| |h|, on dense fields, sources, fields whose spins, colours or sites differ by powers of ten, and
// links near 1: 3.2 u here, 4.0 u in FP64; 7.4 u with a line at 1/32 and 3.2 u with one at 1/8.
// Norm-wise the hop on 8^4 (random and smooth links) is 5.8e-17 off, and 1.5e-16 with the FP64 kernel.
// What is not finite or beyond 2^976 takes slow_site too, and what is below 2^-894, as it is small
// beside the least block.
//
// It needs links with |u| <= 1 and rows and columns of 1-norm <= 2.75 (SU(3): <= 2.45), which
// bounds every sum below 2^63, and with a real of at least 1/4 (link_fixed_check_kernel, when a handle is
// made); other links keep the FP64 kernel.
//
// Layout: two threads a site, one for each spin of the half spinors; lanes 0-15 and 16-31 of a
// warp share 16 sites.  A site's neighbour spinor (192 B) and link (144 B) come by cp.async into
// one shared-memory slot each: the next spinor is requested as soon as this one is converted,
// the next link when this one is used up, so the products (conversions) of a direction cover the
// latency.  With one thread a site, 168 registers and the 8 directions unrolled, the 120 KB of
// code kept warps waiting for instructions (240 us against 215); one looped body with run-time
// directions took 236 us.
//
// Measured: D on 32^3 x 16 (as many sites as an even-odd hop of 32^4): 0.92 ms in FP64, 0.214 ms
// here; its bytes take 0.12 ms.  What bounds it is the integer pipes: without its products,
// conversions and sums the kernel takes 0.123 ms; the multiplier is busy 68 % of the time, the
// ALU 49 %, with warps waiting on fixed latencies (ncu).  The sizes cost 1.3 % of a dense field's
// time.  Where every site takes slow_site (one spin and colour alone on every site): 0.97 ms; the
// zero field 0.234, a point source 0.267.
#pragma once

#include <cuda_pipeline.h>

#include "fixed.cuh"
#include "hop.cuh"

namespace lq {

constexpr int kFixEmin = 128;    // biased exponents the block may have
constexpr int kFixEmax = 2000;
// A sum is kept where its terms, one for each direction, add up to this many 2^-10 of the block
// (larger of the real and the imaginary part of each); others are formed in FP64.  1/16: see above; plain
// FP64 CG from a point source on 16^3 x 32 takes 23.2 ms, 20.4 with a line at 1/32, 30.8 at 1/8 and
// 60.9 with the FP64 kernel.
constexpr int kFixWeak = 64;

// ------------------------------------------------- sites summed in FP64

// z, negated for a set flag
__device__ __forceinline__ cplx<double> flip_sign(cplx<double> z, bool f) {
    const int m = f ? (int)0x80000000 : 0;
    return {__hiloint2double(__double2hiint(z.re) ^ m, __double2loint(z.re)),
            __hiloint2double(__double2hiint(z.im) ^ m, __double2loint(z.im))};
}

// The hop sums of one site with the FP64 unit, from the links as the handle was given them: for
// sums that the fixed-point ones do not hold well enough, and neighbours that are not finite or out
// of their range.  Each of the site's two threads does the half of its spin, so that a warp's
// instructions do as much as those of the FP64 kernel.  To shared memory, NT apart: in s the
// sums of spin s and then those of spin 2 + s without the other thread's part, in l that part.
template <bool DAG, int NT>
__device__ __noinline__ void slow_site(const HopArgs& a, int p, int spin, const char* in, int i, const int* nbr,
                                       int flips, double2* s, double2* l) {
    cplx<double> up[3], lx[3], ly[3];
#pragma unroll
    for (int c = 0; c < 3; ++c) up[c] = lx[c] = ly[c] = {0.0, 0.0};
    const size_t own = lexi_of(a.g, i, p);
    auto dir = [&](auto dtag) {
        constexpr int D = decltype(dtag)::value, MU = D >> 1;
        constexpr bool FWD = (D & 1) == 0;
        constexpr int S = (FWD == DAG) ? 1 : -1;
        const int n = nbr[D * NT];
        const double2* q = reinterpret_cast<const double2*>(in) + n;
        const size_t link = ((FWD ? own : lexi_of(a.g, n, 1 - p)) * 4 + MU) * 9;
        cplx<double> h[3], u[9];
#pragma unroll
        for (int c = 0; c < 3; ++c) {  // the projector, as in project()
            const double2 x = __ldg(q + (size_t)(3 * spin + c) * a.g.Vh);
            const double2 y = __ldg(q + (size_t)((MU < 2 ? 9 - 3 * spin : 6 + 3 * spin) + c) * a.g.Vh);
            cplx<double> z = {y.x, y.y};
            if constexpr (MU == 0) z = cneg(cmul_i(z));
            else if constexpr (MU == 1) z = flip_sign(z, spin == 0);
            else if constexpr (MU == 2) z = flip_sign(cmul_i(z), spin == 0);
            h[c] = flip_sign(cadds<S>(cplx<double>{x.x, x.y}, z), (flips >> D) & 1);
        }
#pragma unroll
        for (int k = 0; k < 9; ++k) {
            if (a.u_f32) {
                const float2 v = __ldg(reinterpret_cast<const float2*>(a.u_sm) + link + k);
                u[k] = {widen(v.x), widen(v.y)};
            } else {
                const double2 v = __ldg(reinterpret_cast<const double2*>(a.u_sm) + link + k);
                u[k] = {v.x, v.y};
            }
        }
#pragma unroll
        for (int c = 0; c < 3; ++c) {  // reconstruct_add()
            cplx<double> w = {0.0, 0.0};
#pragma unroll
            for (int j = 0; j < 3; ++j) {
                if constexpr (FWD) cmac(w, u[3 * c + j], h[j]);
                else cmac_conj(w, u[3 * j + c], h[j]);
            }
            up[c] = cadd(up[c], w);
            if constexpr (MU == 0) lx[c] = cadds<S>(lx[c], cmul_i(w));
            else if constexpr (MU == 1) lx[c] = cadds<S>(lx[c], flip_sign(w, spin == 0));
            else if constexpr (MU == 2) ly[c] = cadds<S>(ly[c], flip_sign(cmul_i(w), spin == 1));
            else ly[c] = cadds<S>(ly[c], w);
        }
    };
    dir(std::integral_constant<int, 0>());
    dir(std::integral_constant<int, 1>());
    dir(std::integral_constant<int, 2>());
    dir(std::integral_constant<int, 3>());
    dir(std::integral_constant<int, 4>());
    dir(std::integral_constant<int, 5>());
    dir(std::integral_constant<int, 6>());
    dir(std::integral_constant<int, 7>());
#pragma unroll
    for (int c = 0; c < 3; ++c) {
        s[(6 * spin + c) * NT] = make_double2(up[c].re, up[c].im);
        s[(6 * spin + 3 + c) * NT] = make_double2(ly[c].re, ly[c].im);
        l[(3 * spin + c) * NT] = make_double2(lx[c].re, lx[c].im);
    }
}

// Do the half spinors of spin `spin` hold anything but zeros?  Nonzero x for the x and y
// directions, y for z and t (there after the projection in FP64, as in the kernel).
template <bool DAG, int NT>
__device__ __noinline__ uint2 nonzero_halves(const HopArgs& a, int spin, const char* in, const int* nbr) {
    uint2 seen = {0, 0};
    auto bits = [](uint4 v) { return v.x | v.z | (v.y | v.w) << 1; };
    for (int d = 0; d < 8; ++d) {
        const uint4* q = reinterpret_cast<const uint4*>(in) + nbr[d * NT];
        const int o = d < 4 ? 9 - 3 * spin : 6 + 3 * spin;
        const bool minus = ((d & 1) == 0) != DAG;
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            uint4 x = __ldg(q + (size_t)(3 * spin + c) * a.g.Vh);
            const uint4 y = __ldg(q + (size_t)(o + c) * a.g.Vh);
            if (d < 4) {
                seen.x |= bits(x) | bits(y);
            } else if (d < 6) {
                seen.y |= bits(x) | bits(y);
            } else {
                const uint32_t f = minus ? 0x80000000u : 0;
                const uint2 re = words(value(make_uint2(x.x, x.y)) + value(make_uint2(y.x, y.y ^ f)));
                const uint2 im = words(value(make_uint2(x.z, x.w)) + value(make_uint2(y.z, y.w ^ f)));
                seen.y |= bits(make_uint4(re.x, re.y, im.x, im.y));
            }
        }
    }
    return seen;
}

// ------------------------------------------------------------------ kernel

constexpr int kFixThreads = 2 * kHopThreads;  // two threads a site

struct FixSmem {
    static constexpr int PL = 16 * kHopThreads;  // bytes of a plane: 16 a site
    static constexpr int SPINOR = 0;
    static constexpr int LINK = 12 * PL;
    static constexpr int NBR = LINK + 9 * PL;
    static constexpr int BYTES = NBR + 8 * 4 * kHopThreads;
};

template <bool DAG, int EPI, bool RED>
__global__ void __launch_bounds__(kFixThreads, 3) wilson_hop_fixed_kernel(const __grid_constant__ HopArgs a) {
    constexpr int NT = kHopThreads, PL = FixSmem::PL;
    extern __shared__ __align__(16) unsigned char smem[];
    // lane 16 s + j: spin s of the half spinors of the warp's site j
    const int spin = (threadIdx.x >> 4) & 1;
    const int t = (threadIdx.x >> 5) * 16 + (threadIdx.x & 15);
    // grid.x = (rhs, output parity, site tile), rhs fastest (see wilson_hop_kernel)
    const int rhs = blockIdx.x % a.nrhs;
    const int pt = blockIdx.x / a.nrhs;
    const Geom& g = a.g;
    const int end = a.nsite ? a.site0 + a.nsite : g.Vh;
    const int i0 = a.site0 + (pt / a.nparity) * NT + t;
    const bool active = i0 < end;
    const int i = active ? i0 : end - 1;  // past the end: recomputes the last site, stores nothing
    const int p = a.parity0 + pt % a.nparity;
    pdl_enter();
    if (a.skip && a.skip[(EPI == EPI_DWF ? 0 : rhs) * a.skip_stride]) return;

    const char* __restrict__ in = a.in[p] + (size_t)rhs * a.in_rhs;
    unsigned char* sp = smem + FixSmem::SPINOR + t * 16;
    unsigned char* lk = smem + FixSmem::LINK + t * 16;
    int* nbr = reinterpret_cast<int*>(smem + FixSmem::NBR) + t;  // neighbour of direction d at d NT
    int flips = 0;                                               // bit d: direction d crosses a boundary with sign -1
    {
        int x[4], n[8];
        cb_coords(g, i, p, x);
        const int xh = x[0] >> 1;
        const bool top0 = x[0] + 1 == g.L[0], bot0 = x[0] == 0;
        n[0] = i - xh + ((top0 ? 0 : x[0] + 1) >> 1);
        n[1] = i - xh + ((bot0 ? g.L[0] - 1 : x[0] - 1) >> 1);
        if (g.bc[0] < 0) flips |= (top0 ? 1 : 0) | (bot0 ? 2 : 0);
        int step = g.Lh0;
#pragma unroll
        for (int mu = 1; mu < 4; ++mu) {
            const bool top = x[mu] == g.L[mu] - 1, bot = x[mu] == 0;
            n[2 * mu] = top ? i - (g.L[mu] - 1) * step : i + step;
            n[2 * mu + 1] = bot ? i + (g.L[mu] - 1) * step : i - step;
            if (g.bc[mu] < 0) flips |= (top ? 1 << (2 * mu) : 0) | (bot ? 2 << (2 * mu) : 0);
            step *= g.L[mu];
        }
        if (spin == 0) {
#pragma unroll
            for (int d = 0; d < 8; ++d) nbr[d * NT] = check_site(n[d], g.Vh);
        }
    }
    __syncwarp();
    const char* __restrict__ links = a.links + (size_t)(p * 4) * a.link_block;
    const ptrdiff_t other = (p ? -4 : 4) * (ptrdiff_t)a.link_block;  // to the other parity's links
    const size_t plane = (size_t)g.Vh * 16;

    // the site's two threads copy half of its planes each
    auto issue_spinor = [&](const char* blk, int site) {
        const char* src = blk + (size_t)(6 * spin) * plane + (size_t)site * 16;
        unsigned char* dst = sp + 6 * spin * PL;
#pragma unroll
        for (int k = 0; k < 6; ++k) __pipeline_memcpy_async(dst + k * PL, src + k * plane, 16);
    };
    auto issue_link = [&](int d) {
        const bool bwd = d & 1;
        const char* src = links + (bwd ? other : 0) + (size_t)(d >> 1) * a.link_block + (size_t)(5 * spin) * plane +
                          (size_t)(bwd ? nbr[d * NT] : i) * 16;
        unsigned char* dst = lk + 5 * spin * PL;
#pragma unroll
        for (int k = 0; k < 4; ++k) __pipeline_memcpy_async(dst + k * PL, src + k * plane, 16);
        if (spin == 0) __pipeline_memcpy_async(dst + 4 * PL, src + 4 * plane, 16);
    };
    // this thread's groups up to the last but one are complete, and so are its partner's
    auto wait_one = [&]() {
        __pipeline_wait_prior(1);
        __syncwarp();
    };

    // sums over directions, [2 c + {re, im}]: up of spin s, low of a lower spin: 2 + (1 - s) for the x
    // and y hops, after which the site's threads exchange theirs, and 2 + s from then on
    long long up[6], low[6];
#pragma unroll
    for (int k = 0; k < 6; ++k) up[k] = low[k] = 0;
    int eb = 0;  // the block's biased exponent: |neighbour components| < 2^(eb - 1022)
    bool slow = false;
    // sums over directions of the larger part of each term of colour c in units of 2^-10 of the block (at
    // most 8 * 5.5 * 2^10): for up in the upper, for low in the lower 16 bits (x and y: both the lower)
    uint32_t size[3] = {0, 0, 0};

    issue_spinor(in, nbr[NT]);
    __pipeline_commit();
    issue_link(1);
    __pipeline_commit();

    // One body per dimension, run backward, then forward: with one for each of the 8 directions
    // the SM waited for instructions.  With w_b, w_f the results of the two, a sum that takes
    // w_f - w_b is formed as sum = w - sum both times.
    const int sg0 = spin ? 0 : -1, sg1 = ~sg0;  // minus for spin 0 / for spin 1
    auto dimension = [&](auto mtag) {
        constexpr int MU = decltype(mtag)::value;
#pragma unroll 1
        for (int d = 2 * MU + 1; d >= 2 * MU; --d) {
            const int bwd = -(d & 1);  // -1: backward, U^dag h = conj(U^T conj(h))
            const int flip = -((flips >> d) & 1), fim = flip ^ bwd;
            const int neg = DAG ? bwd : ~bwd;  // -1: projector sign S = -1
            Fix2 h[6];                         // [2 c + {re, im}] of spin s (backward: of the conjugate)
            wait_one();
            {
                // this spin and the one that the projector adds to it, times i in x and z
                constexpr bool SW = (MU & 1) == 0;
                uint2 r[6], q[6];
                const unsigned char* rp = sp + 3 * spin * PL;
                const unsigned char* qp = sp + (MU < 2 ? 9 - 3 * spin : 6 + 3 * spin) * PL;
#pragma unroll
                for (int c = 0; c < 3; ++c) {
                    const uint4 v = *reinterpret_cast<const uint4*>(rp + c * PL);
                    const uint4 x = *reinterpret_cast<const uint4*>(qp + c * PL);
                    r[2 * c] = make_uint2(v.x, v.y);
                    r[2 * c + 1] = make_uint2(v.z, v.w);
                    q[2 * c + (SW ? 1 : 0)] = make_uint2(x.x, x.y);
                    q[2 * c + (SW ? 0 : 1)] = make_uint2(x.z, x.w);
                }
                if constexpr (MU == 3) {
                    // the time direction is projected in FP64: a ghost spinor rebuilt from its
                    // spin-projected face (halo.cu) has this half spinor and no other component
                    // right, and gives the same sums bit for bit.  (The FP64 unit has time for
                    // these additions; for those of all directions it has not.)
#pragma unroll
                    for (int k = 0; k < 6; ++k)
                        r[k] = words(value(r[k]) + value(make_uint2(q[k].x, q[k].y ^ ((uint32_t)neg << 31))));
                }
                float m = 0.f;
                if constexpr (MU < 3) {
#pragma unroll
                    for (int k = 0; k < 6; ++k) m = max_hi(m, r[k].y, q[k].y);
                } else {
#pragma unroll
                    for (int k = 0; k < 3; ++k) m = max_hi(m, r[2 * k].y, r[2 * k + 1].y);
                }
                m = max_hi(m, __float_as_uint(__shfl_xor_sync(0xffffffffu, m, 16)), 0u);
                const int e = __float_as_int(m) >> 20;
                if (e > eb) {  // one bit of headroom: later neighbours seldom move the sums
                    const int to = max(e + 1, kFixEmin);
                    const uint32_t n = (uint32_t)(to - eb);
#pragma unroll
                    for (int k = 0; k < 6; ++k) {
                        up[k] = sar64(up[k], n);
                        low[k] = sar64(low[k], n);
                    }
#pragma unroll
                    for (int c = 0; c < 3; ++c) size[c] = shr32(size[c], 16 + n) << 16 | shr32(size[c] & 0xffffu, n);
                    eb = to;
                    slow = slow || to > kFixEmax;
                }
                const uint32_t e2 = ((uint32_t)max(eb, kFixEmin) << 21) + 0x1fffffu + (5u << 21);
                // what is added: x: S(im, -re); y: -S (s = 0), S (s = 1); z: as x (s = 0), the
                // opposite (s = 1)
                const int tre = flip ^ neg ^ (MU == 1 ? sg0 : MU == 2 ? sg1 : 0);
                const int tim = fim ^ neg ^ (MU == 0 ? -1 : sg0);
#pragma unroll
                for (int k = 0; k < 6; ++k) {
                    if constexpr (MU == 3) h[k] = fix_one(r[k], e2, k & 1 ? fim : flip);
                    else h[k] = fix_pair(r[k], q[k], e2, k & 1 ? fim : flip, k & 1 ? tim : tre);
                }
            }
            __syncwarp();  // the site's spinor has been read
            const int next = bwd ? d - 1 : d + 3;
            if (MU < 3 || bwd) issue_spinor(in, nbr[next * NT]);
            else if constexpr (EPI >= EPI_DIAG) issue_spinor(a.x[p] + (size_t)rhs * a.x_rhs, i);
            __pipeline_commit();
            wait_one();
            // w = U h (backward: U^T conj(h), the conjugate of U^dag h), rows of U or U^T
            long long w[6];
            const unsigned char* l0 = lk;
            const unsigned char* l1 = lk + (bwd ? 3 : 1) * PL;
            const unsigned char* l2 = lk + (bwd ? 6 : 2) * PL;
            const int sc = (bwd ? 1 : 3) * PL;
#pragma unroll
            for (int c = 0; c < 3; ++c) {
                const int4 a0 = *reinterpret_cast<const int4*>(l0 + c * sc);
                const int4 a1 = *reinterpret_cast<const int4*>(l1 + c * sc);
                const int4 a2 = *reinterpret_cast<const int4*>(l2 + c * sc);
                const Fix2 u[6] = {{a0.y, a0.x}, {a1.y, a1.x}, {a2.y, a2.x}, {a0.w, a0.z}, {a1.w, a1.z}, {a2.w, a2.z}};
                const Fix2 x[6] = {h[0], h[2], h[4], {-h[1].hi, -h[1].lo}, {-h[3].hi, -h[3].lo}, {-h[5].hi, -h[5].lo}};
                const Fix2 y[6] = {h[1], h[3], h[5], h[0], h[2], h[4]};
                w[2 * c] = fix_dot(u, x);
                w[2 * c + 1] = fix_dot(u, y);
            }
            __syncwarp();  // the site's link has been read
            if (MU < 3 || bwd) issue_link(next);
            __pipeline_commit();
            // sums += [uh; S A_mu^dag uh], uh = w, or conj(w) backward; the lower half as if S > 0
            // forward (it changes sign at the end otherwise).  Spin s of uh goes, times S, to
            //   x: i uh of the other lower spin;   y: -uh (s = 0), uh (s = 1) of the other;
            //   z: i uh (s = 0), -i uh (s = 1) of its own;   t: uh of its own.
            const long long n = MU == 1 ? (long long)sg0 : (long long)sg1;
#pragma unroll
            for (int c = 0; c < 3; ++c) {
                const long long re = w[2 * c], im = w[2 * c + 1];
                const uint32_t part = (uint32_t)max(abs((int)(re >> 32)), abs((int)(im >> 32)));
                size[c] += (part >> 15) * (MU < 2 ? 1 : 0x10001);
                up[2 * c] += re;
                up[2 * c + 1] = im - up[2 * c + 1];
                if constexpr (MU == 0) {
                    low[2 * c] -= im;
                    low[2 * c + 1] = re - low[2 * c + 1];
                } else if constexpr (MU == 1) {
                    low[2 * c] = ((re ^ n) - n) - low[2 * c];
                    low[2 * c + 1] += (im ^ n) - n;
                } else if constexpr (MU == 2) {
                    low[2 * c] -= (im ^ n) - n;
                    low[2 * c + 1] = ((re ^ n) - n) - low[2 * c + 1];
                } else {
                    low[2 * c] = re - low[2 * c];
                    low[2 * c + 1] += im;
                }
            }
        }
    };
    dimension(std::integral_constant<int, 0>());
    dimension(std::integral_constant<int, 1>());
#pragma unroll
    for (int k = 0; k < 6; ++k) low[k] = __shfl_xor_sync(0xffffffffu, low[k], 16);
#pragma unroll
    for (int c = 0; c < 3; ++c) size[c] = size[c] << 16 | __shfl_xor_sync(0xffffffffu, size[c], 16);
    dimension(std::integral_constant<int, 2>());
    dimension(std::integral_constant<int, 3>());

    // c_hop, and S of the forward projectors for the lower spins; a power of two (all but the second
    // hop of the Schur complement) goes into the exponent
    const double ch = a.c_hop;
    const uint32_t cw = (uint32_t)__double2hiint(ch);
    const int ce = (int)((cw >> 20) & 0x7ffu) - 1023;
    const bool pow2 = (cw & 0xfffffu) == 0 && __double2loint(ch) == 0 && ce >= -64 && ce <= 16;
    const int ef = eb + (pow2 ? ce : 0);
    const uint32_t fu = pow2 ? cw : 0u, fl = DAG ? fu : ~fu;
    double o[12];  // [2 c + {re, im}] of spin s, then of spin 2 + s
#pragma unroll
    for (int k = 0; k < 6; ++k) {
        o[k] = fix_to_double(up[k], ef, fu);
        o[6 + k] = fix_to_double(low[k], ef, fl);
    }
    if (!pow2) {
#pragma unroll
        for (int k = 0; k < 12; ++k) o[k] *= ch;
    }
    // Where the terms of a sum are small beside the block (a neighbour of much larger other spins,
    // colours or sites, links with small entries, neighbours that are subnormal or out of the fixed-point
    // range), the block's bits are too few for it: the site takes the FP64 sums.  Sums of exact zeros
    // (around sources) are zero already; they are told apart by reading the neighbours once more.
    bool weak_up = false, weak_low = false;
#pragma unroll
    for (int c = 0; c < 3; ++c) {
        weak_up |= size[c] >> 16 < kFixWeak;
        weak_low |= (size[c] & 0xffffu) < kFixWeak;
    }
    bool mine = slow || weak_up || weak_low;
    if (__any_sync(0xffffffffu, mine)) {
        mine = __shfl_xor_sync(0xffffffffu, mine, 16) || mine;  // the same for a site's two threads
        uint2 seen = {0, 0};
        if (mine) seen = nonzero_halves<DAG, NT>(a, spin, in, nbr);
        const uint32_t seen_xy = __shfl_xor_sync(0xffffffffu, seen.x, 16);
        mine = slow || (weak_up && (seen.x | seen.y)) || (weak_low && (seen_xy | seen.y));
        mine = __shfl_xor_sync(0xffffffffu, mine, 16) || mine;
        __pipeline_wait_prior(0);
        __syncwarp();
        double2* v = reinterpret_cast<double2*>(sp);
        double2* x = reinterpret_cast<double2*>(lk);
        if (mine) slow_site<DAG, NT>(a, p, spin, in, i, nbr, flips, v, x);
        __syncwarp();
        if (mine) {
#pragma unroll
            for (int c = 0; c < 3; ++c) {
                const double2 b = v[(6 * spin + c) * NT], l = v[(6 * spin + 3 + c) * NT];
                const double2 m = x[(3 - 3 * spin + c) * NT];
                o[2 * c] = ch * b.x;
                o[2 * c + 1] = ch * b.y;
                o[6 + 2 * c] = ch * (l.x + m.x);
                o[6 + 2 * c + 1] = ch * (l.y + m.y);
            }
        }
        __syncwarp();
        if constexpr (EPI >= EPI_DIAG) issue_spinor(a.x[p] + (size_t)rhs * a.x_rhs, i);
        __pipeline_commit();
    }
    if constexpr (EPI >= EPI_DIAG) {
        __pipeline_wait_prior(0);
        __syncwarp();
        const double cd = a.c_diag;
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            const double2 b = *reinterpret_cast<const double2*>(sp + (3 * spin + c) * PL);
            const double2 l = *reinterpret_cast<const double2*>(sp + (6 + 3 * spin + c) * PL);
            o[2 * c] = fma(cd, b.x, o[2 * c]);
            o[2 * c + 1] = fma(cd, b.y, o[2 * c + 1]);
            o[6 + 2 * c] = fma(cd, l.x, o[6 + 2 * c]);
            o[6 + 2 * c + 1] = fma(cd, l.y, o[6 + 2 * c + 1]);
        }
    }
    if constexpr (EPI == EPI_DWF) {
        const HopShift<double> sh = hop_shift<DAG, double>(a, rhs);
        const double2* xu = reinterpret_cast<const double2*>(a.x[p] + (size_t)sh.up * a.x_rhs);
        const double2* xd = reinterpret_cast<const double2*>(a.x[p] + (size_t)sh.dn * a.x_rhs);
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            const double2 b = __ldg(xu + (size_t)(3 * spin + c) * g.Vh + i);
            const double2 l = __ldg(xd + (size_t)(6 + 3 * spin + c) * g.Vh + i);
            o[2 * c] = fma(sh.c_up, b.x, o[2 * c]);
            o[2 * c + 1] = fma(sh.c_up, b.y, o[2 * c + 1]);
            o[6 + 2 * c] = fma(sh.c_dn, l.x, o[6 + 2 * c]);
            o[6 + 2 * c + 1] = fma(sh.c_dn, l.y, o[6 + 2 * c + 1]);
        }
    }
    if (active) {
        double2* out = reinterpret_cast<double2*>(a.out[p] + (size_t)rhs * a.out_rhs);
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            out[(size_t)(3 * spin + c) * g.Vh + i] = make_double2(o[2 * c], o[2 * c + 1]);
            out[(size_t)(6 + 3 * spin + c) * g.Vh + i] = make_double2(o[6 + 2 * c], o[6 + 2 * c + 1]);
        }
    }
    if constexpr (RED) {
        // a partial for every 32 sites (two warps), group-major (see hop_norm_site)
        __shared__ double half[kFixThreads / 64];
        double v = 0;
        if (active) {
#pragma unroll
            for (int k = 0; k < 12; ++k) v = fma(o[k], o[k], v);
        }
#pragma unroll
        for (int s = 16; s > 0; s >>= 1) v += __shfl_xor_sync(0xffffffffu, v, s);
        const int w = threadIdx.x >> 5;
        if ((w & 1) && (threadIdx.x & 31) == 0) half[w >> 1] = v;
        __syncthreads();
        if (!(w & 1) && (threadIdx.x & 31) == 0) {
            const int wpb = NT >> 5;
            const int grp = EPI == EPI_DWF ? 0 : rhs;
            const int nblk = EPI == EPI_DWF ? gridDim.x : gridDim.x / a.nrhs;
            const int bidx = EPI == EPI_DWF ? blockIdx.x : pt;
            a.red_partial[(size_t)grp * nblk * wpb + bidx * wpb + (w >> 1)] = v + half[w >> 1];
        }
    }
}

template <bool DAG, int EPI, bool RED>
cudaError_t launch_fixed_one(const HopArgs& a, cudaStream_t st) {
    constexpr int NT = kHopThreads, smem = FixSmem::BYTES;
    auto kern = wilson_hop_fixed_kernel<DAG, EPI, RED>;
    static bool configured = false;  // attribute set once per process (per instantiation)
    if (!configured) {
        cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
        if (e != cudaSuccess) return e;
        configured = true;
    }
    const int nsite = a.nsite ? a.nsite : a.g.Vh;
    return launch_pdl(kern, dim3(((nsite + NT - 1) / NT) * a.nrhs * a.nparity), dim3(kFixThreads), smem, st, a);
}

inline cudaError_t launch_hop_fixed(const HopArgs& a, bool dag, int epi, cudaStream_t st) {
    const bool red = a.red_partial != nullptr;
    if (red && epi == EPI_HOP) return cudaErrorInvalidValue;
#define LQ_F_EPI(D)                                                                                    \
    switch (epi) {                                                                                     \
    case EPI_HOP: return launch_fixed_one<D, EPI_HOP, false>(a, st);                                   \
    case EPI_DIAG: return red ? launch_fixed_one<D, EPI_DIAG, true>(a, st)                             \
                              : launch_fixed_one<D, EPI_DIAG, false>(a, st);                           \
    default: return red ? launch_fixed_one<D, EPI_DWF, true>(a, st) : launch_fixed_one<D, EPI_DWF, false>(a, st); \
    }
    if (dag) { LQ_F_EPI(true) } else { LQ_F_EPI(false) }
#undef LQ_F_EPI
}

}  // namespace lq
