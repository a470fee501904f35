// elbm_kernels.cuh -- kernels of the essentially entropic lattice Boltzmann
// step and its companions, instantiated once per lattice by elbm_d2q9.cu and
// elbm_d3q27.cu (include this file after defining ELBM_DIM and ELBM_SUFFIX).
//
//   k_step     fused pull-stream + collide + store (Eq. advection, Eq.
//              fstar_def, path length of Sec. III / Appendix C-D), one node per
//              thread (D2Q9 in FP32 arithmetic: two), ping-pong buffers
//   k_step_tile  several steps of a small D2Q9 domain in shared memory
//   k_init     f = f^eq(rho, u) (Sec. I equilibrium, in FP64 or, for the FP32-arithmetic
//              storages, in double-float; rounded once to storage)
//   k_moments  rho and u of the stored state (FP64; exact sums of FP32 values, split into
//              two FP32 parts or in fixed point)
//   k_alpha    path length of the next collision (no write-back)
//   k_diag     domain reductions: mass, momentum, H (Eq. hdef), alpha statistics
//              and per-node H[f*] - H[f] (Eq. deltaH3) in FP64; warp shuffles,
//              then shared memory, then one atomic per block and quantity
#pragma once

#include <algorithm>
#include <type_traits>

#include "elbm_device.cuh"
#include "elbm_launch.h"
#include "elbm_tma.cuh"
#include "elbm_adjoint.cuh"

namespace eelbm {
namespace ELBM_SUFFIX {

constexpr int D = ELBM_DIM;
constexpr int Q = Lattice<D>::Q;
// Threads per block of the direct step kernel (a tuning knob: block sizes that are
// not a multiple of the register allocation unit leave resident warps unused).
#ifndef ELBM_STEP_BLOCK_D3
#define ELBM_STEP_BLOCK_D3 128
#endif
constexpr int kStepBlock = D == 2 ? 256 : ELBM_STEP_BLOCK_D3;
constexpr int kAuxBlock = 256;


__device__ __forceinline__ void node_coords(int64_t n, const Geometry &g, int &x, int &y, int &z)
{
    if (g.N <= 0xffffffffll) { // 32-bit division where the indices fit (the common case)
        const uint32_t m = uint32_t(n), nx = uint32_t(g.nx), ny = uint32_t(g.ny);
        const uint32_t t = m / nx;
        x = int(m - t * nx);
        z = int(t / ny);
        y = int(t - uint32_t(z) * ny);
        return;
    }
    const int64_t t = n / g.nx;
    x = int(n - t * g.nx);
    z = int(t / g.ny);
    y = int(t - (int64_t)z * g.ny);
}

// Addressing of the direct step kernel (template parameter kAddr), chosen by the launcher
// from the size of the domain:
//   kAddrBytes  Q N elements fill less than 2^32 bytes: 32-bit byte offsets from the buffer
//   kAddrElems  Q N < 2^32 elements: 32-bit element offsets, scaled by the load and store
//   kAddrWide   anything else: a 1D grid over all nodes, 64-bit indices
// One node per thread: blocks of consecutive nodes of an xy-plane (blockIdx.y = z), so that
// a width that is no multiple of the block leaves no idle warps; x and y come from one
// multiplication by a precomputed reciprocal (RowDiv).  D3Q27, ms per step, one block row per
// x-row and element offsets against this: 0.569 and 0.543 (256^3 FP32, Taylor-Green start),
// 0.185 and 0.1525 (203 x 150 x 131, developed flow; a fifth of the threads of its rows of 256
// were idle), 0.2125 and 0.165 (176 x 144 x 160, FP16 deviations).  The addresses cost
// either the multiply-add pipe that the collision needs (a scaled 32-bit offset is one wide
// multiply-add per access) or two additions on the integer pipe, which is less busy: byte
// offsets are 0.543 against 0.550 (256^3) and 0.165 against 0.175 (FP16 deviations).  Two
// nodes per thread (D2Q9): blocks along x-rows, y = blockIdx.y; byte offsets there are 55.8
// against 59.0 us per step (2048^2 FP32, developed flow) and 24.6 against 26.5 (1501 x 997,
// FP32 and FP16 deviations), and leave the DRAM-bound shear layers as they were.
// (Developed flows here and below, both sides, with the Omega- sums as half differences; the
// direct sums of PowerSums add 1 to 2.5 % to each.)
// Minimum resident blocks per SM requested from the register allocator for the direct step
// kernel.  D3Q27 with FP32 storage: 7 blocks of 128 (72 registers).  A step from DRAM is bound
// by the bytes in flight, and the extra resident warps outweigh the spills (256^3, Taylor-Green
// start: 0.544 ms with 7 blocks, 0.551 with 6, 0.579 with 5, 0.566 with 8).  FP32 deviations: 6
// (80 registers).  A step whose two buffers stay in the L2 is bound by instructions and latency
// instead: 5 blocks there (kL2Blocks, up to 102 registers, 4 bytes of spills; us per step, 7 or 6 blocks
// and 5, near-equilibrium and developed flow: FP32 32^3 3.20, 3.04 and 3.33, 3.07; 64^3 10.96,
// 10.45 and 14.69, 14.01; 80^3 20.7, 20.5 and 27.5, 26.4; 96^3, beyond the L2, 34.1, 35.3 and
// 44.8, 43.5; FP32 deviations 32^3 3.54, 3.24, 72^3 16.2, 15.2 and 21.6, 20.8).  The 16-bit
// storages take 5 everywhere, the allocation they had unbounded.  FP64: no bound.
// ELBM_STEP_MIN_BLOCKS overrides.
#ifndef ELBM_STEP_MIN_BLOCKS
#define ELBM_STEP_MIN_BLOCKS 0
#endif
// D2Q9 with FP32 arithmetic runs two nodes per thread (node_collide_x2), in blocks of
// kStepBlock / 2 threads: 8 of them per SM (at most 64 registers) for FP32 and 16-bit
// storage, 6 (80 registers) for FP32 deviations, whose collision keeps d_i and spills at 64
// (4096^2 shear layer: 0.190 against 0.193 ms; FP32 storage loses with 80: 0.188 against
// 0.179).
#ifndef ELBM_PAIR_MIN_BLOCKS
#define ELBM_PAIR_MIN_BLOCKS 8
#endif
#ifndef ELBM_PAIR_MIN_BLOCKS_DEV
#define ELBM_PAIR_MIN_BLOCKS_DEV 6
#endif
template <class ST>
constexpr int step_min_blocks()
{
    return ELBM_STEP_MIN_BLOCKS > 0 ? ELBM_STEP_MIN_BLOCKS
                                    : (sizeof(typename ST::T) != 4 ? 1
                                       : D == 2 ? (ST::kDevCollide ? ELBM_PAIR_MIN_BLOCKS_DEV : ELBM_PAIR_MIN_BLOCKS)
                                       : ST::kDevCollide          ? 6
                                       : sizeof(typename ST::S) == 4 ? 7 : 5);
}
// Two-node kernels: warp w of a block takes the aligned run of kPairSpan nodes
// [kPairSpan w, kPairSpan (w + 1)) of the block's nodes, lane l nodes l and l + 32 of
// it.  A warp's nodes (and so its coefficient form) are then the same whatever the
// block width, and each of its loads covers 32 consecutive nodes.
constexpr uint32_t kPairSpan = 64;
__device__ __forceinline__ uint32_t pair_node(uint32_t t) { return (t >> 5) * kPairSpan + (t & 31u); }
// threads per block of the direct step kernel
template <class ST>
constexpr int step_threads()
{
    return kStepBlock / nodes_per_thread<D, ST>();
}
constexpr int kL2Blocks = 5;
// Bytes of the two population buffers up to which a step is taken to run from the L2 (129 MB).
constexpr uint64_t kL2Bytes = 112ull << 20;

enum { kAddrBytes = 0, kAddrElems = 1, kAddrWide = 2 };

// Exact n / d for n < 2^31: (umulhi(magic, n) + n) >> shift with shift = ceil(log2 d) and
// magic = floor(2^32 (2^shift - d) / d) + 1 (Granlund and Montgomery; the sum stays below
// 2^32 because magic < 2^32 makes umulhi(magic, n) < n).
struct RowDiv {
    uint32_t magic, shift;
};
inline RowDiv row_div(uint32_t d)
{
    RowDiv r{0, 0};
    while ((uint64_t(1) << r.shift) < d) ++r.shift;
    r.magic = uint32_t(((uint64_t(1) << 32) * ((uint64_t(1) << r.shift) - d)) / d + 1);
    return r;
}
// Element at offset o of a buffer: o in bytes (kAddrBytes) or elements.
template <int kAddr, class S>
__device__ __forceinline__ S *at(S *base, uint32_t o)
{
    using C = std::conditional_t<std::is_const_v<S>, const char, char>;
    if constexpr (kAddr == kAddrBytes) return reinterpret_cast<S *>(reinterpret_cast<C *>(base) + o);
    else return base + o;
}
__device__ __forceinline__ uint32_t div_row(uint32_t n, RowDiv r) { return (__umulhi(r.magic, n) + n) >> r.shift; }

// Two nodes x = xa and xa + 32 of row y of a D2Q9 domain (nx by ny, N nodes, populations at
// in / out): pull, collide (node_collide_x2), store.  Where the warp's 64-node run lies inside
// the row, clear of its ends, the second node's addresses are the first's plus 32 elements, an
// immediate offset (32-bit byte offsets cost three integer instructions per address, 108 of
// the 460 instructions of 64 nodes).  Else the columns wrap, and a second node past the end
// of the row is a copy of the first, collided and not stored.  Plain loads when kCoherent
// (buffers written during the launch), else ld_pop.
template <class ST, int kAddr, bool kCoherent = false, bool kForce = false>
__device__ __forceinline__ void step2_row(const typename ST::S *in, typename ST::S *out, uint32_t nx, uint32_t ny,
                                          uint32_t N, uint32_t xa, uint32_t y, const CollideParams &p)
{
    using S = typename ST::S;
    using T = typename ST::T;
    constexpr uint32_t H = kPairSpan / 2;
    constexpr uint32_t B = kAddr == kAddrBytes ? uint32_t(sizeof(S)) : 1u;
    auto ld = [](const S *q) { return kCoherent ? *q : ld_pop<false>(q); };
    const uint32_t sy[3] = {y == ny - 1 ? 0 : (y + 1) * nx, y * nx, (y == 0 ? ny - 1 : y - 1) * nx};
    auto row = [&](int i) { return (uint32_t(i) * N + sy[vel(D, i, 1) + 1]) * B; };
    const uint32_t run = xa & ~(H - 1); // first node of the warp's run (the same for the whole warp)
    const bool inside = run >= 1 && run + kPairSpan < nx, hasb = xa + H < nx;
    T fa[Q], fb[Q];
    if (inside) {
#pragma unroll
        for (int i = 0; i < Q; ++i) {
            const S *q = at<kAddr>(in, (xa - uint32_t(vel(D, i, 0))) * B + row(i));
            fa[i] = ST::raw(ld(q));
            fb[i] = ST::raw(ld(q + H));
        }
    } else {
        const uint32_t xb = hasb ? xa + H : xa;
        const uint32_t ca[3] = {xa == nx - 1 ? 0 : xa + 1, xa, xa == 0 ? nx - 1 : xa - 1};
        const uint32_t cb[3] = {xb == nx - 1 ? 0 : xb + 1, xb, xb == 0 ? nx - 1 : xb - 1};
#pragma unroll
        for (int i = 0; i < Q; ++i) fa[i] = ST::raw(ld(at<kAddr>(in, ca[vel(D, i, 0) + 1] * B + row(i))));
#pragma unroll
        for (int i = 0; i < Q; ++i) fb[i] = ST::raw(ld(at<kAddr>(in, cb[vel(D, i, 0) + 1] * B + row(i))));
    }
    collide2_stored<D, ST, true>(fa, fb, p);
    if constexpr (kForce) {
        add_force<D, T, ST::kDev>(fa, p);
        add_force<D, T, ST::kDev>(fb, p);
    }
    const uint32_t na = (y * nx + xa) * B;
    auto st = [](S *q, S v) {
        if (kCoherent) *q = v;
        else __stcs(q, v);
    };
#pragma unroll
    for (int i = 0; i < Q; ++i) {
        S *q = at<kAddr>(out, uint32_t(i) * N * B + na);
        st(q, ST::pack(fa[i]));
        if (hasb) st(q + H, ST::pack(fb[i]));
    }
}

// Node (x, y, z) of a domain: pull, collide, store.  The offsets of the nine (c_x, c_y) sources
// in a plane are the thread's; the rest of an address is the same for the whole block.
template <class ST, int kAddr, bool kForce = false>
__device__ __forceinline__ void step1_node(const typename ST::S *in, typename ST::S *out, uint32_t nx, uint32_t ny,
                                           uint32_t nz, uint32_t N, uint32_t x, uint32_t y, uint32_t z, const CollideParams &p)
{
    using S = typename ST::S;
    using T = typename ST::T;
    T f[Q], xd[Q]; // the stored values (deviations for deviation storage)
    int br;
    const uint32_t plane = nx * ny;
    constexpr uint32_t B = kAddr == kAddrBytes ? uint32_t(sizeof(S)) : 1u;
    const uint32_t sx[3] = {x == nx - 1 ? 0 : x + 1, x, x == 0 ? nx - 1 : x - 1};
    const uint32_t sy[3] = {y == ny - 1 ? 0 : (y + 1) * nx, y * nx, (y == 0 ? ny - 1 : y - 1) * nx};
    const uint32_t sz[3] = {z == nz - 1 ? 0 : z + 1, z, z == 0 ? nz - 1 : z - 1};
#pragma unroll
    for (int i = 0; i < Q; ++i) {
        const int cx = vel(D, i, 0), cy = vel(D, i, 1), cz = D == 3 ? vel(D, i, 2) : 0;
        const uint32_t o = (sy[cy + 1] + sx[cx + 1]) * B;
        const uint32_t b = (uint32_t(i) * N + sz[cz + 1] * plane) * B;
        f[i] = ST::raw(ld_pop<D == 3>(at<kAddr>(in, o + b)));
    }
    collide_stored<D, ST, true>(f, xd, p, &br);
    if constexpr (kForce) add_force<D, T, ST::kDev>(f, p);
    const uint32_t n = (z * plane + y * nx + x) * B;
#pragma unroll
    for (int i = 0; i < Q; ++i) __stcs(at<kAddr>(out, uint32_t(i) * N * B + n), ST::pack(f[i]));
}

template <class ST, int kAddr, bool kForce = false, int kBlocks = step_min_blocks<ST>()>
__global__ void __launch_bounds__(step_threads<ST>(), kBlocks) k_step(const typename ST::S *__restrict__ fin,
                                                    typename ST::S *__restrict__ fout, Geometry g,
                                                    CollideParams p, RowDiv rd)
{
    wait_previous_kernel();
    using S = typename ST::S;
    using T = typename ST::T;
    if constexpr (nodes_per_thread<D, ST>() == 2) {
        // Two nodes per thread (pair_node); a second node past the end of the row (or of
        // the domain) is a copy of the first, collided and not stored.
        if constexpr (kAddr != kAddrWide) {
            const uint32_t xa = blockIdx.x * kStepBlock + pair_node(threadIdx.x);
            if (xa >= uint32_t(g.nx)) return;
            step2_row<ST, kAddr, false, kForce>(fin, fout, uint32_t(g.nx), uint32_t(g.ny), uint32_t(g.N), xa, blockIdx.y, p);
        } else {
            constexpr uint32_t H = kPairSpan / 2;
            T fa[Q], fb[Q];
            const int64_t na = (int64_t)blockIdx.x * kStepBlock + pair_node(threadIdx.x);
            if (na >= g.N) return;
            const bool hasb = na + H < g.N;
            const int64_t nb = hasb ? na + H : na;
            int x, y, z;
            node_coords(na, g, x, y, z);
            pull_load<D, ST, true>(fin, g, x, y, z, p.dunit_f, fa);
            node_coords(nb, g, x, y, z);
            pull_load<D, ST, true>(fin, g, x, y, z, p.dunit_f, fb);
            collide2_stored<D, ST, true>(fa, fb, p);
            if constexpr (kForce) {
                add_force<D, T, ST::kDev>(fa, p);
                add_force<D, T, ST::kDev>(fb, p);
            }
#pragma unroll
            for (int i = 0; i < Q; ++i) __stcs(fout + (int64_t)i * g.N + na, ST::pack(fa[i]));
            if (hasb) {
#pragma unroll
                for (int i = 0; i < Q; ++i)
                    __stcs(fout + (int64_t)i * g.N + nb, ST::pack(fb[i]));
            }
        }
        return;
    }
    if constexpr (kAddr != kAddrWide) {
        const uint32_t nx = uint32_t(g.nx), ny = uint32_t(g.ny), nz = uint32_t(g.nz), N = uint32_t(g.N);
        const uint32_t plane = nx * ny, xy = blockIdx.x * blockDim.x + threadIdx.x, z = blockIdx.y;
        if (xy >= plane) return;
        const uint32_t y = div_row(xy, rd), x = xy - y * nx;
        step1_node<ST, kAddr, kForce>(fin, fout, nx, ny, nz, N, x, y, z, p);
    } else {
        T f[Q], xd[Q]; // the stored values (deviations for deviation storage)
        int br;
        const int64_t n = (int64_t)blockIdx.x * kStepBlock + threadIdx.x;
        if (n >= g.N) return;
        int x, y, z;
        node_coords(n, g, x, y, z);
        pull_load<D, ST, true>(fin, g, x, y, z, p.dunit_f, f);
        collide_stored<D, ST, true>(f, xd, p, &br);
        if constexpr (kForce) add_force<D, T, ST::kDev>(f, p);
#pragma unroll
        for (int i = 0; i < Q; ++i) __stcs(fout + (int64_t)i * g.N + n, ST::pack(f[i]));
    }
}

// FP64 equilibrium from rho and u (same product form as node_collide): per axis
// phi(-1) = Y den / (6 num) and phi(+1) = Y num / (6 den); kDivide = false takes the same
// factors as (1 + 2t -+ 3u) / 6 with t = s - 1 (to about 2^-51 f^eq), for the nodes that
// k_init evaluates again before rounding them to FP32.
template <bool kDivide>
__device__ __forceinline__ void equilibrium64(double rho, const double (&u)[3], double (&feq)[Q])
{
    double phi[3][3];
#pragma unroll
    for (int a = 0; a < D; ++a) {
        const double s = sqrt(1.0 + 3.0 * u[a] * u[a]);
        if constexpr (kDivide) {
            const double Y = 2.0 - s;
            const double num = 2.0 * u[a] + s, den = 1.0 - u[a];
            phi[a][0] = Y * den / (6.0 * num);
            phi[a][1] = Y * (4.0 / 6.0);
            phi[a][2] = Y * num / (6.0 * den);
        } else {
            const double q = fma(2.0, s, -1.0);
            phi[a][0] = fma(-3.0, u[a], q);
            phi[a][1] = fma(-4.0, s, 8.0);
            phi[a][2] = fma(3.0, u[a], q);
        }
    }
    if constexpr (!kDivide) rho *= weight_unit(D);
#pragma unroll
    for (int i = 0; i < Q; ++i) {
        double v = rho;
#pragma unroll
        for (int a = 0; a < D; ++a) v *= phi[a][vel(D, i, a) + 1];
        feq[i] = v;
    }
}

// Double-length FP32 arithmetic ("double-float": a value hi + lo with |lo| <= ulp(hi)/2):
// Dekker's product with a fused multiply-add for the exact error of hi * hi, Knuth's
// two-sum and Dekker's fast two-sum for additions, and one Newton correction on the FP32
// square root and quotient.  About 44 significant bits, at FP32 instruction rates.
struct DF {
    float hi, lo;
};
__device__ __forceinline__ DF df_fast_two_sum(float a, float b) // |a| >= |b|
{
    const float s = a + b;
    return {s, b - (s - a)};
}
// An FP64 value as hi, the nearest FP32 number, and lo, the rest rounded to FP32, on the
// integer pipe: a conversion or an FP64 addition occupies GB300's FP64 pipe for 16 cycles per
// warp and SM, and four values converted through it (16 such instructions) bounded the whole
// kernel.  Below 2^-74, where lo is no normal FP32 number for some, the conversions; values
// beyond FP32's range, infinities and NaN give infinities and NaN.
__device__ __forceinline__ DF df_from_double(double x)
{
    const uint64_t b = (uint64_t)__double_as_longlong(x);
    const uint32_t top = uint32_t(b >> 32), sign = top & 0x80000000u;
    const int e = int((top >> 20) & 0x7ffu) - 896; // FP32's biased exponent
    if (e <= 52) {
        if ((b << 1) == 0) return {__uint_as_float(sign), 0.0f};
        const float h = __double2float_rn(x);
        return {h, __double2float_rn(x - double(h))};
    }
    if (e >= 255) { // NaN stays NaN, anything else is infinite
        const bool nan = (top & 0x7fffffffu) > 0x7ff00000u || ((top & 0x7fffffffu) == 0x7ff00000u && uint32_t(b) != 0);
        return {__uint_as_float(sign | (nan ? 0x7fc00000u : 0x7f800000u)), 0.0f};
    }
    // the 23 leading bits of the significand, rounded to nearest even by the other 29 (a carry
    // runs into the exponent, as it should)
    const uint32_t m = (uint32_t(e) << 23) | (uint32_t(b >> 29) & 0x7fffffu), low = uint32_t(b) & 0x1fffffffu;
    const uint32_t up = low > 0x10000000u || (low == 0x10000000u && (m & 1u)) ? 1u : 0u;
    const float rest = float(int(low) - int(up << 29)); // in units of 2^(e - 127 - 52)
    return {__uint_as_float(sign | (m + up)), rest * __uint_as_float(sign | (uint32_t(e - 52) << 23))};
}
__device__ __forceinline__ DF df_add(DF a, DF b)
{
    const float s = a.hi + b.hi, bb = s - a.hi;
    const float e = (a.hi - (s - bb)) + (b.hi - bb); // two-sum error
    return df_fast_two_sum(s, e + (a.lo + b.lo));
}
__device__ __forceinline__ DF df_mul(DF a, DF b)
{
    const float p = a.hi * b.hi;
    float e = fmaf(a.hi, b.hi, -p);
    e = fmaf(a.hi, b.lo, e);
    e = fmaf(a.lo, b.hi, e);
    return df_fast_two_sum(p, e);
}
__device__ __forceinline__ DF df_mulf(DF a, float b)
{
    const float p = a.hi * b;
    return df_fast_two_sum(p, fmaf(a.lo, b, fmaf(a.hi, b, -p)));
}
__device__ __forceinline__ DF df_neg(DF a) { return {-a.hi, -a.lo}; }
__device__ __forceinline__ DF df_div(DF a, DF b)
{
    const float q = a.hi / b.hi;
    const DF qb = df_mulf(b, q);
    const float r = ((a.hi - qb.hi) - qb.lo) + a.lo; // a - q b, to the first order
    return df_fast_two_sum(q, r / b.hi);
}
__device__ __forceinline__ DF df_sqrt(DF a)
{
    const float r = sqrtf(a.hi);
    const float e = fmaf(-r, r, a.hi) + a.lo; // a - r^2
    return df_fast_two_sum(r, e / (2.0f * r));
}

// v + err, where |err| is at most half a unit in the last place of v, rounded to odd: v if the
// sum is exact or v is odd, else v's odd neighbour on the side of err.  The 13 or more bits that
// a conversion to 16 bits then drops still tell on which side of a midpoint the sum lies, so
// that the conversion rounds the sum itself (Boldo and Melquiond, Emulation of FMA and correctly
// rounded sums, 2008).
__device__ __forceinline__ float to_odd(float v, float err)
{
    const uint32_t b = __float_as_uint(v);
    if (err == 0.0f || (b & 1u)) return v;
    return __uint_as_float((err < 0.0f) == (v < 0.0f) ? b + 1u : b - 1u);
}

// The equilibrium in double-float, less k_i R (R = 0: populations), rounded once to the storage:
// |error| <= half a unit in the last place + about 2^-44 f^eq.  Per axis phi(-1) = Y den / (6 num)
// and phi(+1) = Y num / (6 den) share one division, r = Y / (6 num den), phi(-1) = r den^2,
// phi(+1) = r num^2.  Returns whether every value is known to be the correctly rounded one (asked
// of the deviations only: f^eq - k_i R is small, so 2^-44 f^eq can reach its last bit): what the
// stored value leaves of the sum is further than 2^-44 f^eq from half a unit in its last place.
template <class ST>
__device__ __forceinline__ bool equilibrium_df(DF rho, const DF (&u)[3], float R, typename ST::S (&feq)[Q])
{
    constexpr double kTwoThirds = 2.0 / 3.0;
    const DF two3 = {float(kTwoThirds), float(kTwoThirds - double(float(kTwoThirds)))};
    DF phi[3][3];
#pragma unroll
    for (int a = 0; a < D; ++a) {
        const DF U = u[a];
        const DF S = df_sqrt(df_add({1.0f, 0.0f}, df_mulf(df_mul(U, U), 3.0f)));
        const DF Y = df_add({2.0f, 0.0f}, df_neg(S));
        const DF num = df_add({2.0f * U.hi, 2.0f * U.lo}, S), den = df_add({1.0f, 0.0f}, df_neg(U));
        const DF r = df_div(Y, df_mulf(df_mul(num, den), 6.0f));
        phi[a][0] = df_mul(r, df_mul(den, den));
        phi[a][1] = df_mul(Y, two3);
        phi[a][2] = df_mul(r, df_mul(num, num));
    }
    bool sure = true;
    DF v[Q / 3]; // rho times the factors of all axes but the last
#pragma unroll
    for (int x = 0; x < 3; ++x) {
        const DF rx = df_mul(rho, phi[0][x]);
        if constexpr (D == 2) {
            v[x] = rx;
        } else {
#pragma unroll
            for (int y = 0; y < 3; ++y) v[3 * x + y] = df_mul(rx, phi[1][y]);
        }
    }
    // the last axis: c = -1 and +1 on packed pairs; en = -(error of p)
    const DF b0 = phi[D - 1][0], b1 = phi[D - 1][1], b2 = phi[D - 1][2];
    const float2 bh = f2(b0.hi, b2.hi), bl = f2(b0.lo, b2.lo);
    auto put = [&](int i, float p, float en) {
        if constexpr (!ST::kDev) {
            feq[i] = ST::pack(p - en);
        } else {
            const float c = -float(weight_k(D, i)) * R, d = p + c, dd = d - p;
            const float w = ((p - (d - dd)) + (c - dd)) - en; // what p + c - d lost, and p's error
            const float r1 = d + w, err = w - (r1 - d);
            const uint32_t expo = __float_as_uint(r1) & 0x7f800000u;
            float gap; // what the stored value leaves of the sum, less half a unit in its last place
            if constexpr (sizeof(typename ST::S) == 4) {
                feq[i] = ST::pack(r1);
                gap = fabsf(err) - __uint_as_float(max(expo, 24u << 23) - (24u << 23));
            } else {
                constexpr uint32_t bits = ST::kBits, low = ST::kMinExponent;
                feq[i] = ST::pack(to_odd(r1, err));
                const float t = r1 - ST::raw(feq[i]);
                gap = (fabsf(t) - __uint_as_float(max(expo, max(low, bits + 1u) << 23) - (bits << 23))) + (t < 0.0f ? -err : err);
            }
            sure = sure && fabsf(gap) > 0x1p-44f * p;
        }
    };
#pragma unroll
    for (int k = 0; k < Q / 3; ++k) {
        const DF a = v[k];
        const float2 p2 = pmul(f2(a.hi), bh);
        const float2 e2 = pfma(f2(-a.lo), bh, pfma(f2(-a.hi), bl, pfma(f2(-a.hi), bh, p2)));
        const float p1 = a.hi * b1.hi, e1 = fmaf(-a.lo, b1.hi, fmaf(-a.hi, b1.lo, fmaf(-a.hi, b1.hi, p1)));
        put(3 * k, p2.x, e2.x);
        put(3 * k + 1, p1, e1);
        put(3 * k + 2, p2.y, e2.y);
    }
    return sure;
}

// f = f^eq(rho, u) for the nodes n0 .. n0 + count - 1 (SoA with stride g.N).  FP64 storage
// in FP64; the FP32-arithmetic storages in double-float (equilibrium_df), rounded once, but for
// a node whose deviations are not sure to be rounded as FP64 would (FP32: a few nodes in a
// hundred, 16 bits: one in millions): FP64 again.  4.8 M D3Q27 nodes: 145 us for FP32
// populations (158 with FP64 conversions), 228 for FP32 deviations and 254 for FP16 (1 433 in
// FP64; 151 when FP16 is rounded twice, first to FP32, which gives another value at 6 in 10^5);
// 8 M D2Q9 nodes: 133, 171 and 188 (184, 1 249, 1 250).  Bound by the FP32 arithmetic and its
// issue slots.  The factors without divisions (1 + 2t -+ 3u) take 122 and 108 us, but round
// a few values in 10^8 the other way than this form, which would show in FP64 moments.
template <class ST>
__global__ void __launch_bounds__(kAuxBlock) k_init(const double *__restrict__ rho,
                                                   const double *__restrict__ u,
                                                   typename ST::S *__restrict__ f, Geometry g,
                                                   double rho_uniform, double rho0, int64_t n0, int64_t count)
{
    wait_previous_kernel();
    const int64_t k = (int64_t)blockIdx.x * kAuxBlock + threadIdx.x;
    if (k >= count) return;
    const int64_t n = n0 + k;
    const double r = rho ? __ldcs(rho + n) : rho_uniform;
    double un[3] = {0.0, 0.0, 0.0};
#pragma unroll
    for (int a = 0; a < D; ++a) un[a] = __ldcs(u + (int64_t)a * g.N + n);
    if constexpr (sizeof(typename ST::T) == 4) {
        const DF ud[3] = {df_from_double(un[0]), df_from_double(un[1]), df_from_double(un[2])};
        typename ST::S fe[Q];
        if (equilibrium_df<ST>(df_from_double(r), ud, ST::kDev ? dev_unit<D>(rho0) : 0.0f, fe)) {
#pragma unroll
            for (int i = 0; i < Q; ++i) f[(int64_t)i * g.N + n] = fe[i];
            return;
        }
    }
    double feq[Q];
    equilibrium64<sizeof(typename ST::T) == 8>(r, un, feq);
    const double R = double(dev_unit<D>(rho0));
#pragma unroll
    for (int i = 0; i < Q; ++i) f[(int64_t)i * g.N + n] = ST::store64(feq[i], weight_k(D, i) * R);
}

// Exact sums of FP32 values in 64-bit fixed point.  A finite FP32 value is m 2^(e - 150),
// e its biased exponent (taken as 1 for subnormals) and m its significand (with the hidden
// bit for normal numbers).  Scaled to a common exponent E0 = e_max - 33 of the values summed,
// each becomes an integer below 2^57 (a value more than 2^33 below the largest loses its low
// bits), 32 of them add without overflow, and the integer sum converts to FP64 with one
// rounding (none while it stays below 2^53).
__device__ __forceinline__ int f32_expo(float v)
{
    const int e = int((__float_as_uint(v) >> 23) & 0xffu);
    return e ? e : 1;
}
__device__ __forceinline__ long long f32_fixed(float v, int E0)
{
    const uint32_t b = __float_as_uint(v);
    const int e = int((b >> 23) & 0xffu);
    const uint32_t m = (b & 0x7fffffu) | (e ? 0x800000u : 0u);
    const int sh = (e ? e : 1) - E0;
    const unsigned long long mag =
        sh >= 0 ? (unsigned long long)m << sh : (sh > -24 ? (unsigned long long)(m >> -sh) : 0ull);
    return (b >> 31) ? -(long long)mag : (long long)mag;
}
__device__ __forceinline__ double fixed_to_f64(long long q, int E0)
{
    return double(q) * __longlong_as_double((long long)(E0 - 150 + 1023) << 52);
}

// A finite FP32 value that is zero or normal as FP64, on the integer pipe.
__device__ __forceinline__ double f32_to_f64(float v)
{
    const uint32_t b = __float_as_uint(v);
    const uint32_t hi = (b & 0x80000000u) | (((b >> 3) & 0x0fffffffu) + (896u << 20));
    return (b << 1) ? __hiloint2double(int(hi), int(b << 29)) : 0.0;
}

// Sums of a over the node (r) and of c_a a (j), any order (the values add exactly).
__device__ __forceinline__ void lattice_sums(const float (&a)[Q], float &r, float (&j)[3])
{
    constexpr int P = Q / 3;
    float s0[P], s1[P];
#pragma unroll
    for (int k = 0; k < P; ++k) s0[k] = a[3 * k] + a[3 * k + 1] + a[3 * k + 2], s1[k] = a[3 * k + 2] - a[3 * k];
    if constexpr (D == 2) {
        r = s0[0] + s0[1] + s0[2];
        j[0] = s0[2] - s0[0];
        j[1] = s1[0] + s1[1] + s1[2];
    } else {
        float t[3], ty[3], tz[3];
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            t[k] = s0[3 * k] + s0[3 * k + 1] + s0[3 * k + 2];
            ty[k] = s0[3 * k + 2] - s0[3 * k];
            tz[k] = s1[3 * k] + s1[3 * k + 1] + s1[3 * k + 2];
        }
        r = t[0] + t[1] + t[2];
        j[0] = t[2] - t[0];
        j[1] = ty[0] + ty[1] + ty[2];
        j[2] = tz[0] + tz[1] + tz[2];
    }
}

// rho and rho u of a node from its stored FP32 values (populations, or deviations d_i of the
// reference c_i = k_i R with sum_i c_i = 6^D R and sum_i c_i c_i = 0): the exact sums rounded
// once to FP64.
//
// Error-free extraction (Rump): adding and subtracting sigma = 1.5 2^(E + 4), where
// |v_i| < 2^E, splits each value into a multiple q of 2^(E - 19) and a rest l below 2^(E - 20).
// At most 27 q's add without rounding in FP32, and so do the l's as long as they are multiples
// of 2^(E - 39), that is no value but zero is more than 15 binades below the largest; both
// sums then meet in one FP64 addition.  Everything else (rare in a flow) goes through 64-bit
// fixed point.  Returns false for a node that holds a value that is not finite.
// The FP64 pipe takes 16 cycles per warp and SM for each instruction: 4 of them here, where
// conversions and scalings took 12; the integer shifts of fixed point were 80 % of the rest.
// Rsum = 6^D R in FP64 (exact).
template <bool kDev>
__device__ __forceinline__ bool exact_sums(const float (&v)[Q], float R, double Rsum, double &rho, double (&j)[3])
{
    float vmax = 0.0f;
    uint32_t umin = 0xffffffffu; // of 2 bits - 1: zero wraps to the top
#pragma unroll
    for (int i = 0; i < Q; ++i) {
        vmax = fmaxf(vmax, fabsf(v[i]));
        umin = min(umin, 2u * __float_as_uint(v[i]) - 1u);
    }
    const int eb = int(__float_as_uint(vmax) >> 23), el = int((umin + 1u) >> 24);
    bool nan = false;
#pragma unroll
    for (int i = 0; i < Q; ++i) nan = nan || v[i] != v[i]; // fmaxf drops NaN
    if (!nan && eb >= 64 && eb < 192 && el >= eb - 15) {
        const float sigma = __uint_as_float((uint32_t(eb + 5) << 23) | 0x400000u);
        float q[Q], l[Q], rq, rl, jq[3], jl[3];
#pragma unroll
        for (int i = 0; i < Q; ++i) {
            q[i] = (sigma + v[i]) - sigma;
            l[i] = v[i] - q[i];
        }
        lattice_sums(q, rq, jq);
        lattice_sums(l, rl, jl);
        rho = f32_to_f64(rq) + f32_to_f64(rl);
        if (kDev) rho += Rsum;
#pragma unroll
        for (int a = 0; a < D; ++a) j[a] = f32_to_f64(jq[a]) + f32_to_f64(jl[a]);
        return true;
    }
    int emax = 1;
#pragma unroll
    for (int i = 0; i < Q; ++i) emax = max(emax, f32_expo(v[i]));
    if (kDev) emax = max(emax, f32_expo(R) + 8); // 6^D R < 2^8 R
    if (emax >= 255) return false;
    const int E0 = emax - 33;
    long long r = 0, jf[3] = {0, 0, 0};
#pragma unroll
    for (int i = 0; i < Q; ++i) {
        const long long f = f32_fixed(v[i], E0);
        r += f;
#pragma unroll
        for (int a = 0; a < D; ++a) {
            if (vel(D, i, a) == 1) jf[a] += f;
            if (vel(D, i, a) == -1) jf[a] -= f;
        }
    }
    if (kDev) r += f32_fixed(R, E0) * (Q == 9 ? 36 : 216);
    rho = fixed_to_f64(r, E0);
#pragma unroll
    for (int a = 0; a < D; ++a) j[a] = fixed_to_f64(jf[a], E0);
    return true;
}

// 1 / rho to FP64 from the FP32 approximation r0 (relative error e < 2^-22): r0 (1 + e + e^2),
// off by e^3 before its one rounding, so at most one in 2^12 is not the correctly rounded
// reciprocal but the next number (none of 2^21 tried)
__device__ __forceinline__ double rcp64(double rho)
{
    const float h = __double2float_rn(rho);
    if (!(fabsf(h) > 1e-30f && fabsf(h) < 1e30f)) return 1.0 / rho;
    const double r0 = f32_to_f64(rcp_(h)), e = fma(-rho, r0, 1.0);
    return fma(r0, fma(e, e, e), r0);
}

// rho and u of the stored state (FP64) for the nodes n0 .. n0 + count - 1: FP64 storage in
// FP64, the FP32-arithmetic storages by exact_sums (a node holding a value that is not finite
// is summed in FP64).  4.8 M D3Q27 nodes of FP32 populations: 114 us = 5.9 TB/s (202 with
// 64-bit fixed point for every value), FP32 deviations 133, FP16 131 (199); 8 M D2Q9 nodes 145,
// 162, 162 (207, 237, 236; bound by the FP64 pipe).  Five blocks of 256 are asked for: at their 48
// registers the D3Q27 sums spill 152 bytes, but without that bound too few loads are in flight
// (same box: FP32 107 and 133 us, FP32 deviations 124 and 149, FP16 118 and 139; D2Q9 alike).
template <class ST>
__global__ void __launch_bounds__(kAuxBlock, 5) k_moments(const typename ST::S *f, Geometry g, float Rf, double Rsum,
                                                      double *rho_out, double *u_out, int64_t n0, int64_t count)
{
    wait_previous_kernel();
    const int64_t k = (int64_t)blockIdx.x * kAuxBlock + threadIdx.x;
    if (k >= count) return;
    const int64_t n = n0 + k;
    if constexpr (sizeof(typename ST::T) == 4) {
        float v[Q];
#pragma unroll
        for (int i = 0; i < Q; ++i) v[i] = ST::raw(f[(int64_t)i * g.N + n]);
        double rho, j[3];
        if (exact_sums<ST::kDev>(v, Rf, Rsum, rho, j)) {
            if (rho_out) rho_out[n] = rho;
            if (u_out) {
                const double ir = rcp64(rho);
#pragma unroll
                for (int a = 0; a < D; ++a) u_out[(int64_t)a * g.N + n] = j[a] * ir;
            }
            return;
        }
    }
    double r = 0.0, j[3] = {0.0, 0.0, 0.0};
#pragma unroll
    for (int i = 0; i < Q; ++i) {
        const double v = ST::load64(f[(int64_t)i * g.N + n], weight_k(D, i) * double(Rf));
        r += v;
#pragma unroll
        for (int a = 0; a < D; ++a) j[a] += vel(D, i, a) * v;
    }
    if (rho_out) rho_out[n] = r;
    if (u_out) {
#pragma unroll
        for (int a = 0; a < D; ++a) u_out[(int64_t)a * g.N + n] = j[a] / r;
    }
}

// Path length of the next collision; optionally the subgrid viscosity of Sec. VI,
// nu_T = theta dt (2 - alpha) / (2 alpha beta) (Eq. nuT, theta = 1/3, dt = 1).
template <class ST>
__global__ void __launch_bounds__(kStepBlock) k_alpha(const typename ST::S *__restrict__ fin,
                                                     Geometry g, CollideParams p,
                                                     double *__restrict__ alpha_out,
                                                     uint8_t *__restrict__ flags,
                                                     double *__restrict__ nut_out)
{
    wait_previous_kernel();
    using T = typename ST::T;
    const int64_t n = (int64_t)blockIdx.x * kStepBlock + threadIdx.x;
    if (n >= g.N) return;
    int x, y, z;
    node_coords(n, g, x, y, z);
    T f[Q], xd[Q];
    pull_load<D, ST, true>(fin, g, x, y, z, p.dunit_f, f); // stored values, as the step collides them
    int br;
    const T alpha = collide_stored<D, ST, false>(f, xd, p, &br);
    if (alpha_out) alpha_out[n] = double(alpha);
    if (flags) flags[n] = uint8_t(br);
    if (nut_out) nut_out[n] = (1.0 / 3.0) * (2.0 - double(alpha)) / (2.0 * double(alpha) * p.beta);
}

// --------------------------------------------------------------------------
// Diagnostics reduction.
// --------------------------------------------------------------------------
__device__ __forceinline__ double warp_sum(double v)
{
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}
__device__ __forceinline__ unsigned long long warp_sum(unsigned long long v)
{
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}
__device__ __forceinline__ unsigned long long warp_max(unsigned long long v)
{
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        const unsigned long long w = __shfl_xor_sync(0xffffffffu, v, o);
        v = w > v ? w : v;
    }
    return v;
}
__device__ __forceinline__ unsigned long long warp_min(unsigned long long v)
{
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        const unsigned long long w = __shfl_xor_sync(0xffffffffu, v, o);
        v = w < v ? w : v;
    }
    return v;
}

// Per-thread accumulation of the domain diagnostics of a node and of the collision
// it undergoes (used by k_diag and by the step fused with diagnostics).  Partial sums
// in the compute type of the small parts (deviations, H + 1, alpha - 2) over the
// thread's nodes; the exact parts (one per node, 2 per alpha) and the conversion to
// FP64 are added once per thread in diag_finish (FP64 arithmetic is slow on this GPU,
// and per node it was a third of the pass).
template <class T>
struct DiagThread {
    double sum[6] = {0, 0, 0, 0, 0, 0};
    unsigned long long cnt[kDiagCounts] = {0, 0, 0, 0, 0, 0, 0, 0, 0};
    unsigned long long dmax = 0ULL, amin = ~0ULL, amax = 0ULL;
    T p_dr = T(0), p_j[3] = {T(0), T(0), T(0)}, p_h = T(0), p_al = T(0);
    T p_dmax = -INFINITY, p_amin = INFINITY, p_amax = -INFINITY;
    unsigned long long p_nodes = 0, p_hnodes = 0;

    // fc: the node's pre-collision populations; xd, alpha_t, br: departures, path length
    // and branch of its collision; s_hist: the block's histogram in shared memory.
    __device__ __forceinline__ void node(const T (&fc)[Q], const T (&xd)[Q], const T alpha_t, const int br,
                                         const CollideParams &p, unsigned int *s_hist)
    {
        bool bad = false;
#pragma unroll
        for (int i = 0; i < Q; ++i) bad |= !(fc[i] > T(0)) || !isfinite(fc[i]);

        // Mass and momentum through the deviations d_i = f_i - w_i (small numbers).
        T dr = T(0), jt[3] = {T(0), T(0), T(0)};
#pragma unroll
        for (int i = 0; i < Q; ++i) {
            const T di = fc[i] - T(weight(D, i));
            dr += di;
#pragma unroll
            for (int a = 0; a < D; ++a) jt[a] += T(vel(D, i, a)) * di;
        }
        p_nodes += 1;
        p_dr += dr;
        for (int a = 0; a < D; ++a) p_j[a] += jt[a];
        if (bad) {
            cnt[3] += 1;
        } else {
            // H[f] = <f, log(f/w)> - rho (Eq. hdef), with log(f/w) = log1p(d/w), and
            // the entropy change of this node's collision (Eq. deltaH3, with <f,x> = 0
            // removing alpha beta <f,x> from both sums):
            // H[f*] - H[f] = <f, g(ab x)> - ab <f, x log(1+x)>, g(y) = (1+y) log(1+y) - y.
            // Per-node sums in the path's compute type, domain sums in FP64.
            const T ab = alpha_t * beta_of<T>(p);
            T hl = T(0), s3 = T(0), xa = T(0);
#pragma unroll
            for (int i = 0; i < Q; ++i) {
                const T fi = fc[i], xi = xd[i];
                hl += fi * log1p((fi - T(weight(D, i))) * T(1.0 / weight(D, i)));
                s3 += fi * xi * xi;
                xa = fmax(xa, fabs(xi));
            }
            T dH;
            if (xa < T(0.1) && ab <= T(2.2)) {
                // g(ab x) - ab x log(1+x) = sum_{k>=2} c_k x^k,
                // c_k = (-1)^k ab/(k-1) (ab^(k-1)/k - 1), summed to k = kTop (for |x| < 0.1
                // and ab <= 2.2 the rest is below 5e-10 x^2).  c_2 = ab (ab - 2)/2 takes
                // ab - 2 from one rounding of alpha beta - 2; the two sums of the direct
                // form cancel to that small leading coefficient instead.
                constexpr int kTop = 13;
                T ck[kTop + 1];
                ck[2] = T(0.5) * ab * fma(alpha_t, beta_of<T>(p), T(-2));
                T abk = ab * ab; // ab^(k-1) at k = 3
#pragma unroll
                for (int k = 3; k <= kTop; ++k) {
                    const T v = ab * T(1.0 / (k - 1)) * (abk * T(1.0 / k) - T(1));
                    ck[k] = (k & 1) ? -v : v;
                    abk *= ab;
                }
                T sd = T(0);
#pragma unroll
                for (int i = 0; i < Q; ++i) {
                    const T xi = xd[i];
                    T poly = ck[kTop];
#pragma unroll
                    for (int k = kTop - 1; k >= 2; --k) poly = fma(poly, xi, ck[k]);
                    sd += fc[i] * (poly * xi * xi);
                }
                dH = sd;
            } else {
                T s1 = T(0), s2 = T(0);
#pragma unroll
                for (int i = 0; i < Q; ++i) {
                    const T fi = fc[i], xi = xd[i];
                    s1 += fi * g_entropy<T>(ab * xi);
                    s2 += fi * xi * log1p(xi);
                }
                dH = s1 - ab * s2;
            }
            // H of the node + (1 + e_w) (the node's -rho without its exact part)
            p_h += hl - dr;
            p_hnodes += 1;
            p_dmax = fmax(p_dmax, dH);
            if (dH > T(1e-6) * s3 && s3 > T(0)) cnt[4] += 1;
            // |x|max band: the cutoff of Appendix D, then the FP32 coefficient forms
            cnt[xa < T(1e-3) ? 5 : (xa < T(5e-3) ? 6 : (xa < T(4e-2) ? 7 : 8))] += 1;
        }
        p_al += alpha_t - T(2);
        cnt[br == kBranchCutoff ? 0 : (br == kBranchSolved ? 1 : 2)] += 1;
        p_amin = fmin(p_amin, alpha_t);
        p_amax = fmax(p_amax, alpha_t);
        // bin of alpha on [1.9, 2.1): alpha - 1.9 with 1.9 in two parts of T
        constexpr T kLo = T(1.9), kLo2 = T(1.9 - double(T(1.9)));
        const T off = (alpha_t - kLo) - kLo2;
        int bin;
        if (!(off >= T(0))) bin = 0;
        else if (off >= T(0.2)) bin = ELBM_HIST_BINS + 1;
        else bin = 1 + min(ELBM_HIST_BINS - 1, int(off * T(ELBM_HIST_BINS / 0.2)));
        atomicAdd(&s_hist[bin], 1u);
    }
};

// Block reduction of the per-thread diagnostics into the FP64 accumulator (warp
// shuffles, then shared memory, then one atomic per block and quantity).  NT >= 65.
template <int NT, class T>
__device__ __forceinline__ void diag_finish(DiagThread<T> &dt, DiagAcc *__restrict__ acc, unsigned int *s_hist)
{
    constexpr int kWarps = NT / 32;
    __shared__ double s_sum[kWarps][6];
    __shared__ unsigned long long s_cnt[kWarps][kDiagCounts];
    __shared__ unsigned long long s_ext[kWarps][3];
    double (&sum)[6] = dt.sum;
    unsigned long long (&cnt)[kDiagCounts] = dt.cnt;
    unsigned long long &dmax = dt.dmax, &amin = dt.amin, &amax = dt.amax;
    const T &p_dr = dt.p_dr, &p_h = dt.p_h, &p_al = dt.p_al;
    const T(&p_j)[3] = dt.p_j;
    const T &p_dmax = dt.p_dmax, &p_amin = dt.p_amin, &p_amax = dt.p_amax;
    const unsigned long long p_nodes = dt.p_nodes, p_hnodes = dt.p_hnodes;
    // this thread's nodes into the FP64 sums: mass = sum (1 + e_w + dr), H = sum hl - rho
    {
        const double nn = double(p_nodes), one = 1.0 + weight_sum_error<D, T>();
        sum[0] = nn * one + double(p_dr);
        for (int a = 0; a < D; ++a) sum[1 + a] = double(p_j[a]);
        sum[4] = double(p_h) - double(p_hnodes) * one;
        sum[5] = 2.0 * nn + double(p_al);
        if (p_nodes) {
            dmax = p_hnodes ? ordered_bits(double(p_dmax)) : 0ULL;
            amin = ordered_bits(double(p_amin));
            amax = ordered_bits(double(p_amax));
        }
    }

    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
    for (int k = 0; k < 6; ++k) sum[k] = warp_sum(sum[k]);
#pragma unroll
    for (int k = 0; k < kDiagCounts; ++k) cnt[k] = warp_sum(cnt[k]);
    dmax = warp_max(dmax);
    amin = warp_min(amin);
    amax = warp_max(amax);
    if (lane == 0) {
        for (int k = 0; k < 6; ++k) s_sum[warp][k] = sum[k];
        for (int k = 0; k < kDiagCounts; ++k) s_cnt[warp][k] = cnt[k];
        s_ext[warp][0] = dmax;
        s_ext[warp][1] = amin;
        s_ext[warp][2] = amax;
    }
    __syncthreads();
    if (threadIdx.x < 6) {
        double v = 0.0;
        for (int w = 0; w < kWarps; ++w) v += s_sum[w][threadIdx.x];
        atomicAdd(&acc->sum[threadIdx.x], v);
    } else if (threadIdx.x >= 32 && threadIdx.x < 32 + kDiagCounts) {
        const int k = threadIdx.x - 32;
        unsigned long long v = 0;
        for (int w = 0; w < kWarps; ++w) v += s_cnt[w][k];
        atomicAdd(&acc->cnt[k], v);
    } else if (threadIdx.x == 64) {
        unsigned long long a = 0, b = ~0ULL, c = 0;
        for (int w = 0; w < kWarps; ++w) {
            a = max(a, s_ext[w][0]);
            b = min(b, s_ext[w][1]);
            c = max(c, s_ext[w][2]);
        }
        atomicMax(&acc->dH_max_ord, a);
        atomicMin(&acc->amin_ord, b);
        atomicMax(&acc->amax_ord, c);
    }
    for (int b = threadIdx.x; b < ELBM_HIST_BINS + 2; b += NT)
        if (s_hist[b]) atomicAdd(&acc->hist[b], (unsigned long long)s_hist[b]);
}

template <class ST>
__global__ void __launch_bounds__(kAuxBlock) k_diag(const typename ST::S *__restrict__ fin,
                                                   Geometry g, CollideParams p,
                                                   DiagAcc *__restrict__ acc)
{
    wait_previous_kernel();
    using T = typename ST::T;
    __shared__ unsigned int s_hist[ELBM_HIST_BINS + 2];
    for (int b = threadIdx.x; b < ELBM_HIST_BINS + 2; b += kAuxBlock) s_hist[b] = 0u;
    __syncthreads();
    DiagThread<T> dt;
    for (int64_t n = (int64_t)blockIdx.x * kAuxBlock + threadIdx.x; n < g.N;
         n += (int64_t)gridDim.x * kAuxBlock) {
        int x, y, z;
        node_coords(n, g, x, y, z);
        T f[Q], xd[Q], fc[Q];
        pull_load<D, ST, true>(fin, g, x, y, z, p.dunit_f, f); // stored values, as the step collides them
#pragma unroll
        for (int i = 0; i < Q; ++i) fc[i] = ST::kDev ? f[i] + dev_ref<D, T>(i, p.dunit_f) : f[i]; // populations
        int br;
        const T alpha_t = collide_stored<D, ST, false>(f, xd, p, &br);
        dt.node(fc, xd, alpha_t, br, p, s_hist);
    }
    diag_finish<kAuxBlock>(dt, acc, s_hist);
}

// The step fused with the diagnostics of the state it advances (the quantities of
// k_diag, taken from the collision the step performs): 3D-grid addressing with 32-bit
// offsets, one node per thread, a grid of a few blocks per SM looping over the
// (x-block, y, z) items so that each block reduces and posts its sums once.
// Its own register budget: the diagnostics' extra live values spilled heavily under
// the step's 72-register cap (3 blocks of 128 for D3Q27, 2 of 256 for D2Q9; FP64 unbounded).
template <class ST>
constexpr int step_diag_min_blocks()
{
    return sizeof(typename ST::T) != 4 ? 1 : (D == 3 ? 3 : 2);
}
template <class ST>
__global__ void __launch_bounds__(kStepBlock, step_diag_min_blocks<ST>()) k_step_diag(const typename ST::S *__restrict__ fin,
                                             typename ST::S *__restrict__ fout, Geometry g, CollideParams p,
                                             DiagAcc *__restrict__ acc)
{
    wait_previous_kernel();
    using T = typename ST::T;
    __shared__ unsigned int s_hist[ELBM_HIST_BINS + 2];
    for (int b = threadIdx.x; b < ELBM_HIST_BINS + 2; b += kStepBlock) s_hist[b] = 0u;
    __syncthreads();
    DiagThread<T> dt;
    const uint32_t nx = uint32_t(g.nx), ny = uint32_t(g.ny), nz = uint32_t(g.nz), N = uint32_t(g.N);
    const uint32_t xblocks = (nx + kStepBlock - 1) / kStepBlock;
    const uint32_t items = xblocks * ny * nz;
    for (uint32_t it = blockIdx.x; it < items; it += gridDim.x) {
        const uint32_t xb = it % xblocks, yz = it / xblocks;
        const uint32_t y = yz % ny, z = yz / ny;
        const uint32_t x = xb * kStepBlock + threadIdx.x;
        if (x >= nx) continue;
        const uint32_t xm = x == 0 ? nx - 1 : x - 1, xp = x == nx - 1 ? 0 : x + 1;
        const uint32_t ym = y == 0 ? ny - 1 : y - 1, yp = y == ny - 1 ? 0 : y + 1;
        const uint32_t zm = z == 0 ? nz - 1 : z - 1, zp = z == nz - 1 ? 0 : z + 1;
        T f[Q], xd[Q], fc[Q];
        auto src = [&](int i) -> uint32_t {
            const int cx = vel(D, i, 0), cy = vel(D, i, 1), cz = D == 3 ? vel(D, i, 2) : 0;
            const uint32_t sx = cx == 1 ? xm : (cx == -1 ? xp : x);
            const uint32_t sy = cy == 1 ? ym : (cy == -1 ? yp : y);
            const uint32_t sz = cz == 1 ? zm : (cz == -1 ? zp : z);
            return uint32_t(i) * N + (sz * ny + sy) * nx + sx;
        };
#pragma unroll
        for (int i = 0; i < Q; ++i) {
            f[i] = ST::raw(ld_pop<false>(fin + src(i)));
            fc[i] = ST::kDev ? f[i] + dev_ref<D, T>(i, p.dunit_f) : f[i]; // populations
        }
        int br;
        const T alpha_t = collide_stored<D, ST, true>(f, xd, p, &br);
        dt.node(fc, xd, alpha_t, br, p, s_hist);
        const uint32_t n = (z * ny + y) * nx + x;
#pragma unroll
        for (int i = 0; i < Q; ++i) __stcs(fout + (uint32_t(i) * N + n), ST::pack(f[i]));
    }
    diag_finish<kStepBlock>(dt, acc, s_hist);
}

// --------------------------------------------------------------------------
#if ELBM_DIM == 2
// --------------------------------------------------------------------------
// Several steps of a small D2Q9 domain in one launch.  A step of a small domain costs its
// latency, not its work: the launch, one pull from L2, one pass through the collision's chain
// of dependent instructions (64^2: 1.7 us, of which the collision is 0.7).  Here a block
// advances `rows` whole rows by k steps: it computes the first step of its rows and of the
// k - 1 rows on either side from the input, each later step, one row fewer on either side,
// from the one before in shared memory, and the last into the output.  The rows of the halos
// are collided by more than one block, on SMs that would be idle.  A warp takes the same nodes
// of a row as in step2_row and the state between two steps is rounded as it is stored, so the
// result is that of k launches of k_step, bit for bit.  us per step, k_step and this kernel:
// 64^2 1.71, 1.14; 64 x 256 2.33, 1.67; 100 x 90 1.89, 1.53; 128^2 2.56, 2.01.  Strips of
// columns with halos of their own are no faster (64^2 1.05, 128^2 1.79) and would regroup the
// nodes of a warp.
constexpr int kTileThreads = 384;
template <class ST, bool kForce = false>
__global__ void __launch_bounds__(kTileThreads, 1) k_step_tile(const typename ST::S *__restrict__ fin,
                                                              typename ST::S *__restrict__ fout, Geometry g,
                                                              CollideParams p, int k, int rows)
{
    using S = typename ST::S;
    using T = typename ST::T;
    wait_previous_kernel();
    extern __shared__ float s_tile[];
    constexpr int H = int(kPairSpan) / 2;
    const int nx = g.nx, ny = g.ny, R = rows + 2 * (k - 1);
    const int y0 = int(blockIdx.x) * rows, h = min(rows, ny - y0);
    // row r of the tile is row y0 - (k - 1) + r of the domain.  The odd steps write rows 0 .. R - 1
    // of one buffer, the even ones, never the outermost rows, rows 1 .. R - 2 of the other
    S *const odd = reinterpret_cast<S *>(s_tile), *const even = odd + Q * R * nx - nx;
    const int runs = (nx + int(kPairSpan) - 1) / int(kPairSpan);
    const int r0 = int(threadIdx.x >> 5) / runs, xa = (int(threadIdx.x >> 5) - r0 * runs) * int(kPairSpan) + int(threadIdx.x & 31);
    const bool hasb = xa + H < nx;
    const int xb = hasb ? xa + H : xa;
    const int ca[3] = {xa == nx - 1 ? 0 : xa + 1, xa, xa == 0 ? nx - 1 : xa - 1};
    const int cb[3] = {xb == nx - 1 ? 0 : xb + 1, xb, xb == 0 ? nx - 1 : xb - 1};
    for (int step = 1; step <= k; ++step) {
        const bool is_odd = step & 1;
        const S *from = is_odd ? even : odd;
        S *to = is_odd ? odd : even;
        const int from_plane = (is_odd ? R - 2 : R) * nx, to_plane = (is_odd ? R : R - 2) * nx;
        const int halo = k - step, row = r0 + step - 1; // one row of the step per warp run
        if (r0 < h + 2 * halo && xa < nx) {
            T fa[Q], fb[Q];
            if (step == 1) {
                int y = (y0 - halo + r0) % ny;
                if (y < 0) y += ny;
                const int sy[3] = {y == ny - 1 ? 0 : (y + 1) * nx, y * nx, (y == 0 ? ny - 1 : y - 1) * nx};
#pragma unroll
                for (int i = 0; i < Q; ++i) {
                    const S *q = fin + (i * int(g.N) + sy[vel(D, i, 1) + 1]);
                    fa[i] = ST::raw(ld_pop<false>(q + ca[vel(D, i, 0) + 1]));
                    fb[i] = ST::raw(ld_pop<false>(q + cb[vel(D, i, 0) + 1]));
                }
            } else {
#pragma unroll
                for (int i = 0; i < Q; ++i) {
                    const S *q = from + i * from_plane + (row - vel(D, i, 1)) * nx;
                    fa[i] = ST::raw(q[ca[vel(D, i, 0) + 1]]);
                    fb[i] = ST::raw(q[cb[vel(D, i, 0) + 1]]);
                }
            }
            collide2_stored<D, ST, true>(fa, fb, p);
            if constexpr (kForce) {
                add_force<D, T, ST::kDev>(fa, p);
                add_force<D, T, ST::kDev>(fb, p);
            }
            S *q = step < k ? to + row * nx + xa : fout + ((y0 + r0) * nx + xa);
            const int plane = step < k ? to_plane : int(g.N);
#pragma unroll
            for (int i = 0; i < Q; ++i, q += plane) {
                q[0] = ST::pack(fa[i]);
                if (hasb) q[H] = ST::pack(fb[i]);
            }
        }
        if (step < k) __syncthreads();
    }
}
#endif

// --------------------------------------------------------------------------
// Batched ensemble: one launch advances up to kBatchTableDomains domains.  Block
// b is one work item, nodes x0 .. x0 + BX - 1 of one x-row of one domain; the
// block finds its domain in the launch's parameter table (a coarse index, then a
// forward scan over the item counts) and its row by division, both uniform over the
// block, so each thread then addresses its populations as k_step does: 32-bit offsets
// inside the domain, in bytes where every domain of the launch holds less than 2^32 bytes
// (us per step, element offsets and bytes: 64 D2Q9 domains of 3.93 M nodes FP32 52.5, 51.8,
// 16-bit 55.3, 54.1; 20 D3Q27 domains of 1.41 M nodes 73.4, 71.9 and 75.9, 71.5).  Each domain
// has its own beta; everything else is the single-domain step.
// --------------------------------------------------------------------------
// Resident threads per SM requested from the register allocator for the batched ensemble
// kernel (0: no bound).  Two-node D2Q9 kernels: 1024 (at most 64 registers; 74.7 against
// 65.7 GLUPS on the 64-domain ensemble with the 80 the compiler picks unbounded), 768 for
// FP32 deviations (80 registers); one node per thread: no bound.  The persistent kernel
// keeps the compiler's choice (bounded to 64 registers it spills: 60.2 against 62.6 GLUPS).
#ifndef ELBM_BATCH_THREADS_PER_SM
#define ELBM_BATCH_THREADS_PER_SM 0
#endif
template <class ST>
constexpr int batch_threads_per_sm()
{
    return ELBM_BATCH_THREADS_PER_SM > 0 ? ELBM_BATCH_THREADS_PER_SM
           : nodes_per_thread<D, ST>() == 2 ? (ST::kDevCollide ? 768 : 1024)
                                            : 0;
}
template <class ST, int BX>
constexpr int batch_min_blocks()
{
    return batch_threads_per_sm<ST>() / (BX / nodes_per_thread<D, ST>());
}
template <class ST, int BX, int kAddr>
__global__ void __launch_bounds__(BX / nodes_per_thread<D, ST>(), batch_min_blocks<ST, BX>()) k_step_batch(const typename ST::S *__restrict__ fin,
                                                  typename ST::S *__restrict__ fout,
                                                  const __grid_constant__ BatchTable tab, CollideParams p)
{
    wait_previous_kernel();
    using T = typename ST::T;
    const int bid = int(blockIdx.x);
    int lo = tab.coarse[bid >> tab.shift]; // item0[lo] <= bid
    while (tab.item0[lo + 1] <= bid) ++lo;
    const BatchTableDom &dm = tab.dom[lo];
    const uint32_t nx = uint32_t(dm.nx), ny = uint32_t(dm.ny), nz = uint32_t(dm.nz), xb = uint32_t(dm.xblocks);
    const uint32_t it = uint32_t(bid - tab.item0[lo]);
    const uint32_t row = it / xb;
    const uint32_t x = (it - row * xb) * BX + (nodes_per_thread<D, ST>() == 2 ? pair_node(threadIdx.x) : threadIdx.x);
    if (x >= nx) return;
    const uint32_t z = row / ny, y = row - z * ny, N = nx * ny * nz;
    p.beta = dm.beta;
    p.beta_f = dm.beta_f;
    const typename ST::S *in = fin + dm.off;
    typename ST::S *out = fout + dm.off;
    if constexpr (nodes_per_thread<D, ST>() == 2) {
        // two nodes per thread (D2Q9: z = 0), as in k_step
        step2_row<ST, kAddr>(in, out, nx, ny, N, x, y, p);
        return;
    }
    step1_node<ST, kAddr>(in, out, nx, ny, nz, N, x, y, z, p);
}

// --------------------------------------------------------------------------
// Persistent ensemble: one cooperative launch advances every domain by nsteps.
// Blocks draw tickets in order from one counter; ticket k is chunk k mod M of step
// k / M (plan.chunks: runs of work items inside one domain, numbered within it and
// located by division as in k_step_batch).  Domains are independent, so before step
// t on domain d a block waits only until cnt[d] has counted every chunk of d at step
// t - 1 (release: stores, barrier, fence, atomic add; acquire: bounded spin, fence,
// barrier).  The chunks it waits for hold smaller tickets, so the smallest unfinished
// ticket never waits and the launch cannot deadlock; idle blocks take the next chunk
// at once, which balances the domains as the hardware scheduler does for separate
// launches.  Populations are read with plain coherent loads, not through the read-only
// path, since the buffers change during the launch; offsets inside a domain are 32-bit
// (Q N < 2^32 per domain, checked when the batch is created).  Every wait is bounded
// (kWaitLimitNs of %globaltimer, also abandoned once another block has flagged an
// error): on expiry the block records ELBM_ERR_TIMEOUT in *err and returns.
// --------------------------------------------------------------------------
__device__ __forceinline__ bool wait_count(const unsigned *cnt, unsigned target, const int *err)
{
    const unsigned long long t0 = global_ns();
    for (;;) {
        unsigned v;
        asm volatile("ld.acquire.gpu.u32 %0, [%1];" : "=r"(v) : "l"(cnt) : "memory");
        if (v >= target) return true;
        if (*(volatile const int *)err != 0 || global_ns() - t0 > kWaitLimitNs) return false;
        __nanosleep(64);
    }
}

template <class ST, int BX>
__global__ void __launch_bounds__(BX / nodes_per_thread<D, ST>()) k_step_persist(typename ST::S *pop0, typename ST::S *pop1, int cur,
                                                    int nsteps, const BatchTableDom *__restrict__ doms,
                                                    PersistPlan plan, CollideParams p, int *err)
{
    using T = typename ST::T;
    using S = typename ST::S;
    __shared__ unsigned s_ticket;
    __shared__ int s_ok;
    const unsigned M = plan.nchunks, total = unsigned(nsteps) * M; // below 2^32 (host)
    const uint32_t tx = nodes_per_thread<D, ST>() == 2 ? pair_node(threadIdx.x) : threadIdx.x;
    for (;;) {
        if (threadIdx.x == 0) s_ticket = atomicAdd(plan.ticket, 1u);
        __syncthreads();
        const unsigned tk = s_ticket;
        if (tk >= total) return;
        const unsigned t = tk / M;
        const int4 seg = plan.chunks[tk - t * M];
        if (t > 0) {
            if (threadIdx.x == 0) {
                s_ok = wait_count(plan.cnt + seg.x, t * plan.owners[seg.x], err);
                if (!s_ok) atomicExch(err, ELBM_ERR_TIMEOUT);
                __threadfence();
            }
            __syncthreads();
            if (!s_ok) return;
        }
        const bool odd = ((unsigned(cur) + t) & 1u) != 0;
        const S *fin = odd ? pop1 : pop0;
        S *fout = odd ? pop0 : pop1;
        const BatchTableDom dm = doms[seg.x];
        p.beta = dm.beta;
        p.beta_f = dm.beta_f;
        const uint32_t nx = uint32_t(dm.nx), ny = uint32_t(dm.ny), nz = uint32_t(dm.nz), N = nx * ny * nz;
        const uint32_t xb = uint32_t(dm.xblocks);
        const S *in = fin + dm.off;
        S *out = fout + dm.off;
        // the chunk's work items: row-major (z, y), then the x-chunk c; one division for
        // the first item, then counters
        uint32_t row = uint32_t(seg.y) / xb, c = uint32_t(seg.y) - row * xb;
        uint32_t z = row / ny, y = row - z * ny;
        for (uint32_t w = uint32_t(seg.y); w < uint32_t(seg.z); ++w) {
            const uint32_t x = c * BX + tx;
            const uint32_t yc = y, zc = z;
            if (++c == xb) { // next row
                c = 0;
                if (++y == ny) {
                    y = 0;
                    ++z;
                }
            }
            if (x >= nx) continue;
            if constexpr (nodes_per_thread<D, ST>() == 2) {
                step2_row<ST, kAddrElems, true>(in, out, nx, ny, N, x, yc, p);
                continue;
            }
            const uint32_t y = yc, z = zc;
            const uint32_t xm = x == 0 ? nx - 1 : x - 1, xp = x == nx - 1 ? 0 : x + 1;
            const uint32_t ym = y == 0 ? ny - 1 : y - 1, yp = y == ny - 1 ? 0 : y + 1;
            const uint32_t zm = z == 0 ? nz - 1 : z - 1, zp = z == nz - 1 ? 0 : z + 1;
            T f[Q], xd[Q];
            auto src = [&](int i) -> uint32_t {
                const int cx = vel(D, i, 0), cy = vel(D, i, 1), cz = D == 3 ? vel(D, i, 2) : 0;
                const uint32_t sx = cx == 1 ? xm : (cx == -1 ? xp : x);
                const uint32_t sy = cy == 1 ? ym : (cy == -1 ? yp : y);
                const uint32_t sz = cz == 1 ? zm : (cz == -1 ? zp : z);
                return uint32_t(i) * N + (sz * ny + sy) * nx + sx;
            };
#pragma unroll
            for (int i = 0; i < Q; ++i) f[i] = ST::raw(in[src(i)]);
            int br;
            collide_stored<D, ST, true>(f, xd, p, &br);
            const uint32_t n = (z * ny + y) * nx + x;
#pragma unroll
            for (int i = 0; i < Q; ++i) out[uint32_t(i) * N + n] = ST::pack(f[i]);
        }
        __syncthreads(); // every store of this chunk issued; s_ticket and s_ok read by all
        if (threadIdx.x == 0) {
            __threadfence();
            atomicAdd(plan.cnt + seg.x, 1u);
        }
    }
}

// --------------------------------------------------------------------------
// Adjoint of one step (f^{t+1} = collide(stream(f^t))): given gnext = dL/df^{t+1},
// write gout = dL/df^t.  Per node x: the pre-collision populations F(x) are
// pulled from f^t as in the step, h = J^T gnext(x) is the collision's VJP, and
// the transpose of pull streaming sends h_i(x) to node x - c_i (a push).
// Gradient arrays are SoA [Q][N] in the compute type.
// --------------------------------------------------------------------------
// FP32: nodes on the power series (node_vjp_series); the others go through node_vjp, kept
// out of line so that its registers do not bound the kernel's occupancy.
template <bool kForce>
__device__ __noinline__ void node_vjp_general(const float (&F)[Q], const float (&g)[Q], const CollideParams &p, float (&h)[Q],
                                              float *dforce)
{
    node_vjp<D, float, kForce>(F, g, p, h, dforce);
}

template <class ST>
constexpr int adjoint_block()
{
    return sizeof(typename ST::T) == 4 ? 128 : kAuxBlock;
}
template <class ST, int kAddr, bool kForce = false>
__global__ void __launch_bounds__(adjoint_block<ST>(), sizeof(typename ST::T) == 4 ? 4 : 1)
    k_step_adjoint(const typename ST::S *__restrict__ fin, const typename ST::T *__restrict__ gnext,
                   typename ST::T *__restrict__ gout, Geometry g, CollideParams p, RowDiv rd, double *__restrict__ dforce)
{
    wait_previous_kernel();
    using T = typename ST::T;
    using S = typename ST::S;
    constexpr int kBlock = adjoint_block<ST>();
    T dfl[3] = {T(0), T(0), T(0)};
    T F[Q], gl[Q], h[Q];
    // J^T g of the node
    auto vjp = [&]() {
        if constexpr (sizeof(T) == 4) {
            if (!node_vjp_series<D, kForce>(F, gl, p, h, dfl)) {
                float Fm[Q], gm[Q], hm[Q], dm[3] = {0.0f, 0.0f, 0.0f}; // in memory for the call; the rest stays in registers
#pragma unroll
                for (int i = 0; i < Q; ++i) Fm[i] = F[i], gm[i] = gl[i];
                node_vjp_general<kForce>(Fm, gm, p, hm, dm);
#pragma unroll
                for (int i = 0; i < Q; ++i) h[i] = hm[i];
#pragma unroll
                for (int a = 0; a < 3; ++a) dfl[a] += dm[a];
            }
        } else {
            node_vjp<D, T, kForce>(F, gl, p, h, dfl);
        }
    };
    if constexpr (kAddr == kAddrBytes) {
        // as k_step: consecutive nodes of an xy-plane, byte offsets; the push of h_i goes where
        // the pull of f_i came from
        const uint32_t nx = uint32_t(g.nx), ny = uint32_t(g.ny), nz = uint32_t(g.nz), N = uint32_t(g.N);
        const uint32_t plane = nx * ny, xy = blockIdx.x * kBlock + threadIdx.x, z = blockIdx.y;
        if (xy < plane) {
            const uint32_t y = div_row(xy, rd), x = xy - y * nx;
            const uint32_t sx[3] = {x == nx - 1 ? 0 : x + 1, x, x == 0 ? nx - 1 : x - 1};
            const uint32_t sy[3] = {y == ny - 1 ? 0 : (y + 1) * nx, y * nx, (y == 0 ? ny - 1 : y - 1) * nx};
            const uint32_t sz[3] = {z == nz - 1 ? 0 : z + 1, z, z == 0 ? nz - 1 : z - 1};
            auto src = [&](int i, uint32_t B) {
                const int cx = vel(D, i, 0), cy = vel(D, i, 1), cz = D == 3 ? vel(D, i, 2) : 0;
                return (sy[cy + 1] + sx[cx + 1]) * B + (uint32_t(i) * N + sz[cz + 1] * plane) * B;
            };
#pragma unroll
            for (int i = 0; i < Q; ++i)
                F[i] = ST::load(ld_pop<true>(at<kAddrBytes>(fin, src(i, sizeof(S)))), dev_ref<D, T>(i, p.dunit_f));
            const uint32_t n = (z * plane + xy) * uint32_t(sizeof(T));
#pragma unroll
            for (int i = 0; i < Q; ++i) gl[i] = __ldcs(at<kAddrBytes>(gnext, uint32_t(i) * N * uint32_t(sizeof(T)) + n));
            vjp();
#pragma unroll
            for (int i = 0; i < Q; ++i) *at<kAddrBytes>(gout, src(i, sizeof(T))) = h[i];
        }
    } else {
        const int64_t n = (int64_t)blockIdx.x * kBlock + threadIdx.x;
        if (n < g.N) {
            int x, y, z;
            node_coords(n, g, x, y, z);
            pull_load<D, ST>(fin, g, x, y, z, p.dunit_f, F);
#pragma unroll
            for (int i = 0; i < Q; ++i) gl[i] = __ldcs(gnext + (int64_t)i * g.N + n);
            vjp();
            const int xm = x == 0 ? g.nx - 1 : x - 1, xp = x == g.nx - 1 ? 0 : x + 1;
            const int ym = y == 0 ? g.ny - 1 : y - 1, yp = y == g.ny - 1 ? 0 : y + 1;
            const int zm = z == 0 ? g.nz - 1 : z - 1, zp = z == g.nz - 1 ? 0 : z + 1;
#pragma unroll
            for (int i = 0; i < Q; ++i) {
                const int cx = vel(D, i, 0), cy = vel(D, i, 1), cz = D == 3 ? vel(D, i, 2) : 0;
                const int dx = cx == 1 ? xm : (cx == -1 ? xp : x);
                const int dy = cy == 1 ? ym : (cy == -1 ? yp : y);
                const int dz = cz == 1 ? zm : (cz == -1 ? zp : z);
                gout[(int64_t)i * g.N + ((int64_t)dz * g.ny + dy) * g.nx + dx] = h[i];
            }
        }
    }
    if constexpr (kForce) {
        // d/dF_b summed over the block (FP64), one atomic per block and component
        __shared__ double s_df[kBlock / 32][3];
        const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
        for (int a = 0; a < D; ++a) {
            const double v = warp_sum(double(dfl[a]));
            if (lane == 0) s_df[warp][a] = v;
        }
        __syncthreads();
        if (dforce && threadIdx.x < D) {
            double v = 0.0;
            for (int w = 0; w < kBlock / 32; ++w) v += s_df[w][threadIdx.x];
            atomicAdd(&dforce[threadIdx.x], v);
        }
    }
}

// Kinetic energy L = 1/2 sum rho |u|^2 of a stored field (FP64 sum into acc[0])
// and, optionally, its gradient dL/df_i = c_i . u - |u|^2 / 2.  The FP32-arithmetic storages
// take rho and rho u from exact_sums and form the gradient in double-float, rounded once to
// FP32, or in FP64 where that is not sure to round alike (a node in some 10^4): 4.8 M D3Q27 nodes
// with gradient 284 us (214 without the test, which is wrong where an entry cancels), where FP64 sums and gradients kept the FP64
// pipe busy for 2.38 ms; 137 k nodes 18 (84), 65 k D2Q9 nodes 8 (26).
template <class ST>
__global__ void __launch_bounds__(kAuxBlock, 4) k_kinetic_energy(const typename ST::S *f, Geometry g, float Rf, double Rsum,
                                                             double *__restrict__ acc, typename ST::T *grad)
{
    wait_previous_kernel();
    using T = typename ST::T;
    double e = 0.0;
    for (int64_t n = (int64_t)blockIdx.x * kAuxBlock + threadIdx.x; n < g.N; n += (int64_t)gridDim.x * kAuxBlock) {
        double r = 0.0, j[3] = {0.0, 0.0, 0.0};
        if constexpr (sizeof(T) == 4) {
            float v[Q];
#pragma unroll
            for (int i = 0; i < Q; ++i) v[i] = ST::raw(f[(int64_t)i * g.N + n]);
            if (exact_sums<ST::kDev>(v, Rf, Rsum, r, j)) {
                const double ir = rcp64(r);
                double uu = 0.0, u[3];
#pragma unroll
                for (int a = 0; a < D; ++a) {
                    u[a] = j[a] * ir;
                    uu = fma(u[a], u[a], uu);
                }
                e = fma(0.5 * r, uu, e);
                if (grad) {
                    DF ud[3], base = df_mulf(df_from_double(uu), -0.5f);
                    float size = -base.hi;
#pragma unroll
                    for (int a = 0; a < D; ++a) {
                        ud[a] = df_from_double(u[a]);
                        size += fabsf(ud[a].hi);
                    }
                    // stores an entry; its rounding is sure where what the sum leaves of the FP32
                    // number is further than its error, below 2^-42 of the largest sum, from half
                    // a unit in the last place
                    bool sure = true;
                    const float slack = 0x1p-42f * size;
                    auto put = [&](int i, DF v) {
                        grad[(int64_t)i * g.N + n] = v.hi;
                        const uint32_t expo = __float_as_uint(v.hi) & 0x7f800000u;
                        const float half = __uint_as_float(max(expo, 24u << 23) - (24u << 23));
                        sure = sure && fabsf(fabsf(v.lo) - half) >= slack;
                    };
                    auto along = [](DF b, DF w, int c) { return c == 0 ? b : df_add(b, c > 0 ? w : df_neg(w)); };
#pragma unroll
                    for (int x = 0; x < 3; ++x) {
                        const DF bx = along(base, ud[0], x - 1);
#pragma unroll
                        for (int y = 0; y < 3; ++y) {
                            const DF by = along(bx, ud[1], y - 1);
                            if constexpr (D == 2) {
                                put(3 * x + y, by);
                            } else {
#pragma unroll
                                for (int z = 0; z < 3; ++z) put(9 * x + 3 * y + z, along(by, ud[2], z - 1));
                            }
                        }
                    }
                    if (!sure) { // in FP64 (c . u and |u|^2 / 2 may cancel to any degree)
#pragma unroll
                        for (int i = 0; i < Q; ++i) {
                            double cu = 0.0;
#pragma unroll
                            for (int a = 0; a < D; ++a) cu += vel(D, i, a) * u[a];
                            grad[(int64_t)i * g.N + n] = T(cu - 0.5 * uu);
                        }
                    }
                }
                continue;
            }
        }
        double fv[Q];
#pragma unroll
        for (int i = 0; i < Q; ++i) {
            fv[i] = ST::load64(f[(int64_t)i * g.N + n], weight_k(D, i) * double(Rf));
            r += fv[i];
#pragma unroll
            for (int a = 0; a < D; ++a) j[a] += vel(D, i, a) * fv[i];
        }
        double uu = 0.0, u[3];
#pragma unroll
        for (int a = 0; a < D; ++a) {
            u[a] = j[a] / r;
            uu += u[a] * u[a];
        }
        e += 0.5 * r * uu;
        if (grad) {
#pragma unroll
            for (int i = 0; i < Q; ++i) {
                double cu = 0.0;
#pragma unroll
                for (int a = 0; a < D; ++a) cu += vel(D, i, a) * u[a];
                grad[(int64_t)i * g.N + n] = T(cu - 0.5 * uu);
            }
        }
    }
    __shared__ double s_e[kAuxBlock / 32];
    e = warp_sum(e);
    if ((threadIdx.x & 31) == 0) s_e[threadIdx.x >> 5] = e;
    __syncthreads();
    if (threadIdx.x == 0) {
        for (int w = 1; w < kAuxBlock / 32; ++w) e += s_e[w];
        atomicAdd(acc, e);
    }
}

// Derivatives of f = f^eq(rho, u) (the initial state) with respect to rho and u:
// drho = sum_i g_i feq_i / rho, du_a = sum_i g_i feq_i d log phi_a(c_ia) / du_a.
template <class T>
__global__ void __launch_bounds__(kAuxBlock) k_equilibrium_vjp(const double *__restrict__ rho,
                                                              const double *__restrict__ u,
                                                              const T *__restrict__ gf, Geometry g, double rho_uniform,
                                                              double *__restrict__ drho, double *__restrict__ du)
{
    wait_previous_kernel();
    const int64_t n = (int64_t)blockIdx.x * kAuxBlock + threadIdx.x;
    if (n >= g.N) return;
    const double r = rho ? __ldcs(rho + n) : rho_uniform;
    double phi[3][3], dlp[3][3];
#pragma unroll
    for (int a = 0; a < D; ++a) {
        const double ua = __ldcs(u + (int64_t)a * g.N + n);
        const double s = sqrt(1.0 + 3.0 * ua * ua), Y = 2.0 - s, num = 2.0 * ua + s, den = 1.0 - ua;
        const double zz = num / den, dY = -3.0 * ua / s, dlz = (2.0 + 3.0 * ua / s) / num + 1.0 / den;
        phi[a][0] = Y / (6.0 * zz);
        phi[a][1] = Y * (4.0 / 6.0);
        phi[a][2] = Y * zz / 6.0;
        dlp[a][0] = dY / Y - dlz;
        dlp[a][1] = dY / Y;
        dlp[a][2] = dY / Y + dlz;
    }
    double sr = 0.0, su[3] = {0.0, 0.0, 0.0};
#pragma unroll
    for (int i = 0; i < Q; ++i) {
        double v = r;
#pragma unroll
        for (int a = 0; a < D; ++a) v *= phi[a][vel(D, i, a) + 1];
        const double gv = double(__ldcs(gf + (int64_t)i * g.N + n)) * v;
        sr += gv;
#pragma unroll
        for (int a = 0; a < D; ++a) su[a] += gv * dlp[a][vel(D, i, a) + 1];
    }
    if (drho) drho[n] = sr / r;
    if (du) {
#pragma unroll
        for (int a = 0; a < D; ++a) du[(int64_t)a * g.N + n] = su[a];
    }
}

// --------------------------------------------------------------------------
// Launchers (storage dispatch).
// --------------------------------------------------------------------------
#define ELBM_STORAGE_SWITCH(storage, CALL)                                                     \
    switch (storage) {                                                                         \
    case ELBM_STORE_F64: { using ST = StoreF64; CALL; }                                        \
    case ELBM_STORE_F32: { using ST = StoreF32; CALL; }                                        \
    case ELBM_STORE_F32DEV: { using ST = StoreF32Dev; CALL; }                                  \
    case ELBM_STORE_F16DEV: { using ST = StoreF16Dev; CALL; }                                  \
    case ELBM_STORE_BF16DEV: { using ST = StoreBF16Dev; CALL; }                                \
    default: return cudaErrorInvalidValue;                                                     \
    }

static inline uint64_t storage_bytes(int storage)
{
    return storage == ELBM_STORE_F64 ? 8 : storage == ELBM_STORE_F32 || storage == ELBM_STORE_F32DEV ? 4 : 2;
}
static inline unsigned blocks_for(int64_t N, int block) { return unsigned((N + block - 1) / block); }

} // namespace ELBM_SUFFIX

#define ELBM_CAT2(a, b) a##_##b
#define ELBM_CAT(a, b) ELBM_CAT2(a, b)

// Each lattice is compiled in three units: ELBM_PART 1 holds the step launcher (and the
// row pipeline), ELBM_PART 3 the launchers of the batched ensemble, ELBM_PART 2 every other
// launcher; without ELBM_PART one unit holds all.
#if !defined(ELBM_PART) || ELBM_PART == 1
namespace ELBM_SUFFIX {

// Row-staged instantiations: (NXMAX, stages) per storage element size.
constexpr int kRowThreads = 256;
template <class S>
constexpr int row_stages()
{
    return sizeof(S) >= 4 ? (D == 3 ? 3 : 3) : 5;
}

template <class ST, int NXMAX>
cudaError_t launch_rows(const void *fin, void *fout, const Geometry &g, const CollideParams &p, int num_sms,
                        int *err, cudaStream_t s)
{
    using S = typename ST::S;
    constexpr int STAGES = (D == 3 && NXMAX > 256) ? 2 : row_stages<S>();
    constexpr size_t smem = rows_smem_bytes<Q, S, NXMAX, STAGES>();
    auto kern = k_step_rows<D, ST, NXMAX, kRowThreads, STAGES>;
    // one-time set-up per instantiation (single-device library use)
    static int per_sm = 0;
    if (per_sm == 0) {
        cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, int(smem));
        if (e != cudaSuccess) return e;
        int n = 0;
        e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, kern, kRowThreads, smem);
        if (e != cudaSuccess) return e;
        per_sm = n < 1 ? 1 : n;
    }
    const int rows = g.ny * g.nz;
    int grid = per_sm * (num_sms > 0 ? num_sms : 1);
    if (grid > rows) grid = rows;
    kern<<<grid, kRowThreads, smem, s>>>(static_cast<const S *>(fin), static_cast<S *>(fout), g, p, err);
    return cudaGetLastError();
}

template <class ST>
int rows_nxmax(const Geometry &g)
{
    using S = typename ST::S;
    if (ST::kRows == 0) return 0;
    if ((size_t(g.nx) * sizeof(S)) % 16 != 0) return 0;
    const int cands[3] = {D == 3 ? 128 : 256, D == 3 ? 256 : 1024, D == 3 ? 512 : 0};
    for (int c : cands)
        if (c && g.nx <= c) return c;
    return 0;
}

} // namespace ELBM_SUFFIX

bool ELBM_CAT(rows_kernel_applies, ELBM_SUFFIX)(int storage, const Geometry &g)
{
    using namespace ELBM_SUFFIX;
    switch (storage) {
    case ELBM_STORE_F32: return rows_nxmax<StoreF32>(g) > 0;
    case ELBM_STORE_F32DEV: return rows_nxmax<StoreF32Dev>(g) > 0;
    case ELBM_STORE_F16DEV: return rows_nxmax<StoreF16Dev>(g) > 0;
    case ELBM_STORE_BF16DEV: return rows_nxmax<StoreBF16Dev>(g) > 0;
    default: return false;
    }
}

// Most steps that one launch_step takes with this kernel choice (1 but for k_step_tile).
// k_step_tile is for domains whose work one wave of blocks of two rows can take several times:
// rows of at most two warps and no more row pairs than SMs.  Rows of more warps lose the
// latency again to the halo's work (203 x 177: 2.95 us per step by k_step, 2.89 so; 203 x 100
// 2.64, 2.85).  Four steps for rows of one warp, three for two (128^2: 2.01 us per step
// against 2.07 with four, and within 48 KB of shared memory).
constexpr int kTileRows = 2;
int ELBM_CAT(steps_per_launch, ELBM_SUFFIX)(int storage, const Geometry &g, int kernel, int num_sms)
{
    using namespace ELBM_SUFFIX;
    if (D != 2 || storage == ELBM_STORE_F64 || kernel != ELBM_KERNEL_AUTO) return 1;
    if (g.N == 0 || g.nx > 2 * int(kPairSpan) || (g.ny + kTileRows - 1) / kTileRows > num_sms) return 1;
    return g.nx <= int(kPairSpan) ? 4 : 3;
}

cudaError_t ELBM_CAT(launch_step, ELBM_SUFFIX)(int storage, const void *fin, void *fout,
                                               const Geometry &g, const CollideParams &p, int kernel,
                                               int steps, int num_sms, int *err, cudaStream_t s)
{
    using namespace ELBM_SUFFIX;
    if (g.N == 0) return cudaSuccess;
    const bool forced = p.force[0] != 0.0 || p.force[1] != 0.0 || p.force[2] != 0.0;
    // AUTO takes DIRECT, or several steps at once (steps_per_launch): on GB300 DIRECT is faster
    // than ROWS at every size measured.  The body force runs on DIRECT only.
    if (kernel == ELBM_KERNEL_ROWS && forced) return cudaErrorNotSupported;
    if (kernel == ELBM_KERNEL_ROWS && ELBM_CAT(rows_kernel_applies, ELBM_SUFFIX)(storage, g)) {
        // the row pipeline is only instantiated for the FP32 and 16-bit storages
#define ELBM_ROWS_FOR(STT)                                                                        \
    {                                                                                             \
        const int nm = rows_nxmax<STT>(g);                                                        \
        if (nm == (D == 3 ? 128 : 256))                                                           \
            return launch_rows<STT, (D == 3 ? 128 : 256)>(fin, fout, g, p, num_sms, err, s);      \
        if (nm == (D == 3 ? 256 : 1024))                                                          \
            return launch_rows<STT, (D == 3 ? 256 : 1024)>(fin, fout, g, p, num_sms, err, s);     \
        if (D == 3 && nm == 512) return launch_rows<STT, 512>(fin, fout, g, p, num_sms, err, s);  \
    }
        switch (storage) {
        case ELBM_STORE_F32: ELBM_ROWS_FOR(StoreF32) break;
        case ELBM_STORE_F32DEV: ELBM_ROWS_FOR(StoreF32Dev) break;
        case ELBM_STORE_F16DEV: ELBM_ROWS_FOR(StoreF16Dev) break;
        case ELBM_STORE_BF16DEV: ELBM_ROWS_FOR(StoreBF16Dev) break;
        default: break;
        }
#undef ELBM_ROWS_FOR
    }
    if (kernel == ELBM_KERNEL_ROWS) return cudaErrorNotSupported;
    if (steps > 1) {
        if (steps > ELBM_CAT(steps_per_launch, ELBM_SUFFIX)(storage, g, kernel, num_sms)) return cudaErrorInvalidValue;
#if ELBM_DIM == 2
        const unsigned R = unsigned(kTileRows + 2 * (steps - 1)), nx = unsigned(g.nx);
        const unsigned threads = R * ((nx + kPairSpan - 1) / kPairSpan) * 32u; // at most kTileThreads
        const size_t shared = size_t(Q) * (R + R - 2) * nx * storage_bytes(storage);
        const unsigned grid = unsigned((g.ny + kTileRows - 1) / kTileRows);
#define ELBM_TILE(FORCE)                                                                                    \
    switch (storage) {                                                                                      \
    case ELBM_STORE_F32: { using ST = StoreF32; ELBM_TILE_ONE(FORCE); }                                     \
    case ELBM_STORE_F32DEV: { using ST = StoreF32Dev; ELBM_TILE_ONE(FORCE); }                               \
    case ELBM_STORE_F16DEV: { using ST = StoreF16Dev; ELBM_TILE_ONE(FORCE); }                               \
    default: { using ST = StoreBF16Dev; ELBM_TILE_ONE(FORCE); }                                             \
    }
#define ELBM_TILE_ONE(FORCE)                                                                                \
    return launch_shared(k_step_tile<ST, FORCE>, grid, threads, shared, s,                                  \
                         static_cast<const typename ST::S *>(fin), static_cast<typename ST::S *>(fout), g,  \
                         p, steps, kTileRows)
        if (forced) ELBM_TILE(true)
        ELBM_TILE(false)
#undef ELBM_TILE
#undef ELBM_TILE_ONE
#endif
    }
    const uint64_t elems = uint64_t(Q) * uint64_t(g.N);
    const RowDiv rd = row_div(uint32_t(g.nx));
    // Steps with a body force take element offsets at every size, and no L2 instantiation: the
    // force's two equilibria make them 1.5 times as long and byte offsets give 1 to 4 % of that (us
    // per step, elements and bytes: D3Q27 201 x 160 x 150 FP32 294, 287, FP32 deviations 295, 283, FP16
    // 284, 277, 60 x 52 x 44 11.1, 10.9; D2Q9 4000 x 2000 FP32 161.6, 159.6), for five more kernels
    // per lattice to build.
#define ELBM_DIRECT_STEP(ADDR, GRID)                                                                   \
    if (forced) {                                                                                      \
        ELBM_STORAGE_SWITCH(storage, return launch(k_step<ST, (ADDR == kAddrBytes ? kAddrElems : ADDR), true>, \
                                                   GRID, threads, s,                                   \
                                                   static_cast<const typename ST::S *>(fin),           \
                                                   static_cast<typename ST::S *>(fout), g, p, rd))     \
    } else {                                                                                           \
        ELBM_STORAGE_SWITCH(storage, return launch(k_step<ST, ADDR>, GRID, threads, s,                 \
                                                   static_cast<const typename ST::S *>(fin),           \
                                                   static_cast<typename ST::S *>(fout), g, p, rd))     \
    }
    const bool pair = D == 2 && storage != ELBM_STORE_F64; // two nodes per thread, blocks along rows
    const int64_t plane = int64_t(g.nx) * g.ny;
    if (elems > 0xffffffffull || (pair ? g.ny : g.nz) > 65535) {
        const unsigned threads = pair ? step_threads<StoreF32>() : kStepBlock;
        ELBM_DIRECT_STEP(kAddrWide, blocks_for(g.N, kStepBlock))
    } else {
        // one node per thread: smaller blocks where full ones would leave SMs without work (D2Q9
        // FP64, 96^2: 55 us per step in blocks of 256, 28 so); FP64 is bound by each SM's FP64
        // pipe and takes 64 from the start, which divides the nodes more evenly over the SMs
        unsigned threads = pair ? step_threads<StoreF32>() : storage == ELBM_STORE_F64 ? 64u : unsigned(kStepBlock);
        if (!pair)
            while (threads > 32 && int64_t(blocks_for(plane, threads)) * g.nz < 2 * int64_t(num_sms)) threads /= 2;
        const dim3 grid = pair ? dim3(blocks_for(g.nx, kStepBlock), unsigned(g.ny))
                               : dim3(blocks_for(plane, threads), unsigned(g.nz));
#if ELBM_DIM == 3 // the tighter register bounds are for DRAM
        if (!forced && 2 * elems * storage_bytes(storage) <= kL2Bytes) {
#define ELBM_L2_STEP(STT)                                                                              \
    return launch(k_step<STT, kAddrBytes, false, kL2Blocks>, grid, threads, s,                         \
              static_cast<const float *>(fin), static_cast<float *>(fout), g, p, rd)
            if (storage == ELBM_STORE_F32) ELBM_L2_STEP(StoreF32);
            if (storage == ELBM_STORE_F32DEV) ELBM_L2_STEP(StoreF32Dev);
#undef ELBM_L2_STEP
        }
#endif
        if (elems * storage_bytes(storage) <= 0xffffffffull) {
            ELBM_DIRECT_STEP(kAddrBytes, grid)
        } else {
            ELBM_DIRECT_STEP(kAddrElems, grid)
        }
    }
#undef ELBM_DIRECT_STEP
}

#endif

#if !defined(ELBM_PART) || ELBM_PART == 2
cudaError_t ELBM_CAT(launch_step_diag, ELBM_SUFFIX)(int storage, const void *fin, void *fout, const Geometry &g,
                                                    const CollideParams &p, DiagAcc *acc, int num_sms,
                                                    cudaStream_t s)
{
    using namespace ELBM_SUFFIX;
    if (g.N == 0) return cudaSuccess;
    const bool forced = p.force[0] != 0.0 || p.force[1] != 0.0 || p.force[2] != 0.0;
    if (forced || uint64_t(Q) * uint64_t(g.N) > 0xffffffffull) return cudaErrorNotSupported;
    const uint64_t items = uint64_t((g.nx + kStepBlock - 1) / kStepBlock) * uint64_t(g.ny) * uint64_t(g.nz);
    const uint64_t cap = uint64_t(num_sms > 0 ? num_sms : 1) * 8u;
    const unsigned grid = unsigned(items < cap ? items : cap);
    ELBM_STORAGE_SWITCH(storage, return launch(k_step_diag<ST>, grid, kStepBlock, s,
                                               static_cast<const typename ST::S *>(fin),
                                               static_cast<typename ST::S *>(fout), g, p, acc))
}

#endif

#if !defined(ELBM_PART) || ELBM_PART == 3
cudaError_t ELBM_CAT(launch_step_batch, ELBM_SUFFIX)(int storage, const void *fin, void *fout,
                                                     const BatchTable &tab, int bx, const CollideParams &p,
                                                     cudaStream_t s)
{
    using namespace ELBM_SUFFIX;
    const int nitems = tab.item0[tab.n];
    if (tab.n <= 0 || nitems <= 0) return cudaSuccess;
    int64_t most = 0; // nodes of the largest domain
    for (int d = 0; d < tab.n; ++d) most = std::max(most, int64_t(tab.dom[d].nx) * tab.dom[d].ny * tab.dom[d].nz);
    const bool bytes = uint64_t(Q) * uint64_t(most) * storage_bytes(storage) <= 0xffffffffull;
#define ELBM_BATCH_BX(BXV, ADDR)                                                                       \
    ELBM_STORAGE_SWITCH(storage, return launch(k_step_batch<ST, BXV, ADDR>, unsigned(nitems), BXV / nodes_per_thread<D, ST>(), s, \
                                               static_cast<const typename ST::S *>(fin),               \
                                               static_cast<typename ST::S *>(fout), tab, p))
#define ELBM_BATCH_ADDR(ADDR)                                                                          \
    switch (bx) {                                                                                      \
    case 64: ELBM_BATCH_BX(64, ADDR); break;                                                           \
    case 128: ELBM_BATCH_BX(128, ADDR); break;                                                         \
    case 256: ELBM_BATCH_BX(256, ADDR); break;                                                         \
    }
    if (bytes) {
        ELBM_BATCH_ADDR(kAddrBytes)
    } else {
        ELBM_BATCH_ADDR(kAddrElems)
    }
    return cudaErrorInvalidValue; // bx
#undef ELBM_BATCH_ADDR
#undef ELBM_BATCH_BX
}

cudaError_t ELBM_CAT(persist_blocks_per_sm, ELBM_SUFFIX)(int storage, int bx, int *blocks)
{
    using namespace ELBM_SUFFIX;
    *blocks = 0;
#define ELBM_PERSIST_OCC(BXV)                                                                          \
    ELBM_STORAGE_SWITCH(storage, return cudaOccupancyMaxActiveBlocksPerMultiprocessor(blocks,           \
                                                                             k_step_persist<ST, BXV>, BXV / nodes_per_thread<D, ST>(), 0))
    switch (bx) {
    case 64: ELBM_PERSIST_OCC(64); break;
    case 128: ELBM_PERSIST_OCC(128); break;
    case 256: ELBM_PERSIST_OCC(256); break;
    default: return cudaErrorInvalidValue;
    }
#undef ELBM_PERSIST_OCC
    return cudaErrorInvalidValue;
}

cudaError_t ELBM_CAT(launch_step_persist, ELBM_SUFFIX)(int storage, void *pop0, void *pop1, int cur, int nsteps,
                                                       const BatchTableDom *doms, const PersistPlan &plan, int bx,
                                                       const CollideParams &p, int *err, cudaStream_t s)
{
    using namespace ELBM_SUFFIX;
    if (nsteps <= 0 || plan.grid <= 0) return cudaSuccess;
    cudaLaunchConfig_t cfg = {};
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeCooperative; // all blocks resident: they wait on one another
    attr[0].val.cooperative = 1;
    cfg.gridDim = dim3(unsigned(plan.grid));
    cfg.dynamicSmemBytes = 0;
    cfg.stream = s;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
#define ELBM_PERSIST_BX(BXV)                                                                           \
    ELBM_STORAGE_SWITCH(storage, cfg.blockDim = dim3(BXV / nodes_per_thread<D, ST>());                 \
                                 return cudaLaunchKernelEx(&cfg, k_step_persist<ST, BXV>,               \
                                                           static_cast<typename ST::S *>(pop0),        \
                                                           static_cast<typename ST::S *>(pop1), cur,   \
                                                           nsteps, doms, plan, p, err))
    switch (bx) {
    case 64: ELBM_PERSIST_BX(64); break;
    case 128: ELBM_PERSIST_BX(128); break;
    case 256: ELBM_PERSIST_BX(256); break;
    default: return cudaErrorInvalidValue;
    }
#undef ELBM_PERSIST_BX
    return cudaErrorInvalidValue;
}

#endif

#if !defined(ELBM_PART) || ELBM_PART == 2
cudaError_t ELBM_CAT(launch_step_adjoint, ELBM_SUFFIX)(int storage, const void *fin, const void *gnext,
                                                       void *gout, const Geometry &g, const CollideParams &p,
                                                       double *dforce, cudaStream_t s)
{
    using namespace ELBM_SUFFIX;
    if (g.N == 0) return cudaSuccess;
    const bool forced = dforce || p.force[0] != 0.0 || p.force[1] != 0.0 || p.force[2] != 0.0;
    // byte offsets where the gradient (and so the state) fills less than 2^32 bytes; FP64, bound
    // by its arithmetic, keeps the 1D grid
    const bool bytes = storage != ELBM_STORE_F64 && uint64_t(Q) * uint64_t(g.N) * 4u <= 0xffffffffull && g.nz <= 65535;
    const int64_t plane = int64_t(g.nx) * g.ny;
    const RowDiv rd = row_div(uint32_t(g.nx));
#define ELBM_ADJOINT(ADDR, FORCE, GRID)                                                                \
    return launch(k_step_adjoint<ST, ADDR, FORCE>, GRID, adjoint_block<ST>(), s,                       \
                  static_cast<const typename ST::S *>(fin), static_cast<const typename ST::T *>(gnext), \
                  static_cast<typename ST::T *>(gout), g, p, rd, dforce)
    if (storage == ELBM_STORE_F64) {
        using ST = StoreF64;
        if (forced) ELBM_ADJOINT(kAddrWide, true, blocks_for(g.N, adjoint_block<ST>()));
        ELBM_ADJOINT(kAddrWide, false, blocks_for(g.N, adjoint_block<ST>()));
    }
#define ELBM_ADJOINT_32(STT)                                                                           \
    {                                                                                                  \
        using ST = STT;                                                                                \
        const dim3 planes(blocks_for(plane, adjoint_block<ST>()), unsigned(g.nz));                     \
        const unsigned line = blocks_for(g.N, adjoint_block<ST>());                                    \
        if (bytes && forced) ELBM_ADJOINT(kAddrBytes, true, planes);                                   \
        if (bytes) ELBM_ADJOINT(kAddrBytes, false, planes);                                            \
        if (forced) ELBM_ADJOINT(kAddrWide, true, line);                                               \
        ELBM_ADJOINT(kAddrWide, false, line);                                                          \
    }
    switch (storage) {
    case ELBM_STORE_F32: ELBM_ADJOINT_32(StoreF32)
    case ELBM_STORE_F32DEV: ELBM_ADJOINT_32(StoreF32Dev)
    case ELBM_STORE_F16DEV: ELBM_ADJOINT_32(StoreF16Dev)
    case ELBM_STORE_BF16DEV: ELBM_ADJOINT_32(StoreBF16Dev)
    default: return cudaErrorInvalidValue;
    }
#undef ELBM_ADJOINT_32
#undef ELBM_ADJOINT
}

cudaError_t ELBM_CAT(launch_kinetic_energy, ELBM_SUFFIX)(int storage, const void *f, const Geometry &g, double rho0,
                                                         double *acc, void *grad, int num_sms, cudaStream_t s)
{
    using namespace ELBM_SUFFIX;
    if (g.N == 0) return cudaSuccess;
    unsigned blocks = blocks_for(g.N, kAuxBlock);
    const unsigned cap = unsigned(num_sms > 0 ? num_sms : 1) * 8u;
    if (blocks > cap) blocks = cap;
    const float Rf = dev_unit<D>(rho0);
    const double Rsum = (Q == 9 ? 36.0 : 216.0) * double(Rf);
    ELBM_STORAGE_SWITCH(storage, return launch(k_kinetic_energy<ST>, blocks, kAuxBlock, s,
                                               static_cast<const typename ST::S *>(f), g, Rf, Rsum, acc,
                                               static_cast<typename ST::T *>(grad)))
}

cudaError_t ELBM_CAT(launch_equilibrium_vjp, ELBM_SUFFIX)(int storage, const double *rho, const double *u,
                                                          const void *gf, const Geometry &g, double rho_uniform,
                                                          double *drho, double *du, cudaStream_t s)
{
    using namespace ELBM_SUFFIX;
    if (g.N == 0) return cudaSuccess;
    if (storage == ELBM_STORE_F64)
        return launch(k_equilibrium_vjp<double>, blocks_for(g.N, kAuxBlock), kAuxBlock, s, rho, u, static_cast<const double *>(gf), g,
                      rho_uniform, drho, du);
    return launch(k_equilibrium_vjp<float>, blocks_for(g.N, kAuxBlock), kAuxBlock, s, rho, u, static_cast<const float *>(gf), g,
                  rho_uniform, drho, du);
}

cudaError_t ELBM_CAT(launch_init, ELBM_SUFFIX)(int storage, const double *rho, const double *u,
                                               void *f, const Geometry &g, double rho_uniform,
                                               double rho0, int64_t n0, int64_t count, cudaStream_t s)
{
    using namespace ELBM_SUFFIX;
    if (count <= 0) return cudaSuccess;
    ELBM_STORAGE_SWITCH(storage, return launch(k_init<ST>, blocks_for(count, kAuxBlock), kAuxBlock, s, rho,
                                               u, static_cast<typename ST::S *>(f), g, rho_uniform, rho0, n0,
                                               count))
}

cudaError_t ELBM_CAT(launch_moments, ELBM_SUFFIX)(int storage, const void *f, const Geometry &g,
                                                  double rho0, double *rho_out, double *u_out,
                                                  int64_t n0, int64_t count, cudaStream_t s)
{
    using namespace ELBM_SUFFIX;
    if (count <= 0) return cudaSuccess;
    const float Rf = dev_unit<D>(rho0);
    const double Rsum = (Q == 9 ? 36.0 : 216.0) * double(Rf);
    ELBM_STORAGE_SWITCH(storage, return launch(k_moments<ST>, blocks_for(count, kAuxBlock), kAuxBlock, s,
                                               static_cast<const typename ST::S *>(f), g, Rf, Rsum, rho_out,
                                               u_out, n0, count))
}

cudaError_t ELBM_CAT(launch_alpha, ELBM_SUFFIX)(int storage, const void *f, const Geometry &g,
                                                const CollideParams &p, double *alpha_out,
                                                uint8_t *flags, double *nut_out, cudaStream_t s)
{
    using namespace ELBM_SUFFIX;
    if (g.N == 0) return cudaSuccess;
    ELBM_STORAGE_SWITCH(storage, return launch(k_alpha<ST>, blocks_for(g.N, kStepBlock), kStepBlock, s,
                                               static_cast<const typename ST::S *>(f), g, p, alpha_out,
                                               flags, nut_out))
}

cudaError_t ELBM_CAT(launch_diag, ELBM_SUFFIX)(int storage, const void *f, const Geometry &g,
                                               const CollideParams &p, DiagAcc *acc, int num_sms,
                                               cudaStream_t s)
{
    using namespace ELBM_SUFFIX;
    if (g.N == 0) return cudaSuccess;
    unsigned blocks = blocks_for(g.N, kAuxBlock);
    const unsigned cap = unsigned(num_sms > 0 ? num_sms : 1) * 8u;
    if (blocks > cap) blocks = cap;
    ELBM_STORAGE_SWITCH(storage, return launch(k_diag<ST>, blocks, kAuxBlock, s,
                                               static_cast<const typename ST::S *>(f), g, p, acc))
}

#endif

} // namespace eelbm
